// Test infrastructure: the bit-sliced classification (tc_sliced.cuh) compiled
// for the host, a block of sign vectors at a time: every phase is run for
// all threads of the block before the next begins, as the kernels' barriers
// order them, over areas of exactly the sizes the kernels reserve, against
// the oracle.  Usage: run_sliced_sweep <d> <edges file> <blocks>; the last
// block starts with the special sign vectors of run_table_sweep.cpp (constant,
// Harnack's distribution, parities).  Exit 0 when all codes agree.
#define main run_table_sweep_main
#include "run_table_sweep.cpp"
#undef main
#define TC_SL_EMULATE
#include "tc_sliced.cuh"

static uint64_t special(int d, int which, u32 w) {
  uint64_t x = 0;
  for (int j = 0; j <= d; ++j)
    for (int i = 0; i + j <= d; ++i) {
      const int k = j * (d + 1) - j * (j - 1) / 2 + i;
      const bool b[8] = {false, true, i % 2 == 0 && j % 2 == 0, i % 2 == 1 && j % 2 == 1,
                         (i + j) % 2 == 0, i % 2 == 0, k % 2 == 0, (i % 2 == 0) != (j % 2 == 0)};
      if (b[which] && (u32)(k >> 6) == w) x |= 1ull << (k & 63);
    }
  return x;
}

template <class K>
static void emulate_events(const TcSlMem &m, u32 chunks) {
  for (u32 k = 0; k < chunks * K::NG; ++k) {  // tc_sl_events
    u32 *const p = m.ev + k * TC_SL_GROUP;
    u32 o[32];
    for (u32 r = 0; r < 32; ++r) {
      o[r] = 0;
      for (u32 s = 0; s < 32; ++s) o[r] |= ((p[s] >> r) & 1u) << s;
    }
    for (u32 r = 0; r < 32; ++r) p[r] = o[r];
  }
}

template <int D, int NG>
int run_sliced(const char *edge_file, int blocks) {
  typedef TcSlK<D, NG> K;
  std::vector<int32_t> e;
  {
    std::ifstream f(edge_file);
    int a;
    while (f >> a) e.push_back(a);
  }
  const int ne = (int)e.size() / 4;
  std::vector<std::array<Pt, 3>> tris;
  ts_tri t;
  if (!triangles_of(D, e.data(), ne, tris) || !build_diamond(D, tris, t.dia) || !pack_tables(t.dia, &t))
    return 2;
  std::vector<int32_t> otri(6 * D * D);
  if (orc_triangles_from_edges(D, ne, e.data(), otri.data(), D * D) != D * D) return 2;
  const u32 *tab = t.host_stables.data();
  const u32 nch = t.slay.chunks, words = tc_sl_words<K>(nch);
  std::vector<TcQuad> area(words / 4 + 2, TcQuad{0xA5A5A5A5u, 0xA5A5A5A5u, 0xA5A5A5A5u, 0xA5A5A5A5u});
  u32 *const base = reinterpret_cast<u32 *>(area.data());
  for (u32 i = words; i < 4 * area.size(); ++i) base[i] = 0xC3C3C3C3u;  // behind the areas: not to be written
  const int cw = orc_code_words(D);
  int bad = 0;
  for (int blk = 0; blk < blocks; ++blk) {
    std::vector<TcSig<K::W>> sig(K::T);
    for (u32 i = 0; i < K::T; ++i) {
      for (u32 w = 0; w < K::W; ++w)
        sig[i].w[w] = blk == blocks - 1 && i < 8 ? special(D, (int)i, w)
                                                 : mix64(7000003ull * D + ((uint64_t)blk * K::T + i) * K::W + w);
      sig[i].w[K::W - 1] &= tc_top_mask(K::NPOINTS, K::W);
    }
    const TcSlMem m = tc_sl_carve<K>(tab, base, nch);
    for (u32 i = 0; i < K::T; ++i) tc_sl_clear<K>(m, i);
    for (u32 k = 0; k < K::NPOINTS; ++k)  // tc_sl_planes: bit i % 32 of the group's word
      for (u32 g = 0; g < K::NG; ++g) {
        u32 x = 0;
        for (u32 i = 0; i < 32; ++i) x |= sig[32 * g + i].bit(k) << i;
        m.x[k * K::NG + g] = x;
      }
    for (u32 i = 0; i < K::T; ++i) tc_sl_logic<K>(m, i);
    for (u32 i = 0; i < K::T; ++i) tc_sl_tiles<K>(m, i);
    emulate_events<K>(m, nch);
    std::vector<u64> code((size_t)K::T * K::CW, 0);
    std::vector<u32> R(K::T), root(K::T), err(K::T, 0);
    std::vector<char> star(K::T);
    for (u32 i = 0; i < K::T; ++i) {
      const TcSlInst<K> I(m, i);
      bool st = false;
      tc_sl_labels<K>(I, K::V);
      R[i] = tc_sl_regions<K>(m, I, root[i], st, err[i]);
      star[i] = st;
    }
    for (u32 i = 0; i < K::T; ++i) {
      const u32 at = tc_sl_instance<K>(i);
      const TcSlInst<K> I(m, i);
      tc_sl_finish<K>(m, I, i, R[i], root[i], star[i], err[i], &code[(size_t)at * K::CW]);
      if (err[i]) ++bad;
    }
    for (u32 i = 0; i < K::T; ++i) {
      uint64_t want[4] = {0, 0, 0, 0};
      const int rc = orc_real_scheme(D, otri.data(), (const uint64_t *)sig[i].w, want, cw, nullptr);
      bool same = rc == 0;
      for (int w = 0; w < cw; ++w) same &= code[(size_t)i * K::CW + w] == want[w];
      if (!same && bad++ < 3) printf("block %d instance %u differs (oracle status %d)\n", blk, i, rc);
    }
  }
  for (u32 i = words; i < 4 * area.size(); ++i)
    if (base[i] != 0xC3C3C3C3u) ++bad;
  printf("d=%d sliced NG=%d instances=%d differing=%d\n", D, NG, blocks * (int)K::T, bad);
  return bad != 0;
}

#ifndef TC_SL_NO_MAIN
int main(int argc, char **argv) {
  const int d = atoi(argv[1]), n = atoi(argv[3]);
  switch (d) {
#define TC_CASE(x) \
  case x: return run_sliced<x, TC_SL_GROUPS>(argv[2], n);
    TC_CASE(1) TC_CASE(2) TC_CASE(3) TC_CASE(4) TC_CASE(5) TC_CASE(6) TC_CASE(7) TC_CASE(8)
    TC_CASE(9) TC_CASE(10) TC_CASE(11) TC_CASE(12) TC_CASE(13) TC_CASE(14) TC_CASE(15) TC_CASE(16)
  }
  return 2;
}
#endif
