// Test infrastructure: the bit-sliced block sweep (tc_block_sweep.cuh)
// compiled for the host: 128 high parts by the phases of the kernel, every
// phase for all threads before the next, then the middle row of each, its
// histogram against the oracle's over the same masks.  Usage: run_block_sliced
// <d> <edges file> <plain|flip|reduced|orbits> <seed>; exit 0 when all agree.
// Prints how many high parts the middle phase took (the others are left to
// the per-mask phases).
#define TC_SL_NO_MAIN
#include "run_sliced_sweep.cpp"
static inline unsigned atomicAdd(unsigned *p, unsigned v) { auto o = *p; *p += v; return o; }
#include "tc_block_sweep.cuh"
#include <string>

template <int D>
int run_blocks(const char *edge_file, const std::string &mode, uint64_t seed) {
  typedef TcSbK<D> K;
  typedef typename K::Base B;
  std::vector<int32_t> e;
  {
    std::ifstream f(edge_file);
    std::string line;
    while (std::getline(f, line)) {
      if (line.empty() || line[0] == '#') continue;
      int q[4];
      if (sscanf(line.c_str(), "%d %d %d %d", q, q + 1, q + 2, q + 3) == 4) e.insert(e.end(), q, q + 4);
    }
  }
  std::vector<std::array<Pt, 3>> tris;
  ts_tri t;
  if (!triangles_of(D, e.data(), (int)e.size() / 4, tris) || !build_diamond(D, tris, t.dia) ||
      !pack_tables(t.dia, &t))
    return 2;
  std::vector<int32_t> otri(6 * D * D);
  if (orc_triangles_from_edges(D, (int)e.size() / 4, e.data(), otri.data(), D * D) != D * D) return 2;
  u32 ib = D + 1, oshift = D + 1, ishift = 0, oflags = 0;
  if (mode == "flip") { ib = D; ishift = 1; }
  if (mode == "reduced") { ib = D - 1; ishift = 2; oshift = D + 2; }
  if (mode == "orbits") {
    int p1 = 0, p2 = 0;
    if (!tc_orbit_pivots(D, &p1, &p2)) return 2;
    oshift = D + 2;
    oflags = 8u | ((u32)p1 << 8) | ((u32)p2 << 16);
  }
  if (ib < 5) return 2;
  const int np = (D + 1) * (D + 2) / 2;
  const uint64_t hmax = 1ull << (np - oshift - (oflags ? 2 : 0));
  const u32 *tab = t.host_stables.data();
  const u32 words = tc_sb_words<K>(t.slay.chunks);
  std::vector<TcQuad> area(words / 4 + 2, TcQuad{0xA5A5A5A5u, 0xA5A5A5A5u, 0xA5A5A5A5u, 0xA5A5A5A5u});
  u32 *const base = reinterpret_cast<u32 *>(area.data());
  for (u32 i = words; i < 4 * area.size(); ++i) base[i] = 0xC3C3C3C3u;
  const TcSbMem M = tc_sb_carve<K>(tab, base, t.slay.chunks);
  const TcSlMem &m = M.s;
  std::vector<uint64_t> mask(K::T);
  for (u32 i = 0; i < K::T; ++i) {
    const uint64_t u = i == 0 ? 0 : i == 1 ? hmax - 1 : mix64(seed * 1000 + i) % hmax;
    mask[i] = (oflags ? tc_orbit_high(u, oflags) : u) << oshift;
  }
  for (u32 i = 0; i < K::T; ++i) tc_sl_clear<B>(m, i);
  for (u32 k = 0; k < B::NPOINTS; ++k)
    for (u32 g = 0; g < B::NG; ++g) {
      u32 x = 0;
      for (u32 i = 0; i < 32; ++i) x |= (u32)((mask[32 * g + i] >> k) & 1) << i;
      m.x[k * B::NG + g] = x;
    }
  for (u32 i = 0; i < K::T; ++i) tc_sl_logic<B>(m, i);
  for (u32 i = 0; i < K::T; ++i) tc_sl_tiles<B>(m, i);
  emulate_events<B>(m, t.slay.chunks);
  for (u32 i = 0; i < K::T; ++i) tc_sb_record<K>(M, i, mask[tc_sl_instance<B>(i)]);
  int bad = 0, valid = 0;
  for (u32 hl = 0; hl < K::T; ++hl) {
    const uint64_t mk = mask[tc_sl_instance<B>(hl)];
    if (!((M.rec[K::R_HDR * K::T + hl] >> 25) & 1u)) continue;
    ++valid;
    std::vector<u64> hk(K::HASH, 0), gk(16, 0);
    std::vector<u32> hc(K::HASH, 0);
    std::vector<unsigned long long> gc(16, 0);
    u32 gerr = 0, err = 0;
    unsigned long long failed = 0;
    for (u32 i = 0; i < K::STARS; ++i) M.stars[i] = 0;
    *M.queued = 0;
    const TcSbOut out{hk.data(), hc.data(), gk.data(), gc.data(), 16, &gerr};
    const u32 N = (M.rec[K::R_HDR * K::T + hl] >> 8) & 255u;
    for (u32 w = 0; w < (1u << ib) / 32; ++w) {
      const u32 th = (hl * 7 + w) % K::T;
      if (N <= K::NA && w % 2) tc_sb_middle<K, K::NA>(M, th, hl, w, ishift, out, err, failed);
      else tc_sb_middle<K, K::NB>(M, th, hl, w, ishift, out, err, failed);
      if (w % 4 == 3 || w + 1 == (1u << ib) / 32) {  // the kernel's queue of deep trees
        for (u32 i = 0; i < std::min(*M.queued, K::QUEUE); ++i) {
          const u32 *const q = M.queue + 4 * i;
          tc_sb_deep<K>(M, i % K::T, q[2] & 0xFFFFu, ((u64)q[1] << 32) | q[0], q[2] >> 16, q[3], out, err, failed);
        }
        *M.queued = 0;
      }
    }
    std::map<u64, unsigned long long> got, want;
    for (u32 s = 0; s < K::HASH; ++s)
      if (hk[s]) got[hk[s]] += hc[s];
    for (u32 R = 1; R < K::STARS; ++R)
      if (M.stars[R]) got[tc_sb_star_code(R)] += M.stars[R];
    for (uint64_t p = 0; p < (1ull << ib); ++p) {
      const uint64_t x = mk | (p << ishift);
      uint64_t code = 0;
      if (orc_real_scheme(D, otri.data(), &x, &code, 1, nullptr) != 0) return 3;
      want[code] += 1;
    }
    if (got != want || err || gerr || failed) {
      if (bad++ < 3)
        printf("high part %llx differs (N %u, %zu codes, oracle %zu, err %u, failed %llu)\n",
               (unsigned long long)mk, N, got.size(), want.size(), err, failed);
    }
  }
  for (u32 i = words; i < 4 * area.size(); ++i)
    if (base[i] != 0xC3C3C3C3u) ++bad;
  printf("d=%d map=%s high parts=%u in the middle phase=%d differing=%d\n", D, mode.c_str(), K::T, valid, bad);
  return bad != 0;
}

int main(int argc, char **argv) {
  const int d = atoi(argv[1]);
  const uint64_t seed = argc > 4 ? atoi(argv[4]) : 1;
  switch (d) {
    case 4: return run_blocks<4>(argv[2], argv[3], seed);
    case 5: return run_blocks<5>(argv[2], argv[3], seed);
    case 6: return run_blocks<6>(argv[2], argv[3], seed);
    case 7: return run_blocks<7>(argv[2], argv[3], seed);
    case 8: return run_blocks<8>(argv[2], argv[3], seed);
    case 9: return run_blocks<9>(argv[2], argv[3], seed);
  }
  return 2;
}
