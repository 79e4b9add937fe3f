// tc_block_sweep.cuh -- exhaustive sweeps in whole blocks of middle-row
// patterns, bit-sliced twice (d <= 9; block_sweep.cu).
//
// The masks of a block share their high bits (the lattice points off the
// x-axis); its 2^ib masks differ in the middle row only.  No edge of
// T^diamond crosses the x-axis, so the two half-diamonds depend on the high
// bits alone, and what they leave to the middle row is small: the components
// ("comps") that touch it, which of them are next to which middle vertex with
// which sign, and the tree they hang in.  A thread block takes 128 high parts:
//
//   halves   the half-diamonds of 128 high parts by the phases of
//            tc_sliced.cuh, then one high part per thread: the half joins, and
//            a record of the comps (TcSb below)
//   middle   32 middle-row patterns of one high part per thread, one bit each.
//            The open comps (about d + 1 of them) are the nodes of a graph;
//            the middle row is walked once, joining all nodes of a run of one
//            sign, and the graph is closed transitively (Warshall): a region
//            is a class of nodes, or a closed comp.  The root needs no
//            orientation parity: a region X other than the root is a disk with
//            holes, so chi(X) + (its neighbours in the region tree) is even,
//            and it is odd for the root (one Moebius band more, or the
//            pseudoline's two sides), where chi counts label starts minus join
//            events.  Both are sums over nodes, kept modulo 2 as bit planes.
//            Patterns whose regions all border the root (a star) are counted
//            by their number of regions.  Trees of depth two are told by that
//            number and how many children of the root have 1, 2, ... children
//            of their own: the regions' degrees are sums over classes too,
//            three bit planes each, and one code is made for all patterns of a
//            word with the same numbers.  Deeper trees are coded one by one
//            from their classes.
//
// Every middle vertex has half-diamond neighbours of both signs: the triangle
// over an edge of the x-axis has its apex at height 1, and the reflections
// (x, 1) and (x, -1) have opposite signs (Eq. 2).  So no region lies in the
// middle row alone, and every run has a node.
//
// The open comps are as many under every high part (open_components, engine.h):
// d on the standard triangulation, 12 on a seeded one at d = 9, up to 29 with
// long edges at the x-axis.  Above K::NB of them the block sweep is not launched
// (block_range).  High parts with more than 32 comps (none seen with up to K::NB
// open ones) take the per-mask phases of tc_sliced.cuh.
#pragma once

#include "tc_sliced.cuh"

// Traits: TcSlK's, two sizes of the middle phase (nodes), the areas.
template <int D_>
struct TcSbK : TcSlK<D_, 4> {
  typedef TcSlK<D_, 4> Base;
  static constexpr u32 D = D_, M = 2 * D_ + 1;  // middle vertices
  static constexpr u32 NA = D_ <= 8 ? D_ + 1 : 13, NB = tc_block_nodes(D_);
  // record of a high part (words, one column per thread)
  static constexpr u32 R_HDR = 0,          // comps | nodes << 8 | closed comps << 16 | star impossible << 24
                                           // | valid << 25 | corner edge signs << 26, 27
                                           // | some closed comp is no leaf << 28
                       R_NODE = 1,         // nodes that must be in the root | chi parities << 16
                       R_ADJ = 2,          // per middle vertex: nodes next to it with sigma 0 | with sigma 1 << 16
                       R_TOG = R_ADJ + M,  // per middle vertex 4 bits: chi changes by an odd number; bit
                                           // sigma + 2 * (same sign as the vertex before)
                       R_NPAR = R_TOG + (4 * M + 31) / 32,  // parent of a node (byte): node, 254 closed, 255 none
                       R_NCOMP = R_NPAR + 4,                // comp of a node (byte)
                       R_KIDS = R_NCOMP + 4,                // closed leaves at a node (byte)
                       R_CPAR = R_KIDS + 4,                 // parent of a comp (byte)
                       R_CNODE = R_CPAR + 8,                // node of a comp (byte; 255: closed)
                       R_WORDS = R_CNODE + 8;
  static constexpr u32 T = Base::T;
  // areas (words): the label area also holds, per thread, the degree planes
  // (3 NB words) or a tree code's children masks and parents (32 + 8 words);
  // scratch: M words per thread; the event chunks also hold the queue of deep
  // trees
  static constexpr u32 LAB = Base::LABW > 48 * T ? Base::LABW : 48 * T;
  static constexpr u32 QUEUE = 512;  // deep trees in waiting (four words each)
  static constexpr u32 HASH = D_ <= 7 ? 256 : 512;
  static constexpr u32 SW = (M > 16 ? M : 16) * T;
  static constexpr u32 STARS = 48;  // star patterns by number of regions
};

struct TcSbMem {
  TcSlMem s;     // tables, labels, events, sign planes
  u32 *rec;      // K::R_WORDS words per thread
  u32 *scr;      // K::SW words
  u32 *stars;    // K::STARS counters
  u32 *queue;    // K::QUEUE deep trees: two words of node classes, high part | root node << 16, patterns
  u32 *queued;   // their number
};

template <class K>
__host__ __device__ constexpr u32 tc_sb_evwords(u32 chunks) {
  return chunks * K::NG * TC_SL_GROUP > 4 * K::QUEUE ? chunks * K::NG * TC_SL_GROUP : 4 * K::QUEUE;
}

template <class K>
__host__ __device__ constexpr u32 tc_sb_words(u32 chunks) {
  return K::LAB + tc_sb_evwords<K>(chunks) + K::XW +
         K::R_WORDS * K::T + K::SW + K::STARS + 4;
}

template <class K>
__device__ __forceinline__ TcSbMem tc_sb_carve(const u32 *tab, u32 *area, u32 chunks) {
  TcSbMem m;
  m.s.tab = tab;
  m.s.lab = area;
  m.s.ev = m.s.lab + K::LAB;
  m.queue = m.s.ev;
  m.s.x = m.s.ev + tc_sb_evwords<K>(chunks);
  m.rec = m.s.x + K::XW;
  m.scr = m.rec + K::R_WORDS * K::T;
  m.stars = m.scr + K::SW;
  m.queued = m.stars + K::STARS;
  return m;
}

template <class K>
__device__ __forceinline__ u8 *tc_sb_byte(u32 *rec, u32 off, u32 i, u32 t) {
  return reinterpret_cast<u8 *>(rec + (off + (i >> 2)) * K::T + t) + (i & 3u);
}

// ---- halves: one high part per thread (thread t: instance
// tc_sl_instance<K>(t) of the block), after the phases of tc_sliced.cuh up to
// the tiles.  sig: its mask, middle-row bits zero.
template <class K>
__device__ __forceinline__ void tc_sb_record(const TcSbMem &m, u32 t, u64 sig) {
  typedef TcSlInst<typename K::Base> Inst;
  const Inst I(m.s, t);
  const u32 *const tab = m.s.tab;
  const u32 nc1 = tab[1];
  // label starts and joins of the half-diamonds only.  The first pair behind
  // a corner is joined whatever the corner's sign; the corner pair is not.
  constexpr u32 HB = 2 * K::H;
  if constexpr (HB % 32 != 0) I.set_event(HB / 32, I.event(HB / 32) & ((1u << (HB % 32)) - 1u));
  for (u32 c = (HB + 31) / 32; c < K::NCB; ++c) I.set_event(c, 0);
  const u32 be = (I.event(K::NCB + nc1) | 1u) & ((1u << (2 * K::D - 1)) - 1u);
  I.set_event(K::NCB + nc1, be);
  tc_sl_labels<typename K::Base>(I, 2 * K::H);
  tc_sl_joins<typename K::Base>(I, tab + tab[5], 0, nc1 + 1);
  u32 *const rec = m.rec + t;
  rec[K::R_HDR * K::T] = 0;
  // comps in the order of their smallest starts; chi of every comp modulo 2:
  // label starts plus join events
  static_assert(kBlockComps == 32 && Inst::MARK + 32 <= 256, "comps in label bytes, sets of them in words");
  u32 C = 0;
  {
    u32 n = 0;  // roots, before they are numbered
#pragma unroll
    for (u32 c = 0; c < K::NCB; ++c)
      for (u32 w = I.event(c); w; w &= w - 1u) {
        const u32 v = 32u * c + (u32)__ffs(w) - 1u;
        n += I.raw(v) == v;
      }
    if (n > kBlockComps) return;  // not valid: the block's masks one by one
  }
  u32 chis = 0;
  C = tc_sl_number<typename K::Base>(I, [&](u32 r) { chis ^= 1u << r; });
  auto comp_of = [&](u32 v) -> u32 { return I.region(v); };
  {
    const u32 *const site = tab + tab[5];
    u32 c = 0, w = 0;
    for (;;) {
      while (w == 0 && c <= nc1) w = I.event(K::NCB + c++);
      if (w == 0) break;
      const u32 s = site[32u * (c - 1u) + (u32)__ffs(w) - 1u];
      w &= w - 1u;
      chis ^= 1u << comp_of(s & 0xFFFFu);
    }
  }
  // the middle vertices' neighbours: comps next to them by sign, and whether
  // chi changes by an odd number when the vertex joins: 1 minus the runs of
  // its same-sign earlier neighbours, for either sign and with or without the
  // vertex before it
  u32 open = 0, tog = 0, vi = 0;
  {
    // The four choices of the vertex at once, a bit each (choice k: sigma = k &
    // 1, of one sign with the vertex before if k & 2): the ones for which the
    // last entry had the vertex's sign, and 1 minus the runs modulo 2.  A fan
    // may have any length.
    u32 m0 = 0, m1 = 0, same = 0, runs = 15;
    const TcQuad *f = reinterpret_cast<const TcQuad *>(tab + tab[3]) + 2 * tab[0];
    for (u32 s = 2 * tab[0]; s < tab[8]; ++s, ++f) {
      const TcQuad q = *f;
#pragma unroll
      for (u32 i = 0; i < 4; ++i) {
        const u32 e = i == 0 ? q.a : i == 1 ? q.b : i == 2 ? q.c : q.d, u = (e >> 8) & 0xFFFFu;
        if (e & (1u << 26)) continue;  // padding
        u32 now = 12;
        if (u < 2 * K::H) {
          // sigma of the middle vertex for which the two have one sign
          const u32 b = ((u32)(sig >> (e & 63u)) ^ (e >> 31) ^ 1u) & 1u;
          const u32 c = 1u << comp_of(u);
          m0 |= b ? 0u : c;
          m1 |= b ? c : 0u;
          now = 5u << b;
        }
        runs ^= now & ~(same & tc_bitmask(e, 30));
        same = now;
      }
      if (q.a & (1u << 25)) continue;  // another step of this vertex
      tog |= runs << ((4u * vi) & 31u);
      rec[(K::R_ADJ + vi) * K::T] = m0;
      m.scr[vi * K::T + t] = m1;
      open |= m0 | m1;
      if ((vi & 7u) == 7u || vi + 1u == K::M) {
        rec[(K::R_TOG + (vi >> 3)) * K::T] = tog;
        tog = 0;
      }
      ++vi;
      m0 = m1 = same = 0;
      runs = 15;
    }
  }
  const u32 N = (u32)__popc(open);
  if (N > K::NB) return;
  // neighbours in node numbers
  for (u32 v = 0; v < K::M; ++v) {
    const u32 a = rec[(K::R_ADJ + v) * K::T], b = m.scr[v * K::T + t];
    u32 x = 0, k = 0;
    for (u32 o = open; o; o &= o - 1u, ++k) {
      const u32 c = (u32)__ffs(o) - 1u;
      x |= (((a >> c) & 1u) | (((b >> c) & 1u) << 16)) << k;
    }
    rec[(K::R_ADJ + v) * K::T] = x;
  }
  // comps in order: parents, chi, what a star needs
  auto node_of = [&](u32 c) -> u32 { return (open >> c) & 1u ? (u32)__popc(open & ((1u << c) - 1u)) : 255u; };
  u32 need = 0, chi = 0, nostar = 0, inner = 0;
  u32 zkids = 0, zkid = 255u;  // comp 0's children, one of them
  for (u32 k = 0; k < 4; ++k) rec[(K::R_KIDS + k) * K::T] = 0;
  const u32 *const vd = tab + tab[4];
  {
    u32 ch = 0, w = 0;
    for (u32 c = 0; c < C; ++c) {
      while (w == 0) w = I.event(ch++);
      const u32 v = 32u * (ch - 1u) + (u32)__ffs(w) - 1u;
      w &= w - 1u;
      const u32 p = c ? comp_of(vd[v] & 0x7FFFu) : 255u, nc = node_of(c),
                np = c ? node_of(p) : 255u;
      *tc_sb_byte<K>(m.rec, K::R_CPAR, c, t) = (u8)p;
      *tc_sb_byte<K>(m.rec, K::R_CNODE, c, t) = (u8)nc;
      if (p == 0) {
        ++zkids;
        zkid = nc;
      }
      if (nc != 255u) {
        *tc_sb_byte<K>(m.rec, K::R_NPAR, nc, t) = (u8)(c == 0 ? 255u : np == 255u ? 254u : np);
        *tc_sb_byte<K>(m.rec, K::R_NCOMP, nc, t) = (u8)c;
        chi ^= ((chis >> c) & 1u) << nc;
        need |= c && np == 255u ? 1u << nc : 0u;
        inner |= c && np == 255u && p != 0 ? 1u : 0u;
      } else if (c) {  // a closed comp: one more neighbour of its parent
        if (np == 255u) {
          nostar = inner = 1;
        } else {
          chi ^= 1u << np;
          need |= 1u << np;
          u8 *const k = tc_sb_byte<K>(m.rec, K::R_KIDS, np, t);
          inner |= *k == 7u;
          ++*k;
        }
      }
    }
  }
  if (node_of(0) == 255u) {
    if (zkids == 1u && zkid != 255u) {  // comp 0 is a closed leaf at its one child
      *tc_sb_byte<K>(m.rec, K::R_NPAR, zkid, t) = 255u;
      chi ^= 1u << zkid;
      u8 *const k = tc_sb_byte<K>(m.rec, K::R_KIDS, zkid, t);
      inner |= *k == 7u;
      ++*k;
    } else {
      inner = 1;
    }
  }
  // sigma of each corner for which its half-diamond boundary edge is not
  // crossed: edge 0 at (d, 0), edge 2d - 1 at (-d, 0)
  const u32 *const bx = tab + tab[6];
  const u32 e0 = bx[0], e1 = bx[2 * K::D - 1];
  const u32 s0 = ((u32)(sig >> ((e0 >> 8) & 63u)) ^ (e0 >> 16)) & 1u;
  const u32 s1 = ((u32)(sig >> (e1 & 63u)) ^ (e1 >> 16)) & 1u;
  rec[K::R_NODE * K::T] = need | (chi << 16);
  rec[K::R_HDR * K::T] = C | (N << 8) | ((C - N) << 16) | (nostar << 24) | (1u << 25) | (s0 << 26) | (s1 << 27) |
                         (inner << 28);
}

// ---- middle: 32 patterns per thread ----

// Bit plane of pattern bit j of the 32 patterns of word w.
__device__ __forceinline__ u32 tc_sb_plane(u32 j, u32 w) {
  switch (j) {
    case 0: return 0xAAAAAAAAu;
    case 1: return 0xCCCCCCCCu;
    case 2: return 0xF0F0F0F0u;
    case 3: return 0xFF00FF00u;
    case 4: return 0xFFFF0000u;
    default: return (w >> (j - 5u)) & 1u ? ~0u : 0u;
  }
}

// Add cnt to key in the block's hash table, or in the device's if that is full.
// The block's counts have 32 bits (a 64-bit add in shared memory is a
// compare-and-swap loop) and are moved to the device every few work items.
template <u32 HASH>
__device__ __forceinline__ void tc_sb_insert(u64 key, u32 cnt, u64 *hkeys, u32 *hcnt, u64 *gkeys,
                                             unsigned long long *gcnt, u64 gslots, u32 *gerr) {
  u32 s = tc_hash_slot(key, HASH - 1);
  for (u32 probe = 0; probe < HASH; ++probe) {
    unsigned long long *kp = reinterpret_cast<unsigned long long *>(hkeys + s);
    unsigned long long k = *reinterpret_cast<volatile unsigned long long *>(kp);
    if (k == 0) k = atomicCAS(kp, 0ull, (unsigned long long)key);
    if (k == 0 || k == key) {
      atomicAdd(hcnt + s, cnt);
      return;
    }
    s = (s + 1) & (HASH - 1);
  }
  tc_global_add(gkeys, gcnt, gslots, gerr, key, cnt);
}

// Code of a star: R - 1 ovals, none in another.
__device__ __forceinline__ u64 tc_sb_star_code(u32 R) {
  const u32 q = 2 * (R - 1);
  return (1ull << q) | (0xAAAAAAAAAAAAAAAAull & ((1ull << q) - 1));
}

// Where the codes of a sweep go.
struct TcSbOut {
  u64 *hkeys;
  u32 *hcnt;
  u64 *gkeys;
  unsigned long long *gcnt;
  u64 gslots;
  u32 *gerr;
};

// Code and count cnt patterns of high part hl: low = the smallest node of every
// node's class, 4 bits each, rootn a node of the root's class.
template <class K>
__device__ __noinline__ void tc_sb_deep(const TcSbMem &m, u32 t, u32 hl, u64 low, u32 rootn, u32 cnt,
                                        const TcSbOut &out, u32 &err, unsigned long long &failed) {
  u8 *const par = reinterpret_cast<u8 *>(m.s.lab + 32 * K::T + t);  // byte i: word i / 4 of the thread
  const u32 C = m.rec[K::R_HDR * K::T + hl] & 255u;
  auto comp = [&](u32 c) -> u32 {  // the region of comp c: its smallest comp
    const u32 k = *tc_sb_byte<K>(m.rec, K::R_CNODE, c, hl);
    return k == 255u ? c : (u32)*tc_sb_byte<K>(m.rec, K::R_NCOMP, (u32)(low >> (4 * k)) & 15u, hl);
  };
  u32 alive = 0;
  for (u32 c = 0; c < C; ++c) {
    if (comp(c) != c) continue;
    alive |= 1u << c;
    if (c) par[(c >> 2) * 4 * K::T + (c & 3u)] = (u8)comp(*tc_sb_byte<K>(m.rec, K::R_CPAR, c, hl));
  }
  const u32 root = *tc_sb_byte<K>(m.rec, K::R_NCOMP, rootn, hl);
  const u64 key = tc_sl_tree_code<1, K::T, 4 * K::T, K::RMAX>(par, m.s.lab + t, alive, root, err);
  if (key)
    tc_sb_insert<K::HASH>(key, cnt, out.hkeys, out.hcnt, out.gkeys, out.gcnt, out.gslots, out.gerr);
  else
    failed += cnt;
}

// Word w of the patterns of high part hl (a column of the records), at most
// NN nodes; ishift: the lowest middle-row bit that varies.
template <class K, u32 NN>
__device__ __forceinline__ void tc_sb_middle(const TcSbMem &m, u32 t, u32 hl, u32 w, u32 ishift,
                                             const TcSbOut &out, u32 &err, unsigned long long &failed) {
  const u32 *const rec = m.rec + hl;
  const u32 hdr = rec[K::R_HDR * K::T], N = (hdr >> 8) & 255u, nd = rec[K::R_NODE * K::T];
  u32 *const tg = m.scr + t;  // chi + degree of the nodes, modulo 2, one plane each
  u32 conn[NN * (NN - 1) / 2], T[NN], n[NN], first[NN];
  auto pair = [](u32 a, u32 b) constexpr -> u32 { return b * (b - 1) / 2 + a; };  // a < b
#pragma unroll
  for (u32 i = 0; i < NN * (NN - 1) / 2; ++i) conn[i] = 0;
#pragma unroll
  for (u32 c = 0; c < NN; ++c) {
    T[c] = 0;
    tg[c * K::T] = tc_bitmask(nd, 16 + c);
  }
  u32 prev = 0, S = 0, sfirst = 0, togw = 0, adj = 0;
  for (u32 v = 0; v < K::M; ++v) {
    const u32 x = v < K::D ? K::D - v : v - K::D;
    S = x < ishift ? 0u : tc_sb_plane(x - ishift, w);
    // same sign as the vertex before: left of the origin Eq. 2's constant
    // |x| mod 2 changes from vertex to vertex, up to (-1, 0) -> (0, 0)
    const u32 same = v ? ~(S ^ prev ^ (v <= K::D ? ~0u : 0u)) : 0u;
    adj = rec[(K::R_ADJ + v) * K::T];
#pragma unroll
    for (u32 c = 0; c < NN; ++c) {
      n[c] = (tc_bitmask(adj, c) & ~S) | (tc_bitmask(adj, 16 + c) & S);
      T[c] = (T[c] & same) | n[c];
    }
#pragma unroll
    for (u32 b = 1; b < NN; ++b)
#pragma unroll
      for (u32 a = 0; a < b; ++a) conn[pair(a, b)] |= (n[a] & T[b]) | (n[b] & T[a]);
    if ((v & 7u) == 0) togw = rec[(K::R_TOG + (v >> 3)) * K::T];
    const u32 tb = togw >> (4u * (v & 7u));
    const u32 od0 = (tc_bitmask(tb, 0) & ~same) | (tc_bitmask(tb, 2) & same),
              od1 = (tc_bitmask(tb, 1) & ~same) | (tc_bitmask(tb, 3) & same);
    tg[((u32)__ffs(adj & 0xFFFFu) - 1u) * K::T] ^= od0 & ~S;
    tg[((u32)__ffs(adj >> 16) - 1u) * K::T] ^= od1 & S;
    if (v == 0) {
      sfirst = S;
#pragma unroll
      for (u32 c = 0; c < NN; ++c) first[c] = n[c];
    }
    prev = S;
  }
  // the corners (d, 0) and (-d, 0) are one point; identifying them and the
  // uncrossed boundary edges next to them changes chi by -1 + those edges
#pragma unroll
  for (u32 b = 1; b < NN; ++b)
#pragma unroll
    for (u32 a = 0; a < b; ++a) conn[pair(a, b)] |= (first[a] & n[b]) | (first[b] & n[a]);
  {
    const u32 od = ~(tc_bitmask(hdr, 26) ^ S) ^ ~(tc_bitmask(hdr, 27) ^ sfirst) ^ ~0u;
    tg[((u32)__ffs(adj & 0xFFFFu) - 1u) * K::T] ^= od & ~S;
    tg[((u32)__ffs(adj >> 16) - 1u) * K::T] ^= od & S;
  }
#pragma unroll
  for (u32 k = 0; k < NN; ++k)
#pragma unroll
    for (u32 b = 1; b < NN; ++b)
#pragma unroll
      for (u32 a = 0; a < b; ++a)
        if (a != k && b != k)
          conn[pair(a, b)] |= conn[a < k ? pair(a, k) : pair(k, a)] & conn[b < k ? pair(b, k) : pair(k, b)];
  // region roots (the smallest node of a class), the tree edges they hang on,
  // the number of regions as a 5-bit number per pattern
  u32 cnt[5] = {0, 0, 0, 0, 0};
#pragma unroll
  for (u32 c = 0; c < NN; ++c) {
    u32 r = c < N ? ~0u : 0u;
#pragma unroll
    for (u32 a = 0; a < c; ++a) r &= ~conn[pair(a, c)];
    const u32 p = c < N ? (u32)*tc_sb_byte<K>(m.rec, K::R_NPAR, c, hl) : 255u;
    if (p != 255u) tg[c * K::T] ^= r;
    if (p < 254u) tg[p * K::T] ^= r;
    first[c] = r;
    u32 carry = r;
#pragma unroll
    for (u32 i = 0; i < 5; ++i) {
      const u32 s = cnt[i] & carry;
      cnt[i] ^= carry;
      carry = s;
    }
  }
  // the root region's nodes: chi + degree of their class is odd
#pragma unroll
  for (u32 c = 0; c < NN; ++c) n[c] = tg[c * K::T];
#pragma unroll
  for (u32 c = 0; c < NN; ++c) {
    u32 x = n[c];
#pragma unroll
    for (u32 a = 0; a < NN; ++a)
      if (a != c) x ^= conn[a < c ? pair(a, c) : pair(c, a)] & n[a];
    T[c] = c < N ? x : 0u;
  }
#pragma unroll
  for (u32 c = 0; c < NN; ++c) tg[c * K::T] = T[c];
  u32 star = (hdr >> 24) & 1u ? 0u : ~0u, any = 0;
#pragma unroll
  for (u32 c = 0; c < NN; ++c) {
    any |= T[c];
    if (c < N) {
      const u32 p = *tc_sb_byte<K>(m.rec, K::R_NPAR, c, hl);
      if ((nd >> c) & 1u) star &= T[c];
      if (p < 254u) star &= T[c] | tg[p * K::T];
    }
  }
  const u32 closed = (hdr >> 16) & 255u;
#pragma unroll
  for (u32 k = 1; k <= NN; ++k) {
    u32 x = star & any;
#pragma unroll
    for (u32 i = 0; i < 5; ++i) x &= (k >> i) & 1u ? cnt[i] : ~cnt[i];
    if (x) atomicAdd(m.stars + closed + k, (u32)__popc(x));
  }
  if (~any) {  // no root: counted as failed, not inserted
    failed += (u32)__popc(~any);
    err |= TC_ERR_INTERNAL;
  }
  u32 rest = any & ~star;
  // Trees of depth two: every edge that does not touch the root has an end of
  // degree one.  Degrees as three bit planes, by node (area: the label area,
  // 3 NN + words per thread), then by class.
  static_assert(3 * NN <= K::LAB / K::T, "degree planes");
  {
    if (rest && !((hdr >> 28) & 1u)) {
      u32 *const A = m.s.lab + t;
      u32 over = 0;  // patterns with a number too large for its planes
      auto bump = [&](u32 c, u32 x) {
#pragma unroll
        for (u32 i = 0; i < 3; ++i) {
          const u32 y = A[(3 * c + i) * K::T];
          A[(3 * c + i) * K::T] = y ^ x;
          x &= y;
        }
        over |= x;
      };
#pragma unroll
      for (u32 c = 0; c < NN; ++c) {
        const u32 k = c < N ? (u32)*tc_sb_byte<K>(m.rec, K::R_KIDS, c, hl) : 0u;
#pragma unroll
        for (u32 i = 0; i < 3; ++i) A[(3 * c + i) * K::T] = tc_bitmask(k, i);
      }
#pragma unroll
      for (u32 c = 0; c < NN; ++c)
        if (c < N) {
          const u32 p = *tc_sb_byte<K>(m.rec, K::R_NPAR, c, hl);
          if (p < 254u) {
            bump(c, first[c]);
            bump(p, first[c]);
          }
        }
      u32 num[13];  // regions off the root with 1 (three planes), 2 .. 6 (two planes) children
#pragma unroll
      for (u32 i = 0; i < 13; ++i) num[i] = 0;
#pragma unroll
      for (u32 c = 0; c < NN; ++c) {
        u32 d0 = A[(3 * c) * K::T], d1 = A[(3 * c + 1) * K::T], d2 = A[(3 * c + 2) * K::T], o = 0;
#pragma unroll
        for (u32 b = c + 1; b < NN; ++b) {
          const u32 mk = conn[pair(c, b)];
          const u32 x0 = A[(3 * b) * K::T] & mk, x1 = A[(3 * b + 1) * K::T] & mk, x2 = A[(3 * b + 2) * K::T] & mk;
          const u32 c0 = d0 & x0, c1 = (d1 & x1) | (c0 & (d1 ^ x1)), c2 = (d2 & x2) | (c1 & (d2 ^ x2));
          d0 ^= x0;
          d1 ^= x1 ^ c0;
          d2 ^= x2 ^ c1;
          o |= c2;
        }
        over |= o & first[c];
        n[c] = first[c] & d0 & ~d1 & ~d2;  // the class is a leaf (by its smallest node)
        const u32 x = first[c] & ~T[c];
        const u32 e2 = x & ~d0 & d1 & ~d2;
        const u32 c0 = num[0] & e2, c1 = num[1] & c0;
        num[0] ^= e2;
        num[1] ^= c0;
        over |= num[2] & c1;
        num[2] ^= c1;
#pragma unroll
        for (u32 k = 3; k < 8; ++k) {
          const u32 e = x & (k & 1u ? d0 : ~d0) & (k & 2u ? d1 : ~d1) & (k & 4u ? d2 : ~d2);
          const u32 y = num[2 * k - 3] & e;
          num[2 * k - 3] ^= e;
          over |= num[2 * k - 2] & y;
          num[2 * k - 2] ^= y;
        }
      }
#pragma unroll
      for (u32 c = 0; c < NN; ++c) {  // leaf planes of all nodes
        u32 x = n[c];
#pragma unroll
        for (u32 a = 0; a < c; ++a) x |= conn[pair(a, c)] & n[a];
        A[3 * c * K::T] = x;
      }
      u32 deep = over;
#pragma unroll
      for (u32 c = 0; c < NN; ++c)
        if (c < N) {
          const u32 p = *tc_sb_byte<K>(m.rec, K::R_NPAR, c, hl);
          if (p < 254u) deep |= first[c] & ~(T[c] | tg[p * K::T] | A[3 * c * K::T] | A[3 * p * K::T]);
        }
      for (u32 f = rest & ~deep; f;) {  // patterns with the numbers of the first one
        const u32 i = (u32)__ffs(f) - 1u;
        u32 eq = f, R = closed, ovals = 0;
        auto bit = [&](u32 x) -> u32 {
          const u32 b = (x >> i) & 1u;
          eq &= b ? x : ~x;
          return b;
        };
#pragma unroll
        for (u32 k = 0; k < 5; ++k) R += bit(cnt[k]) << k;
        u32 q[8];
        q[2] = bit(num[0]);
        q[2] += bit(num[1]) << 1;
        q[2] += bit(num[2]) << 2;
#pragma unroll
        for (u32 k = 3; k < 8; ++k) {
          q[k] = bit(num[2 * k - 3]);
          q[k] += bit(num[2 * k - 2]) << 1;
        }
        u64 key = 1;
#pragma unroll
        for (u32 k = 7; k >= 2; --k)  // a region with k - 1 leaves: 1 (10)^(k-1) 0
          for (u32 j = 0; j < q[k]; ++j) {
            key = (key << (2 * k)) | (1ull << (2 * k - 1)) | ((0xAAAAu & ((1u << (2 * k - 2)) - 1u)) << 1);
            ovals += k;
          }
        const u32 leaves = R - 1u - ovals;
        key = (key << (2 * leaves)) | (0xAAAAAAAAAAAAAAAAull & ((1ull << (2 * leaves)) - 1));
        tc_sb_insert<K::HASH>(key, (u32)__popc(eq), out.hkeys, out.hcnt, out.gkeys, out.gcnt,
                              out.gslots, out.gerr);
        f &= ~eq;
      }
      rest &= deep;
    }
  }
  // deeper trees, one by one (patterns of the word with the same classes and
  // root together): queued for the whole block to code, so that its lanes have
  // one each, or coded here when the queue is full
  while (rest) {
    const u32 i = (u32)__ffs(rest) - 1u;
    u64 low = 0;  // smallest node of every node's class, 4 bits each
    u32 rootn = 0, have = 0, eq = rest;
#pragma unroll
    for (u32 c = 0; c < NN; ++c) {
      u32 row = 1u << c;
#pragma unroll
      for (u32 a = 0; a < c; ++a) {
        const u32 x = conn[pair(a, c)], b = (x >> i) & 1u;
        row |= b << a;
        eq &= x ^ (b - 1u);
      }
      low |= (u64)((u32)__ffs(row) - 1u) << (4 * c);
      const u32 g = (T[c] >> i) & 1u;
      eq &= T[c] ^ (g - 1u);
      rootn = g && !have ? c : rootn;
      have |= g;
    }
    rest &= ~eq;
    const u32 at = atomicAdd(m.queued, 1u);
    if (at < K::QUEUE) {
      m.queue[4 * at] = (u32)low;
      m.queue[4 * at + 1] = (u32)(low >> 32);
      m.queue[4 * at + 2] = hl | (rootn << 16);
      m.queue[4 * at + 3] = (u32)__popc(eq);
    } else {
      tc_sb_deep<K>(m, t, hl, low, rootn, (u32)__popc(eq), out, err, failed);
    }
  }
}

#ifndef TC_SL_EMULATE
// Barrier; then code the queued trees when there are enough of them for the
// block's lanes, or (last) all of them.  All threads call it.  The choice is
// one for the block: a thread that went on may already queue trees of its next
// word, so it is thread 0's look before the barrier, not each thread's after it.
template <class K>
__device__ __forceinline__ void tc_sb_flush_queue(const TcSbMem &m, u32 t, bool last, const TcSbOut &out,
                                                  u32 &err, unsigned long long &failed) {
  volatile u32 *const queued = m.queued;
  if (!__syncthreads_or(last || (t == 0 && *queued >= K::QUEUE / 2))) return;
  u32 nq = *queued;
  if (nq > K::QUEUE) nq = K::QUEUE;
  for (u32 i = t; i < nq; i += K::T) {
    const u32 *const q = m.queue + 4 * i;
    tc_sb_deep<K>(m, t, q[2] & 0xFFFFu, ((u64)q[1] << 32) | q[0], q[2] >> 16, q[3], out, err, failed);
  }
  __syncthreads();
  if (t == 0) *queued = 0;
  __syncthreads();
}
#endif
