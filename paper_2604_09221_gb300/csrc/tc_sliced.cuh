// tc_sliced.cuh -- Algorithm 1 for a block of sign vectors at once, bit-sliced
// (the table-driven query, sweep and batch kernels).
//
// A block of NG warps classifies T = 32 NG sign vectors together.  The part
// of the method that looks at every edge of T^diamond (crossing tests, which
// earlier neighbour gives a vertex its label, where two runs of a fan have to
// be joined) is plain logic, so it runs on 32 sign vectors per instruction:
// bit i of a word is instance i of a group of 32.  Only the few events it
// leaves (about one vertex in eight starts a label, about one in eight joins
// two) are handled one instance per thread.  Phases, a barrier between each:
//
//   planes   sign vectors -> one word per lattice point and group (32 x 32
//            bit transposes across the warp)
//   logic    (vertex, group) per thread, vertices in order of fan length:
//            for every fan entry the mask of the instances that take their
//            label from it (first same-sign entry), hence the number of that
//            neighbour (of the vertex itself if it starts a label) as bit
//            planes; per vertex the mask of the instances in which it starts a
//            label, per entry that can start a second run the mask of the
//            instances that have to join
//   tiles    planes -> one byte (d >= 11: half-word) per vertex and
//            instance, in place; event masks -> one word per instance
//   labels   one instance per thread: vertices in sweep order, every vertex
//            gets the label of the neighbour its byte names (a label is the
//            number of the vertex that starts it)
//   trees    one instance per thread: joins in a union-find over the label
//            bytes themselves (a vertex that starts a label points at itself),
//            regions (whose numbers then replace the bytes of the starts),
//            region tree, root and code
//
// Everything a block touches is in shared memory; nothing is allocated.
//
// Root of even degree (Alg. 1 lines 6-7), without orientation parities: a
// region X that is a disk with holes has Euler number chi(X) = 2 - (its
// neighbours in the region tree), the non-orientable region 1 less.  So the
// root is the one region for which chi plus degree is odd; chi of a region
// counts its label starts minus its join events (a vertex with k runs of
// same-sign earlier neighbours adds 1 - k; identifying a run of boundary
// vertices with its antipodes takes one away).
//
// Antipodal joins.  Consecutive boundary vertices of one sign are joined by
// their boundary edge, and so are their antipodes; so a pair is joined only
// where the boundary edge in front of it is crossed.  Those crossed edges are
// also the pseudoline's candidates (odd d).
#pragma once

#include "tc_layout.h"
#include "tc_runtime.cuh"

// Table words (host.cpp, pack_sliced_tables), staged into shared memory:
//   header   [0] steps of a half-diamond  [1] event chunks of half-diamond
//            joins  [2] event chunks in all  [3] off_fan  [4] off_vd
//            [5] off_site  [6] off_bx  [7] off_be  [8] steps in all
//   task[V]  two words per vertex, in order of fan length: k(v) (8 bits) |
//            fan steps << 8 (8 bits) | first fan entry << 16, and
//            v | first join site << 16
//   fan[]    in steps of four entries, vertices in sweep order, a vertex's
//            last step padded (one step for an empty fan): k(u) (8 bits) |
//            u << 8 (16 bits) | "can start a second run" << 24 | "another step
//            of this vertex follows" << 25 | link << 30 |
//            (c(u) ^ c(v) ^ 1) << 31; padding: k(v) (never of v's sign) | 1 << 26
//   vd[V]    u of the first fan entry | "the fan is not empty" << 15
//   site[]   32 per chunk of join events: v | u << 16: the half-diamonds'
//            sites, one chunk of boundary pairs, the middle row's sites
//   bx[2d]   k(a) | k(b) << 8 | (c(a) ^ c(b)) << 16 | event slot << 17 of the
//            boundary edges of half the boundary, in cyclic order
//   be[2d]   a | b << 16 of the same edges
#define TC_SL_HEADER 12u
#define TC_SL_GROUP 40u  // words of one group's event chunk: 32 and a pad
                         // (the trees phase reads it conflict-free)

template <int D_, int NG_>
struct TcSlK {
  static constexpr TcLayout L = tc_layout(D_, true, 32);
  static constexpr u32 D = D_, NG = NG_, T = 32 * NG_, V = L.V, NPOINTS = L.np, W = L.sw,
                       CW = L.cw, RMAX = L.rmax, WIDE = L.wide, HASH = L.hash, CODE64 = L.code64;
  static constexpr u32 H = D * D;                 // vertices of one half-diamond
  static constexpr u32 LB = V <= 256 ? 1 : 2;     // bytes per label
  static constexpr u32 NPL = V <= 128 ? 7 : V <= 256 ? 8 : V <= 512 ? 9 : 10;  // label planes
  static constexpr u32 TW = 8 * LB;               // words of a vertex's tile per group
  static constexpr u32 NCB = (V + 31) / 32;       // birth chunks
  static constexpr bool EVEN = D % 2 == 0;
  static constexpr u32 LABW = V * TW * NG;        // words of the label area
  static constexpr u32 PAR_WORDS = (RMAX + 3) / 4 * T;  // region parents, a byte each
  static constexpr u32 PLANES = (NPOINTS * NG + 3) & ~3u;
  // d = 10 (one-byte labels, more regions than spare byte values) keeps the
  // roots' words apart from the starts' (NCB per thread)
  static constexpr u32 ROOT_WORDS = LB == 1 && !(V < 224 && RMAX <= 32) ? NCB * T : 0;
  static constexpr u32 XW = PLANES > PAR_WORDS + ROOT_WORDS ? PLANES : PAR_WORDS + ROOT_WORDS;
  // tree codes: the wide back end's scratch lies over the label area
  static constexpr u32 THREADS = T;
  static constexpr u32 WB = (RMAX + 3) / 4, WARENA = L.warena_words;
  static constexpr u32 OFF_WPAR = 0, OFF_WFC = WB, OFF_WNS = 2 * WB, OFF_WENT = 3 * WB,
                       OFF_WARENA = 3 * WB + (RMAX / 2 + 2 + 1) / 2,
                       OFF_WTEMP = OFF_WARENA + WARENA, WIDE_WORDS = OFF_WTEMP + WARENA;
  // up to 57 regions (d <= 12): tree codes in two words, children sets of two
  // words each over the label area and the event chunks (AREA words of them).
  // Against the byte-tree back end (tc_backend_wide's code): 2^18 queries at
  // d = 12 562 -> 437 us, 2^21 sampled vectors at d = 10 1914 -> 1546 us.
  static constexpr bool TREE2 = WIDE && RMAX <= 58;
  static constexpr u32 AREA = TREE2 && 2 * RMAX * T > LABW ? 2 * RMAX * T - LABW : 0;
  static_assert(!TREE2 || CW == 2, "tree codes of two words");
  static_assert(WIDE || RMAX * T <= LABW, "the narrow tree code's children masks fit the label area");
  static_assert(!WIDE || WIDE_WORDS * T <= LABW, "the wide back end's scratch fits the label area");
  // unused members TcScratch names
  static constexpr u32 LBYTES = LB, OFF_LPAR = 0, OFF_CAND = 0;
};

// Shared-memory areas of a block.
struct TcSlMem {
  const u32 *tab;  // staged tables
  u32 *lab;        // label planes, then label bytes (K::LABW words)
  u32 *ev;         // event chunks (chunks x NG x TC_SL_GROUP words)
  u32 *x;          // sign planes, then region parents
};

// Words of a block's areas behind the tables (chunks of events).  The last
// area holds the sign planes, in the trees phase the region parents.
template <class K>
__host__ __device__ constexpr u32 tc_sl_evwords(u32 chunks) {
  return chunks * K::NG * TC_SL_GROUP > K::AREA ? chunks * K::NG * TC_SL_GROUP : K::AREA;
}
template <class K>
__host__ __device__ constexpr u32 tc_sl_words(u32 chunks) {
  return K::LABW + tc_sl_evwords<K>(chunks) + K::XW;
}

template <class K>
__device__ __forceinline__ TcSlMem tc_sl_carve(const u32 *tab, u32 *area, u32 chunks) {
  TcSlMem m;
  m.tab = tab;
  m.lab = area;
  m.ev = m.lab + K::LABW;
  m.x = m.ev + tc_sl_evwords<K>(chunks);
  return m;
}

struct alignas(16) TcQuad {
  u32 a, b, c, d;
};
struct alignas(8) TcPair {
  u32 a, b;
};

// 32 x 32 bit transpose across a warp: lane r's word is row r; lane r gets
// column r.  Stage j exchanges words with the lane at distance j and swaps the
// off-diagonal j x j blocks: one shuffle, one rotate (by the lane's side), one
// bitwise select.
#ifndef TC_SL_EMULATE
struct TcTranspose {
  u32 keep[5], rot[5];
  __device__ __forceinline__ explicit TcTranspose(u32 lane) {
#pragma unroll
    for (u32 s = 0; s < 5; ++s) {
      const u32 j = 16u >> s, m = 0xFFFFFFFFu / ((1u << j) + 1u);  // low halves of the 2j-bit blocks
      keep[s] = (lane & j) ? ~m : m;
      rot[s] = (lane & j) ? 32u - j : j;
    }
  }
  __device__ __forceinline__ u32 operator()(u32 x) const {
#pragma unroll
    for (u32 s = 0; s < 5; ++s) {
      const u32 y = __shfl_xor_sync(0xffffffffu, x, 16u >> s);
      x = (x & keep[s]) | (__funnelshift_l(y, y, rot[s]) & ~keep[s]);
    }
    return x;
  }
};
#endif

// Instance (of the block's T) that thread t holds in the trees phase: label
// bytes of one vertex are T consecutive bytes, four instances to a word, and
// a warp's threads read 32 different words, so that any mix of vertices is
// free of bank conflicts.
template <class K>
__device__ __forceinline__ u32 tc_sl_instance(u32 t) {
  constexpr u32 WR = K::TW * K::NG;  // words per vertex
  const u32 word = t % WR, part = t / WR, g = word / K::TW, q = word % K::TW;
  return 32u * g + (K::LB == 1 ? 8u * part + q : 8u * (2u * (q >> 3) + part) + (q & 7u));
}

// ---- planes: clear the event chunks; transpose the sign words ----
template <class K>
__device__ __forceinline__ void tc_sl_clear(const TcSlMem &m, u32 t) {
  const u32 n = m.tab[2] * K::NG * TC_SL_GROUP;
  for (u32 i = t; i < n; i += K::T) m.ev[i] = 0;
}

// sg: the sign vector of instance t of the block (warp t / 32 is a group).
#ifndef TC_SL_EMULATE
template <class K>
__device__ __forceinline__ void tc_sl_planes(const TcSlMem &m, const TcSig<K::W> &sg, u32 t) {
  const u32 g = t >> 5, lane = t & 31u;
  const TcTranspose transpose(lane);
#pragma unroll
  for (u32 j = 0; j < (K::NPOINTS + 31) / 32; ++j) {
    const u32 half = (u32)(sg.w[j / 2] >> (32 * (j & 1)));
    const u32 p = transpose(half);
    if (32 * j + lane < K::NPOINTS) m.x[(32 * j + lane) * K::NG + g] = p;
  }
}
#endif

// All ones if bit b of f is set, else zero.
__device__ __forceinline__ u32 tc_bitmask(u32 f, u32 b) { return (u32)((int)(f << (31u - b)) >> 31); }

template <class K>
__device__ __forceinline__ u32 *tc_sl_event(const TcSlMem &m, u32 slot, u32 g) {
  return m.ev + ((slot >> 5) * K::NG + g) * TC_SL_GROUP + (slot & 31u);
}

// ---- logic: one (vertex, group) at a time, four fan entries a step ----
template <class K>
__device__ __forceinline__ void tc_sl_logic(const TcSlMem &m, u32 t) {
  const u32 g = t % K::NG;
  const u32 *const P = m.x + g;
  const TcPair *task = reinterpret_cast<const TcPair *>(m.tab + TC_SL_HEADER) + t / K::NG;
  const u32 *const fan = m.tab + m.tab[3];
  for (u32 k = t / K::NG; k < K::V; k += 32u, task += 32) {
    const TcPair w = *task;
    const u32 sv = P[(w.a & 255u) * K::NG], steps = (w.a >> 8) & 255u, v = w.b & 0xFFFFu;
    u32 site = w.b >> 16, any = 0, prev = 0;
    const TcQuad *f = reinterpret_cast<const TcQuad *>(fan + (w.a >> 16));
    u32 plane[K::NPL];  // of the number of the vertex the label comes from
#pragma unroll
    for (u32 i = 0; i < K::NPL; ++i) plane[i] = 0;
    auto from = [&](u32 mask, u32 u) {
#pragma unroll
      for (u32 i = 0; i < K::NPL; ++i)
        if (u & (1u << i)) plane[i] |= mask;
    };
    for (u32 j = 0; j < steps; ++j, ++f) {
      const TcQuad q = *f;
      // the four entries' masks "same sign as v"
      const u32 ea = P[(q.a & 255u) * K::NG] ^ sv ^ (u32)((int)q.a >> 31);
      const u32 eb = P[(q.b & 255u) * K::NG] ^ sv ^ (u32)((int)q.b >> 31);
      const u32 ec = P[(q.c & 255u) * K::NG] ^ sv ^ (u32)((int)q.c >> 31);
      const u32 ed = P[(q.d & 255u) * K::NG] ^ sv ^ (u32)((int)q.d >> 31);
      auto entry = [&](u32 f, u32 e) {
        if (f & (1u << 24)) {  // a run that may follow another one
          *tc_sl_event<K>(m, site, g) = e & any & ~(prev & tc_bitmask(f, 30));
          ++site;
        }
        from(e & ~any, f >> 8);
        any |= e;
        prev = e;
      };
      entry(q.a, ea);
      entry(q.b, eb);
      entry(q.c, ec);
      entry(q.d, ed);
    }
    from(~any, v);
    u32 *const out = m.lab + (v * K::NG + g) * K::TW;
    if constexpr (K::LB == 1) {
      TcQuad *const o = reinterpret_cast<TcQuad *>(out);
      o[0] = TcQuad{plane[0], plane[1], plane[2], plane[3]};
      o[1] = TcQuad{plane[4], plane[5], plane[6], K::NPL > 7 ? plane[K::NPL - 1] : 0u};
    } else {
      TcQuad *const o = reinterpret_cast<TcQuad *>(out);
      o[0] = TcQuad{plane[0], plane[1], plane[2], plane[3]};
      o[1] = TcQuad{plane[4], plane[5], plane[6], plane[7]};
      o[2] = TcQuad{plane[8], K::NPL > 9 ? plane[K::NPL - 1] : 0u, 0u, 0u};
    }
    *tc_sl_event<K>(m, v, g) = ~any;  // v starts a label
  }
  // crossed boundary edges
  const u32 *const bx = m.tab + m.tab[6];
  for (u32 k = t / K::NG; k < 2 * K::D; k += 32u) {
    const u32 w = bx[k];
    *tc_sl_event<K>(m, w >> 17, g) = P[(w & 255u) * K::NG] ^ P[((w >> 8) & 255u) * K::NG] ^ tc_bitmask(w, 16);
  }
}

// ---- tiles ----
// Bytes c = 0..3 of the words p[0..7] as four 8 x 8 bit matrices, transposed:
// byte c of word r gets bit s of p[s]'s byte c, bit r.
__device__ __forceinline__ void tc_transpose8(u32 (&p)[8]) {
#pragma unroll
  for (u32 j = 4, mk = 0x0F0F0F0Fu; j; j >>= 1, mk ^= mk << j) {
#pragma unroll
    for (u32 r = 0; r < 8; ++r)
      if (!(r & j)) {
        const u32 x = ((p[r] >> j) ^ p[r + j]) & mk;
        p[r + j] ^= x;
        p[r] ^= x << j;
      }
  }
}

template <class K>
__device__ __forceinline__ void tc_sl_tiles(const TcSlMem &m, u32 t) {
  for (u32 k = t; k < K::V * K::NG; k += K::T) {
    TcQuad *const q = reinterpret_cast<TcQuad *>(m.lab + k * K::TW);
    const TcQuad x = q[0], y = q[1];
    u32 lo[8] = {x.a, x.b, x.c, x.d, y.a, y.b, y.c, K::NPL > 7 ? y.d : 0u};
    tc_transpose8(lo);
    if constexpr (K::LB == 1) {
      q[0] = TcQuad{lo[0], lo[1], lo[2], lo[3]};
      q[1] = TcQuad{lo[4], lo[5], lo[6], lo[7]};
    } else {  // planes 8 and 9: two more bits per label
      const TcQuad z = q[2];
      u32 h[8] = {z.a, K::NPL > 9 ? z.b : 0u, 0, 0, 0, 0, 0, 0};
      tc_transpose8(h);
      u32 o[16];
#pragma unroll
      for (u32 r = 0; r < 8; ++r) {  // bytes 0, 1 and bytes 2, 3 with their high bytes
        o[r] = (lo[r] & 0xFFu) | ((h[r] & 0xFFu) << 8) | ((lo[r] & 0xFF00u) << 8) | ((h[r] & 0xFF00u) << 16);
        o[8 + r] = ((lo[r] >> 16) & 0xFFu) | (((h[r] >> 16) & 0xFFu) << 8) | (((lo[r] >> 24) & 0xFFu) << 16) |
                   (h[r] & 0xFF000000u);
      }
#pragma unroll
      for (u32 r = 0; r < 4; ++r) q[r] = TcQuad{o[4 * r], o[4 * r + 1], o[4 * r + 2], o[4 * r + 3]};
    }
  }
}

#ifndef TC_SL_EMULATE
template <class K>
__device__ __forceinline__ void tc_sl_events(const TcSlMem &m, u32 t) {
  const TcTranspose transpose(t & 31u);
  u32 *p = m.ev + (t >> 5) * TC_SL_GROUP + (t & 31u);
  u32 *const end = m.ev + m.tab[2] * K::NG * TC_SL_GROUP;
  for (; p < end; p += K::NG * TC_SL_GROUP) *p = transpose(*p);
}
#endif

// ---- trees: one instance per thread ----
template <u32 LB>
struct TcSlLab;
template <>
struct TcSlLab<1> {
  typedef u8 T;
};
template <>
struct TcSlLab<2> {
  typedef u16 T;
};

// One thread's labels, event words and region parents.
template <class K>
struct TcSlInst {
  typedef typename TcSlLab<K::LB>::T lab_t;
  static constexpr u32 ROW = K::T;  // labels per vertex
  // A start's region number replaces its label byte, marked by bits that no
  // vertex number has set; at d = 10 there are too few spare numbers, and a
  // start is told by its event bit.
  static constexpr u32 MARK = K::LB == 2 ? 0x8000u : K::V < 224 && K::RMAX <= 32 ? 224u : 0u;
  lab_t *l;
  u32 *ev;
  u8 *par;  // region r: byte r % 4 of word r / 4
  __device__ __forceinline__ TcSlInst(const TcSlMem &m, u32 t) {
    constexpr u32 WR = K::TW * K::NG;
    const u32 i = tc_sl_instance<K>(t);
    l = reinterpret_cast<lab_t *>(m.lab + t % WR) + t / WR;
    ev = m.ev + (i >> 5) * TC_SL_GROUP + (i & 31u);
    par = reinterpret_cast<u8 *>(m.x + t);
  }
  // roots among the starts of chunk c: over the starts' word, but at d = 10
  __device__ __forceinline__ u32 *root_word(u32 c) const {
    return MARK ? ev + c * (K::NG * TC_SL_GROUP) : reinterpret_cast<u32 *>(par) + K::PAR_WORDS + c * K::T;
  }
  __device__ __forceinline__ u8 &parent(u32 r) const { return par[(r >> 2) * 4 * K::T + (r & 3u)]; }
  __device__ __forceinline__ u32 raw(u32 v) const { return l[v * ROW]; }
  __device__ __forceinline__ void set(u32 v, u32 x) const { l[v * ROW] = (lab_t)x; }
  __device__ __forceinline__ u32 event(u32 chunk) const { return ev[chunk * (K::NG * TC_SL_GROUP)]; }
  __device__ __forceinline__ void set_event(u32 chunk, u32 w) const { ev[chunk * (K::NG * TC_SL_GROUP)] = w; }
  // region of vertex v, once the starts up to it (or its label) have theirs
  __device__ __forceinline__ u32 region(u32 v) const {
    const u32 x = raw(v);
    if constexpr (MARK != 0)
      return (x < MARK ? raw(x) : x) - MARK;
    else
      return (event(v >> 5) >> (v & 31u)) & 1u ? x : raw(x);
  }
};

// ---- labels: vertices [0, n) in sweep order ----
// A vertex's neighbour comes before it, so that one's entry is its label
// already.  Four vertices' entries are loaded ahead of their labels.
template <class K>
__device__ __forceinline__ void tc_sl_labels(const TcSlInst<K> &I, u32 n) {
  u32 v = 0;
  for (; v + 4 <= n; v += 4) {
    u32 p[4];
#pragma unroll
    for (u32 i = 0; i < 4; ++i) p[i] = I.raw(v + i);
#pragma unroll
    for (u32 i = 0; i < 4; ++i) I.set(v + i, I.raw(p[i]));
  }
  for (; v < n; ++v) I.set(v, I.raw(I.raw(v)));
}

// Joins of the event chunks [c0, c1) without parity.  The next event and its
// two labels are loaded before the present join's roots are known (a label
// read early is still a label of the same set).
template <class K>
__device__ __forceinline__ void tc_sl_joins(const TcSlInst<K> &I, const u32 *site, u32 c0, u32 c1) {
  u32 c = c0, w = 0;
  while (w == 0 && c < c1) w = I.event(K::NCB + c++);
  if (w == 0) return;
  u32 s = site[32u * (c - 1u) + (u32)__ffs(w) - 1u];
  w &= w - 1u;
  u32 na = I.raw(s & 0xFFFFu), nb = I.raw(s >> 16);
  for (;;) {
    u32 a = na, b = nb, pa, pb;
    while (w == 0 && c < c1) w = I.event(K::NCB + c++);
    const bool more = w != 0;
    if (more) {
      s = site[32u * (c - 1u) + (u32)__ffs(w) - 1u];
      w &= w - 1u;
      na = I.raw(s & 0xFFFFu);
      nb = I.raw(s >> 16);
    }
    do {
      pa = a;
      pb = b;
      a = I.raw(pa);
      b = I.raw(pb);
    } while (a != pa || b != pb);
    if (a != b) I.set(a < b ? b : a, a < b ? a : b);
    if (!more) return;
  }
}

// Region numbers in the order of the regions' smallest labels: every start
// gets its region (a parent is smaller, so it has its region already), and
// the roots' words the starts that are roots.  on_start(r): called for every
// start with its region.  Returns the number of regions.
template <class K, class F>
__device__ __forceinline__ u32 tc_sl_number(const TcSlInst<K> &I, F on_start) {
  constexpr u32 MARK = TcSlInst<K>::MARK;
  u32 R = 0, left = 0;
#pragma unroll
  for (u32 c = 0; c < K::NCB; ++c) left += (u32)__popc(I.event(c));
  u32 c = 0, w = 0, roots = 0;
  for (; left; --left) {
    while (w == 0) {
      if (c) *I.root_word(c - 1u) = roots;
      roots = 0;
      w = I.event(c++);
    }
    const u32 bit = (u32)__ffs(w) - 1u, v = 32u * (c - 1u) + bit;
    w &= w - 1u;
    const u32 p = I.raw(v);
    const bool is_root = p == v;
    const u32 x = is_root ? MARK + R : I.raw(p);
    I.set(v, x);
    on_start(x - MARK);
    roots |= is_root ? 1u << bit : 0u;
    R += is_root;
  }
  *I.root_word(c - 1u) = roots;
  return R;
}

// Joins, regions and the region tree of one instance.  Returns the number of
// regions R (0: failed, err set) with their parents in I.parent(r) (< r, r >=
// 1) and the region the tree is rooted at; star (narrow back end): every oval
// is outermost.
template <class K>
__device__ __forceinline__ u32 tc_sl_regions(const TcSlMem &m, const TcSlInst<K> &I, u32 &root, bool &star,
                                             u32 &err) {
  const u32 *const tab = m.tab;
  const u32 *const site = tab + tab[5];
  const u32 nc1 = tab[1], nc = tab[2] - K::NCB;
  tc_sl_joins<K>(I, site, 0, nc);
  // chi + degree of the regions modulo 2, a bit each (even d)
  u64 odd = 0, odd1 = 0;
  auto toggle = [&](u32 r) {
    if constexpr (K::RMAX <= 32) {
      odd ^= 1u << (r & 31u);
    } else if constexpr (K::RMAX <= 64) {
      odd ^= 1ull << (r & 63u);
    } else {
      const u64 b = 1ull << (r & 63u);
      odd ^= r < 64u ? b : 0ull;
      odd1 ^= r < 64u ? 0ull : b;
    }
  };
  u32 R;
  if constexpr (K::EVEN) {
    R = tc_sl_number<K>(I, toggle);
    u32 c = 0, w = 0;
    for (;;) {
      while (w == 0 && c < nc) w = I.event(K::NCB + c++);
      if (w == 0) break;
      const u32 s = site[32u * (c - 1u) + (u32)__ffs(w) - 1u];
      w &= w - 1u;
      toggle(I.region(s & 0xFFFFu));
    }
  } else {
    R = tc_sl_number<K>(I, [](u32) {});
    // the pseudoline's region: both ends of a crossed boundary edge in one
    // region; the near end of a crossed edge is in the region of the far end
    // of the one before
    const u32 *const be = tab + tab[7];
    u32 prev = I.region(be[0] & 0xFFFFu), rv = ~0u;
    bool two = false;
    for (u32 w = I.event(K::NCB + nc1); w; w &= w - 1u) {
      const u32 a = I.region(be[(u32)__ffs(w) - 1u] >> 16);
      two |= a == prev && rv != ~0u && rv != a;
      rv = a == prev ? a : rv;
      prev = a;
    }
    if (two || rv == ~0u) {
      err |= TC_ERR_INTERNAL;
      return 0;
    }
    root = rv;
  }
  if (R > K::RMAX) {
    err |= TC_ERR_OVERFLOW;
    return 0;
  }
  // the tree hanging from region 0: the parent of region r is the region of
  // the first earlier neighbour of its smallest label's vertex
  const u32 *const vd = tab + tab[4];
  bool bad = false;
  u32 internal = 0, kids0 = 0, c = 0, w = 0;
  for (u32 r = 0; r < R; ++r) {
    while (w == 0) w = *I.root_word(c++);
    const u32 v = 32u * (c - 1u) + (u32)__ffs(w) - 1u;
    w &= w - 1u;
    if (r) {
      const u32 d = vd[v], p = I.region(d & 0x7FFFu);
      bad |= !(d & 0x8000u) || p >= r;  // no earlier neighbour, or not a tree
      I.parent(r) = (u8)p;
      if constexpr (K::EVEN) {
        toggle(r);
        toggle(p);
      }
      if constexpr (!K::WIDE) {
        internal |= 1u << (p & 31u);
        kids0 |= p == 0 ? 1u << r : 0u;
      }
    }
  }
  if constexpr (K::EVEN) {
    bad |= __popcll(odd) + __popcll(odd1) != 1;
    root = odd ? (u32)__ffsll(odd) - 1u : 63u + (u32)__ffsll(odd1);
  }
  if (bad) {
    err |= TC_ERR_INTERNAL;
    return 0;
  }
  if constexpr (!K::WIDE)
    star = !(internal & ~(1u | (1u << root))) && (root == 0 || kids0 == 1u << root);
  return R;
}

// Sets of regions and codes of the tree codes below: up to 32 regions with
// codes of up to 56 bits, or up to 64 with codes of up to 112 bits.
template <u32 WORDS>
struct TcTreeSet;
template <>
struct TcTreeSet<1> {
  typedef u32 set_t;
  typedef u64 code_t;
  static __device__ __forceinline__ u32 low(set_t x) { return (u32)__ffs(x) - 1u; }
  static __device__ __forceinline__ u32 high(set_t x) { return 31u - (u32)__clz(x); }
  static __device__ __forceinline__ u32 size(set_t x) { return (u32)__popc(x); }
};
template <>
struct TcTreeSet<2> {
  typedef u64 set_t;
  typedef unsigned __int128 code_t;
  static __device__ __forceinline__ u32 low(set_t x) { return (u32)__ffsll(x) - 1u; }
  static __device__ __forceinline__ u32 high(set_t x) {
    return x >> 32 ? 63u - (u32)__clz((u32)(x >> 32)) : 31u - (u32)__clz((u32)x);
  }
  static __device__ __forceinline__ u32 size(set_t x) { return (u32)__popcll(x); }
};

// Canonical code of a region tree that is no star.  alive: the regions'
// numbers (region 0 or the smallest one first); parent of region r: byte r % 4
// of par's group r / 4 (PW bytes apart), smaller than r; adj: children sets,
// word w of region r's at adj[(WORDS r + w) AW], written here.  The tree is
// re-rooted by reversing the path from the root to the first region; AHU codes
// follow for the regions with children, those off the path by falling number
// (children have larger ones), then along the path.  A code is left-aligned
// with its length in the low byte; a leaf's code '10' is the smallest.  The
// halves of a region's code take the place of its children set and of one
// child's (whose code is used by then), that child's number the place of its
// parent: no local memory.
// Returns (1 << bits) | bits, zero with err set on failure.
template <u32 WORDS, u32 AW, u32 PW, u32 RMAX>
__device__ __forceinline__ typename TcTreeSet<WORDS>::code_t tc_sl_tree_code(
    u8 *par, u32 *adj, typename TcTreeSet<WORDS>::set_t alive, u32 root, u32 &err) {
  typedef TcTreeSet<WORDS> TS;
  typedef typename TS::set_t set_t;
  typedef typename TS::code_t code_t;
  constexpr u32 BITS = 64 * WORDS, NONE = 255;
  static_assert(2 * RMAX <= BITS - 6 && RMAX <= 32 * WORDS, "tree codes");
  auto up_of = [&](u32 r) -> u8 & { return par[(r >> 2) * PW + (r & 3u)]; };
  auto kids_of = [&](u32 r) -> set_t {
    if constexpr (WORDS == 1) return adj[r * AW];
    else return (set_t)adj[2 * r * AW] | ((set_t)adj[(2 * r + 1) * AW] << 32);
  };
  auto set_kids = [&](u32 r, set_t x) {
    adj[WORDS * r * AW] = (u32)x;
    if constexpr (WORDS == 2) adj[(2 * r + 1) * AW] = (u32)(x >> 32);
  };
  const set_t one = 1;
  const u32 first = TS::low(alive);
  for (set_t a = alive; a; a &= a - 1u) set_kids(TS::low(a), 0);
  set_t internal = 0, path = 0;
  for (set_t a = alive & (alive - 1u); a; a &= a - 1u) {
    const u32 r = TS::low(a), p = up_of(r);
    adj[(WORDS * p + (r >> 5)) * AW] |= 1u << (r & 31u);
    internal |= one << p;
  }
  for (u32 x = root, prev = NONE;;) {  // reverse the path root -> first region
    const u32 up = x == first ? NONE : (u32)up_of(x);
    set_t kids = kids_of(x);
    if (prev != NONE) kids &= ~(one << prev);
    if (x != first) kids |= one << up;
    set_kids(x, kids);
    internal = kids ? internal | (one << x) : internal & ~(one << x);
    path |= one << x;
    up_of(x) = (u8)prev;
    if (x == first) break;
    prev = x;
    x = up;
  }
  const u32 nb2 = 2u * (TS::size(alive) - 1u);
  if (nb2 == 0) return 1;  // no ovals (the pseudoline alone)
  code_t tens = 0xAAAAAAAAAAAAAAAAull;
  if constexpr (WORDS == 2) tens |= tens << 64;
  set_t off = internal & ~path;
  u32 x = 0, next = first;
  for (;;) {
    if (off) {
      x = TS::high(off);
      off &= ~(one << x);
    } else if (path) {  // from the first region towards the root
      x = next;
      next = up_of(x);
      path &= ~(one << x);
      if (!((internal >> x) & 1u)) continue;
    } else {
      break;
    }
    const set_t kids = kids_of(x);
    code_t v = 0;
    u32 len = 0;
    for (set_t big = kids & internal; big;) {  // larger codes first
      u32 best = 0;
      code_t bv = 0;
      for (set_t y = big; y; y &= y - 1u) {
        const u32 k = TS::low(y);
        const code_t cv = ((code_t)kids_of(k) << (BITS / 2)) | (code_t)kids_of(up_of(k));
        if (cv > bv) {
          bv = cv;
          best = k;
        }
      }
      v |= (bv & ~(code_t)255) >> len;
      len += (u32)bv & 255u;
      big &= ~(one << best);
    }
    const u32 nl = 2u * TS::size(kids & ~internal);
    if (nl) v |= (tens & ~(~(code_t)0 >> nl)) >> len;
    len += nl;
    if (x == root) {
      if (len != nb2) break;
      return ((code_t)1 << len) | (v >> (BITS - len));
    }
    const u32 slot = TS::low(kids);
    const code_t c = ((code_t)1 << (BITS - 1)) | (v >> 1) | (code_t)(len + 2u);
    set_kids(x, (set_t)(c >> (BITS / 2)));
    set_kids(slot, (set_t)c);
    up_of(x) = (u8)slot;
  }
  err |= TC_ERR_INTERNAL;
  return 0;
}

// Code of thread t's instance from tc_sl_regions' result (all zero if it
// failed).  The tree codes work over the label area, so every thread of the
// block must be done with tc_sl_regions.
template <class K>
__device__ __forceinline__ void tc_sl_finish(const TcSlMem &m, const TcSlInst<K> &I, u32 t, u32 R, u32 root,
                                             bool star, u32 &err, u64 *code) {
  if constexpr (!K::WIDE) {
    const u32 q = 2 * (R - 1);
    code[0] = R == 0 ? 0ull
              : star ? (1ull << q) | (0xAAAAAAAAAAAAAAAAull & ((1ull << q) - 1))
                     : tc_sl_tree_code<1, K::T, 4 * K::T, K::RMAX>(I.par, m.lab + t,
                                                                   R >= 32 ? ~0u : (1u << R) - 1u, root, err);
  } else if constexpr (K::TREE2) {
    code[0] = code[1] = 0;
    if (R == 0) return;
    const unsigned __int128 c = tc_sl_tree_code<2, K::T, 4 * K::T, K::RMAX>(
        I.par, m.lab + t, R >= 64 ? ~0ull : (1ull << R) - 1ull, root, err);
    code[0] = (u64)c;
    code[1] = (u64)(c >> 64);
  } else {
#pragma unroll
    for (u32 w = 0; w < K::CW; ++w) code[w] = 0;
    if (R == 0) return;
    const TcScratch<K> S{m.lab + t};
    for (u32 r = 1; r < R; ++r) *S.byte(K::OFF_WPAR, r) = I.parent(r);
    tc_wide_tree_code(S, R, (int)root, err, code);
  }
}

#ifndef TC_SL_EMULATE
// The whole classification: sg is the sign vector of instance t of the block,
// code receives that of instance tc_sl_instance<K>(t) (zero if it failed).
// All T threads call it, after a barrier behind the last use of the areas.
template <class K>
__device__ __forceinline__ void tc_sl_classify(const TcSlMem &m, const TcSig<K::W> &sg, u32 t, u32 &err,
                                               u64 *code) {
  tc_sl_clear<K>(m, t);
  tc_sl_planes<K>(m, sg, t);
  __syncthreads();
  tc_sl_logic<K>(m, t);
  __syncthreads();
  tc_sl_tiles<K>(m, t);
  tc_sl_events<K>(m, t);
  __syncthreads();
  const TcSlInst<K> I(m, t);
  tc_sl_labels<K>(I, K::V);
  u32 root = 0;
  bool star = false;
  const u32 R = tc_sl_regions<K>(m, I, root, star, err);
  __syncthreads();  // tree codes are made over the label area
  tc_sl_finish<K>(m, I, t, R, root, star, err, code);
}
#endif

// ---- launch shape of the query, sweep and batch kernels ----
// Bytes of shared memory of a block: tables, mbarrier and work slot, areas.
template <class K>
constexpr size_t tc_sl_bytes(u32 table_words, u32 chunks) {
  return ((size_t)table_words * 4 + 127) / 128 * 128 + 128 + (size_t)tc_sl_words<K>(chunks) * 4;
}
// Blocks of 128 sign vectors; from d = 13 (130 to 195 KB) of 64, what limits
// them being the sign vectors a multiprocessor's shared memory holds (d = 13:
// three blocks of 64, one of 128; 0.40 against 0.28e9 schemes/s).
template <int D>
using TcSlNarrow = TcSlK<D, D <= 12 ? 4 : 2>;
// Or, at d = 13 and 14, of 192 where that is more, so that the n sign vectors of
// a launch are fewer waves of blocks (152 multiprocessors): one block of 192
// against two of 64 at d = 14 (2^21 queries 10.2 -> 7.4 ms, one thread per sign
// vector with scratch in global memory 8.6; 2^16 0.42 -> 0.35; as many waves,
// 2^13 0.136 against 0.142, 2^15 0.23 against 0.24).  Bound by latency: six
// warps per multiprocessor issue in 26 % of the slots.  Above, 192 do not fit.
template <int D>
using TcSlWide = TcSlK<D, D == 13 || D == 14 ? 6 : D <= 12 ? 4 : 2>;
template <int D>
constexpr bool tc_sl_wide(u32 table_words, u32 chunks, u64 n) {
  constexpr size_t BLOCK = 227 * 1024, SM = 228 * 1024, RESERVED = 1024;  // of a block
  constexpr u32 NT = TcSlNarrow<D>::T, WT = TcSlWide<D>::T;
  const size_t nb = tc_sl_bytes<TcSlNarrow<D>>(table_words, chunks), wb = tc_sl_bytes<TcSlWide<D>>(table_words, chunks);
  if (WT <= NT || wb > BLOCK) return false;
  const u64 narrow = SM / (nb + RESERVED) * NT * 152, wide = SM / (wb + RESERVED) * WT * 152;  // a wave
  return (n + wide - 1) / wide < (n + narrow - 1) / narrow;
}
