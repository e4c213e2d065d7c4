// escg_patch.cuh -- the elementary step (Alg. 3) on sub-blocks held in
// registers, and the shared-memory layout that makes loading them cheap.
//
// Layout.  Along one axis the fine segments k = 0, 1, ... are 2 or 3 sites
// wide.  A "slot" of the axis holds two sites that sit on either side of a
// segment boundary: joint slot J(k) holds the last site of segment k - 1
// (half 0) and the first site of segment k (half 1); a segment of 3 sites
// also has a slot of its own, J(k) + 1, for its middle site (half 0).  A
// "macro" is the 2 x 2 sites of a row slot and a column slot, in a byte (2
// bits per site, states 0..3: S <= 3) or two (4 bits per site); the site of
// row half h and column half g is its field 2h + g.
//
// Why.  Everything the attempts of a 2 x 2 sub-block read or write -- its
// four sites and their neighbours, diagonal ones included -- are the sites of
// the four macros at its corners, and in one fine phase every macro belongs
// to exactly one sub-block.  So a visit of a sub-block is four loads, four
// steps on one or two 32-bit registers, four stores, with no byte shared
// between threads; the edges of a periodic lattice need no halo (the joint
// slot 0 holds the last and the first site).  A step is then a table entry
// (mask and distance of the pair, known from the random word alone) and four
// logic operations per plane in a chain of about 18 cycles, where two shared
// loads and two shared stores of single bytes took about 28 cycles of latency
// and 8 address instructions.
#pragma once

#include <cstdint>

#include "escg_device.cuh"

namespace escg_impl {

// PL = 1: 2 bits per site, states 0..3, every dominance edge certain.
// PL = 2: 4 bits per site, any states and edge probabilities.
//
inline int patch_planes(const LatticeDesc& d) { return d.S <= 3 && d.certain ? 1 : 2; }

// A sub-block in registers.  lo: the four corner macros, k = 0 (top row slot,
// left column slot), 1 (top, right), 2 (bottom, left), 3 (bottom, right), 8 PL
// bits each.  hi, only for sub-blocks with a 3-site side: macro 0 the top
// row slot's macro of the middle column, 1 the bottom row slot's, 2 the
// middle row's macro of the left column, 3 of the right one; the site of the
// middle row and the middle column takes the second site of macro 0, which a
// middle column's macro leaves free.
//
// Position (0..63; lo below 32) of site (r, c), r in [-1, h], c in [-1, w],
// of a w x h sub-block (sides 2 or 3), in bits of a PL = 1 patch; twice that
// in a PL = 2 patch.
__host__ __device__ inline int patch_bit(int r, int c, int w, int h) {
  const int rs = r <= 0 ? 0 : (r >= h - 1 ? 1 : 2), rh = (r == 0 || r == h) ? 1 : 0;   // slot, half; 2: middle
  const int cs = c <= 0 ? 0 : (c >= w - 1 ? 1 : 2), ch = (c == 0 || c == w) ? 1 : 0;
  if (rs < 2 && cs < 2) return 8 * (2 * rs + cs) + 4 * rh + 2 * ch;
  if (cs == 2 && rs < 2) return 32 + 8 * rs + 4 * rh;
  if (rs == 2 && cs < 2) return 48 + 8 * cs + 2 * ch;
  return 34;
}

// Row and column step of direction dir (0 up, 1 down, 2 left, 3 right, 4
// up-left, 5 up-right, 6 down-left, 7 down-right).
__host__ __device__ inline void dir_step(uint32_t dir, int* dr, int* dc) {
  *dr = (int)((0xA058u >> (2 * dir)) & 3u) - 1;
  *dc = (int)((0x8885u >> (2 * dir)) & 3u) - 1;
}

// Positions of the selected site (x) and its neighbour (y) of entry e = site *
// nbh + direction of a w x h sub-block.
__host__ __device__ inline uint2 patch_pair(int e, int w, int h, int nbh) {
  const int site = e / nbh, r = site / w, c = site - r * w;
  int dr, dc;
  dir_step((uint32_t)(e % nbh), &dr, &dc);
  uint2 v;
  v.x = (uint32_t)patch_bit(r, c, w, h);
  v.y = (uint32_t)patch_bit(r + dr, c + dc, w, h);
  return v;
}

// The tables of a launch, in shared memory.  Entries e as above; irr: shapes
// 3 x 2 from entry 0, 2 x 3 from 6 nbh, 3 x 3 from 12 nbh.
//  swap  (PL = 1) x = 3 << the higher position of the pair, y = distance
//  pair  2 x 2: the two positions; PL = 1 as rotations that bring the
//        selected site to bits 2, 3 and its neighbour to bits 4, 5
//  irr   the two positions
//  act   (PL = 1) action -> 16 fields of 4 bits: field 4 b + a (a the selected
//        site) at bits 4 (4 b + a) + 2: a ^ a' (low two bits) and b ^ b'
//        (the top field, of two equal states, is 0 and lies beyond bit 63)
//  rule  (PL = 2) 16 b + a: x = a ^ a' | (b ^ b') << 4 per action, one byte
//        each (0 exchange, 1 interaction, 2 reproduction); y = the pair's
//        interaction threshold
constexpr int kPatchMaxNbh = 8;
struct PatchTables {
  uint2 swap[4 * kPatchMaxNbh];
  uint2 pair[4 * kPatchMaxNbh];
  uint2 irr[21 * kPatchMaxNbh];
  uint2 act[3];
  uint2 rule[256];
};

__host__ __device__ inline uint2 patch_swap_entry(uint2 p) {
  const uint32_t top = p.x > p.y ? p.x : p.y, dist = p.x > p.y ? p.x - p.y : p.y - p.x;
  uint2 v;
  v.x = 3u << top;
  v.y = dist;
  return v;
}

// The XOR of pair (a, b) under action act, from the host's table.
__device__ __forceinline__ uint32_t patch_delta(const LatticeDesc& d, uint32_t a, uint32_t b, uint32_t act) {
  const uint32_t n = d.trans[(a * (uint32_t)(d.S + 1) + b) * 4u + act];
  return (a ^ (n & 15u)) | ((b ^ (n >> 4)) << 4);
}

// Entries of the rule tables.
__device__ __forceinline__ uint2 patch_act_entry(const LatticeDesc& d, uint32_t act) {
  uint64_t f = 0;
  for (int b = 0; b <= d.S; ++b)
    for (int a = 0; a <= d.S; ++a) {
      if (a == b) continue;
      const uint32_t x = patch_delta(d, (uint32_t)a, (uint32_t)b, act);
      f |= (uint64_t)((x & 3u) | (((x >> 4) & 3u) << 2)) << (4 * (4 * b + a) + 2);
    }
  return make_uint2((uint32_t)f, (uint32_t)(f >> 32));
}
__device__ __forceinline__ uint2 patch_rule_entry(const LatticeDesc& d, uint32_t a, uint32_t b) {
  uint32_t x = 0;
  for (uint32_t c = 0; c < 3u; ++c) x |= patch_delta(d, a, b, c) << (8u * c);
  return make_uint2(x, reinterpret_cast<const uint32_t*>(d.trans)[kTransPairs + a * (uint32_t)(d.S + 1) + b]);
}

// Fills the tables of the geometry, then all; threads t0, t0 + n, ... of the
// caller.
template <int PL>
__device__ __forceinline__ void patch_tables_geometry(PatchTables& T, int nbh, int t0, int n) {
  for (int e = t0; e < 4 * nbh; e += n) {
    const uint2 p = patch_pair(e, 2, 2, nbh);
    if (PL == 1) {
      T.swap[e] = patch_swap_entry(p);
      T.pair[e] = make_uint2((p.x - 2u) & 31u, (p.y - 4u) & 31u);
    } else {
      T.pair[e] = make_uint2(2u * p.x, 2u * p.y);
    }
  }
  for (int e = t0; e < 21 * nbh; e += n) {
    const uint2 p = e < 6 * nbh ? patch_pair(e, 3, 2, nbh)
                                : (e < 12 * nbh ? patch_pair(e - 6 * nbh, 2, 3, nbh) : patch_pair(e - 12 * nbh, 3, 3, nbh));
    T.irr[e] = make_uint2((uint32_t)PL * p.x, (uint32_t)PL * p.y);
  }
}
template <int PL>
__device__ __forceinline__ void patch_tables_fill(PatchTables& T, const LatticeDesc& d, int t0, int n) {
  patch_tables_geometry<PL>(T, d.nbh == 8 ? 8 : 4, t0, n);
  const int S1 = d.S + 1;
  if (PL == 1) {
    for (int k = t0; k < 3; k += n) T.act[k] = patch_act_entry(d, (uint32_t)k);
  } else {
    for (int k = t0; k < S1 * S1; k += n) {
      const uint32_t a = (uint32_t)(k % S1), b = (uint32_t)(k / S1);
      T.rule[16u * b + a] = patch_rule_entry(d, a, b);
    }
  }
}

// Mirrors entry e of a w-wide, h-high sub-block whose sides `edge` (1 top,
// 2 bottom, 4 left, 8 right) are edges of a reflecting lattice: a step that
// would leave the lattice goes the other way in that coordinate.
__host__ __device__ constexpr uint32_t patch_mirror(uint32_t e, int w, int h, int lg, uint32_t edge) {
  const uint32_t dir = e & ((1u << lg) - 1u), site = e >> lg;
  const int r = (int)(site / (uint32_t)w), c = (int)site - r * w;
  int dr = (int)((0xA058u >> (2 * dir)) & 3u) - 1, dc = (int)((0x8885u >> (2 * dir)) & 3u) - 1;   // dir_step
  if (((edge & 1u) && r == 0 && dr < 0) || ((edge & 2u) && r == h - 1 && dr > 0)) dr = -dr;
  if (((edge & 4u) && c == 0 && dc < 0) || ((edge & 8u) && c == w - 1 && dc > 0)) dc = -dc;
  // directions by 3 (dr + 1) + dc + 1: 4 0 5 2 . 3 6 1 7
  const uint32_t nd = (uint32_t)(0x716302504ull >> (4 * (3 * (dr + 1) + dc + 1))) & 15u;
  return (site << lg) | nd;
}

// The same for every entry and edge, by neighbourhood: 2 x 2 from entry 0, then
// the shapes of PatchTables::irr.  A mirrored step is one load here (6 KB, in
// the L1 of every SM that runs such a lattice); worked out step by step, with a
// division by w, it took longer than the step itself.  us per MCS of reflecting
// lattices, byte kernels, worked out, table: L = 100 34.6, 31.0, 12.3; 150 (S = 5)
// 39.5, 49.2, 33.0; 191 39.5, 41.4, 29.7; 3200 26.9, 25.3, 23.0, (S = 5) 27.1, 28.2,
// 26.2.
struct MirrorTable {
  uint8_t e[2][16][25 * kPatchMaxNbh];
};
constexpr MirrorTable make_mirror_table() {
  MirrorTable t{};
  constexpr int kShape[4][3] = {{0, 2, 2}, {4, 3, 2}, {10, 2, 3}, {16, 3, 3}};   // first site, width, height
  for (int lg = 2; lg <= 3; ++lg)
    for (uint32_t edge = 0; edge < 16u; ++edge)
      for (int k = 0; k < 4; ++k)
        for (int e = 0; e < (kShape[k][1] * kShape[k][2]) << lg; ++e)
          t.e[lg - 2][edge][(kShape[k][0] << lg) + e] =
              (uint8_t)patch_mirror((uint32_t)e, kShape[k][1], kShape[k][2], lg, edge);
  return t;
}
static __device__ const MirrorTable g_mirror = make_mirror_table();

// The four attempts of a 2 x 2 sub-block as the tables give them from the
// random words alone: L the pair's entry (swap if `general` is false, else
// pair).  PL = 1: A the action's fields; PL = 2: A.x = 8 * action, A.y the
// action draw.  Almost every attempt of a large lattice with movement is an
// exchange (epsilon = 2 M N), so four exchanges take a path of their own:
// four logic operations a step instead of ten.  (A choice per step was
// slower: its branches cost more than the steps they shorten.)
template <int PL>
struct Steps2 {
  uint2 L[4], A[4];
  bool general;
};

// LG: log2 of the neighbourhood.
template <int PL, int LG, bool REFLECT>
__device__ __forceinline__ Steps2<PL> patch_steps2(uint4 x, const PatchTables& T, uint32_t tx, uint32_t txi,
                                                   uint32_t edge) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
  uint32_t e[4], u[4];
  Steps2<PL> s;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    e[t] = w[t] >> (30 - LG);
    if (REFLECT && edge) e[t] = g_mirror.e[LG - 2][edge][e[t]];
    u[t] = w[t] << (2 + LG);
  }
  // one choice for the lanes that come here together: a mixed warp would
  // step through both paths (any split of the warp gives the same states)
  s.general = __any_sync(__activemask(), max(max(u[0], u[1]), max(u[2], u[3])) >= tx);
  if (!s.general) {
#pragma unroll
    for (int t = 0; t < 4; ++t) s.L[t] = PL == 1 ? T.swap[e[t]] : T.pair[e[t]];
  } else {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      s.L[t] = T.pair[e[t]];
      const uint32_t act = u[t] < tx ? 0u : (u[t] < txi ? 1u : 2u);
      s.A[t] = PL == 1 ? T.act[act] : make_uint2(8u * act, u[t]);
    }
  }
  return s;
}

// The XOR of the pair (a, b) of a PL = 2 step.
__device__ __forceinline__ uint32_t patch_rule(const uint2* __restrict__ rule, uint32_t a, uint32_t b, uint2 A) {
  const uint2 e = rule[16u * b + a];
  return (A.x == 8u && A.y >= e.y) ? 0u : e.x >> A.x;
}

template <int PL>
__device__ __forceinline__ void patch_run2(uint32_t (&v)[PL], const Steps2<PL>& s, const PatchTables& T) {
  if (PL == 1) {
    if (!s.general) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const uint32_t z = (v[0] ^ __funnelshift_l(0u, v[0], s.L[t].y)) & s.L[t].x;
        v[0] ^= z ^ __funnelshift_r(z, 0u, s.L[t].y);
      }
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const uint32_t a = __funnelshift_r(v[0], v[0], s.L[t].x), b = __funnelshift_r(v[0], v[0], s.L[t].y);
        const uint32_t f = ((a & 0xCu) | (b & 0xFFFFFFF3u)) & 0x3Cu;
        const uint32_t x = (uint32_t)((((uint64_t)s.A[t].y << 32) | s.A[t].x) >> f);
        const uint32_t da = x & 0xCu, db = x & 0x30u;
        v[0] ^= __funnelshift_l(da, da, s.L[t].x) ^ __funnelshift_l(db, db, s.L[t].y);
      }
    }
  } else {
    uint64_t V = ((uint64_t)v[PL - 1] << 32) | v[0];
    if (!s.general) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const uint64_t x = (uint64_t)(((uint32_t)(V >> s.L[t].x) ^ (uint32_t)(V >> s.L[t].y)) & 15u);
        V ^= (x << s.L[t].x) ^ (x << s.L[t].y);
      }
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const uint32_t a = (uint32_t)(V >> s.L[t].x) & 15u, b = (uint32_t)(V >> s.L[t].y) & 15u;
        const uint32_t x = patch_rule(T.rule, a, b, s.A[t]);
        V ^= ((uint64_t)(x & 15u) << s.L[t].x) ^ ((uint64_t)((x >> 4) & 15u) << s.L[t].y);
      }
    }
    v[0] = (uint32_t)V;
    v[PL - 1] = (uint32_t)(V >> 32);
  }
}

// One attempt (entry e, action draw u) of a sub-block with a 3-site side; lut the
// shape's entries.  V, W: its bits (PL = 1: V alone).
template <int PL>
__device__ __forceinline__ void patch_attempt(uint64_t& V, uint64_t& W, uint32_t e, uint32_t u,
                                              const uint2* __restrict__ lut, const PatchTables& T, uint32_t tx,
                                              uint32_t txi) {
  const uint2 L = lut[e];
  const uint32_t act = u < tx ? 0u : (u < txi ? 1u : 2u);
  if (PL == 1) {
    const uint2 A = T.act[act];
    const uint32_t a = (uint32_t)(V >> L.x) & 3u, b = (uint32_t)(V >> L.y) & 3u;
    const uint32_t x = (uint32_t)((((uint64_t)A.y << 32) | A.x) >> (4u * a + 16u * b));
    V ^= ((uint64_t)((x >> 2) & 3u) << L.x) ^ ((uint64_t)((x >> 4) & 3u) << L.y);
  } else {
    const bool ha = L.x >= 64u, hb = L.y >= 64u;
    const uint32_t sa = L.x & 63u, sb = L.y & 63u;
    const uint32_t a = (uint32_t)((ha ? W : V) >> sa) & 15u, b = (uint32_t)((hb ? W : V) >> sb) & 15u;
    const uint32_t x = patch_rule(T.rule, a, b, make_uint2(8u * act, u));
    const uint64_t fa = (uint64_t)(x & 15u) << sa, fb = (uint64_t)((x >> 4) & 15u) << sb;
    V ^= (ha ? 0ull : fa) ^ (hb ? 0ull : fb);
    W ^= (ha ? fa : 0ull) ^ (hb ? fb : 0ull);
  }
}

// Where a sub-block's macros are: i00 the index of the top left one, dc and
// dr the index distances of the right column slot and the bottom row slot
// (negative across the periodic wrap); a middle column or row slot follows
// the left or top one (distance 1 or the row pitch).
template <int PL>
struct MacroOf;
template <>
struct MacroOf<1> {
  typedef uint8_t type;
};
template <>
struct MacroOf<2> {
  typedef uint16_t type;
};

template <int PL>
__device__ __forceinline__ void patch_load2(const typename MacroOf<PL>::type* __restrict__ M, int i00, int dc, int dr,
                                            uint32_t (&v)[PL]) {
  const uint32_t a = M[i00], b = M[i00 + dc], c = M[i00 + dr], e = M[i00 + dr + dc];
  if (PL == 1) {
    v[0] = __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, e, 0x0040), 0x5410);
  } else {
    v[0] = __byte_perm(a, b, 0x5410);
    v[PL - 1] = __byte_perm(c, e, 0x5410);
  }
}

template <int PL>
__device__ __forceinline__ void patch_store2(typename MacroOf<PL>::type* __restrict__ M, int i00, int dc, int dr,
                                             const uint32_t (&v)[PL]) {
  typedef typename MacroOf<PL>::type MT;
  if (PL == 1) {
    M[i00] = (MT)v[0];
    M[i00 + dc] = (MT)(v[0] >> 8);
    M[i00 + dr] = (MT)(v[0] >> 16);
    M[i00 + dr + dc] = (MT)(v[0] >> 24);
  } else {
    M[i00] = (MT)v[0];
    M[i00 + dc] = (MT)(v[0] >> 16);
    M[i00 + dr] = (MT)v[PL - 1];
    M[i00 + dr + dc] = (MT)(v[PL - 1] >> 16);
  }
}

// Entries of a sub-block with a 3-site side: nbh times its sites, and the first
// of its shape in PatchTables::irr.
template <int LG>
__device__ __forceinline__ uint32_t patch_entries(bool wc, bool wr) {
  return (uint32_t)((wc ? 3 : 2) * (wr ? 3 : 2)) << LG;
}
template <int LG>
__device__ __forceinline__ uint32_t patch_first(bool wc, bool wr) {
  return !wr ? 0u : (!wc ? 6u << LG : 12u << LG);
}

// All attempts (words w[0 .. 5] or w[0 .. 8]) of a sub-block with a 3-site
// side (wc: 3 wide, wr: 3 high), from and to its macros.  REFLECT: their entries
// are the bytes of ent, else the words give them.
template <int PL, int LG, bool REFLECT>
__device__ __forceinline__ void patch_irregular(typename MacroOf<PL>::type* __restrict__ M, int i00, int dc, int dr,
                                                int pitch, bool wc, bool wr, const uint32_t (&w)[9],
                                                const uint32_t (&ent)[3], const PatchTables& T, uint32_t tx,
                                                uint32_t txi) {
  typedef typename MacroOf<PL>::type MT;
  constexpr int kB = 8 * PL;                          // bits of a macro
  constexpr uint32_t kMid = PL == 1 ? 0x33u : 0x0F0Fu;   // sites of a middle column's macro
  uint32_t lo[PL], m0 = 0, m1 = 0, m2 = 0, m3 = 0, m4 = 0;
  patch_load2<PL>(M, i00, dc, dr, lo);
  if (wc) {
    m0 = M[i00 + 1];
    m1 = M[i00 + dr + 1];
  }
  if (wr) {
    m2 = M[i00 + pitch];
    m3 = M[i00 + pitch + dc];
  }
  if (wc && wr) m4 = M[i00 + pitch + 1];
  m0 |= m4 << (kB / 4);
  uint64_t V, W = 0;
  if (PL == 1) {
    V = ((uint64_t)(m0 | (m1 << 8) | (m2 << 16) | (m3 << 24)) << 32) | lo[0];
  } else {
    V = ((uint64_t)lo[PL - 1] << 32) | lo[0];
    W = ((uint64_t)(m2 | (m3 << 16)) << 32) | (m0 | (m1 << 16));
  }
  const uint32_t n = patch_entries<LG>(wc, wr);
  const uint2* lut = T.irr + patch_first<LG>(wc, wr);
#pragma unroll
  for (int t = 0; t < 9; ++t) {
    if (t >= 6 && !(wc && wr)) break;
    const uint32_t e = REFLECT ? (ent[t >> 2] >> (8 * (t & 3))) & 255u : __umulhi(w[t], n);
    patch_attempt<PL>(V, W, e, w[t] * n, lut, T, tx, txi);
  }
  lo[0] = (uint32_t)V;
  if (PL == 2) lo[PL - 1] = (uint32_t)(V >> 32);
  patch_store2<PL>(M, i00, dc, dr, lo);
  const uint64_t H = PL == 1 ? V >> 32 : W;
  if (wc) {
    M[i00 + 1] = (MT)((uint32_t)H & kMid);
    M[i00 + dr + 1] = (MT)(H >> kB);
  }
  if (wr) {
    M[i00 + pitch] = (MT)(H >> (2 * kB));
    M[i00 + pitch + dc] = (MT)(H >> (3 * kB));
  }
  if (wc && wr) M[i00 + pitch + 1] = (MT)((uint32_t)(H >> (kB / 4)) & (PL == 1 ? 3u : 15u));
}

// The part of the Philox call of attempts 0..3 (counter (0, g, m, STEP)) that
// does not depend on the sub-block g: of the call's twenty wide multiplies
// four have operands fixed by m and the key, so a thread takes them once per
// MCS and a draw costs sixteen.
struct StepKeys {
  uint32_t x1;   // round 1: first word = x1 ^ g
  uint32_t x3;   // round 3: first word = hi(M1 z) ^ x3
  uint32_t z3, w3;
};

template <class RK>
__host__ __device__ __forceinline__ StepKeys step_keys(uint32_t m, RK rk) {
  const uint64_t p1 = (uint64_t)0xCD9E8D57u * m;
  const uint64_t q1 = (uint64_t)0xCD9E8D57u * (kTagStep ^ rk[1]);          // round 2, third word of round 1
  const uint32_t x2 = (uint32_t)(q1 >> 32) ^ (uint32_t)p1 ^ rk[2];         // round 2, first word
  const uint64_t q0 = (uint64_t)0xD2511F53u * x2;                          // round 3
  StepKeys k;
  k.x1 = (uint32_t)(p1 >> 32) ^ rk[0];
  k.x3 = (uint32_t)q1 ^ rk[4];
  k.z3 = (uint32_t)(q0 >> 32) ^ rk[5];
  k.w3 = (uint32_t)q0;
  return k;
}

// philox10_rk((0, g, m, STEP)) from the keys of MCS m.
template <class RK>
__host__ __device__ __forceinline__ uint4 philox_step(const StepKeys& k, uint32_t g, RK rk) {
  const uint64_t p0 = (uint64_t)0xD2511F53u * (k.x1 ^ g);                  // round 2
  const uint64_t p1 = (uint64_t)0xCD9E8D57u * ((uint32_t)(p0 >> 32) ^ rk[3]);   // round 3
  uint4 c = make_uint4((uint32_t)(p1 >> 32) ^ k.x3, (uint32_t)p1, k.z3 ^ (uint32_t)p0, k.w3);
#pragma unroll
  for (int r = 3; r < 10; ++r) {
    const uint64_t a = (uint64_t)0xD2511F53u * c.x;
    const uint64_t b = (uint64_t)0xCD9E8D57u * c.z;
    c = make_uint4((uint32_t)(b >> 32) ^ c.y ^ rk[2 * r], (uint32_t)b, (uint32_t)(a >> 32) ^ c.w ^ rk[2 * r + 1],
                   (uint32_t)a);
  }
  return c;
}

// One sub-block of a fine phase with what is known of it before the phase:
// for a 2 x 2 one its steps, for one with a 3-site side its random words, in
// the same registers (word t in s.L[t / 2], the last one in i8; with a
// reflecting boundary the entries in s.A).
template <int PL>
struct PatchItem {
  Steps2<PL> s;
  uint32_t i8;
  int i00, dc, dr;
  uint32_t fl;   // 1 present, 2 three wide, 4 three high, edge flags << 4
};

// The random words of sub-block g in MCS m and, for a 2 x 2 one, its steps;
// fl and the macro indexes are set.
// WIDE = false: every sub-block is 2 x 2.
template <int PL, int LG, bool REFLECT, bool WIDE = true, class RK>
__device__ __forceinline__ void patch_item_draw(PatchItem<PL>& I, const StepKeys& key, uint32_t g, uint32_t m,
                                                RK rk, const PatchTables& T, uint32_t tx, uint32_t txi) {
  if (!WIDE || !(I.fl & 6u)) {
    I.s = patch_steps2<PL, LG, REFLECT>(philox_step(key, g, rk), T, tx, txi, REFLECT ? I.fl >> 4 : 0u);
  } else {
    // the three calls side by side, also where a 2 x 3 sub-block needs two:
    // the phase waits for the 3 x 3 one
    uint4 x = make_uint4(0u, g, m, kTagStep), y = x, z = x;
    y.x = 1u;
    z.x = 2u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
      x = philox_round(x, rk[2 * r], rk[2 * r + 1]);
      y = philox_round(y, rk[2 * r], rk[2 * r + 1]);
      z = philox_round(z, rk[2 * r], rk[2 * r + 1]);
    }
    I.s.L[0] = make_uint2(x.x, x.y);
    I.s.L[1] = make_uint2(x.z, x.w);
    I.s.L[2] = make_uint2(y.x, y.y);
    I.s.L[3] = make_uint2(y.z, y.w);
    I.i8 = z.x;
    if (REFLECT) {
      // the entries now: a mirrored one must not wait in the chain of the steps
      const bool wc = (I.fl & 2u) != 0u, wr = (I.fl & 4u) != 0u;
      const uint32_t n = patch_entries<LG>(wc, wr), edge = I.fl >> 4;
      const uint32_t w[9] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w, z.x};
      const uint8_t* mir = g_mirror.e[LG - 2][edge] + (4u << LG) + patch_first<LG>(wc, wr);
      uint32_t ent[3] = {0u, 0u, 0u};
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        uint32_t e = __umulhi(w[t], n);
        if (edge) e = mir[e];
        ent[t >> 2] |= e << (8 * (t & 3));
      }
      I.s.A[0] = make_uint2(ent[0], ent[1]);
      I.s.A[1].x = ent[2];
    }
  }
}

// All its attempts, from and to its macros.
template <int PL, int LG, bool REFLECT, bool WIDE = true>
__device__ __forceinline__ void patch_item_run(typename MacroOf<PL>::type* __restrict__ M, int pitch,
                                               const PatchItem<PL>& I, const PatchTables& T, uint32_t tx,
                                               uint32_t txi) {
  if (!WIDE || !(I.fl & 6u)) {
    uint32_t v[PL];
    patch_load2<PL>(M, I.i00, I.dc, I.dr, v);
    patch_run2<PL>(v, I.s, T);
    patch_store2<PL>(M, I.i00, I.dc, I.dr, v);
  } else {
    const uint32_t w[9] = {I.s.L[0].x, I.s.L[0].y, I.s.L[1].x, I.s.L[1].y, I.s.L[2].x, I.s.L[2].y, I.s.L[3].x,
                           I.s.L[3].y, I.i8};
    const uint32_t ent[3] = {I.s.A[0].x, I.s.A[0].y, I.s.A[1].x};
    patch_irregular<PL, LG, REFLECT>(M, I.i00, I.dc, I.dr, pitch, (I.fl & 2u) != 0u, (I.fl & 4u) != 0u, w, ent, T, tx,
                                     txi);
  }
}

// ---------------------------------------------------------------------------
// One axis of a partition by slots (segments of 2 or 3 sites).
__host__ __device__ inline bool slot_axis_ok(const AxisGeom& g) {
  // all segments 2 or 3 sites wide
  const bool a = g.r == 0 || (g.Qa > 0 && g.fqa >= 2 && g.fqa + (g.fra > 0 ? 1 : 0) <= 3);
  const bool b = g.Qb > 0 && g.fqb >= 2 && g.fqb + (g.frb > 0 ? 1 : 0) <= 3;
  return a && b;
}
// 3-site segments of a wide (a) or narrow block.
__host__ __device__ inline int block_wide(const AxisGeom& g, bool a) {
  return a ? (g.fqa == 3 ? g.Qa : g.fra) : (g.fqb == 3 ? g.Qb : g.frb);
}
// Slots of a whole periodic axis: segments plus middle slots.
__host__ __device__ inline int axis_slots(const AxisGeom& g, int P) {
  return g.r * (g.Qa + block_wide(g, true)) + (P - g.r) * (g.Qb + block_wide(g, false));
}

// Segment k of the whole axis: its left joint slot, whether it is 3 wide and
// its first site.
__host__ __device__ inline void axis_segment(const AxisGeom& g, int k, int& slot, bool& wide, int& first) {
  const int ka = g.r * g.Qa;
  const bool a = k < ka;
  const int b = a ? k / g.Qa : g.r + (k - ka) / g.Qb;
  const int j = a ? k - b * g.Qa : k - ka - (b - g.r) * g.Qb;
  const int fq = a ? g.fqa : g.fqb, fr = a ? g.fra : g.frb;
  const int na = b < g.r ? b : g.r;
  const int before = na * block_wide(g, true) + (b - na) * block_wide(g, false) + (fq == 3 ? j : (j < fr ? j : fr));
  wide = fq == 3 || j < fr;
  slot = k + before;
  first = b * g.q + na + j * fq + (j < fr ? j : fr);
}

// Quads (pairs of segments) of the blocks of one parity along an axis: the
// regular ones (both segments 2 wide) first.  total, regular.
__host__ __device__ inline void axis_quads(const AxisGeom& g, int P, int par, int* total, int* regular) {
  const int nblk = (P - par + 1) / 2, na0 = (g.r - par + 1) / 2, na = na0 < 0 ? 0 : (na0 < nblk ? na0 : nblk);
  const int wa = block_wide(g, true), wb = block_wide(g, false);
  const int ha = g.Qa >> 1, hb = g.Qb >> 1, ia = (wa + 1) >> 1, ib = (wb + 1) >> 1;
  *total = na * ha + (nblk - na) * hb;
  *regular = na * (ha - ia) + (nblk - na) * (hb - ib);
}

// Quad k2 (0 .. G/2 - 1) of the axis: its block, first segment and position
// in the order of its block's parity.
__host__ __device__ inline void axis_quad(const AxisGeom& g, int P, int k2, int& b, int& seg, int& pos) {
  const int ha = g.Qa >> 1, hb = g.Qb >> 1, ka = g.r * ha;
  const bool a = k2 < ka;
  b = a ? k2 / ha : g.r + (k2 - ka) / hb;
  const int q = a ? k2 - b * ha : k2 - ka - (b - g.r) * hb;
  seg = 2 * k2;
  const int par = b & 1, i = b >> 1;
  const int na0 = (g.r - par + 1) / 2, na1 = na0 < 0 ? 0 : na0, na = i < na1 ? i : na1;
  const int ia = (block_wide(g, true) + 1) >> 1, ib = (block_wide(g, false) + 1) >> 1;
  int total, regular;
  axis_quads(g, P, par, &total, &regular);
  const int irr = a ? ia : ib;
  pos = q >= irr ? na * (ha - ia) + (i - na) * (hb - ib) + (q - irr) : regular + na * ia + (i - na) * ib + q;
}

// First joint slot of block b of an axis, and its slots up to the next block's.
__host__ __device__ inline int block_slot(const AxisGeom& g, int b) {
  const int na = b < g.r ? b : g.r;
  return na * (g.Qa + block_wide(g, true)) + (b - na) * (g.Qb + block_wide(g, false));
}
__host__ __device__ inline int block_slots(const AxisGeom& g, int b) {
  return b < g.r ? g.Qa + block_wide(g, true) : g.Qb + block_wide(g, false);
}

// Quad i of a block of hx x hy quads with frx and fry leading segments of 3
// sites, those of 2 x 2 sub-blocks only first (so that warps are of one kind),
// then the leading rows, then the leading columns: its top left macro (base
// added; 16 bits) | qx << 16 | qy << 22 (6 bits each) | 3-site segments (2 qx, 2 qx + 1
// at bits 28, 29; 2 qy, 2 qy + 1 at bits 30, 31).
__device__ __forceinline__ uint32_t quad_entry(int i, int hx, int hy, int frx, int fry, int pitch, int base) {
  const int ix = (frx + 1) >> 1, iy = (fry + 1) >> 1, rx = hx - ix, nreg = rx * (hy - iy), top = hx * iy;
  int qx, qy;
  if (i < nreg) {
    qy = i / rx;
    qx = i - qy * rx + ix;
    qy += iy;
  } else if (i < nreg + top) {
    qy = (i - nreg) / hx;
    qx = i - nreg - qy * hx;
  } else {
    qy = (i - nreg - top) / ix;
    qx = i - nreg - top - qy * ix;
    qy += iy;
  }
  const int fx = 2 * qx, fy = 2 * qy;
  const uint32_t wide = (fx < frx ? 1u : 0u) | (fx + 1 < frx ? 2u : 0u) | (fy < fry ? 4u : 0u) | (fy + 1 < fry ? 8u : 0u);
  return (uint32_t)(base + (fy + min(fy, fry)) * pitch + fx + min(fx, frx)) | ((uint32_t)qx << 16) | ((uint32_t)qy << 22) |
         (wide << 28);
}

}  // namespace escg_impl
