// escg_group.cu -- block owners on macros: partitions with fine segments of 2 or
// 3 sites, both neighbourhoods, any number of species, any bits per site (see
// group_fn for which of them it runs).
//
// CTA g owns coarse group g -- the 2 x 2 blocks (2 gx + cx, 2 gy + cy), one of
// each colour -- for a whole cooperative launch and keeps their macros
// (escg_patch.cuh) in shared memory as one array: the joint slots between
// its own blocks need no exchange, and each block has one vertical and one
// horizontal joint line that it shares with another group.  A visit
//  1. waits for what it reads of other groups: the macros of those two lines
//     and of their three end points, each from its latest writer and only
//     where that is not the group itself;
//  2. runs the four fine phases (escg_patch.cuh: sub-blocks in registers);
//  3. publishes its two lines.
// A line travels as 64-bit words, 4 macro bytes and the epoch (MCS + 1) of the
// visit that wrote them, each read and written with one single-copy-atomic
// access: the data is its own flag.  Every macro of the lattice is written back
// by the last visitor of the blocks that share it, so the end of a launch
// needs no exchange.
//
// Why no record is overwritten before it is read: a block's next visit
// depends on every visit of the blocks it shares macros with that came
// before it, either because it reads that visit's line (edge neighbours) or
// because it waits for a later visit of a block next to both (diagonals).
//
// What bounds a visit is a chain: the record round trip through L2, then four
// fine phases, each four macro loads, the steps of its longest sub-block
// and a barrier.  Random words, table entries and addresses depend on the
// schedule only, so 2 or 4 groups of threads take the fine phases in turn
// where an SM holds one or two CTAs and prepare their next sub-block while
// the others run (escg_resident_patch.cuh), and one warp does all of the
// exchange.
#include "escg_internal.h"
#include "escg_patch.cuh"
#include "escg_sync.cuh"

namespace escg_impl {

constexpr int kLineWords = 32;    // record words per line: 45 macros of 2 bytes at most (80-site blocks) or, in a
                                  // lattice of 2 blocks, 51 (96 sites)
static_assert(kGroupRecordWords == 2 * kLineWords, "record layout: the vertical line's words, then the horizontal's");
constexpr int kGroupWords = 2 * 26 + 3;   // record words a visit reads, at most

// One of the group's four blocks.
struct GroupBlock {
  int32_t id, bx, by;
  int32_t base;          // its top left macro in the tile array
  int32_t ncx, ncy;      // joint slots 0 .. ncx, 0 .. ncy (middle slots among them)
  int32_t frx, fry;      // leading segments of 3 sites
  int32_t f0x, f0y;      // first fine segment of each axis
  int32_t hx, hy, nq;    // quads: pairs of segments of each axis, all
  int32_t nw;            // record words of a visit
};

// A record word of a visit: where it is read, where this block publishes
// its own of the same macros (lines only), and the macros.
enum : uint32_t { kVLine = 0, kHLine = 1, kCorner = 2 };
struct GroupWord {
  uint32_t src, own;
  uint16_t dst, stride;   // first macro in the tile array and the step to the next
  uint8_t n, kind;
  uint8_t sub;            // position of the (single) macro in the word read
  uint8_t ends;           // 1: the first, 2: the last macro is an end of the line
};

template <int PL>
struct GroupSmem {
  PatchTables T;
  GroupBlock b[4];
  GroupWord w[4][kGroupWords];
  uint32_t fo[2][4];   // by MCS parity: fine orders of the blocks by colour,
  StepKeys key[2];     // the step keys
  uint32_t hist[kMaxStates];
  uint32_t quit;
};

// Threads of a CTA of ng groups, at most: with 3-site segments a thread needs the
// registers that two groups leave it, without them four groups fit.
__host__ __device__ constexpr int group_max_threads(int ng) { return ng == 1 ? 288 : (ng == 2 ? 640 : 1024); }

struct GroupArgs {
  PersistentArgs p;
  int32_t gs, pitch, gpitch, nsx, nsy, gqy;
  int32_t quads, nq_max;   // byte offset of the quad tables in shared memory, entries of each
};

__device__ __forceinline__ void group_block(const LatticeDesc& d, int gx, int gy, int c, int pitch, GroupBlock& B) {
  const int cx = c & 1, cy = c >> 1, bx = 2 * gx + cx, by = 2 * gy + cy;
  const BlockSpan X = block_span(d.ax, bx), Y = block_span(d.ay, by);
  B.id = by * d.P + bx;
  B.bx = bx;
  B.by = by;
  B.ncx = block_slots(d.ax, bx);
  B.ncy = block_slots(d.ay, by);
  B.base = (cy ? block_slots(d.ay, by - 1) : 0) * pitch + (cx ? block_slots(d.ax, bx - 1) : 0);
  B.frx = B.ncx - X.Q;
  B.fry = B.ncy - Y.Q;
  B.f0x = X.f0;
  B.f0y = Y.f0;
  B.hx = X.Q >> 1;
  B.hy = Y.Q >> 1;
  B.nq = B.hx * B.hy;
}

__device__ __forceinline__ uint32_t group_quad(const GroupBlock& B, int pitch, int i) {
  return quad_entry(i, B.hx, B.hy, B.frx, B.fry, pitch, B.base);
}

// Record word i of block c; false if there is none.
template <int PL>
__device__ __forceinline__ bool group_word(const LatticeDesc& d, const GroupBlock& B, int pitch, int i, GroupWord& W) {
  constexpr int kPer = 4 / PL;   // macros per word
  const int P = d.P, Py = d.Py, bx = B.bx, by = B.by, cx = bx & 1, cy = by & 1;
  const int xo = cx ? (bx == P - 1 ? 0 : bx + 1) : (bx == 0 ? P - 1 : bx - 1);     // the other groups' blocks beside
  const int yo = cy ? (by == Py - 1 ? 0 : by + 1) : (by == 0 ? Py - 1 : by - 1);   // and above or below
  const int wv = B.ncx / kPer + 1, wh = B.ncy / kPer + 1;
  const int row = B.base + (cy ? B.ncy * pitch : 0), col = B.base + (cx ? B.ncx : 0);   // the lines' first macros
  W.ends = 0;
  W.sub = 0;
  W.own = 0;
  W.stride = 0;
  W.n = 1;
  if (i < wv) {
    W.kind = kVLine;
    W.src = (uint32_t)((yo * P + bx) * kGroupRecordWords + i);
    W.own = (uint32_t)(B.id * kGroupRecordWords + i);
    W.dst = (uint16_t)(row + i * kPer);
    W.stride = 1;
    W.n = (uint8_t)min(kPer, B.ncx + 1 - i * kPer);
    W.ends = (uint8_t)((i == 0 ? 1 : 0) | (i == wv - 1 ? 2 : 0));
    return true;
  }
  i -= wv;
  if (i < wh) {
    W.kind = kHLine;
    W.src = (uint32_t)((by * P + xo) * kGroupRecordWords + kLineWords + i);
    W.own = (uint32_t)(B.id * kGroupRecordWords + kLineWords + i);
    W.dst = (uint16_t)(col + i * kPer * pitch);
    W.stride = (uint16_t)pitch;
    W.n = (uint8_t)min(kPer, B.ncy + 1 - i * kPer);
    W.ends = (uint8_t)((i == 0 ? 1 : 0) | (i == wh - 1 ? 2 : 0));
    return true;
  }
  i -= wh;
  if (i >= 3) return false;
  // the diagonal blocks' macros at the lines' end points: 0 where both lines
  // meet, 1 the vertical line's other end, 2 the horizontal line's
  int e, id, line = 0;
  if (i == 0) {
    id = yo * P + xo;
    e = cx ? 0 : block_slots(d.ax, xo);
    W.dst = (uint16_t)(row + (cx ? B.ncx : 0));
  } else if (i == 1) {
    id = yo * P + (bx ^ 1);
    e = cx ? block_slots(d.ax, bx ^ 1) : 0;
    W.dst = (uint16_t)(row + (cx ? 0 : B.ncx));
  } else {
    id = (by ^ 1) * P + xo;
    e = cy ? block_slots(d.ay, by ^ 1) : 0;
    W.dst = (uint16_t)(col + (cy ? 0 : B.ncy * pitch));
    line = kLineWords;
  }
  W.kind = kCorner;
  W.src = (uint32_t)(id * kGroupRecordWords + line + e / kPer);
  W.sub = (uint8_t)(e % kPer);
  return true;
}

// Counts of a block's visit, slot k against its vertical, horizontal and
// diagonal neighbours': a macro is counted by the last visit of the blocks
// that share it, the non-empty states only.  Threads t of nt (whole warps).
// Out of line, as is the log entry: their registers must not count against
// the visit's 64.
template <int PL>
__device__ __noinline__ void group_count(const typename MacroOf<PL>::type* M, int pitch, const GroupBlock& B, int S,
                                            int k, int sV, int sH, int sD, uint32_t* hist, int t, int nt) {
  constexpr int kPer = 4 / PL;
  constexpr uint32_t kMacro = PL == 1 ? 0xFFu : 0xFFFFu;
  const uint32_t* W = reinterpret_cast<const uint32_t*>(M);
  const int r0 = B.base / pitch, c0 = B.base - r0 * pitch, w0 = c0 / kPer, used = (c0 + B.ncx) / kPer - w0 + 1;
  uint32_t cnt[kMaxStates];
#pragma unroll
  for (int v = 0; v < kMaxStates; ++v) cnt[v] = 0;
  for (int i = t; i < (B.ncy + 1) * used; i += nt) {
    const int r = i / used, w = w0 + i - r * used;
    uint32_t x = W[(r0 + r) * (pitch / kPer) + w], mask = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int col = kPer * w + j - c0;
      const bool lr = r == 0 || r == B.ncy, lc = col == 0 || col == B.ncx;
      const bool mine = col >= 0 && col <= B.ncx && (!lr || sV < k) && (!lc || sH < k) && (!(lr && lc) || sD < k);
      if (mine) mask |= kMacro << (8 * PL * j);
    }
    x &= mask;
#pragma unroll
    for (int v = 1; v < (PL == 1 ? 4 : kMaxStates); ++v) {
      if (v > S) break;
      if (PL == 1) {
        const uint32_t z = x ^ (uint32_t)(v * 0x55555555u);
        cnt[v] += __popc(~(z | (z >> 1)) & 0x55555555u);
      } else {
        const uint32_t z = x ^ (uint32_t)(v * 0x11111111u), n = z | (z >> 1);
        cnt[v] += __popc(~(n | (n >> 2)) & 0x11111111u);
      }
    }
  }
#pragma unroll
  for (int v = 1; v < (PL == 1 ? 4 : kMaxStates); ++v) {
    if (v > S) break;
    const uint32_t s = __reduce_add_sync(0xFFFFFFFFu, cnt[v]);
    if ((t & 31) == 0 && s) atomicAdd(&hist[v], s);
  }
}

// Adds a visit's counts (hist, zeroed for the next) to the open log point of
// MCS m_end; the last of the nb blocks writes the entry, the empty sites being
// the rest of the n.  One warp.
static __device__ __noinline__ void group_log(RunState* st, LogBuffers lb, int S, uint32_t m_end, uint32_t log_every,
                                              int stop_at_extinction, uint32_t nb, uint32_t* hist,
                                              unsigned long long n) {
  const int lane = threadIdx.x & 31;
  const uint32_t ring = (m_end / log_every) % (uint32_t)kPendRing;
  if (lane >= 1 && lane <= S && hist[lane]) {
    atomicAdd(&st->acc[ring][lane], (unsigned long long)hist[lane]);
    hist[lane] = 0;
  }
  __syncwarp();
  if (lane == 0) {
    __threadfence();
    if (atomicAdd(&st->pend[ring], 1u) == nb - 1u) {
      __threadfence();   // every contribution is in acc
      unsigned long long c[kMaxStates];
      for (int s = 1; s < kMaxStates; ++s) {
        c[s] = atomicExch(&st->acc[ring][s], 0ull);
        n -= c[s];
      }
      c[0] = n;
      st->pend[ring] = 0;
      write_log_entry(st, lb, S, m_end, log_every, c, stop_at_extinction);
    }
  }
  __syncwarp();
}

// Item `it` (a quad) of fine phase fi of the visit of the group's block c in
// MCS m: its sub-block of that phase's colour.
template <int PL, int LG, bool REFLECT, bool WIDE>
__device__ __forceinline__ PatchItem<PL> group_prepare(const GroupArgs& ga, const GroupSmem<PL>& sm,
                                                       const uint32_t* __restrict__ quads, int it, int c, int fi,
                                                       uint32_t m) {
  const LatticeDesc& d = ga.p.d;
  PatchItem<PL> I;
  const GroupBlock& B = sm.b[c];
  I.fl = it < B.nq ? 1u : 0u;
  if (!I.fl) return I;
  const int pitch = ga.pitch;
  const uint32_t q = quads[c * ga.nq_max + it], fcol = sm.fo[m & 1u][c] >> (2 * fi), fx = fcol & 1u, fy = (fcol >> 1) & 1u;
  I.i00 = (int)(q & 0xFFFFu) + (int)fx + (fy ? pitch : 0);
  I.dc = 1;
  I.dr = pitch;
  if (WIDE) {
    const uint32_t wc = (q >> (28u + fx)) & 1u, wr = (q >> (30u + fy)) & 1u;
    I.i00 += (fx & (q >> 28)) + (fy & (q >> 30) ? pitch : 0);
    I.dc += (int)wc;
    I.dr += wr ? pitch : 0;
    I.fl |= wc << 1 | wr << 2;
  }
  const uint32_t GQ = (uint32_t)d.GQ;
  const uint32_t kx = (uint32_t)B.f0x + 2u * ((q >> 16) & 63u) + fx, ky = (uint32_t)B.f0y + 2u * ((q >> 22) & 63u) + fy;
  if (REFLECT)
    I.fl |= (ky == 0u ? 16u : 0u) | (ky == (uint32_t)ga.gqy - 1u ? 32u : 0u) | (kx == 0u ? 64u : 0u) |
            (kx == GQ - 1u ? 128u : 0u);
  patch_item_draw<PL, LG, REFLECT, WIDE>(I, sm.key[m & 1u], ky * GQ + kx, m, d.rk, sm.T, d.tx, d.txi);
  return I;
}

// Named barriers: 1 + f hands the macros to fine phase f, kBarDone ends a
// visit's last phase, kBarCount its count.
constexpr int kBarDone = 6, kBarCount = 7;

// With one group the phase is a constant; a barrier id in a register makes a
// CTA reserve all 16.
template <int NG>
__device__ __forceinline__ void phase_sync(int fi, uint32_t n) {
  if (NG > 1)
    bar_named(1u + (uint32_t)fi, n);
  else if (fi == 0)
    bar_named<1>(n);
  else if (fi == 1)
    bar_named<2>(n);
  else if (fi == 2)
    bar_named<3>(n);
  else
    bar_named<4>(n);
}

// NG (1, 2 or 4) groups of ga.gs threads; group i runs the fine phases
// i, i + NG, ...; the last warp of the last group (which runs the
// last fine phase) does the exchange.
//
// WIDE: some fine segments have 3 sites.
template <int PL, int LG, bool REFLECT, bool WIDE, int NG>
__global__ void __launch_bounds__(group_max_threads(NG), NG == 1 ? 3 : 1)
    persistent_group_kernel(const __grid_constant__ GroupArgs ga) {
  typedef typename MacroOf<PL>::type MT;
  constexpr int kPer = 4 / PL;
  constexpr int kItems = (kGroupWords * PL + 63) / 64;   // record words per lane of the exchanging warp
  extern __shared__ __align__(16) uint8_t group_dyn[];
  __shared__ GroupSmem<PL> sm;
  const PersistentArgs& a = ga.p;
  const LatticeDesc& d = a.d;
  RunState* st = a.st;
  unsigned long long* ob = a.ob;
  MT* M = reinterpret_cast<MT*>(group_dyn);
  MT* G = reinterpret_cast<MT*>(a.macros);
  const int tid = threadIdx.x, nt = (int)blockDim.x, lane = tid & 31, pitch = ga.pitch;
  const bool run = !ld_volatile(&st->stopped);
  if (run) {
    patch_tables_fill<PL>(sm.T, d, tid, nt);
    const int half = d.P >> 1, gx = (int)blockIdx.x % half, gy = (int)blockIdx.x / half;
    if (tid < 4) group_block(d, gx, gy, tid, pitch, sm.b[tid]);
    if (tid < 4)
      sm.fo[a.m_begin & 1u][tid] = fine_order(d, 2 * gx + (tid & 1), 2 * gy + (tid >> 1), a.m_begin);
    if (tid == 4) sm.key[a.m_begin & 1u] = step_keys(a.m_begin, d.rk);
    if (tid < kMaxStates) sm.hist[tid] = 0;
    if (tid == 0) sm.quit = 0;
    __syncthreads();
    if (tid < 4) {
      const GroupBlock& B = sm.b[tid];
      sm.b[tid].nw = B.ncx / kPer + 1 + B.ncy / kPer + 1 + 3;
    }
    uint32_t* quads = reinterpret_cast<uint32_t*>(group_dyn + ga.quads);
    for (int i = tid; i < 4 * ga.nq_max; i += nt) {
      const int c = i / ga.nq_max, q = i - c * ga.nq_max;
      if (q < sm.b[c].nq) quads[i] = group_quad(sm.b[c], pitch, q);
    }
    for (int i = tid; i < 4 * kGroupWords; i += nt) {
      GroupWord W;
      if (group_word<PL>(d, sm.b[i / kGroupWords], pitch, i % kGroupWords, W)) sm.w[i / kGroupWords][i % kGroupWords] = W;
    }
    const int sx0 = block_slot(d.ax, 2 * gx), sy0 = block_slot(d.ay, 2 * gy);
    {
      const int nx = sm.b[0].ncx + sm.b[1].ncx + 1, ny = sm.b[0].ncy + sm.b[2].ncy + 1;
      for (int r = tid >> 5; r < ny; r += nt >> 5) {
        const int y = sy0 + r == ga.nsy ? 0 : sy0 + r;
        for (int c = lane; c < nx; c += 32)
          M[r * pitch + c] = __ldcg(G + (size_t)y * ga.gpitch + (sx0 + c == ga.nsx ? 0 : sx0 + c));
      }
    }
    __syncthreads();

    const int gs = ga.gs, grp = NG == 1 ? 0 : tid / gs, t = tid - grp * gs;
    const bool comm = grp == NG - 1, commw = comm && t >= gs - 32;
    const uint32_t m_end = a.m_begin + a.n_mcs, nb = (uint32_t)(d.P * d.Py);

    auto order = [&](uint32_t m) {
      return colour_order(philox10_rk(make_uint4(0u, 0u, m, kTagOrder), d.rk).x, d.perm24);
    };
    // What the visit (m, k) reads of other groups, by the exchanging warp; o,
    // op: the coarse orders of MCS m and m - 1.  A block's key is its slot if
    // it visited in MCS m - 1 only, 4 + its slot in m; in the launch's first
    // MCS the array as loaded stands for every earlier visit (this block's
    // key 3, the others' -1).
    auto receive = [&](uint32_t m, int k, uint32_t o, uint32_t op) {
      const int c = order_at(o, k);
      const bool first = m == a.m_begin;
      const int sV = slot_of(o, c ^ 2), sH = slot_of(o, c ^ 1), sD = slot_of(o, c ^ 3);
      const int kV = sV < k ? sV + 4 : (first ? -1 : slot_of(op, c ^ 2));
      const int kH = sH < k ? sH + 4 : (first ? -1 : slot_of(op, c ^ 1));
      const int kD = sD < k ? sD + 4 : (first ? -1 : slot_of(op, c ^ 3));
      const int kX = first ? 3 : slot_of(op, c), best = max(max(kV, kH), max(kD, kX));
      const int nw = sm.b[c].nw;
      GroupWord W[kItems];
      uint32_t epoch[kItems];
      unsigned long long v[kItems];
      bool need[kItems], got[kItems];
#pragma unroll
      for (int j = 0; j < kItems; ++j) {
        const int i = lane + 32 * j;
        need[j] = false;
        epoch[j] = 0;
        v[j] = 0;
        if (i < nw) {
          W[j] = sm.w[c][i];
          const int s = W[j].kind == kVLine ? sV : (W[j].kind == kHLine ? sH : sD);
          const int key = W[j].kind == kVLine ? kV : (W[j].kind == kHLine ? kH : kD);
          need[j] = W[j].kind == kCorner ? kD == best : key > kX;
          epoch[j] = s < k ? m + 1u : m;
          if (need[j]) v[j] = ld_word(ob + W[j].src);
        }
        got[j] = !need[j];
      }
      uint32_t spins = 0;
      for (;;) {
        bool all = true;
#pragma unroll
        for (int j = 0; j < kItems; ++j) {
          got[j] = got[j] || (uint32_t)(v[j] >> 32) == epoch[j];
          all = all && got[j];
        }
        if (all) break;
        // the abort flag every 16th round: a read of it in every round would
        // put a second L2 round trip between two polls
        if ((spins & 15u) == 15u && ld_volatile(&st->abort)) {
          sm.quit = 1;
          break;
        }
        if (++spins > a.spin_limit) {
          atomicOr(&st->error, kErrTimeout);
          atomicExch(&st->abort, 1u);
          sm.quit = 1;
          break;
        }
#pragma unroll
        for (int j = 0; j < kItems; ++j)
          if (!got[j]) v[j] = ld_word(ob + W[j].src);
      }
      __syncwarp();
#pragma unroll
      for (int j = 0; j < kItems; ++j) {
        if (!need[j]) continue;
        const int key = W[j].kind == kVLine ? kV : (W[j].kind == kHLine ? kH : kD);
        const uint32_t data = (uint32_t)v[j] >> (8 * PL * W[j].sub);
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
          const bool end = (e == 0 && (W[j].ends & 1u)) || (e == W[j].n - 1 && (W[j].ends & 2u));
          if (e < W[j].n && (!end || key == best)) M[W[j].dst + e * W[j].stride] = (MT)(data >> (8 * PL * e));
        }
      }
      __syncwarp();
    };

    uint32_t ordp = 0, ord = order(a.m_begin), ord_next = order(a.m_begin + 1u);
    PatchItem<PL> cur = group_prepare<PL, LG, REFLECT, WIDE>(ga, sm, quads, t, order_at(ord, 0), grp, a.m_begin);
    if (NG > 1 && commw) bar_arrive(1u, (uint32_t)(gs + 32));   // the launch's first visit reads no one
    bool quit = false;
    uint32_t m = a.m_begin;
    int k = 0;
    for (;;) {   // one visit
      const int colour = order_at(ord, k);
      const bool last = k == 3 && m + 1u == m_end;
#pragma unroll
      for (int f = 0; f < 4 / NG; ++f) {
        const int fi = NG == 1 ? f : grp + f * NG;
        phase_sync<NG>(fi, (uint32_t)(NG == 1 ? gs : (fi == 0 ? gs + 32 : 2 * gs)));
        if (f == 0 && sm.quit) {
          if (fi + 1 < NG) bar_arrive(2u + (uint32_t)fi, (uint32_t)(2 * gs));
          quit = true;
          break;
        }
        if (cur.fl) patch_item_run<PL, LG, REFLECT, WIDE>(M, pitch, cur, sm.T, d.tx, d.txi);
        // the item prepared next
        const bool turn = f == 4 / NG - 1, pn = turn && k == 3;   // of the next visit, the next MCS
        const int pc = turn ? (pn ? order_at(ord_next, 0) : order_at(ord, k + 1)) : colour;
        if (NG > 1 && fi < 3) bar_arrive(2u + (uint32_t)fi, (uint32_t)(2 * gs));
        if (turn && comm) {
          const bool log_point = a.fuse_counts && ((m + 1u) % a.log_every) == 0u;
          if (commw || log_point)
            bar_named<kBarDone>((uint32_t)gs);
          else
            bar_arrive<kBarDone>((uint32_t)gs);
          if (commw) {
            const GroupBlock& B = sm.b[colour];
            if (B.id != a.stall_block)
              for (int i = lane; i < B.nw - 3; i += 32) {
                const GroupWord W = sm.w[colour][i];
                uint32_t x = 0;
#pragma unroll
                for (int e = 0; e < kPer; ++e)
                  if (e < W.n) x |= (uint32_t)M[W.dst + e * W.stride] << (8 * PL * e);
                st_word(ob + W.own, ((unsigned long long)(m + 1u) << 32) | x);
              }
            __syncwarp();
          }
          if (log_point) {
            group_count<PL>(M, pitch, sm.b[colour], d.S, k, slot_of(ord, colour ^ 2), slot_of(ord, colour ^ 1),
                            slot_of(ord, colour ^ 3), sm.hist, t, gs);
            if (commw)
              bar_named<kBarCount>((uint32_t)gs);
            else
              bar_arrive<kBarCount>((uint32_t)gs);
            if (commw)
              group_log(st, a.lb, d.S, m + 1u, a.log_every, a.stop_at_extinction, nb, sm.hist,
                        (unsigned long long)d.L * (unsigned long long)d.H);
          }
          if (commw && !last) {
            receive(k < 3 ? m : m + 1u, (k + 1) & 3, k < 3 ? ord : ord_next, k < 3 ? ordp : ord);
            if (NG > 1) bar_arrive(1u, (uint32_t)(gs + 32));
          }
        }
        if (fi == 0 && k == 0) {   // read from this MCS's last visit on
          if (t < 4) sm.fo[(m + 1u) & 1u][t] = fine_order(d, sm.b[t].bx, sm.b[t].by, m + 1u);
          if (t == 4) sm.key[(m + 1u) & 1u] = step_keys(m + 1u, d.rk);
        }
        cur = group_prepare<PL, LG, REFLECT, WIDE>(ga, sm, quads, t, pc, turn ? grp : fi + NG, pn ? m + 1u : m);
      }
      if (quit || last) break;
      if (++k == 4) {
        k = 0;
        ++m;
        ordp = ord;
        ord = ord_next;
        ord_next = order(m + 1u);
      }
    }
    __syncthreads();
    if (!quit) {
      // every macro from the last visitor of the blocks that share it
      for (int c = 0; c < 4; ++c) {
        const GroupBlock& B = sm.b[c];
        const int kc = slot_of(ord, c), bx0 = sx0 + ((c & 1) ? sm.b[0].ncx : 0), by0 = sy0 + ((c >> 1) ? sm.b[0].ncy : 0);
        const bool v = slot_of(ord, c ^ 2) < kc, h = slot_of(ord, c ^ 1) < kc, dg = slot_of(ord, c ^ 3) < kc;
        for (int r = tid >> 5; r <= B.ncy; r += nt >> 5) {
          const bool lr = r == 0 || r == B.ncy;
          if (lr && !v) continue;
          const int y = by0 + r == ga.nsy ? 0 : by0 + r;
          for (int q = lane; q <= B.ncx; q += 32) {
            const bool lc = q == 0 || q == B.ncx;
            if ((lc && !h) || (lr && lc && !dg)) continue;
            G[(size_t)y * ga.gpitch + (bx0 + q == ga.nsx ? 0 : bx0 + q)] = M[B.base + r * pitch + q];
          }
        }
      }
    }
  }
  // The last CTA to leave publishes the MCS number.
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(&st->exited, 1u) == gridDim.x - 1u) {
      st->exited = 0;
      st->ticket = 0;
      if (!st->stopped && !st->abort) st->mcs = a.m_begin + a.n_mcs;
    }
  }
}

// ---------------------------------------------------------------------------
// Lattice array <-> macros of any partition (escg_flag.cu has the kernels of
// the uniform one).

// Sites of slot s of an axis (P blocks, n sites): half 0 and half 1, -1 none.
__device__ __forceinline__ int2 slot_sites(const AxisGeom& g, int n, int s) {
  const int wa = g.Qa + block_wide(g, true), wb = g.Qb + block_wide(g, false), ka = g.r * wa;
  const bool a = s < ka;
  const int b = a ? s / wa : g.r + (s - ka) / wb, o = a ? s - b * wa : s - ka - (b - g.r) * wb;
  const int fr = a ? block_wide(g, true) : block_wide(g, false), x0 = b * g.q + min(b, g.r);
  const bool wide = o < 2 * fr;   // slots of the block's leading 3-site segments
  const int j = wide ? o >> 1 : o - fr, x = x0 + (wide ? 3 * j : 2 * j + fr);   // the segment's first site
  if (wide && (o & 1)) return make_int2(x + 1, -1);
  return make_int2(x == 0 ? n - 1 : x - 1, x);
}
// Slot and half of site x of an axis with ns slots: 2 slot + half.
__device__ __forceinline__ int site_slot(const AxisGeom& g, int ns, int x) {
  const int ka = g.r * (g.q + 1);
  const bool a = x < ka;
  const int b = a ? x / (g.q + 1) : g.r + (x - ka) / g.q, o = a ? x - b * (g.q + 1) : x - ka - (b - g.r) * g.q;
  const int fr = block_wide(g, a), na = min(b, g.r);
  const int s0 = na * (g.Qa + block_wide(g, true)) + (b - na) * (g.Qb + block_wide(g, false));
  if (o < 3 * fr) {
    const int j = o / 3, r = o - 3 * j;
    return r == 0 ? 2 * (s0 + 2 * j) + 1 : (r == 1 ? 2 * (s0 + 2 * j + 1) : 2 * (s0 + 2 * j + 2 == ns ? 0 : s0 + 2 * j + 2));
  }
  const int p = o - 3 * fr, s = s0 + 2 * fr + (p >> 1);
  return (p & 1) ? 2 * (s + 1 == ns ? 0 : s + 1) : 2 * s + 1;
}

// A block moves 32 columns (of slots, or of groups of 4 sites) of kConvRows
// rows: a thread works out its columns once, the block its rows once (the
// divisions of the closed form cost more than the loads).
constexpr int kConvRows = 64;

template <int PL>
__global__ void __launch_bounds__(256)
    macro_fill_any_kernel(LatticeDesc d, int nsx, int nsy, int gpitch, typename MacroOf<PL>::type* G, RunState* st) {
  const bool off = macro_fill_off(st);
  typedef typename MacroOf<PL>::type MT;
  __shared__ int2 rows[kConvRows];
  const int x = blockIdx.x * 32 + threadIdx.x, y0 = blockIdx.y * kConvRows, t = threadIdx.y * 32 + threadIdx.x;
  if (t < kConvRows && y0 + t < nsy) rows[t] = slot_sites(d.ay, d.H, y0 + t);
  __syncthreads();
  if (x >= nsx) return;
  const int2 c = slot_sites(d.ax, d.L, x);
  if (off) return;   // asked for above: its load passes beside the divisions
  auto site = [&](int row, int col) -> uint32_t {
    if (row < 0 || col < 0) return 0u;
    const uint8_t* p = d.lat + (size_t)row * d.pitch;
    if (d.bits == 8) return p[col];
    const uint32_t bit = (uint32_t)col * (uint32_t)d.bits;
    return ((uint32_t)p[bit >> 3] >> (bit & 7u)) & ((1u << d.bits) - 1u);
  };
#pragma unroll 4
  for (int k = threadIdx.y; k < kConvRows; k += 8) {
    if (y0 + k >= nsy) break;
    const int2 r = rows[k];
    G[(size_t)(y0 + k) * gpitch + x] = (MT)(site(r.x, c.x) | (site(r.x, c.y) << (2 * PL)) | (site(r.y, c.x) << (4 * PL)) |
                                            (site(r.y, c.y) << (6 * PL)));
  }
}

template <int PL>
__global__ void __launch_bounds__(256)
    macro_drain_any_kernel(LatticeDesc d, int nsx, int nsy, int gpitch, const typename MacroOf<PL>::type* G,
                           const RunState* st) {
  const bool on = st->on_macros != 0u;
  __shared__ int rows[kConvRows];
  const int c0 = 4 * (blockIdx.x * 32 + threadIdx.x), y0 = blockIdx.y * kConvRows, t = threadIdx.y * 32 + threadIdx.x;
  if (t < kConvRows && y0 + t < d.H) rows[t] = site_slot(d.ay, nsy, y0 + t);
  __syncthreads();
  if (c0 >= d.L) return;
  int mx[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) mx[e] = c0 + e < d.L ? site_slot(d.ax, nsx, c0 + e) : -1;
  if (!on) return;
#pragma unroll 4
  for (int k = threadIdx.y; k < kConvRows; k += 8) {
    const int y = y0 + k;
    if (y >= d.H) break;
    const int my = rows[k];
    const typename MacroOf<PL>::type* row = G + (size_t)(my >> 1) * gpitch;
    uint32_t u = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (mx[e] >= 0)
        u |= (((uint32_t)row[mx[e] >> 1] >> (2 * PL * (2 * (my & 1) + (mx[e] & 1)))) & (PL == 1 ? 3u : 15u)) << (8 * e);
    uint8_t* out = d.lat + (size_t)y * d.pitch;
    if (d.bits == 8 && c0 + 4 > d.L) {   // no row padding written
      for (int e = 0; c0 + e < d.L; ++e) out[c0 + e] = (uint8_t)(u >> (8 * e));
    } else {
      store_group(out, c0, d.bits, pack4(u, d.bits));
    }
  }
}

// ---------------------------------------------------------------------------
int macro_pitch(const LatticeDesc& d) { return (axis_slots(d.ax, d.P) + 15) & ~15; }
size_t macro_bytes(const LatticeDesc& d) {
  return (size_t)macro_pitch(d) * (size_t)axis_slots(d.ay, d.Py) * (size_t)patch_planes(d);
}

cudaError_t launch_macro_fill_any(const LatticeDesc& d, void* macros, RunState* st, cudaStream_t stream) {
  const int nsx = axis_slots(d.ax, d.P), nsy = axis_slots(d.ay, d.Py);
  const dim3 cb(32, 8), cg((nsx + 31) / 32, (nsy + kConvRows - 1) / kConvRows);
  if (patch_planes(d) == 1)
    macro_fill_any_kernel<1><<<cg, cb, 0, stream>>>(d, nsx, nsy, macro_pitch(d), reinterpret_cast<uint8_t*>(macros), st);
  else
    macro_fill_any_kernel<2><<<cg, cb, 0, stream>>>(d, nsx, nsy, macro_pitch(d), reinterpret_cast<uint16_t*>(macros), st);
  return cudaGetLastError();
}
cudaError_t launch_macro_drain_any(const LatticeDesc& d, const void* macros, const RunState* st, cudaStream_t stream) {
  const int nsx = axis_slots(d.ax, d.P), nsy = axis_slots(d.ay, d.Py);
  const dim3 cb(32, 8), cg(((d.L + 3) / 4 + 31) / 32, (d.H + kConvRows - 1) / kConvRows);
  if (patch_planes(d) == 1)
    macro_drain_any_kernel<1><<<cg, cb, 0, stream>>>(d, nsx, nsy, macro_pitch(d), reinterpret_cast<const uint8_t*>(macros), st);
  else
    macro_drain_any_kernel<2><<<cg, cb, 0, stream>>>(d, nsx, nsy, macro_pitch(d),
                                                     reinterpret_cast<const uint16_t*>(macros), st);
  return cudaGetLastError();
}

static int fine_rows(const LatticeDesc& d) { return d.ay.r * d.ay.Qa + (d.Py - d.ay.r) * d.ay.Qb; }

// The build for a lattice and a number of groups, or null: those that beat
// the other kernels.  us per MCS at M = 1e-4, one CTA per SM unless stated,
// against the byte kernels in parentheses:
//  * von Neumann, periodic, 3-site segments, 2 bits per site: L = 200 15.3
//    (25.6), 400 18.1 (26.5), 800 18.2 (24.1); at 4 bits (S = 5) 24.9 (24.1), and at
//    two CTAs per SM (L = 2200) 27.9 (27.2): not built.
//  * Moore, periodic: L = 400 18.1 (39.5), S = 5 26.3 (40.4); 64 x 64 blocks, L =
//    1024, against the flag kernel on macros 12.5 (15.5), S = 5 13.7 (17.9); two
//    CTAs per SM, 2 bits per site: 1600 28.7 (40.8), 2200 26.9 (39.2).
//  * reflecting on 64 x 64 blocks, L = 1024: 12.9 (22.2), S = 5 13.9.  With 3-site
//    segments the mirrored steps were slower, L = 800 35.0 (28.2), before their
//    entries came from a table (not measured since): not built.
//  * 64 x 64 blocks, von Neumann, periodic: L = 1024 12.5 (12.6), 1536 12.3 (11.9):
//    not built.
static const void* group_fn(const LatticeDesc& d, int groups) {
#define GROUP_FN(PL, LG, RF, WIDE, NG) reinterpret_cast<const void*>(&persistent_group_kernel<PL, LG, RF, WIDE, NG>)
  const bool wide = axis_slots(d.ax, d.P) > d.GQ || axis_slots(d.ay, d.Py) > fine_rows(d);
  const bool one = patch_planes(d) == 1, moore = d.nbh == 8, refl = d.reflect != 0;
  if (wide && !refl) {
    if (groups == 2) return moore ? (one ? GROUP_FN(1, 3, false, true, 2) : GROUP_FN(2, 3, false, true, 2))
                                  : (one ? GROUP_FN(1, 2, false, true, 2) : nullptr);
    if (groups == 1) return moore && one ? GROUP_FN(1, 3, false, true, 1) : nullptr;
  } else if (!wide && groups == (one ? 4 : 2)) {   // 4 bits per site: 64 registers would spill
    if (moore && !refl) return one ? GROUP_FN(1, 3, false, false, 4) : GROUP_FN(2, 3, false, false, 2);
    if (!moore && refl) return one ? GROUP_FN(1, 2, true, false, 4) : GROUP_FN(2, 2, true, false, 2);
  }
  return nullptr;
#undef GROUP_FN
}

int persistent_group_config(const LatticeDesc& d, int device, GroupConfig* cfg, int min_per_sm) {
  if (d.P < 2 || d.Py < 2 || !slot_axis_ok(d.ax) || !slot_axis_ok(d.ay)) return 0;
  auto wider = [](const AxisGeom& g, bool slots) {   // of the axis's two block widths
    const int a = g.r > 0 ? g.Qa + (slots ? block_wide(g, true) : 0) : 0;
    const int b = g.Qb + (slots ? block_wide(g, false) : 0);
    return a > b ? a : b;
  };
  const int nq = (wider(d.ax, false) / 2) * (wider(d.ay, false) / 2);
  const int nsx = wider(d.ax, true), nsy = wider(d.ay, true);
  const int planes = patch_planes(d), groups = (d.P / 2) * (d.Py / 2);
  // a tile row: whole 32-byte sectors, the rows of two quads 32 or 96 bytes apart modulo the banks
  const int pitch = ((2 * nsx + 1 + 15) & ~31) + 16;
  const int quads = ((2 * nsy + 1) * pitch * planes + 15) & ~15, need = (quads + 16 * nq + 15) & ~15;
  if (nsx / (4 / planes) + 1 > 26 || nsy / (4 / planes) + 1 > 26) return 0;   // kGroupWords
  int sms = 0, smem_sm = 0, reserved = 0, optin = 0, coop = 0;
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device);
  if (!coop) return 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device);
  cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, device);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (sms <= 0) return 0;
  int per_sm = (groups + sms - 1) / sms;
  if (per_sm < min_per_sm) per_sm = min_per_sm;
  const int full = (nq + 31) & ~31;
  struct {
    int groups, gs;
  } const cand[] = {{4, full}, {2, full + 32}, {2, full}, {1, full + 32}};
  for (const auto& c : cand) {
    const int nt = c.groups * c.gs;
    if (nt > group_max_threads(c.groups)) continue;
    const void* fn = group_fn(d, c.groups);
    if (!fn) continue;
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) return 0;
    const int stat = (int)fa.sharedSizeBytes;
    if (optin - stat < need ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - stat) != cudaSuccess)
      return 0;
    // padding: per_sm + 1 CTAs just do not fit an SM, so the grid spreads over
    // all SMs and the rest of the SM's memory stays L1 cache
    int pad = (smem_sm / (per_sm + 1) - reserved - stat + 256) & ~127;
    if (pad > optin - stat) pad = optin - stat;
    if (pad < need) pad = need;
    for (int dyn = pad;; dyn = dyn - 1024 > need ? dyn - 1024 : need) {
      int occ = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, nt, (size_t)dyn) != cudaSuccess) return 0;
      if (occ >= per_sm) {
        cfg->dyn_bytes = dyn;
        cfg->groups = c.groups;
        cfg->group_threads = c.gs;
        cfg->ctas_per_sm = per_sm;
        cfg->pitch = pitch;
        cfg->quads = quads;
        cfg->nq_max = nq;
        return groups;
      }
      if (dyn == need) break;   // the grid cannot be resident at once
    }
  }
  return 0;
}

// A cooperative launch: the runtime starts the grid only with every CTA
// resident, also while kernels of other streams hold part of the device.
cudaError_t launch_persistent_group(const PersistentArgs& a, const GroupConfig& cfg, cudaStream_t stream) {
  GroupArgs arg;
  arg.p = a;
  arg.gs = cfg.group_threads;
  arg.pitch = cfg.pitch;
  arg.quads = cfg.quads;
  arg.nq_max = cfg.nq_max;
  arg.gpitch = macro_pitch(a.d);
  arg.gqy = fine_rows(a.d);
  arg.nsx = axis_slots(a.d.ax, a.d.P);
  arg.nsy = axis_slots(a.d.ay, a.d.Py);
  cudaError_t e = cudaSuccess;
  if (a.fill)
    e = a.d.blocks64 ? launch_macro_fill(a.d, a.macros, a.st, stream)
                     : launch_macro_fill_any(a.d, a.macros, a.st, stream);
  if (e != cudaSuccess) return e;
  void* params[] = {&arg};
  e = cudaLaunchCooperativeKernel(group_fn(a.d, cfg.groups), dim3((a.d.P / 2) * (a.d.Py / 2)), dim3(cfg.groups * cfg.group_threads),
                                  params, (size_t)cfg.dyn_bytes, stream);
  if (e != cudaSuccess || !a.drain) return e;
  return a.d.blocks64 ? launch_macro_drain(a.d, a.macros, a.st, stream)
                      : launch_macro_drain_any(a.d, a.macros, a.st, stream);
}

}  // namespace escg_impl
