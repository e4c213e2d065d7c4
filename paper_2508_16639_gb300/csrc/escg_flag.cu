// escg_flag.cu -- the epoch-flag kernel on macros: uniform partitions (blocks
// of 64 x 64 sites, 2 x 2 sub-blocks), any rule, any number of species, any
// bits per site.
//
// persistent_kernel's work items and flags (escg_kernels.cu), on the layout
// of escg_patch.cuh.  For the time of a call the lattice is kept as an
// array of macros, row slot ky, column slot kx at ky * GQ + kx (a byte or two
// bytes for 2 x 2 sites): macro_fill_kernel makes it from the caller's array
// before the call's first launch and macro_drain_kernel writes the caller's
// array after its last.  A block's tile is the 33 x 33 macros of its joint slots -- 1.1 or 2.2 KB,
// one 16-byte load per thread, no conversion -- and holds its 64 x 64 sites,
// its rim lines and its corners, so the Moore rule needs nothing more.  At
// L = 12800 the macros are 41 or 82 MB and stay in the L2, where the array of
// one byte per site (164 MB) does not.
//
// Blocks of one colour never share a macro (two of them are a block apart),
// and a visit writes its whole tile back, so a macro always holds what the
// last visit of the up to four blocks around it left.
#include "escg_internal.h"
#include "escg_patch.cuh"
#include "escg_sync.cuh"

namespace escg_impl {

constexpr int kFlagSlots = 33;    // joint slots of a block along an axis
constexpr int kFlagPitch = 48;    // macros per tile row: 16-byte aligned rows, and the two quad rows of
                                  // a warp fall into different shared-memory banks

template <int PL>
struct FlagSmem {
  alignas(16) typename MacroOf<PL>::type tile[kFlagSlots * kFlagPitch];
  PatchTables T;
  uint32_t hist[kMaxStates];
  uint4 dec;   // the item's (m, k, bx, by), decoded by the ticket thread
  uint32_t ord, forder, quit, abort;
};

// 16-byte pieces of a tile's rows (32 macros), then one piece per row for its
// last macro.
template <int PL>
struct FlagPieces {
  static constexpr int kVec = 2 * PL * kFlagSlots;
  static constexpr int kAll = kVec + kFlagSlots;
};

// Piece i of the tile of block (bx, by): its address in the macro array and
// in the tile.
template <int PL>
__device__ __forceinline__ void flag_piece(const LatticeDesc& d, int bx, int by, int i, uint32_t& g, int& t) {
  const int GQ = d.GQ, GQy = d.H >> 1;
  const bool vec = i < FlagPieces<PL>::kVec;
  const int r = vec ? i / (2 * PL) : i - FlagPieces<PL>::kVec, c = vec ? (16 / PL) * (i % (2 * PL)) : 32;
  int gy = 32 * by + r, gx = 32 * bx + c;
  if (gy == GQy) gy = 0;
  if (gx == GQ) gx = 0;
  g = (uint32_t)gy * (uint32_t)GQ + (uint32_t)gx;   // < 2^27: L, H <= 16384
  t = r * kFlagPitch + c;
}

// Counts of a visit: a macro is counted by the last visit of the blocks that
// share it (slot k against the vertical, horizontal and diagonal neighbours'),
// the non-empty states only (the empty sites are the rest of the lattice).
template <int PL, int NT>
__device__ __forceinline__ void flag_count(FlagSmem<PL>& sm, int S, int k, int sV, int sH, int sD) {
  constexpr int kPerWord = 4 / PL, kWords = kFlagPitch / kPerWord;
  constexpr uint32_t kMacro = PL == 1 ? 0xFFu : 0xFFFFu;
  const uint32_t* W = reinterpret_cast<const uint32_t*>(sm.tile);
  const int used = (kFlagSlots + kPerWord - 1) / kPerWord;
  uint32_t cnt[kMaxStates];
#pragma unroll
  for (int v = 0; v < kMaxStates; ++v) cnt[v] = 0;
  for (int i = threadIdx.x; i < kFlagSlots * used; i += NT) {
    const int r = i / used, c = i % used;
    uint32_t x = W[r * kWords + c], mask = 0;
#pragma unroll
    for (int j = 0; j < kPerWord; ++j) {
      const int col = kPerWord * c + j;
      const bool lr = r == 0 || r == kFlagSlots - 1, lc = col == 0 || col == kFlagSlots - 1;
      const bool mine = col < kFlagSlots && (!lr || sV < k) && (!lc || sH < k) && (!(lr && lc) || sD < k);
      if (mine) mask |= kMacro << (8 * PL * j);
    }
    x &= mask;
#pragma unroll
    for (int v = 1; v < (PL == 1 ? 4 : kMaxStates); ++v) {
      if (v > S) break;
      if (PL == 1) {
        const uint32_t t = x ^ (uint32_t)(v * 0x55555555u);
        cnt[v] += __popc(~(t | (t >> 1)) & 0x55555555u);
      } else {
        const uint32_t t = x ^ (uint32_t)(v * 0x11111111u), n = t | (t >> 1);
        cnt[v] += __popc(~(n | (n >> 2)) & 0x11111111u);
      }
    }
  }
#pragma unroll
  for (int v = 1; v < (PL == 1 ? 4 : kMaxStates); ++v) {
    if (v > S) break;
    const uint32_t s = __reduce_add_sync(0xFFFFFFFFu, cnt[v]);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(&sm.hist[v], s);
  }
}

// A block's counts are in st->acc[ring]; the last of the nb blocks writes the
// log entry of MCS m + 1.
static __device__ __noinline__ void flag_log(RunState* st, const PersistentArgs& a, uint32_t m, uint32_t ring, uint32_t nb) {
  __threadfence();
  if (atomicAdd(&st->pend[ring], 1u) != nb - 1u) return;
  __threadfence();
  unsigned long long c[kMaxStates], rest = (unsigned long long)a.d.L * (unsigned long long)a.d.H;
  for (int v = 1; v < kMaxStates; ++v) {
    c[v] = atomicExch(&st->acc[ring][v], 0ull);
    rest -= c[v];
  }
  c[0] = rest;
  st->pend[ring] = 0;
  write_log_entry(st, a.lb, a.d.S, m + 1u, a.log_every, c, a.stop_at_extinction);
}

// Bound by the colour chain while a phase is one wave (L = 3200: issue active
// 52 %, 39 executed thread instructions per attempt where the byte tile took
// 52), by integer issue once phases are several waves deep.  us per MCS of
// 10-MCS launches, conversions included, against the byte tile: L = 3200 23.2 ->
// 19.2 (4.4e11 -> 5.3e11 site updates/s), Moore 24.5 -> 19.9, L = 12800 304 ->
// 208, at 2 bits per site 337 -> 207; 60-MCS launches: L = 2816 22.2 -> 17.8, 4096
// 35.8 -> 28.0, 6400 77.1 -> 52.9, L = 12800 with S = 5 307 -> 256.
//
// LG: log2 of the neighbourhood.  NT = 256: a sub-block per thread and fine
// phase, 4 CTAs per SM; NT = 128: two, 8 CTAs per SM.
template <int PL, int LG, bool REFLECT, int NT>
__global__ void __launch_bounds__(NT, NT == 128 ? 8 : 4)
    persistent_macro_kernel(const __grid_constant__ PersistentArgs a) {
  typedef typename MacroOf<PL>::type MT;
  constexpr int kSub = 256 / NT;   // sub-blocks per thread and fine phase
  __shared__ FlagSmem<PL> sm;
  const LatticeDesc& d = a.d;
  RunState* st = a.st;
  MT* G = reinterpret_cast<MT*>(a.macros);
  const int tid = threadIdx.x;
  const bool run = !ld_volatile(&st->stopped);
  if (run) {
    patch_tables_fill<PL>(sm.T, d, tid, NT);
    const int P = d.P, half = P >> 1, Py = d.Py;
    const uint32_t nb = (uint32_t)(P * Py), per = nb >> 2;
    const uint64_t total = (uint64_t)a.n_mcs * nb;
    const uint32_t GQ = (uint32_t)d.GQ, GQy = (uint32_t)d.H >> 1, tx = d.tx, txi = d.txi;
    // Tickets as in persistent_kernel: taken in schedule order, one at a time,
    // as the CTA releases the epoch of its previous visit, by a thread of warp
    // 1 (warp 0 releases and polls).
    constexpr int kTicketThread = 32;
    uint32_t c_m = 0xFFFFFFFFu, c_ord = 0;   // ticket thread: coarse order of MCS c_m
    uint32_t t_next = 0, ab_next = 0;        // ticket thread: next ticket, abort flag seen with it
    if (tid == kTicketThread) {
      t_next = atomicAdd(&st->ticket, 1u);
      ab_next = ld_volatile(&st->abort);
    }
    const int qx = tid & 15, qy = tid >> 4;
    for (;;) {
      if (tid == kTicketThread) {
        const uint32_t t = t_next;
        const uint32_t quit = ((uint64_t)t >= total) || ab_next;
        if (!quit) {
          uint32_t rem, j, jx;
          const uint32_t m = a.m_begin + div_by_rcp(t, nb, a.rcp_nb, rem);
          if (m != c_m) {
            c_m = m;
            c_ord = colour_order(philox10_rk(make_uint4(0u, 0u, m, kTagOrder), d.rk).x, d.perm24);
          }
          sm.ord = c_ord;
          const uint32_t kk = div_by_rcp(rem, per, a.rcp_per, j);
          const uint32_t jy = div_by_rcp(j, (uint32_t)half, a.rcp_half, jx);
          const uint32_t col = (uint32_t)order_at(c_ord, (int)kk);
          sm.dec = make_uint4(m, kk, 2u * jx + (col & 1u), 2u * jy + (col >> 1));
        }
        sm.quit = quit;
        sm.abort = 0;
      }
      if (tid < kMaxStates) sm.hist[tid] = 0;
      __syncthreads();
      if (sm.quit) break;
      const uint4 dec = sm.dec;
      const uint32_t m = dec.x, ord = sm.ord;
      const int k = (int)dec.y, bx = (int)dec.z, by = (int)dec.w, colour = (bx & 1) | ((by & 1) << 1);
      if (tid == kTicketThread) sm.forder = fine_order(d, bx, by, m);
      if (tid < 9) {
        // every visit of the block and its 8 neighbours that precedes this one
        // in schedule order
        const int dx = tid % 3 - 1, dy = tid / 3 - 1;
        const int ncol = colour ^ ((dx & 1) | ((dy & 1) << 1));
        const uint32_t need = (tid == 4) ? m : (slot_of(ord, ncol) < k ? m + 1u : m);
        const uint32_t* flag = a.done + wrap(by + dy, Py) * P + wrap(bx + dx, P);
        uint32_t spins = 0;
        while (ld_acquire(flag) < need) {
          // the abort flag every 16th round, not between every two polls
          if ((spins & 15u) == 15u && ld_volatile(&st->abort)) {
            sm.abort = 1;
            break;
          }
          if (++spins > a.spin_limit) {
            atomicOr(&st->error, kErrTimeout);
            atomicExch(&st->abort, 1u);
            sm.abort = 1;
            break;
          }
          __nanosleep(64);
        }
      }
      const StepKeys key = step_keys(m, d.rk);   // while the pollers wait
      __syncthreads();
      if (sm.abort) break;   // uniform across the CTA
      // The tile's loads, then -- while they are in flight -- what the first
      // fine phase needs: the words depend on the schedule only.
      constexpr int kLoads = (FlagPieces<PL>::kAll + NT - 1) / NT;
      uint4 v[kLoads];
      uint32_t g[kLoads];
      int ti[kLoads];
#pragma unroll
      for (int j = 0; j < kLoads; ++j) {
        const int i = tid + j * NT;
        if (i >= FlagPieces<PL>::kAll) continue;
        flag_piece<PL>(d, bx, by, i, g[j], ti[j]);
        if (i < FlagPieces<PL>::kVec)
          v[j] = __ldcg(reinterpret_cast<const uint4*>(G + g[j]));
        else
          v[j].x = __ldcg(G + g[j]);
      }
      const uint32_t ford = sm.forder;
      const uint32_t kx0 = (uint32_t)(32 * bx + 2 * qx), ky0 = (uint32_t)(32 * by + 2 * qy);
      Steps2<PL> s[kSub];
      auto draw = [&](int fi) {
        const uint32_t fcol = (ford >> (2 * fi)) & 3u, kx = kx0 + (fcol & 1u);
#pragma unroll
        for (int j = 0; j < kSub; ++j) {
          const uint32_t ky = ky0 + (fcol >> 1) + (uint32_t)(j * (NT / 8));
          uint32_t edge = 0;
          if (REFLECT)
            edge = (ky == 0u ? 1u : 0u) | (ky == GQy - 1u ? 2u : 0u) | (kx == 0u ? 4u : 0u) | (kx == GQ - 1u ? 8u : 0u);
          s[j] = patch_steps2<PL, LG, REFLECT>(philox_step(key, ky * GQ + kx, d.rk), sm.T, tx, txi, edge);
        }
      };
      draw(0);
#pragma unroll
      for (int j = 0; j < kLoads; ++j) {
        const int i = tid + j * NT;
        if (i < FlagPieces<PL>::kVec)
          *reinterpret_cast<uint4*>(sm.tile + ti[j]) = v[j];
        else if (i < FlagPieces<PL>::kAll)
          sm.tile[ti[j]] = (MT)v[j].x;
      }
      __syncthreads();
#pragma unroll
      for (int fi = 0; fi < 4; ++fi) {
        const uint32_t fcol = (ford >> (2 * fi)) & 3u;
        const int i00 = (2 * qy + (int)(fcol >> 1)) * kFlagPitch + 2 * qx + (int)(fcol & 1u);
        if (fi > 0) draw(fi);
        uint32_t w[kSub][PL];
#pragma unroll
        for (int j = 0; j < kSub; ++j) patch_load2<PL>(sm.tile, i00 + j * (NT / 8) * kFlagPitch, 1, kFlagPitch, w[j]);
#pragma unroll
        for (int j = 0; j < kSub; ++j) patch_run2<PL>(w[j], s[j], sm.T);
#pragma unroll
        for (int j = 0; j < kSub; ++j) patch_store2<PL>(sm.tile, i00 + j * (NT / 8) * kFlagPitch, 1, kFlagPitch, w[j]);
        __syncthreads();
      }
#pragma unroll
      for (int j = 0; j < kLoads; ++j) {
        const int i = tid + j * NT;
        if (i < FlagPieces<PL>::kVec)
          *reinterpret_cast<uint4*>(G + g[j]) = *reinterpret_cast<const uint4*>(sm.tile + ti[j]);
        else if (i < FlagPieces<PL>::kAll)
          G[g[j]] = sm.tile[ti[j]];
      }
      const bool log_point = a.fuse_counts && ((m + 1u) % a.log_every) == 0u;
      if (log_point)
        flag_count<PL, NT>(sm, d.S, k, slot_of(ord, colour ^ 2), slot_of(ord, colour ^ 1), slot_of(ord, colour ^ 3));
      __syncthreads();
      // st.release orders the CTA's stores (made before the barrier above)
      // before the new epoch; the counts follow it, off the neighbours' path
      if (tid == 0 && by * P + bx != a.stall_block) st_release(a.done + by * P + bx, m + 1u);
      if (tid == kTicketThread) {
        t_next = atomicAdd(&st->ticket, 1u);
        ab_next = ld_volatile(&st->abort);
      }
      if (log_point) {
        const uint32_t ring = ((m + 1u) / a.log_every) % (uint32_t)kPendRing;
        if (tid >= 1 && tid <= d.S && sm.hist[tid])
          atomicAdd(&st->acc[ring][tid], (unsigned long long)sm.hist[tid]);
        __syncthreads();
        if (tid == 0) {
          __threadfence();
          if (atomicAdd(&st->pend[ring], 1u) == nb - 1u) {
            // last block of this log point: every contribution is in acc
            // (flag_log in line: a call of it costs L = 3200 1 %)
            __threadfence();
            unsigned long long c[kMaxStates], rest = (unsigned long long)d.L * (unsigned long long)d.H;
            for (int v = 1; v < kMaxStates; ++v) {
              c[v] = atomicExch(&st->acc[ring][v], 0ull);
              rest -= c[v];
            }
            c[0] = rest;
            st->pend[ring] = 0;
            write_log_entry(st, a.lb, d.S, m + 1u, a.log_every, c, a.stop_at_extinction);
          }
        }
      }
    }
  }
  // The last CTA to leave publishes the MCS number and resets the
  // dispensers for the next launch on this stream.
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
// The same on any partition of at least 4 blocks a side whose segments have 2 or
// 3 sites and whose blocks at most 256 quads (escg_patch.cuh).  A tile is the
// block's slots, staged in whole aligned 16-byte pieces: they carry up to 15
// macros of the blocks left and right, which go back unchanged -- those blocks
// are idle during the visit, and a piece never reaches a third block (blocks have
// 24 slots or more).
constexpr int kAnySlots = 45;    // of a block along an axis, right joint included: at most 80 sites
constexpr int kAnyPitch = 80;    // macros per tile row: 16-byte rows; the rows of two quads fall into different banks

template <int PL>
struct AnySmem {
  alignas(16) typename MacroOf<PL>::type tile[kAnySlots * kAnyPitch];
  PatchTables T;
  uint32_t quads[4][256];   // by wider block along the columns (1), along the rows (2)
  uint32_t hist[kMaxStates];
  uint4 dec;
  uint32_t ord, forder, quit, abort;
};

// flag_count for a tile of slots 0 .. ncx, 0 .. ncy from column xoff on.  Out of
// line: its registers must not count against the visit's.
template <int PL>
__device__ __noinline__ void any_count(AnySmem<PL>& sm, int xoff, int ncx, int ncy, int S, int k, int sV, int sH, int sD) {
  constexpr int kPer = 4 / PL;
  constexpr uint32_t kMacro = PL == 1 ? 0xFFu : 0xFFFFu;
  const uint32_t* W = reinterpret_cast<const uint32_t*>(sm.tile);
  const int w0 = xoff / kPer, used = (xoff + ncx) / kPer - w0 + 1;
  uint32_t cnt[kMaxStates];
#pragma unroll
  for (int v = 0; v < kMaxStates; ++v) cnt[v] = 0;
  for (int i = threadIdx.x; i < (ncy + 1) * used; i += 256) {
    const int r = i / used, w = w0 + i - r * used;
    uint32_t x = W[r * (kAnyPitch / kPer) + w], mask = 0;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const int col = kPer * w + e - xoff;
      const bool lr = r == 0 || r == ncy, lc = col == 0 || col == ncx;
      if (col >= 0 && col <= ncx && (!lr || sV < k) && (!lc || sH < k) && (!(lr && lc) || sD < k))
        mask |= kMacro << (8 * PL * e);
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
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(&sm.hist[v], s);
  }
}

// Bound by integer issue where phases are several waves deep, the warps of
// the leading 3-site segments (9 attempts and three Philox calls each) among it;
// a phase's words are drawn before the barrier that ends the one before.  us per
// MCS against the byte tile, 10-MCS counts, M = 1e-4: L = 4800 114.6 -> 90.9 (2.0e11
// -> 2.5e11 site updates/s), 12700 619 -> 406, Moore 115.1 -> 93.8, reflecting 127.6 ->
// 107.8, 6400 x 1600 45.9 -> 35.2; at 2 bits per site 193 -> 93.7, at 4 193 -> 118; S = 5,
// L = 12700 619 -> 478, 8000 287 -> 278, 4800 114.6 -> 115.4 (bytes kept).
template <int PL, int LG, bool REFLECT>
__global__ void __launch_bounds__(256, 4) persistent_macro_any_kernel(const __grid_constant__ PersistentArgs a, int nsx,
                                                                      int nsy, int gp) {
  typedef typename MacroOf<PL>::type MT;
  constexpr int kVec = 16 / PL, kLpr = 4 * PL;   // macros per piece, lanes per tile row
  constexpr int kLoads = (kAnySlots * kLpr + 255) / 256;
  __shared__ AnySmem<PL> sm;
  const LatticeDesc& d = a.d;
  RunState* st = a.st;
  MT* G = reinterpret_cast<MT*>(a.macros);
  const int tid = threadIdx.x;
  const bool run = !ld_volatile(&st->stopped);
  if (run) {
    patch_tables_fill<PL>(sm.T, d, tid, 256);
    for (int i = tid; i < 4 * 256; i += 256) {
      const bool ax = (i >> 8) & 1, ay = (i >> 9) & 1;
      const int Qx = ax ? d.ax.Qa : d.ax.Qb, Qy = ay ? d.ay.Qa : d.ay.Qb, q = i & 255;
      sm.quads[i >> 8][q] = q < (Qx >> 1) * (Qy >> 1)
                                ? quad_entry(q, Qx >> 1, Qy >> 1, block_wide(d.ax, ax), block_wide(d.ay, ay), kAnyPitch, 0)
                                : 0xFFFFFFFFu;
    }
    const int P = d.P, half = P >> 1, Py = d.Py;
    const uint32_t nb = (uint32_t)(P * Py), per = nb >> 2;
    const uint64_t total = (uint64_t)a.n_mcs * nb;
    const uint32_t GQ = (uint32_t)d.GQ, GQy = (uint32_t)(d.ay.r * d.ay.Qa + (Py - d.ay.r) * d.ay.Qb);
    // tickets and flags as in persistent_macro_kernel
    constexpr int kTicketThread = 32;
    uint32_t c_m = 0xFFFFFFFFu, c_ord = 0, t_next = 0, ab_next = 0;
    if (tid == kTicketThread) {
      t_next = atomicAdd(&st->ticket, 1u);
      ab_next = ld_volatile(&st->abort);
    }
    for (;;) {
      if (tid == kTicketThread) {
        const uint32_t t = t_next;
        const uint32_t quit = ((uint64_t)t >= total) || ab_next;
        if (!quit) {
          uint32_t rem, j, jx;
          const uint32_t m = a.m_begin + div_by_rcp(t, nb, a.rcp_nb, rem);
          if (m != c_m) {
            c_m = m;
            c_ord = colour_order(philox10_rk(make_uint4(0u, 0u, m, kTagOrder), d.rk).x, d.perm24);
          }
          sm.ord = c_ord;
          const uint32_t kk = div_by_rcp(rem, per, a.rcp_per, j);
          const uint32_t jy = div_by_rcp(j, (uint32_t)half, a.rcp_half, jx);
          const uint32_t col = (uint32_t)order_at(c_ord, (int)kk);
          sm.dec = make_uint4(m, kk, 2u * jx + (col & 1u), 2u * jy + (col >> 1));
        }
        sm.quit = quit;
        sm.abort = 0;
      }
      if (tid < kMaxStates) sm.hist[tid] = 0;
      __syncthreads();
      if (sm.quit) break;
      const uint4 dec = sm.dec;
      const uint32_t m = dec.x, ord = sm.ord;
      const int k = (int)dec.y, bx = (int)dec.z, by = (int)dec.w, colour = (bx & 1) | ((by & 1) << 1);
      if (tid == kTicketThread) sm.forder = fine_order(d, bx, by, m);
      if (tid < 9) {
        const int dx = tid % 3 - 1, dy = tid / 3 - 1;
        const int ncol = colour ^ ((dx & 1) | ((dy & 1) << 1));
        const uint32_t need = (tid == 4) ? m : (slot_of(ord, ncol) < k ? m + 1u : m);
        const uint32_t* flag = a.done + wrap(by + dy, Py) * P + wrap(bx + dx, P);
        uint32_t spins = 0;
        while (ld_acquire(flag) < need) {
          if ((spins & 15u) == 15u && ld_volatile(&st->abort)) {
            sm.abort = 1;
            break;
          }
          if (++spins > a.spin_limit) {
            atomicOr(&st->error, kErrTimeout);
            atomicExch(&st->abort, 1u);
            sm.abort = 1;
            break;
          }
          __nanosleep(64);
        }
      }
      // the block, while the pollers wait
      const StepKeys key = step_keys(m, d.rk);
      const int sx0 = block_slot(d.ax, bx), sy0 = block_slot(d.ay, by), ncx = block_slots(d.ax, bx), ncy = block_slots(d.ay, by);
      const uint32_t f0x = (uint32_t)(min(bx, d.ax.r) * d.ax.Qa + max(bx - d.ax.r, 0) * d.ax.Qb);
      const uint32_t f0y = (uint32_t)(min(by, d.ay.r) * d.ay.Qa + max(by - d.ay.r, 0) * d.ay.Qb);
      const uint32_t q = sm.quads[(bx < d.ax.r ? 1 : 0) + (by < d.ay.r ? 2 : 0)][tid];
      const int p0 = sx0 / kVec, xoff = sx0 - p0 * kVec;
      const bool wrap_x = sx0 + ncx == nsx;   // the right joint slot is slot 0
      const int np = (xoff + ncx - (wrap_x ? 1 : 0)) / kVec + 1;
      __syncthreads();
      if (sm.abort) break;   // uniform across the CTA
      uint4 v[kLoads];
      uint32_t w[kLoads];
      auto row_at = [&](int i) {
        const int y = sy0 + i / kLpr;
        return G + (size_t)(y == nsy ? 0 : y) * gp;
      };
#pragma unroll
      for (int j = 0; j < kLoads; ++j) {
        const int i = tid + j * 256, p = i % kLpr;
        if (i / kLpr > ncy || p >= np) continue;
        const MT* row = row_at(i);
        v[j] = __ldcg(reinterpret_cast<const uint4*>(row + (p0 + p) * kVec));
        if (wrap_x && p == np - 1) w[j] = __ldcg(row);
      }
      const uint32_t ford = sm.forder;
      PatchItem<PL> I;
      auto draw = [&](int fi) {
        const uint32_t fcol = (ford >> (2 * fi)) & 3u, fx = fcol & 1u, fy = fcol >> 1;
        const uint32_t wc = (q >> (28u + fx)) & 1u, wr = (q >> (30u + fy)) & 1u;
        I.i00 = (int)(q & 0xFFFFu) + xoff + (int)fx + (int)(fx & (q >> 28)) + (fy ? kAnyPitch : 0) +
                (fy & (q >> 30) ? kAnyPitch : 0);
        I.dc = 1 + (int)wc;
        I.dr = wr ? 2 * kAnyPitch : kAnyPitch;
        I.fl = 1u | wc << 1 | wr << 2;
        const uint32_t kx = f0x + 2u * ((q >> 16) & 63u) + fx, ky = f0y + 2u * ((q >> 22) & 63u) + fy;
        if (REFLECT)
          I.fl |= (ky == 0u ? 16u : 0u) | (ky == GQy - 1u ? 32u : 0u) | (kx == 0u ? 64u : 0u) | (kx == GQ - 1u ? 128u : 0u);
        patch_item_draw<PL, LG, REFLECT>(I, key, ky * GQ + kx, m, d.rk, sm.T, d.tx, d.txi);
      };
      const bool item = q != 0xFFFFFFFFu;
      if (item) draw(0);
#pragma unroll
      for (int j = 0; j < kLoads; ++j) {
        const int i = tid + j * 256, r = i / kLpr, p = i % kLpr;
        if (r > ncy || p >= np) continue;
        *reinterpret_cast<uint4*>(sm.tile + r * kAnyPitch + p * kVec) = v[j];
        if (wrap_x && p == np - 1) sm.tile[r * kAnyPitch + xoff + ncx] = (MT)w[j];
      }
      __syncthreads();
#pragma unroll 1
      for (int fi = 0; fi < 4; ++fi) {
        if (item) patch_item_run<PL, LG, REFLECT>(sm.tile, kAnyPitch, I, sm.T, d.tx, d.txi);
        if (item && fi < 3) draw(fi + 1);
        __syncthreads();
      }
      const bool log_point = a.fuse_counts && ((m + 1u) % a.log_every) == 0u;
      if (log_point)
        any_count<PL>(sm, xoff, ncx, ncy, d.S, k, slot_of(ord, colour ^ 2), slot_of(ord, colour ^ 1), slot_of(ord, colour ^ 3));
#pragma unroll
      for (int j = 0; j < kLoads; ++j) {
        const int i = tid + j * 256, r = i / kLpr, p = i % kLpr;
        if (r > ncy || p >= np) continue;
        MT* row = row_at(i);
        *reinterpret_cast<uint4*>(row + (p0 + p) * kVec) = *reinterpret_cast<const uint4*>(sm.tile + r * kAnyPitch + p * kVec);
        if (wrap_x && p == np - 1) row[0] = sm.tile[r * kAnyPitch + xoff + ncx];
      }
      __syncthreads();
      if (tid == 0 && by * P + bx != a.stall_block) st_release(a.done + by * P + bx, m + 1u);
      if (tid == kTicketThread) {
        t_next = atomicAdd(&st->ticket, 1u);
        ab_next = ld_volatile(&st->abort);
      }
      if (log_point) {
        const uint32_t ring = ((m + 1u) / a.log_every) % (uint32_t)kPendRing;
        if (tid >= 1 && tid <= d.S && sm.hist[tid])
          atomicAdd(&st->acc[ring][tid], (unsigned long long)sm.hist[tid]);
        __syncthreads();
        if (tid == 0) flag_log(st, a, m, ring, nb);
      }
    }
  }
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
// Lattice array <-> macros.  One thread moves 16 columns of one row slot: the
// rows 2 ky - 1 and 2 ky (periodic), 8 macros.

// Sites 16 t .. 16 t + 15 of row y as 4 words of bytes.
__device__ __forceinline__ uint4 macro_row16(const LatticeDesc& d, int y, int t) {
  const uint8_t* row = d.lat + (size_t)y * d.pitch;
  if (d.bits == 8) return *(reinterpret_cast<const uint4*>(row) + t);
  if (d.bits == 4) {
    const uint2 w = *(reinterpret_cast<const uint2*>(row) + t);
    return make_uint4(unpack4(w.x, 4), unpack4(w.x >> 16, 4), unpack4(w.y, 4), unpack4(w.y >> 16, 4));
  }
  const uint32_t w = *(reinterpret_cast<const uint32_t*>(row) + t);
  return make_uint4(unpack4(w, 2), unpack4(w >> 8, 2), unpack4(w >> 16, 2), unpack4(w >> 24, 2));
}

// 4 sites (bytes) as 2 PL bits each, first site lowest.
template <int PL>
__device__ __forceinline__ uint32_t macro_pack4(uint32_t w) {
  if (PL == 1) return (w * 0x01041040u) >> 24;   // sites at bits 24, 26, 28, 30 of the product; no carries below
  const uint32_t t = (w | (w >> 4)) & 0x00FF00FFu;
  return (t | (t >> 8)) & 0xFFFFu;
}
// and back
template <int PL>
__device__ __forceinline__ uint32_t macro_unpack4(uint32_t v) {
  return unpack4(v, 2 * PL);
}

template <int PL>
__global__ void __launch_bounds__(256) macro_fill_kernel(LatticeDesc d, typename MacroOf<PL>::type* G, RunState* st) {
  const bool off = macro_fill_off(st);   // asked for before the stores: its load must not hold the others up
  const int nt = d.L >> 4, rows = d.H >> 1;
  const int t = blockIdx.x * blockDim.x + threadIdx.x, ky = blockIdx.y * blockDim.y + threadIdx.y;
  if (t >= nt || ky >= rows) return;
  const int t1 = t == 0 ? nt - 1 : t - 1;
  uint64_t line[2];   // sites 16 t - 1 .. 16 t + 14 of the two rows, 2 PL bits each (PL = 1: the low word)
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int y = h ? 2 * ky : (ky == 0 ? d.H - 1 : 2 * ky - 1);
    const uint4 w = macro_row16(d, y, t);
    const uint32_t prev = macro_row16(d, y, t1).w >> 24;   // site 16 t - 1
    const uint64_t p = (uint64_t)macro_pack4<PL>(w.x) | ((uint64_t)macro_pack4<PL>(w.y) << (8 * PL)) |
                       ((uint64_t)macro_pack4<PL>(w.z) << (16 * PL)) | ((uint64_t)macro_pack4<PL>(w.w) << (24 * PL));
    line[h] = (p << (2 * PL)) | prev;
  }
  if (off) return;
  uint8_t* out = reinterpret_cast<uint8_t*>(G + (size_t)ky * d.GQ + 8 * t);
  if (PL == 1) {
    // nibble i of each row -> byte i
    uint32_t o[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      uint32_t v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t x = (uint32_t)(line[h] >> (16 * q)) & 0xFFFFu;
        x = (x | (x << 8)) & 0x00FF00FFu;
        v[h] = (x | (x << 4)) & 0x0F0F0F0Fu;
      }
      o[q] = v[0] | (v[1] << 4);
    }
    *reinterpret_cast<uint2*>(out) = make_uint2(o[0], o[1]);
  } else {
    const uint32_t a0 = (uint32_t)line[0], a1 = (uint32_t)(line[0] >> 32), b0 = (uint32_t)line[1],
                   b1 = (uint32_t)(line[1] >> 32);
    *reinterpret_cast<uint4*>(out) = make_uint4(__byte_perm(a0, b0, 0x5140), __byte_perm(a0, b0, 0x7362),
                                                __byte_perm(a1, b1, 0x5140), __byte_perm(a1, b1, 0x7362));
  }
}

template <int PL>
__global__ void __launch_bounds__(256) macro_drain_kernel(LatticeDesc d, const typename MacroOf<PL>::type* G,
                                                         const RunState* st) {
  const bool on = st->on_macros != 0u;
  const int nt = d.L >> 4, rows = d.H >> 1;
  const int t = blockIdx.x * blockDim.x + threadIdx.x, ky = blockIdx.y * blockDim.y + threadIdx.y;
  if (t >= nt || ky >= rows) return;
  const typename MacroOf<PL>::type* src = G + (size_t)ky * d.GQ;
  const uint32_t next = src[t == nt - 1 ? 0 : 8 * t + 8];   // holds site 16 t + 15
  uint64_t line[2];
  if (PL == 1) {
    const uint2 m = *reinterpret_cast<const uint2*>(src + 8 * t);
    const uint32_t w[2] = {m.x, m.y};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t x[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t v = (w[q] >> (4 * h)) & 0x0F0F0F0Fu;   // byte i -> nibble i
        v = (v | (v >> 4)) & 0x00FF00FFu;
        x[q] = (v | (v >> 8)) & 0xFFFFu;
      }
      line[h] = (uint64_t)(x[0] | (x[1] << 16)) | ((uint64_t)((next >> (4 * h)) & 15u) << 32);
    }
  } else {
    const uint4 m = *reinterpret_cast<const uint4*>(src + 8 * t);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t sel = h ? 0x7531u : 0x6420u;
      line[h] = (uint64_t)__byte_perm(m.x, m.y, sel) | ((uint64_t)__byte_perm(m.z, m.w, sel) << 32);
    }
  }
  if (!on) return;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    // drop site 16 t - 1, append site 16 t + 15
    uint64_t p = line[h] >> (2 * PL);
    if (PL == 2) p |= (uint64_t)((next >> (8 * h)) & 15u) << 60;
    const uint32_t b0 = macro_unpack4<PL>((uint32_t)p & (PL == 1 ? 0xFFu : 0xFFFFu)),
                   b1 = macro_unpack4<PL>((uint32_t)(p >> (8 * PL)) & (PL == 1 ? 0xFFu : 0xFFFFu)),
                   b2 = macro_unpack4<PL>((uint32_t)(p >> (16 * PL)) & (PL == 1 ? 0xFFu : 0xFFFFu)),
                   b3 = macro_unpack4<PL>((uint32_t)(p >> (24 * PL)) & (PL == 1 ? 0xFFu : 0xFFFFu));
    const int y = h ? 2 * ky : (ky == 0 ? d.H - 1 : 2 * ky - 1);
    uint8_t* row = d.lat + (size_t)y * d.pitch;
    if (d.bits == 8)
      *(reinterpret_cast<uint4*>(row) + t) = make_uint4(b0, b1, b2, b3);
    else if (d.bits == 4)
      *(reinterpret_cast<uint2*>(row) + t) =
          make_uint2(pack4(b0, 4) | (pack4(b1, 4) << 16), pack4(b2, 4) | (pack4(b3, 4) << 16));
    else
      *(reinterpret_cast<uint32_t*>(row) + t) =
          pack4(b0, 2) | (pack4(b1, 2) << 8) | (pack4(b2, 2) << 16) | (pack4(b3, 2) << 24);
  }
}

// ---------------------------------------------------------------------------
cudaError_t launch_macro_fill(const LatticeDesc& d, void* macros, RunState* st, cudaStream_t stream) {
  const dim3 cb(32, 8), cg(((d.L >> 4) + 31) / 32, ((d.H >> 1) + 7) / 8);
  if (patch_planes(d) == 1)
    macro_fill_kernel<1><<<cg, cb, 0, stream>>>(d, reinterpret_cast<uint8_t*>(macros), st);
  else
    macro_fill_kernel<2><<<cg, cb, 0, stream>>>(d, reinterpret_cast<uint16_t*>(macros), st);
  return cudaGetLastError();
}
cudaError_t launch_macro_drain(const LatticeDesc& d, const void* macros, const RunState* st, cudaStream_t stream) {
  const dim3 cb(32, 8), cg(((d.L >> 4) + 31) / 32, ((d.H >> 1) + 7) / 8);
  if (patch_planes(d) == 1)
    macro_drain_kernel<1><<<cg, cb, 0, stream>>>(d, reinterpret_cast<const uint8_t*>(macros), st);
  else
    macro_drain_kernel<2><<<cg, cb, 0, stream>>>(d, reinterpret_cast<const uint16_t*>(macros), st);
  return cudaGetLastError();
}

template <int PL, int NT>
static const void* macro_fn(const LatticeDesc& d) {
#define FLAG_FN(LG, RF) reinterpret_cast<const void*>(&persistent_macro_kernel<PL, LG, RF, NT>)
  if (d.nbh == 8) return d.reflect ? FLAG_FN(3, true) : FLAG_FN(3, false);
  return d.reflect ? FLAG_FN(2, true) : FLAG_FN(2, false);
#undef FLAG_FN
}
static const void* macro_kernel_fn(const LatticeDesc& d, int nt) {
  if (patch_planes(d) == 1) return nt == 128 ? macro_fn<1, 128>(d) : macro_fn<1, 256>(d);
  return nt == 128 ? macro_fn<2, 128>(d) : macro_fn<2, 256>(d);
}

static const void* macro_any_fn(const LatticeDesc& d) {
#define ANY_FN(PL, LG, RF) reinterpret_cast<const void*>(&persistent_macro_any_kernel<PL, LG, RF>)
  if (patch_planes(d) == 1) return d.nbh == 8 ? (d.reflect ? ANY_FN(1, 3, true) : ANY_FN(1, 3, false))
                                              : (d.reflect ? ANY_FN(1, 2, true) : ANY_FN(1, 2, false));
  return d.nbh == 8 ? (d.reflect ? ANY_FN(2, 3, true) : ANY_FN(2, 3, false))
                    : (d.reflect ? ANY_FN(2, 2, true) : ANY_FN(2, 2, false));
#undef ANY_FN
}

int persistent_macro_any_grid(const LatticeDesc& d, int device) {
  if (d.P < 4 || d.Py < 4 || !slot_axis_ok(d.ax) || !slot_axis_ok(d.ay)) return 0;
  const int Qx = d.ax.r > 0 && d.ax.Qa > d.ax.Qb ? d.ax.Qa : d.ax.Qb, Qy = d.ay.r > 0 && d.ay.Qa > d.ay.Qb ? d.ay.Qa : d.ay.Qb;
  if ((Qx >> 1) * (Qy >> 1) > 256) return 0;
  int sms = 0, occ = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, macro_any_fn(d), 256, 0) != cudaSuccess) return 0;
  const int grid = sms * (occ < 4 ? occ : 4);
  // Where it beats the flag kernel on bytes: with 2 bits per site (S <= 3), the
  // reflecting boundary only once a phase is two waves deep (mirrored steps
  // lengthened the chain, L = 800, Moore, 44.1 -> 52.5 us per MCS, before their
  // entries came from a table; not measured since); with 4 bits only
  // past half of the L2, where the bytes no longer stay.  Packed lattices, whose
  // byte tiles cost a conversion each way, always.
  if (d.bits == 8) {
    const bool deep = (int64_t)d.P * d.Py / 4 >= 2 * (int64_t)grid;
    if (patch_planes(d) == 1 ? d.reflect && !deep : d.reflect || (size_t)d.H * d.pitch < (64u << 20)) return 0;
  }
  return grid;
}

int persistent_macro_grid(const LatticeDesc& d, int device, int threads) {
  int sms = 0, occ = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, macro_kernel_fn(d, threads), threads, 0) != cudaSuccess)
    return 0;
  const int cap = threads == 128 ? 8 : 4;
  return sms * (occ < cap ? occ : cap);
}

// A call pays for two conversions (15 us at L = 3200, 300 at 12700), which the
// macros win back at some us per MCS.  Calls below the lines run on bytes.  us per
// MCS of calls of n MCS on bytes and on macros (M = 1e-4 unless stated), the line
// where they meet:
//  * owners: L = 800 n = 1 40.4, 47.5, n = 2 31.7, 33.2, n = 3 29.1, 28.5, n = 5 26.8, 23.5;
//    L = 400 n = 2 33.7, 31.8; L = 2200 Moore 53.5, 64.9 / 45.0, 46.4 / 43.4, 40.0, L = 1600
//    n = 2 48.3, 45.4.  On 64 x 64 blocks with a reflecting
//    boundary n = 1 already gains (L = 1024 1.15 x).
//  * flags, 64 x 64 blocks, 2 bits per site: L = 3200 34.1, 39.6 / 29.4, 29.1 / 25.3,
//    22.7; the Moore bytes are slower and meet at 1 (39.3, 40.5), deep phases (L = 6400)
//    too.
//  * the same at 4 bits: L = 3200 meets at 5 to 8 (26.5 each at n = 5), Moore at 3,
//    reflecting at 5; deep ones at 2 (82.8, 81.2).  With few exchanges (M = 0: every
//    step takes the rule table) the macros gain 0 to 5 % at n = 20 and lose at 10.
//  * packed lattices: the bytes pay a conversion in every visit; the rule variants
//    and ragged blocks always gain (L = 3333, 2 bits, n = 1 1.3 x).
//  * other partitions: L = 3333 56.4, 72.6 / 51.6, 52.7 / n = 3 1.08 x; L = 12700 629, 689 /
//    624, 540.
uint32_t macro_min_mcs(const LatticeDesc& d, bool group, bool deep) {
  const bool one = patch_planes(d) == 1, moore = d.nbh == 8, refl = d.reflect != 0;
  const bool few = d.tx < 0x80000000u;   // fewer than half the attempts exchange
  if (group) {
    if (d.blocks64 && refl) return 1u;
    return !few && (size_t)d.H * d.L > (moore ? 1u << 22 : 1u << 18) ? 3u : 2u;
  }
  if (!d.blocks64) return d.bits != 8 ? 1u : ((size_t)d.H * d.L >= (32u << 20) ? 2u : 3u);
  if (d.bits != 8) {
    if (moore || refl) return 1u;
    return one ? (deep ? 1u : 2u) : (few ? 5u : (deep ? 2u : 3u));
  }
  if (one) return deep || (moore && !refl) ? 1u : 2u;
  if (refl) return moore && deep ? 3u : 5u;
  if (moore) return deep ? 1u : 3u;
  return few ? 16u : (deep ? 2u : 6u);
}

cudaError_t launch_persistent_macro(const PersistentArgs& args, int grid, cudaStream_t stream) {
  PersistentArgs a = args;
  const uint32_t nb = (uint32_t)(a.d.P * a.d.Py);
  a.rcp_nb = div_rcp32(nb);
  a.rcp_per = div_rcp32(nb >> 2);
  a.rcp_half = div_rcp32((uint32_t)(a.d.P >> 1));
  const bool any = !a.d.blocks64;
  cudaError_t e = cudaSuccess;
  if (a.fill)
    e = any ? launch_macro_fill_any(a.d, a.macros, a.st, stream) : launch_macro_fill(a.d, a.macros, a.st, stream);
  if (e != cudaSuccess) return e;
  if (any) {
    int nsx = axis_slots(a.d.ax, a.d.P), nsy = axis_slots(a.d.ay, a.d.Py), gp = macro_pitch(a.d);
    void* params[] = {&a, &nsx, &nsy, &gp};
    e = cudaLaunchKernel(macro_any_fn(a.d), dim3(grid), dim3(256), params, 0, stream);
  } else {
    void* params[] = {&a};
    e = cudaLaunchKernel(macro_kernel_fn(a.d, a.threads), dim3(grid), dim3(a.threads), params, 0, stream);
  }
  if (e != cudaSuccess || !a.drain) return e;
  return any ? launch_macro_drain_any(a.d, a.macros, a.st, stream) : launch_macro_drain(a.d, a.macros, a.st, stream);
}

}  // namespace escg_impl
