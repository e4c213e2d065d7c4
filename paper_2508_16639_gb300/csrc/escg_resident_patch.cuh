// escg_resident_patch.cuh -- whole-lattice residency on the macro layout of
// escg_patch.cuh: one CTA holds the lattice in shared memory, 2 bits per site
// and plane, for every coarse phase of a launch.
//
// A coarse phase runs the blocks of one colour side by side, a fine phase one
// sub-block of every quad of them, one CTA barrier per fine phase and no
// other: the joint slot 0 of an axis holds the lattice's last and first site,
// so a periodic lattice has no halo to refresh or to write back.  What a fine
// phase has to wait for is four macro loads and the chain of its longest
// sub-block's steps; which sub-block, its random words and their table entries
// do not depend on the lattice.  So the threads form 1 to 8 groups that take
// the phases in turn: a group works out its next phase's first sub-block per
// thread while the other groups run theirs, and a named barrier hands the
// macros on.  A lattice whose phases fill the CTA has one group, which works
// one sub-block ahead.
#pragma once

#include "escg_patch.cuh"
#include "escg_sync.cuh"

namespace escg_impl {

struct ResidentPatchSmem {
  PatchTables T;
  uint32_t hist[kMaxStates];
  uint32_t stop;
  int32_t nq[2][2], nr[2][2];   // [axis][parity]: quads and regular quads
  int32_t n[4];                 // by colour: items of a fine phase
};

// Dynamic shared memory: the macros, the items' table, the tables of both axes.
// A lattice of more than kResPatchBytes stays on the one-byte image.
constexpr int kResPatchBytes = 222 * 1024;
struct ResidentLayout {
  int nsx, nsy, pitch;               // slots, macros per row (whole 32-bit words)
  int items;                         // entries of a colour in the items' table (whole warps)
  int table, segx, segy, quadx, quady, slx, sly, mapx, mapy, fo, bytes;   // byte offsets
};

// Sub-blocks of one fine phase, at most (the threads a launch can use).
__host__ __device__ inline int resident_phase_items(const AxisGeom& ax, int P, const AxisGeom& ay, int Py) {
  int n = 0;
  for (int cy = 0; cy < 2; ++cy)
    for (int cx = 0; cx < 2; ++cx) {
      int qx, rx, qy, ry;
      axis_quads(ax, P, cx, &qx, &rx);
      axis_quads(ay, Py, cy, &qy, &ry);
      if (qx * qy > n) n = qx * qy;
    }
  return n;
}

__host__ __device__ inline ResidentLayout resident_layout(const AxisGeom& ax, int P, int L, const AxisGeom& ay, int Py,
                                                          int H, int planes) {
  ResidentLayout R;
  R.nsx = axis_slots(ax, P);
  R.nsy = axis_slots(ay, Py);
  R.pitch = planes == 1 ? (R.nsx + 3) & ~3 : (R.nsx + 1) & ~1;
  const int gx = ax.r * ax.Qa + (P - ax.r) * ax.Qb, gy = ay.r * ay.Qa + (Py - ay.r) * ay.Qb;
  R.items = (resident_phase_items(ax, P, ay, Py) + 31) & ~31;
  int o = (R.nsy * R.pitch * planes + 15) & ~15;
  R.table = o;
  R.segx = o += 32 * R.items;
  R.segy = o += 4 * gx;
  R.quadx = o += 4 * gy;
  R.quady = o += 2 * gx;
  R.slx = o += 2 * gy;
  R.sly = o += 4 * R.nsx;
  R.mapx = o += 4 * R.nsy;
  R.mapy = o += 2 * ((L + 1) & ~1);
  R.fo = o += 2 * ((H + 1) & ~1);
  R.bytes = (o + 2 * P * Py + 15) & ~15;
  if (R.nsy * R.pitch > 65536) R.bytes = 1 << 30;   // past the items' macro indexes
  return R;
}
__host__ __device__ inline ResidentLayout resident_layout(const LatticeDesc& d, int planes) {
  return resident_layout(d.ax, d.P, d.L, d.ay, d.Py, d.H, planes);
}

// Tables of one axis (n sites, P blocks): segment k -> left joint slot |
// right joint slot << 12 | 3 wide << 24; quad position -> left joint slot |
// first segment << 12 | block / 2 << 24, the quads of parity 0, then those of
// parity 1; slot -> its sites (half 0 | half 1 << 16, 0xFFFF none); site -> 2 slot + half.
__device__ __forceinline__ void resident_axis(const AxisGeom& g, int P, int n, uint32_t* seg, uint32_t* quad,
                                              uint32_t* sl, uint16_t* map, int32_t* nq, int32_t* nr) {
  const int G = g.r * g.Qa + (P - g.r) * g.Qb;
  for (int k = threadIdx.x; k < G; k += blockDim.x) {
    int slot, first;
    bool wide;
    axis_segment(g, k, slot, wide, first);
    const int next = slot + 1 + (wide ? 1 : 0), right = k + 1 == G ? 0 : next;
    seg[k] = (uint32_t)slot | ((uint32_t)right << 12) | (wide ? 1u << 24 : 0u);
    sl[slot] = (uint32_t)(first == 0 ? n - 1 : first - 1) | ((uint32_t)first << 16);
    map[first] = (uint16_t)(2 * slot + 1);
    if (wide) {
      sl[slot + 1] = (uint32_t)(first + 1) | 0xFFFF0000u;
      map[first + 1] = (uint16_t)(2 * (slot + 1));
    }
    map[first + (wide ? 2 : 1)] = (uint16_t)(2 * right);
  }
  int t0, r0;
  axis_quads(g, P, 0, &t0, &r0);
  for (int k = threadIdx.x; k < G / 2; k += blockDim.x) {
    int b, s, pos, slot, first;
    bool wide;
    axis_quad(g, P, k, b, s, pos);
    axis_segment(g, s, slot, wide, first);
    quad[((b & 1) ? t0 : 0) + pos] = (uint32_t)slot | ((uint32_t)s << 12) | ((uint32_t)(b >> 1) << 24);
  }
  if (threadIdx.x < 2) {
    int t, r;
    axis_quads(g, P, (int)threadIdx.x, &t, &r);
    nq[threadIdx.x] = t;
    nr[threadIdx.x] = r;
  }
}

// Everything a launch needs besides the macros.  Ends without a barrier.
template <int PL>
__device__ __forceinline__ void resident_setup(const LatticeDesc& d, const ResidentLayout& R, uint8_t* dyn,
                                               ResidentPatchSmem& S) {
  patch_tables_fill<PL>(S.T, d, threadIdx.x, blockDim.x);
  resident_axis(d.ax, d.P, d.L, reinterpret_cast<uint32_t*>(dyn + R.segx), reinterpret_cast<uint32_t*>(dyn + R.quadx),
                reinterpret_cast<uint32_t*>(dyn + R.slx), reinterpret_cast<uint16_t*>(dyn + R.mapx), S.nq[0], S.nr[0]);
  resident_axis(d.ay, d.Py, d.H, reinterpret_cast<uint32_t*>(dyn + R.segy), reinterpret_cast<uint32_t*>(dyn + R.quady),
                reinterpret_cast<uint32_t*>(dyn + R.sly), reinterpret_cast<uint16_t*>(dyn + R.mapy), S.nq[1], S.nr[1]);
  __syncthreads();
  // The items of each colour, a quad each: regular quads first, then the rows
  // and the columns of the others.  x: top left macro (16 bits) | 3-site
  // segments (columns 2 qx, 2 qx + 1 at bits 16, 17, rows at 18, 19) | last column
  // (20) and row (21), first column (22) and row (23) of the lattice | present
  // (31); y: sub-block of fine colour 0 | block << 24.  Worked out here once: an
  // item is 25 instructions of a fine phase otherwise.
  uint2* table = reinterpret_cast<uint2*>(dyn + R.table);
  const uint32_t* segx = reinterpret_cast<const uint32_t*>(dyn + R.segx);
  const uint32_t* segy = reinterpret_cast<const uint32_t*>(dyn + R.segy);
  const uint32_t* quadx = reinterpret_cast<const uint32_t*>(dyn + R.quadx);
  const uint32_t* quady = reinterpret_cast<const uint32_t*>(dyn + R.quady);
  const int GQ = d.GQ, GQy = d.ay.r * d.ay.Qa + (d.Py - d.ay.r) * d.ay.Qb;
  if (threadIdx.x < 4) S.n[threadIdx.x] = S.nq[0][threadIdx.x & 1u] * S.nq[1][threadIdx.x >> 1];
  for (int i = threadIdx.x; i < 4 * R.items; i += blockDim.x) {
    const int c = i / R.items, it = i - c * R.items, cx = c & 1, cy = c >> 1;
    const int nqx = S.nq[0][cx], nqy = S.nq[1][cy], rx = S.nr[0][cx], ry = S.nr[1][cy];
    uint2 v = make_uint2(0u, 0u);
    if (it < nqx * nqy) {
      const int k = it - rx * ry, top = nqx * (nqy - ry);
      int px, py;
      if (k < 0) {
        py = it / rx;
        px = it - py * rx;
      } else if (k < top) {
        py = k / nqx;
        px = k - py * nqx;
        py += ry;
      } else {
        py = (k - top) / (nqx - rx);
        px = k - top - py * (nqx - rx) + rx;
      }
      const uint32_t qx = quadx[(cx ? S.nq[0][0] : 0) + px], qy = quady[(cy ? S.nq[1][0] : 0) + py];
      const uint32_t kx = (qx >> 12) & 0xFFFu, ky = (qy >> 12) & 0xFFFu;
      const uint32_t blk = (2u * (qy >> 24) + (uint32_t)cy) * (uint32_t)d.P + 2u * (qx >> 24) + (uint32_t)cx;
      v.x = ((qy & 0xFFFu) * (uint32_t)R.pitch + (qx & 0xFFFu)) | (segx[kx] >> 24) << 16 | (segx[kx + 1] >> 24) << 17 |
            (segy[ky] >> 24) << 18 | (segy[ky + 1] >> 24) << 19 | ((int)kx + 2 == GQ ? 1u << 20 : 0u) |
            ((int)ky + 2 == GQy ? 1u << 21 : 0u) | (kx == 0u ? 1u << 22 : 0u) | (ky == 0u ? 1u << 23 : 0u) | 1u << 31;
      v.y = (ky * (uint32_t)GQ + kx) | blk << 24;
    }
    table[i] = v;
  }
}

__device__ __forceinline__ uint32_t load_site(const LatticeDesc& d, uint32_t row, uint32_t col) {
  const uint8_t* p = d.lat + (size_t)row * d.pitch;
  if (d.bits == 8) return __ldcg(p + col);
  const uint32_t bit = col * (uint32_t)d.bits;
  return ((uint32_t)__ldcg(p + (bit >> 3)) >> (bit & 7u)) & ((1u << d.bits) - 1u);
}

// Lattice array -> macros (a row slot per warp and pass).
template <int PL>
__device__ __forceinline__ void resident_fill(const LatticeDesc& d, const ResidentLayout& R, uint8_t* dyn) {
  typedef typename MacroOf<PL>::type MT;
  MT* M = reinterpret_cast<MT*>(dyn);
  const uint32_t* slx = reinterpret_cast<const uint32_t*>(dyn + R.slx);
  const uint32_t* sly = reinterpret_cast<const uint32_t*>(dyn + R.sly);
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int r = threadIdx.x >> 5; r < R.nsy; r += nw) {
    const uint32_t ys = sly[r], r0 = ys & 0xFFFFu, r1 = ys >> 16;
    for (int c = lane; c < R.pitch; c += 32) {
      uint32_t v[4] = {0u, 0u, 0u, 0u};
      if (c < R.nsx) {
        const uint32_t xs = slx[c], c0 = xs & 0xFFFFu, c1 = xs >> 16;
        v[0] = load_site(d, r0, c0);
        if (c1 != 0xFFFFu) v[1] = load_site(d, r0, c1);
        if (r1 != 0xFFFFu) {
          v[2] = load_site(d, r1, c0);
          if (c1 != 0xFFFFu) v[3] = load_site(d, r1, c1);
        }
      }
      M[r * R.pitch + c] = (MT)(v[0] | (v[1] << (2 * PL)) | (v[2] << (4 * PL)) | (v[3] << (6 * PL)));
    }
  }
}

// Macros -> lattice array, one group of 4 sites per lane and pass (sites past
// column L written as 0, as in the staging of one-byte images).
template <int PL>
__device__ __forceinline__ void resident_drain(const LatticeDesc& d, const ResidentLayout& R, const uint8_t* dyn) {
  typedef typename MacroOf<PL>::type MT;
  const MT* M = reinterpret_cast<const MT*>(dyn);
  const uint16_t* mapx = reinterpret_cast<const uint16_t*>(dyn + R.mapx);
  const uint16_t* mapy = reinterpret_cast<const uint16_t*>(dyn + R.mapy);
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int r = threadIdx.x >> 5; r < d.H; r += nw) {
    const uint32_t my = mapy[r];
    const MT* row = M + (my >> 1) * R.pitch;
    for (int c0 = 4 * lane; c0 < d.L; c0 += 128) {
      uint32_t u = 0;
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (c0 + e < d.L) {
          const uint32_t mx = mapx[c0 + e], field = 2u * (my & 1u) + (mx & 1u);
          u |= (((uint32_t)row[mx >> 1] >> (2 * PL * field)) & (PL == 1 ? 3u : 15u)) << (8 * e);
        }
      store_group(d.lat + (size_t)r * d.pitch, c0, d.bits, pack4(u, d.bits));
    }
  }
}

// Barrier of the nthr threads that run a resident lattice (barriers 1 .. 8 hand
// its phases on).
__device__ __forceinline__ void res_sync(uint32_t nthr) { bar_named(14u, nthr); }

// Species histogram of the macros into S.hist.  Unused fields hold 0, so the
// empty sites are counted as the rest.
template <int PL>
__device__ __forceinline__ void resident_count_macros(const LatticeDesc& d, const ResidentLayout& R, const uint8_t* dyn,
                                                      ResidentPatchSmem& S, uint32_t nthr) {
  if (threadIdx.x < kMaxStates) S.hist[threadIdx.x] = 0;
  res_sync(nthr);
  const uint32_t* W = reinterpret_cast<const uint32_t*>(dyn);
  const int words = R.nsy * R.pitch * PL / 4;
  uint32_t c[kMaxStates];
#pragma unroll
  for (int v = 0; v < kMaxStates; ++v) c[v] = 0;
  for (int k = threadIdx.x; k < words; k += (int)nthr) {
    const uint32_t x = W[k];
#pragma unroll
    for (int v = 1; v < (PL == 1 ? 4 : kMaxStates); ++v) {
      if (v > d.S) break;
      if (PL == 1) {
        const uint32_t t = x ^ (uint32_t)(v * 0x55555555u);
        c[v] += __popc(~(t | (t >> 1)) & 0x55555555u);
      } else {
        const uint32_t t = x ^ (uint32_t)(v * 0x11111111u), n = t | (t >> 1);
        c[v] += __popc(~(n | (n >> 2)) & 0x11111111u);
      }
    }
  }
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int v = 1; v < (PL == 1 ? 4 : kMaxStates); ++v) {
    if (v > d.S) break;
    const uint32_t s = __reduce_add_sync(0xFFFFFFFFu, c[v]);
    if (lane == 0 && s) atomicAdd(&S.hist[v], s);
  }
  res_sync(nthr);
  if (threadIdx.x == 0) {
    uint32_t rest = (uint32_t)(d.L * d.H);
    for (int v = 1; v <= d.S; ++v) rest -= S.hist[v];
    S.hist[0] = rest;
  }
  res_sync(nthr);
}

// Threads of a group (whole warps) and of a launch of at most max_threads: a
// power of two of groups, so that a group takes the same phases of every MCS.
constexpr int kResMaxGroups = 8;
__host__ __device__ inline void resident_threads(const LatticeDesc& d, int max_threads, int* gs, int* nt) {
  int g = (resident_phase_items(d.ax, d.P, d.ay, d.Py) + 31) & ~31;
  if (g > max_threads) g = max_threads;
  int k = 1;
  while (2 * k <= kResMaxGroups && 2 * k * g <= max_threads) k *= 2;
  *gs = g;
  *nt = k * g;
}

// MCS [m_begin, m_end) on the resident macros, by threads 0 .. nthr - 1 in groups of
// gs; rk: the round keys; on_log as in resident_run of the
// one-byte image.  Returns the MCS
// reached.
template <int PL, int LG, bool REFLECT, class RK, class OnLog>
__device__ uint32_t resident_run_patch(const LatticeDesc& d, RK rk, const ResidentLayout& R, uint8_t* dyn,
                                       ResidentPatchSmem& S, int gs, uint32_t nthr, uint32_t m_begin, uint32_t m_end,
                                       uint32_t log_every, OnLog on_log) {
  typedef typename MacroOf<PL>::type MT;
  MT* M = reinterpret_cast<MT*>(dyn);
  const uint2* table = reinterpret_cast<const uint2*>(dyn + R.table);
  uint8_t* fo = dyn + R.fo;
  const int grp = (int)threadIdx.x / gs, tid = (int)threadIdx.x - grp * gs, groups = (int)nthr / gs;
  const int nblk = d.P * d.Py, pitch = R.pitch;
  const uint32_t tx = d.tx, txi = d.txi, GQ = (uint32_t)d.GQ;

  // item `it` of fine phase fi of coarse colour `colour` in MCS m
  auto prepare = [&](PatchItem<PL>& I, int it, int colour, int fi, uint32_t m, const StepKeys& key) {
    const uint2 e = table[colour * R.items + it];
    I.fl = e.x >> 31;
    if (!I.fl) return;
    // fine order of the quad's block
    const uint32_t fcol = (uint32_t)fo[(m & 1u) * nblk + (e.y >> 24)] >> (2 * fi), fx = fcol & 1u, fy = (fcol >> 1) & 1u;
    const uint32_t wide = e.x >> 16, wc = (wide >> fx) & 1u, wr = (wide >> (2u + fy)) & 1u;
    I.i00 = (int)((e.x & 0xFFFFu) + fx + (fx & wide)) + (fy ? ((wide & 4u) ? 2 * pitch : pitch) : 0);
    I.dc = 1 + (int)wc - ((fx & (e.x >> 20)) ? R.nsx : 0);   // the last column's right joint is slot 0
    I.dr = (1 + (int)wr - ((fy & (e.x >> 21)) ? R.nsy : 0)) * pitch;
    I.fl |= wc << 1 | wr << 2;
    if (REFLECT)
      I.fl |= ((e.x >> 23) & (fy ^ 1u) & 1u) << 4 | ((e.x >> 21) & fy) << 5 | ((e.x >> 22) & (fx ^ 1u) & 1u) << 6 |
              ((e.x >> 20) & fx) << 7;
    patch_item_draw<PL, LG, REFLECT>(I, key, (e.y & 0xFFFFFFu) + fy * GQ + fx, m, rk, S.T, tx, txi);
  };

  auto orders = [&](uint32_t m, int t, int n) {   // the blocks' fine orders of MCS m
    for (int b = t; b < nblk; b += n)
      fo[(m & 1u) * nblk + b] =
          (uint8_t)colour_order(philox10_rk(make_uint4(0u, (uint32_t)b, m, kTagFineOrder), rk).x, d.perm24);
  };
  auto order = [&](uint32_t m) {
    return colour_order(philox10_rk(make_uint4(0u, 0u, m, kTagOrder), rk).x, d.perm24);
  };

  orders(m_begin, (int)threadIdx.x, (int)nthr);
  uint32_t ord = order(m_begin);
  StepKeys key = step_keys(m_begin, rk);
  res_sync(nthr);
  PatchItem<PL> cur;
  prepare(cur, tid, order_at(ord, grp >> 2), grp & 3, m_begin, key);
  bool handed = false;   // the last phase ended with a CTA barrier instead of a hand-over
  uint32_t m = m_begin;
  for (; m < m_end; ++m) {
    const uint32_t ord_next = order(m + 1u);
    const StepKeys key_next = step_keys(m + 1u, rk);
    const bool log_point = ((m + 1u) % log_every) == 0u, joined = log_point || m + 1u == m_end;
#pragma unroll 1
    for (int ph = grp; ph < 16; ph += groups) {
      // the macros as the phase before left them
      if (groups == 1)
        res_sync(nthr);
      else if (ph > 0 || handed)
        bar_named((uint32_t)(1 + grp), (uint32_t)(2 * gs));
      const int colour = order_at(ord, ph >> 2), fi = ph & 3;
      const int n = S.n[colour];
      const int phn = (ph + groups) & 15;   // this group's next phase
      const bool wrap = ph + groups > 15;
      const int colour_n = order_at(wrap ? ord_next : ord, phn >> 2);
      for (int it = tid;; it += gs) {
        // the macros first, then what the other groups' phases hide
        const bool more = it + gs < n;
        if (cur.fl) patch_item_run<PL, LG, REFLECT>(M, pitch, cur, S.T, tx, txi);
        if (groups > 1 && !more && !(joined && ph == 15))
          bar_arrive((uint32_t)(grp + 1 == groups ? 1 : 2 + grp), (uint32_t)(2 * gs));
        const bool nm = wrap && !more;
        prepare(cur, more ? it + gs : tid, more ? colour : colour_n, more ? fi : phn & 3, nm ? m + 1u : m,
                      nm ? key_next : key);
        if (!more) break;
      }
      // read from this MCS's last phases on; the buffer's previous content
      // was last read before phase 0 began
      if (ph == 0) orders(m + 1u, tid, gs);
    }
    handed = !joined;
    ord = ord_next;
    key = key_next;
    if (log_point) {
      res_sync(nthr);
      resident_count_macros<PL>(d, R, dyn, S, nthr);
      if (threadIdx.x == 0) S.stop = on_log(m + 1u, S.hist) ? 1u : 0u;
      res_sync(nthr);
      if (S.stop) {
        ++m;
        break;
      }
    }
  }
  res_sync(nthr);
  return m;
}

}  // namespace escg_impl
