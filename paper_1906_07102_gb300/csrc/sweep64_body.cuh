// Gridding and degridding sweeps of complex128 plans.
//
// A GB300 SM retires about two float64 FMAs a cycle, so one warp FMA holds the SM's float64 pipe
// for some 16 cycles, busy lanes or not: these sweeps are bound by the number of float64 warp
// instructions, and shared memory, integer work and issue are nearly free beside them. So the lanes
// of a warp take the cells of one record's W x W support together (the float32 sweeps' lanes each
// own columns, and wait for the lane with the most records), and the rows they add into or read
// sit in shared memory:
//   * a warp owns a work item (records of some rows of one 32-column strip, sorted by pairs of
//     support-start rows) and holds a ring of W + 1 rows (an even number of slots) of the strip and
//     the W - 1 columns past it, so that no record needs a second copy in the next strip;
//   * 32 records at a time: each lane computes its record's table row, fraction or Lagrange basis
//     and weighted visibility; then 8 records at a time the weights, EW lanes for each axis of a
//     record reading consecutive table entries (rows at random s would each cost a line per lane);
//   * gridding: cell n of the support belongs to lane n mod 32 (ceil(W^2 / 32) cells a lane), each
//     adding Cv_r x (Cu_c w V) in shared memory, two FMAs a cell; rows leave the ring by reductions
//     into the zeroed grid, where neighbouring strips and items overlap;
//   * degridding: lane g W + c sums column c over the rows g, g + G, .. (G = min(32 / W, W)), and
//     four lanes add up a record's partial sums, weighted by Cu.
// Measured against the float32 sweeps' scheme in float64 (one column a lane, ring in registers),
// gridding and degridding in us: 1.03M visibilities, W = 14 cubic, 2048^2: 3194 + 3017 -> 1311 + 1320;
// 0.81M, W = 7 linear, 2048^2: 726 + 827 -> 349 + 400; 0.40M, W = 9, 256^2: 2450 + 2931 -> 275 + 277;
// 0.40M, W = 6, 1024^2: 382 + 458 -> 186 + 221. W = 14 takes about 20 float64 warp instructions a
// record, 325 cycles of an SM's pipe, 1.2 ms in all: the pipe is what bounds it.
#pragma once

#include "sweep_body.cuh"

namespace lmg {
namespace {

constexpr int kThreads64 = 64;  // two warps a CTA: the granularity in which shared memory fills the SM
constexpr int kWarps64 = kThreads64 / 32;
constexpr int kSub = 8;         // records whose weights are staged together

template <int W> struct Lay64 {
  static constexpr int S = strip_width(1);
  static constexpr int RR = (W + 2) & ~1;                    // ring rows: W + 1 rounded up to even
  static constexpr int COLS = S + W - 1;
  static constexpr int TS = COLS + ((W - COLS) % 8 + 8) % 8;  // pitch = W mod 8: cells of successive
                                                              // rows go on through the banks
  static constexpr int EW = W <= 4 ? 4 : (W <= 8 ? 8 : 16);  // lanes a record's axis takes
  static constexpr int RPS = 16 / EW;                        // records a lookup step takes
  static constexpr int NI = (W * W + 31) / 32;               // gridding: cells a lane
  static constexpr int G = 32 / W < W ? 32 / W : W;          // degridding: row groups
  static constexpr int NR = (W + G - 1) / G;                 // rows a lane
  static constexpr int PP = 36;                              // partial sums of a record (pitch)
  // byte offsets in a warp's shared memory
  static constexpr int ring = 0;
  static constexpr int basis = ring + RR * TS * 16;          // [axis][4][32] fraction or Lagrange basis
  static constexpr int val = basis + 2 * 4 * 32 * 8;         // [32] weighted visibility
  static constexpr int off = val + 32 * 16;                  // [axis][32] table offset
  static constexpr int cv = off + 2 * 32 * 4;                // [kSub][EW] Cv
  static constexpr int cu = cv + kSub * EW * 8;              // [kSub][EW] Cu w V, or (degridding) Cu
  static constexpr int part = cu + kSub * EW * 8;            // [kSub][PP] partial sums (degridding)
  static constexpr int grid_bytes = cu + kSub * EW * 16;
  static constexpr int degrid_bytes = part + kSub * PP * 16;
};

// Table offset and the numbers that the lookups of one axis need of a record: the fraction
// (linear), s (direct calculation) or the Lagrange basis at the local coordinate f (the products
// of lagrange_entry, shared by the axis' W entries).
template <bool EXT>
__device__ __forceinline__ void stage_basis(int interp, double f, double* __restrict__ b) {
  if constexpr (EXT) {
    if (interp == 2 || interp == 3) {
      const double x = f, y = f - 1.0, z = f - 2.0;
      if (interp == 2) {
        b[0] = 0.5 * y * z;
        b[32] = -x * z;
        b[64] = 0.5 * x * y;
      } else {
        const double e = f - 3.0, sixth = 1.0 / 6.0;
        b[0] = -sixth * y * z * e;
        b[32] = 0.5 * x * z * e;
        b[64] = -0.5 * x * y * e;
        b[96] = sixth * x * y * z;
      }
      return;
    }
  }
  b[0] = f;
}

// Entry e of the weights of one axis at table offset `off` with basis b (stage_basis).
template <int W, bool EXT>
__device__ __forceinline__ double weight64(const double* __restrict__ tab, int Wp, int interp, int off, int e,
                                           const double* __restrict__ b) {
  if constexpr (EXT) {
    if constexpr (W <= 11) {
      if (interp == 4) return direct_entry(tab, W, e, b[0]);
    }
    const double* p = tab + off + e;
    const double c = b[0] * p[0] + b[32] * p[Wp] + b[64] * p[2 * Wp];
    return interp == 3 ? c + b[96] * p[3 * Wp] : c;
  } else {
    const double* p = tab + off + e;
    const double a = p[0];
    return interp ? a + b[0] * (p[Wp] - a) : a;
  }
}

// The weights of records s0 .. s0 + kSub - 1 of the window (those below n), staged at s_cv and
// s_cu: with GRID the latter times the record's weighted visibility.
template <int W, bool EXT, bool GRID>
__device__ __forceinline__ void stage_weights(const double* __restrict__ tab, int Wp, int interp, unsigned char* my,
                                              int s0, int n, int lane) {
  using L = Lay64<W>;
  const int rp = lane / (2 * L::EW), axis = (lane / L::EW) & 1, e = lane % L::EW;
  const int* off = reinterpret_cast<const int*>(my + L::off) + 32 * axis;
  const double* basis = reinterpret_cast<const double*>(my + L::basis) + 128 * axis;
  const double* val = reinterpret_cast<const double*>(my + L::val);
  double* cv = reinterpret_cast<double*>(my + L::cv);
  double* cu = reinterpret_cast<double*>(my + L::cu);
#pragma unroll
  for (int k = 0; k < kSub; k += L::RPS) {
    const int s = k + rp, l = s0 + s;
    double c = 0.0;
    if (l < n && e < W) c = weight64<W, EXT>(tab, Wp, interp, off[l], e, basis + l);
    if constexpr (GRID) {
      // Cu w V: the lanes of the u axis take the real parts, those of the v axis the imaginary
      const double u = __shfl_sync(0xffffffffu, c, lane & ~L::EW);
      if (l < n) {
        if (axis) cv[s * L::EW + e] = c;
        cu[(s * L::EW + e) * 2 + axis] = u * val[2 * l + axis];
      }
    } else if (l < n) {
      (axis ? cv : cu)[s * L::EW + e] = c;
    }
  }
}

// W = 1: a record is one cell, so a lane takes a whole record, 32 at a time; a record at a time would
// leave 31 lanes idle. Gridding and degridding in us, a record at a time and now: 1.0M visibilities,
// nearest, 512^2: 222 + 226 -> 80 + 64; 4.0M, 4096^2: 906 + 844 -> 356 + 247.
// The weights' product with the record's value: c = Cv (Cu x), Cu and Cv from the lane's own basis.
template <bool EXT>
__device__ __forceinline__ void lane_weights(const SweepArgs& a, unsigned char* my, const Rec& rc, int lane, double& cu,
                                             double& cv) {
  const double* tab = static_cast<const double*>(a.table);
  double* basis = reinterpret_cast<double*>(my + Lay64<1>::basis) + lane;
  int ou, ov;
  double fu, fv;
  record_coords<double, EXT>(a, rc, ou, fu, ov, fv);
  stage_basis<EXT>(a.interp, fu, basis);
  stage_basis<EXT>(a.interp, fv, basis + 128);
  cu = weight64<1, EXT>(tab, a.Wp, a.interp, ou, 0, basis);
  cv = weight64<1, EXT>(tab, a.Wp, a.interp, ov, 0, basis + 128);
}

// Gridding: the records of one pair of rows are added into the pair's cells, those of one cell one
// after another in the order of their lanes (the sums do not depend on the run).
template <bool EXT>
__device__ __forceinline__ void grid_item64_cells(const SweepArgs& a, unsigned char* my, const Item& item, int lane) {
  using L = Lay64<1>;
  const double2* __restrict__ vis = static_cast<const double2*>(a.vis);
  const double* __restrict__ wts = static_cast<const double*>(a.weights);
  double* __restrict__ grid = static_cast<double*>(a.grid);
  double2* ring = reinterpret_cast<double2*>(my + L::ring);
  ring[lane] = ring[L::TS + lane] = make_double2(0.0, 0.0);
  auto flush = [&](int base) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const double2 v = ring[r * L::TS + lane];
      ring[r * L::TS + lane] = make_double2(0.0, 0.0);
      double* dst = grid + (static_cast<size_t>(base + r) * a.N + item.strip * L::S + lane) * 2;
      if (v.x != 0.0) atomicAdd(dst, v.x);
      if (v.y != 0.0) atomicAdd(dst + 1, v.y);
    }
  };
  int base = -1;
  for (int w = 0; w < item.nrec; w += 32) {
    const int n = min(32, item.nrec - w);
    int pair = -1, cell = 0;
    double ar = 0.0, ai = 0.0, cv = 0.0;
    if (lane < n) {
      const Rec rc = a.recs[item.rb + w + lane];
      double cu;
      lane_weights<EXT>(a, my, rc, lane, cu, cv);
      const double2 v = vis[rc.idx];
      const double wt = wts != nullptr ? wts[rc.idx] : 1.0;
      ar = cu * (v.x * wt);
      ai = cu * (v.y * wt);
      const int y = rec_row(rc.rx);
      pair = y & ~1;
      cell = (y & 1) * L::TS + rec_xrel(rc.rx);
    }
    for (unsigned left = __ballot_sync(0xffffffffu, lane < n); left;) {
      const int p = __shfl_sync(0xffffffffu, pair, __ffs(left) - 1);
      const bool mine = pair == p;
      __syncwarp();
      if (p != base) {
        if (base >= 0) flush(base);
        base = p;
        __syncwarp();
      }
      // lanes of one cell, and this lane's place among them
      const unsigned same = __match_any_sync(0xffffffffu, mine ? cell : -1 - lane);
      const int turn = __popc(same & ((1u << lane) - 1u));
      const int turns = __reduce_max_sync(0xffffffffu, mine ? turn : 0);
      for (int t = 0; t <= turns; ++t) {
        if (mine && turn == t) {
          const double2 g = ring[cell];
          ring[cell] = make_double2(fma(cv, ar, g.x), fma(cv, ai, g.y));
        }
        __syncwarp();
      }
      left &= ~__ballot_sync(0xffffffffu, mine);
    }
  }
  if (base >= 0) flush(base);
  __syncwarp();
}

// Degridding: each lane reads its record's cell.
template <bool EXT>
__device__ __forceinline__ void degrid_item64_cells(const SweepArgs& a, unsigned char* my, const Item& item, int lane) {
  const double2* __restrict__ grid = static_cast<const double2*>(a.grid_in);
  double2* __restrict__ out = static_cast<double2*>(a.vis_out);
  for (int l = lane; l < item.nrec; l += 32) {
    const Rec rc = a.recs[item.rb + l];
    const double2 g = grid[static_cast<size_t>(rec_row(rc.rx)) * a.N + item.strip * Lay64<1>::S + rec_xrel(rc.rx)];
    double cu, cv;
    lane_weights<EXT>(a, my, rc, lane, cu, cv);
    atomicAdd(&out[rc.idx].x, cu * (cv * g.x));
    atomicAdd(&out[rc.idx].y, cu * (cv * g.y));
  }
}

template <int W, bool EXT>
__device__ __forceinline__ void grid_item64(const SweepArgs& a, unsigned char* my, const Item& item, int lane) {
  using L = Lay64<W>;
  constexpr int RR = L::RR, TS = L::TS, NI = L::NI;
  const double* tab = static_cast<const double*>(a.table);
  const double2* __restrict__ vis = static_cast<const double2*>(a.vis);
  const double* __restrict__ wts = static_cast<const double*>(a.weights);
  double* __restrict__ grid = static_cast<double*>(a.grid);
  double2* ring = reinterpret_cast<double2*>(my + L::ring);
  double* basis = reinterpret_cast<double*>(my + L::basis);
  double2* val = reinterpret_cast<double2*>(my + L::val);
  int* off = reinterpret_cast<int*>(my + L::off);
  const double* cv = reinterpret_cast<const double*>(my + L::cv);
  const double2* cu = reinterpret_cast<const double2*>(my + L::cu);
  int r[NI], c[NI];
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    const int cell = lane + 32 * i;
    r[i] = cell / W;
    c[i] = cell - W * r[i];
  }
  for (int k = lane; k < RR * TS; k += 32) ring[k] = make_double2(0.0, 0.0);
  // adds ring slot s (grid row `row`, wrapped) to the grid and clears it
  auto flush = [&](int s, int row) {
    if (row >= a.N) row -= a.N;
    double* src = reinterpret_cast<double*>(ring + s * TS);
    for (int k = lane; k < 2 * L::COLS; k += 32) {
      const double v = src[k];
      src[k] = 0.0;
      int col = item.strip * L::S + (k >> 1);
      if (col >= a.N) col -= a.N;
      if (v != 0.0) atomicAdd(grid + (static_cast<size_t>(row) * a.N + col) * 2 + (k & 1), v);
    }
  };
  int base = -1, ps = 0;  // the ring holds rows base .. base + RR - 1, row base in slot ps
  for (int w = 0; w < item.nrec; w += 32) {
    const int n = min(32, item.nrec - w);
    int rx = 0;
    __syncwarp();
    if (lane < n) {
      const Rec rc = a.recs[item.rb + w + lane];
      rx = rc.rx;
      int ou, ov;
      double fu, fv;
      record_coords<double, EXT>(a, rc, ou, fu, ov, fv);
      off[lane] = ou;
      off[32 + lane] = ov;
      stage_basis<EXT>(a.interp, fu, basis + lane);
      stage_basis<EXT>(a.interp, fv, basis + 128 + lane);
      const double2 v = vis[rc.idx];
      const double wt = wts != nullptr ? wts[rc.idx] : 1.0;
      val[lane] = make_double2(v.x * wt, v.y * wt);
    }
    __syncwarp();
    for (int s0 = 0; s0 < n; s0 += kSub) {
      stage_weights<W, EXT, true>(tab, a.Wp, a.interp, my, s0, n, lane);
      __syncwarp();
      const int ns = min(kSub, n - s0);
      for (int s = 0; s < ns; ++s) {
        const int x = __shfl_sync(0xffffffffu, rx, s0 + s);
        const int y = rec_row(x), pair = y & ~1;
        if (pair != base) {
          if (base >= 0) {
            const int steps = min((pair - base) >> 1, RR / 2);
            for (int k = 0; k < steps; ++k) {
              flush(ps, base + 2 * k);
              flush(ps + 1, base + 2 * k + 1);
              ps = ps + 2 == RR ? 0 : ps + 2;
            }
            __syncwarp();
          }
          base = pair;
        }
        const int q0 = ps + (y & 1), x0 = rec_xrel(x);
        const double* pv = cv + s * L::EW;
        const double2* pu = cu + s * L::EW;
        double2* g[NI];
        double2 t[NI], u[NI];
        double b[NI];
        // all loads before the first store: the compiler may not move them across it
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const bool in = 32 * (i + 1) <= W * W || lane + 32 * i < W * W;
          int q = q0 + r[i];
          if (q >= RR) q -= RR;
          g[i] = ring + q * TS + x0 + c[i];
          if (in) {
            b[i] = pv[r[i]];
            u[i] = pu[c[i]];
            t[i] = *g[i];
          }
        }
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          if (32 * (i + 1) <= W * W || lane + 32 * i < W * W)
            *g[i] = make_double2(fma(b[i], u[i].x, t[i].x), fma(b[i], u[i].y, t[i].y));
        }
        __syncwarp();  // the next record's lanes hold other cells
      }
    }
  }
  if (base >= 0)
    for (int k = 0; k < RR; ++k) flush(ps + k >= RR ? ps + k - RR : ps + k, base + k);
  __syncwarp();
}

template <int W, bool EXT>
__device__ __forceinline__ void degrid_item64(const SweepArgs& a, unsigned char* my, const Item& item, int lane) {
  using L = Lay64<W>;
  constexpr int RR = L::RR, TS = L::TS, G = L::G, NR = L::NR;
  const double* tab = static_cast<const double*>(a.table);
  const double2* __restrict__ grid = static_cast<const double2*>(a.grid_in);
  double2* __restrict__ out = static_cast<double2*>(a.vis_out);
  double2* ring = reinterpret_cast<double2*>(my + L::ring);
  double* basis = reinterpret_cast<double*>(my + L::basis);
  int* off = reinterpret_cast<int*>(my + L::off);
  const double* cv = reinterpret_cast<const double*>(my + L::cv);
  const double* cu = reinterpret_cast<const double*>(my + L::cu);
  double2* part = reinterpret_cast<double2*>(my + L::part);
  const int g = lane / W, c = lane - W * g;
  const int rec4 = lane >> 2, q4 = lane & 3;  // final sums: four lanes a record
  // ring slot s holds grid row `row` (wrapped)
  auto load = [&](int s, int row) {
    if (row >= a.N) row -= a.N;
    for (int k = lane; k < L::COLS; k += 32) {
      int col = item.strip * L::S + k;
      if (col >= a.N) col -= a.N;
      ring[s * TS + k] = grid[static_cast<size_t>(row) * a.N + col];
    }
  };
  int base = -RR, ps = 0;  // the ring holds rows base .. base + RR - 1, row base in slot ps
  for (int w = 0; w < item.nrec; w += 32) {
    const int n = min(32, item.nrec - w);
    int rx = 0;
    unsigned idx = 0;
    __syncwarp();
    if (lane < n) {
      const Rec rc = a.recs[item.rb + w + lane];
      rx = rc.rx;
      idx = rc.idx;
      int ou, ov;
      double fu, fv;
      record_coords<double, EXT>(a, rc, ou, fu, ov, fv);
      off[lane] = ou;
      off[32 + lane] = ov;
      stage_basis<EXT>(a.interp, fu, basis + lane);
      stage_basis<EXT>(a.interp, fv, basis + 128 + lane);
    }
    __syncwarp();
    for (int s0 = 0; s0 < n; s0 += kSub) {
      stage_weights<W, EXT, false>(tab, a.Wp, a.interp, my, s0, n, lane);
      __syncwarp();
      const int ns = min(kSub, n - s0);
      for (int s = 0; s < ns; ++s) {
        const int x = __shfl_sync(0xffffffffu, rx, s0 + s);
        const int y = rec_row(x), pair = y & ~1;
        if (pair != base) {
          __syncwarp();
          const int fresh = min(pair - base, RR);  // rows not in the ring
          if (fresh == RR) {
            ps = 0;
          } else {
            ps += fresh;
            if (ps >= RR) ps -= RR;
          }
          for (int k = RR - fresh; k < RR; ++k) load(ps + k >= RR ? ps + k - RR : ps + k, pair + k);
          base = pair;
          __syncwarp();
        }
        if (g < G) {
          const int q0 = ps + (y & 1), x0 = rec_xrel(x) + c;
          const double* pv = cv + s * L::EW;
          double pr = 0.0, pi = 0.0;
#pragma unroll
          for (int i = 0; i < NR; ++i) {
            const int r = g + G * i;
            if (G * (i + 1) <= W || r < W) {
              int q = q0 + r;
              if (q >= RR) q -= RR;
              const double2 t = ring[q * TS + x0];
              const double b = pv[r];
              pr = fma(b, t.x, pr);
              pi = fma(b, t.y, pi);
            }
          }
          part[s * L::PP + lane] = make_double2(pr, pi);
        }
      }
      __syncwarp();
      double vr = 0.0, vi = 0.0;
      if (rec4 < ns) {
#pragma unroll
        for (int k = 0; k < (G * W + 3) / 4; ++k) {
          const int cell = q4 + 4 * k;
          if (4 * (k + 1) <= G * W || cell < G * W) {
            const double2 p = part[rec4 * L::PP + cell];
            const double b = cu[rec4 * L::EW + cell % W];
            vr = fma(b, p.x, vr);
            vi = fma(b, p.y, vi);
          }
        }
      }
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        vr += __shfl_xor_sync(0xffffffffu, vr, o);
        vi += __shfl_xor_sync(0xffffffffu, vi, o);
      }
      const unsigned k = __shfl_sync(0xffffffffu, idx, s0 + rec4);
      if (rec4 < ns && q4 < 2) atomicAdd(&out[k].x + q4, q4 ? vi : vr);
      __syncwarp();
    }
  }
}

template <int W, bool EXT, bool DEGRID>
__global__ void __launch_bounds__(kThreads64) k_sweep64(const SweepArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  using L = Lay64<W>;
  const int lane = threadIdx.x & 31;
  unsigned char* my = smem + (threadIdx.x >> 5) * (DEGRID ? L::degrid_bytes : L::grid_bytes);
  int* work = a.counters + (DEGRID ? kCntDegridWork : kCntGridWork);
  int nfront;
  const int total = work_total(a.counters, a.item_cap, nfront);
  for (int w = next_item(work, lane); w < total; w = next_item(work, lane)) {
    const Item item = a.items[item_slot(w, nfront, a.item_cap)];
    if constexpr (DEGRID) {
      if constexpr (W == 1) degrid_item64_cells<EXT>(a, my, item, lane);
      else degrid_item64<W, EXT>(a, my, item, lane);
    } else {
      if constexpr (W == 1) grid_item64_cells<EXT>(a, my, item, lane);
      else grid_item64<W, EXT>(a, my, item, lane);
    }
  }
}

template <bool EXT, int W> void* pick64(bool degrid) {
  return degrid ? reinterpret_cast<void*>(&k_sweep64<W, EXT, true>) : reinterpret_cast<void*>(&k_sweep64<W, EXT, false>);
}
template <bool EXT> void* sweep64_pick(int W, bool degrid) {
  switch (W) {
    case 1: return pick64<EXT, 1>(degrid);
    case 2: return pick64<EXT, 2>(degrid);
    case 3: return pick64<EXT, 3>(degrid);
    case 4: return pick64<EXT, 4>(degrid);
    case 5: return pick64<EXT, 5>(degrid);
    case 6: return pick64<EXT, 6>(degrid);
    case 7: return pick64<EXT, 7>(degrid);
    case 8: return pick64<EXT, 8>(degrid);
    case 9: return pick64<EXT, 9>(degrid);
    case 10: return pick64<EXT, 10>(degrid);
    case 11: return pick64<EXT, 11>(degrid);
    case 12: return pick64<EXT, 12>(degrid);
    case 13: return pick64<EXT, 13>(degrid);
    case 14: return pick64<EXT, 14>(degrid);
    case 15: return pick64<EXT, 15>(degrid);
    case 16: return pick64<EXT, 16>(degrid);
    default: return nullptr;
  }
}

}  // namespace
}  // namespace lmg
