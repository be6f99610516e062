// Warp strips: the walk over the grid that the FP64 stencils share.
//
// A warp owns 32 neighbouring j and marches along i in one time plane.  Values
// at j +- 1 come from the neighbouring lanes and values at i +- 1 from registers,
// so each value is loaded once per warp and whatever two neighbours have in
// common (a pair sum, a face difference) is formed once: FP64
// instructions are what these kernels have to save.  What lanes 0 and 31 need
// from beyond the strip is gathered once per chunk of at most 32 rows, with lane r
// holding row r, and handed out row by row.
#pragma once

#include <algorithm>

#include "mfg_internal.cuh"

namespace mfg {

// Index of a node beyond the end of an axis: wrapped, or the end itself.
__device__ __forceinline__ int ghost(int i, int N, int per) {
  if (i < 0) return per ? N - 1 : 0;
  return i < N ? i : (per ? 0 : N - 1);
}


// Constant viscosity and at least num/den of the strips' lanes with a column: where an
// operator walks in strips, each by its own measured line; the rest runs point by point.
inline bool strips_filled(const Geom& g, int num, int den) {
  return g.kfy == nullptr && (long long)(g.ny + 31) / 32 * 32 * num <= (long long)g.ny * den;
}

// Launch: 32-column strips x row chunks x planes, one warp each.  A block holds 8
// warps, fewer where that leaves fewer than 4 blocks per SM.  The chunk length (2 to 32 rows) is
// the one with the least waves x (rows + 1.5): whole waves of the per_sm blocks a kernel's
// registers admit per SM, 1.5 rows' worth of work for a chunk's start.  (256^2 x 128: 29
// rows, 1.9 waves, where 26 rows filled 2.1 and left the third wave nearly empty.)
// want scales the wave over kAatWantDefault: AAt passes its tuned Geom::aat_want, which says
// nothing about the other operators (C in strips, 512 x 45 x 100: 102 us by the default, 125 by half of it).
struct StripGrid {
  int strips, chunks, rows, warps, blocks;
};

inline StripGrid strip_grid(const Geom& g, int per_sm, int want = kAatWantDefault) {
  StripGrid a;
  a.strips = (g.ny + 31) / 32;
  const long long base = (long long)a.strips * g.nt, wave = std::max(1, want / 8 * per_sm);
  double best = 1e300;
  for (int most = 32; most >= 2; --most) {
    const int chunks = (g.nx + most - 1) / most, rows = (g.nx + chunks - 1) / chunks;
    const long long blocks = (base * chunks + 7) / 8;
    const double cost = (double)((blocks + wave - 1) / wave) * (rows + 1.5);
    if (cost < best) {
      best = cost;
      a.chunks = chunks;
      a.rows = rows;
    }
  }
  a.chunks = (g.nx + a.rows - 1) / a.rows;
  const long long items = base * a.chunks;
  a.warps = 8;
  while (a.warps > 1 && items < (long long)a.warps * 152 * 4) a.warps >>= 1;
  a.blocks = (int)((items + a.warps - 1) / a.warps);
  return a;
}

// This warp's strip, row chunk and plane; false past the last one.
__device__ __forceinline__ bool strip_item(const StripGrid& ag, const Geom& g, int& j0, int& i0, int& i1, int& k) {
  const long long item = (long long)blockIdx.x * ag.warps + (threadIdx.x >> 5);
  if (item >= (long long)ag.strips * ag.chunks * g.nt) return false;
  const int per = ag.strips * ag.chunks;
  k = (int)(item / per);
  const int rem = (int)(item - (long long)k * per), c = rem / ag.strips;
  j0 = (rem - c * ag.strips) * 32;
  i0 = c * ag.rows;
  i1 = min(g.nx, i0 + ag.rows);
  return true;
}

// Column a lane reads (past the last column: the one beyond the end), and the
// columns beside the strip.
struct StripCols {
  int j, left, right;
};
__device__ __forceinline__ StripCols strip_cols(const Geom& g, int j0) {
  const int j = j0 + (int)(threadIdx.x & 31), beyond = ghost(g.ny, g.ny, g.pery);
  return StripCols{j < g.ny ? j : beyond, ghost(j0 - 1, g.ny, g.pery), j0 + 32 < g.ny ? j0 + 32 : beyond};
}

// v of the lane below (lane 0: lane r's `edge`) and of the lane above (lane 31).
__device__ __forceinline__ double from_left(double v, double edge, int r) {
  const double w = __shfl_up_sync(0xffffffffu, v, 1), e = __shfl_sync(0xffffffffu, edge, r);
  return (threadIdx.x & 31) == 0 ? e : w;
}
__device__ __forceinline__ double from_right(double v, double edge, int r) {
  const double w = __shfl_down_sync(0xffffffffu, v, 1), e = __shfl_sync(0xffffffffu, edge, r);
  return (threadIdx.x & 31) == 31 ? e : w;
}

// The march over one chunk for neighbour sums: f(row, centre value, sum, loaded) with
// sum = (p_S + p_N) + rho (p_W + p_E); ISO (rho = 1): by shared pair sums.  ld(i, j) is
// the value at node (i, j) of this plane; pre(i) loads whatever else f needs for row
// i.  The loads of ROWS rows are issued together, without branches between them
// (rows past the end repeat the last one), so a batch costs one memory latency.
// f is called by all lanes.
template <bool ISO, int ROWS, typename Ld, typename Pre, typename F>
__device__ __forceinline__ void sum_march(const Geom& g, double rho, int i0, int i1, int j0, Ld ld, Pre pre, F f) {
  const int lane = threadIdx.x & 31;
  const StripCols c = strip_cols(g, j0);
  // lane r: what row i0 + r needs from the columns beside the strip
  const int ir = min(i0 + lane, i1 - 1);
  const double left = ld(ir, c.left), right = ld(ir, c.right);
  double hl = left;  // ISO: the pair sum A(i-1, j0-1) of lane 0
  double vm = ld(ghost(i0 - 1, g.nx, g.perx), c.j), vc = ld(i0, c.j), hc = 0.0;
  if (ISO) hc = ld(ghost(ir - 1, g.nx, g.perx), j0);
  double ap = 0.0;
  for (int i = i0; i < i1; i += ROWS) {
    double v[ROWS];
    decltype(pre(0)) x[ROWS];
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      const int it = min(i + t, i1 - 1);
      v[t] = ld(ghost(it + 1, g.nx, g.perx), c.j);
      x[t] = pre(it);
    }
    if (ISO && i == i0) {
      hl += hc;
      ap = __shfl_down_sync(0xffffffffu, vm, 1) + vc;
    }
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      if (i + t >= i1) break;
      const double vp = v[t], e = from_right(vc, right, i + t - i0);
      double sum;
      if (ISO) {
        const double an = e + vp;  // A(i, j)
        sum = an + from_left(ap, hl, i + t - i0);
        ap = an;
      } else {
        sum = fma(rho, vm + vp, from_left(vc, hl, i + t - i0) + e);
      }
      f(i + t, vc, sum, x[t]);
      vm = vc;
      vc = vp;
    }
  }
}

// The march for neighbour differences: f(row, centre p, Diff, loaded).  Each face's
// difference is formed once, and scaled once for the gradient components.  The second
// differences come from the unscaled ones, which are exact where p varies slowly: scaled
// first, they carry an error of the size of the gradient (512^2 Neumann, nu = 1: the m
// row of C^T p 15 times as far off).  A lane gets its left face's two values from the
// neighbour by shuffles, which cost less than a second FP64 multiplication.
struct Diff {
  double yp, ym, xp, xm;  // (p - p_{j+1})/dy, (p_{j-1} - p)/dy, the same in x; 0 across a Neumann end
  double yy, xx;          // 2 p - p_{j-1} - p_{j+1}, the same in x
};

template <int ACTX, int ROWS, typename Ld, typename Pre, typename F>
__device__ __forceinline__ void diff_march(const Geom& g, int i0, int i1, int j0, Ld ld, Pre pre, F f) {
  const int lane = threadIdx.x & 31;
  const StripCols c = strip_cols(g, j0);
  const int ir = min(i0 + lane, i1 - 1);
  const double right = ld(ir, c.right);
  double hd = ld(ir, c.left), hc = ld(ir, j0), hs = 0.0, vc = ld(i0, c.j), dxm = 0.0;
  if (ACTX) dxm = ld(ghost(i0 - 1, g.nx, g.perx), c.j);
  Diff d{};
  for (int i = i0; i < i1; i += ROWS) {
    double v[ROWS];
    decltype(pre(0)) x[ROWS];
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      const int it = min(i + t, i1 - 1);
      if (ACTX) v[t] = ld(ghost(it + 1, g.nx, g.perx), c.j);
      x[t] = pre(it);
    }
    if (i == i0) {
      hd -= hc;
      hs = hd * g.idy;
      if (ACTX) {
        dxm -= vc;
        d.xm = dxm * g.idx;
      }
    }
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      if (i + t >= i1) break;
      const double dyp = vc - from_right(vc, right, i + t - i0);
      d.yp = dyp * g.idy;
      d.ym = from_left(d.yp, hs, i + t - i0);
      d.yy = dyp - from_left(dyp, hd, i + t - i0);
      double dxp = 0.0;
      if (ACTX) {
        dxp = vc - v[t];
        d.xp = dxp * g.idx;
        d.xx = dxp - dxm;
      }
      f(i + t, vc, d, x[t]);
      if (ACTX) {
        dxm = dxp;
        d.xm = d.xp;
        vc = v[t];
      }
    }
  }
}

}  // namespace mfg
