// On-device diagnostics of Secs. 3-4 of arXiv:2009.12584 (declared with
// lbm_diagnostics in include/lbm.h): reductions over the moments that the
// eval pass writes to the staging area (rho^A, rho^B, u_x, u_y as double
// [ny][nx] arrays), in FP64 and a fixed order.
#pragma once

#include "lbm_common.cuh"

namespace lbm {

constexpr int DIAG_BLOCKS = 256;
constexpr int DIAG_THREADS = 256;
// A node per thread until all blocks are in use.
inline int diag_blocks(const Geo& g) {
  const int64_t nb = ((int64_t)g.nx * g.ny + DIAG_THREADS - 1) / DIAG_THREADS;
  return nb < DIAG_BLOCKS ? (int)nb : DIAG_BLOCKS;
}
// reduced quantities: 0 sum w, 1 sum w x, 2 sum w y, 3 sum w u_x,
// 4 sum w u_y, 5 crossings kept, 6..13 the Kasa sums over kept crossings
// (x, y, xx, yy, xy, x r, y r, r with r = x^2 + y^2, coordinates relative to
// the grid centre), 14 max |u|^2 over finite nodes, 15 fluid nodes whose
// rho^A, rho^B or u is not finite, 16 bridge radius (final kernel only)
constexpr int DIAG_NQ = 17;
constexpr int DIAG_NRED = 16;  // quantities reduced over nodes (0..15)

struct DiagArgs {
  double level, rho_out;
  double wx, wy;    // wall point
  double nx_, ny_;  // wall normal towards the fluid
  double exclude;
  double box[4];
  bool use_box;
  double ox, oy;    // origin of the fit coordinates
  int bridge_x, bridge_y0;
};

// Sign of v (0 for either zero) from its bits: a comparison of FP64 values is
// an instruction of the FP64 pipe.
__device__ __forceinline__ int dsgn(double v) {
  const long long b = __double_as_longlong(v);
  return (b << 1) == 0 ? 0 : (b < 0 ? -1 : 1);
}
__device__ __forceinline__ bool dfinite(double v) {
  return (((unsigned)__double2hiint(v) >> 20) & 0x7FFu) != 0x7FFu;
}

// One contour point: drop it near the wall or outside the box, else add it
// to the fit sums.
__device__ __forceinline__ void diag_point(const DiagArgs& a, double px, double py, double acc[DIAG_NRED]) {
  const double dist = (px - a.wx) * a.nx_ + (py - a.wy) * a.ny_;
  if (!(dist > a.exclude)) return;
  if (a.use_box && !(px >= a.box[0] && px <= a.box[1] && py >= a.box[2] && py <= a.box[3])) return;
  const double x = px - a.ox, y = py - a.oy, r = x * x + y * y;
  acc[5] += 1.0;
  acc[6] += x;
  acc[7] += y;
  acc[8] += x * x;
  acc[9] += y * y;
  acc[10] += x * y;
  acc[11] += x * r;
  acc[12] += y * r;
  acc[13] += r;
}

// Per-block partial sums (and max) over a fixed grid-stride assignment of
// the owned nodes; st = [rho^A | rho^B | u_x | u_y], each nx * ny. Bound by the
// FP64 pipe (2 lanes per clock and SM): signs and tests go by the bits, a node
// without weight adds nothing to the weighted sums, and a warp without a
// crossing reduces no fit sums.
static __global__ void __launch_bounds__(DIAG_THREADS) k_diag_partial(const double* __restrict__ st,
                                                                      const uint16_t* __restrict__ flags, Geo g,
                                                                      DiagArgs a, double* __restrict__ partial) {
  __shared__ double red[DIAG_THREADS / 32][DIAG_NRED];
  double acc[DIAG_NRED];
#pragma unroll
  for (int q = 0; q < DIAG_NRED; ++q) acc[q] = 0.0;
  const int64_t N = (int64_t)g.nx * g.ny;
  for (int64_t n = (int64_t)blockIdx.x * DIAG_THREADS + threadIdx.x; n < N; n += (int64_t)gridDim.x * DIAG_THREADS) {
    const int y = (int)((unsigned)n / (unsigned)g.nx), x = (int)((unsigned)n - (unsigned)y * (unsigned)g.nx);
    const int k = g.idx(x, y);
    if (flags[k] & F_SOLID) continue;
    const double rA = st[n], ux = st[2 * N + n], uy = st[3 * N + n];
    if (!dfinite(rA) || !dfinite(st[N + n]) || !dfinite(ux) || !dfinite(uy)) {
      acc[15] += 1.0;  // counted, and left out of every other sum
      continue;
    }
    const double w = rA - a.rho_out;
    if (dsgn(w) > 0) {
      acc[0] += w;
      acc[1] += w * x;
      acc[2] += w * y;
      acc[3] += w * ux;
      acc[4] += w * uy;
    }
    acc[14] = fmax(acc[14], ux * ux + uy * uy);
    const double d = rA - a.level;
    if (x + 1 < g.nx && !(flags[k + 1] & F_SOLID)) {  // edge to (x + 1, y)
      const double e = st[n + 1] - a.level;
      if (dsgn(d) != dsgn(e)) diag_point(a, x + d / (d - e), (double)y, acc);
    }
    if (y + 1 < g.ny && !(flags[k + g.px] & F_SOLID)) {  // edge to (x, y + 1)
      const double e = st[n + g.nx] - a.level;
      if (dsgn(d) != dsgn(e)) diag_point(a, (double)x, y + d / (d - e), acc);
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool fit = __any_sync(0xffffffffu, __double_as_longlong(acc[5]) != 0);
  const bool bad = __any_sync(0xffffffffu, __double_as_longlong(acc[15]) != 0);
#pragma unroll
  for (int q = 0; q < DIAG_NRED; ++q) {
    double v = acc[q];
    if ((q >= 5 && q <= 13 && !fit) || (q == 15 && !bad)) {  // zero in every lane
      if (lane == 0) red[wid][q] = 0.0;
      continue;
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double t = __shfl_down_sync(0xffffffffu, v, o);
      v = q == 14 ? fmax(v, t) : v + t;
    }
    if (lane == 0) red[wid][q] = v;
  }
  __syncthreads();
  if (threadIdx.x < DIAG_NRED) {
    const int q = threadIdx.x;
    double v = red[0][q];
    for (int w = 1; w < DIAG_THREADS / 32; ++w) v = q == 14 ? fmax(v, red[w][q]) : v + red[w][q];
    partial[(size_t)blockIdx.x * DIAG_NRED + q] = v;
  }
}

// One warp per quantity: blocks in a fixed order (a lane takes every 32nd,
// then a tree), and the bridge radius by a scan of one column, 32 rows at a
// time (one thread's dependent loads and FP64 additions took 27 us).
static __global__ void __launch_bounds__(32 * DIAG_NQ) k_diag_final(const double* __restrict__ partial, int nblocks,
                                                                    const double* __restrict__ st, Geo g, DiagArgs a,
                                                                    double* __restrict__ out) {
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q < DIAG_NRED) {
    double v = 0.0;  // also the identity of the maximum of |u|^2
    for (int b = lane; b < nblocks; b += 32) {
      const double t = partial[(size_t)b * DIAG_NRED + q];
      v = q == 14 ? fmax(v, t) : v + t;
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double t = __shfl_down_sync(0xffffffffu, v, o);
      v = q == 14 ? fmax(v, t) : v + t;
    }
    if (lane == 0) out[q] = v;
    return;
  }
  double br = 0.0;
  if (a.bridge_x >= 0) {
    const double* col = st + a.bridge_x;  // rho^A, stride nx
    // first row from bridge_y0 on below the level (or ny)
    int y1 = g.ny;
    for (int y = a.bridge_y0; y < g.ny; y += 32) {
      const bool below = y + lane < g.ny && !(col[(int64_t)(y + lane) * g.nx] >= a.level);
      const unsigned m = __ballot_sync(0xffffffffu, below);
      if (m) {
        y1 = y + __ffs(m) - 1;
        break;
      }
    }
    if (y1 >= g.ny) {
      br = g.ny - (a.bridge_y0 - 0.5);
    } else if (y1 > a.bridge_y0) {
      const int y = y1 - 1;
      const double c0 = col[(int64_t)y * g.nx], c1 = col[(int64_t)y1 * g.nx];
      br = y + (c0 - a.level) / (c0 - c1) - (a.bridge_y0 - 0.5);
    }
  }
  if (lane == 0) out[16] = br;
}

}  // namespace lbm
