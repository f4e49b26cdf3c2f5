// On-device diagnostics of Secs. 3-4 of arXiv:2009.12584 (declared with
// lbm_diagnostics in include/lbm.h): reductions over the moments that the
// eval pass writes to the staging area (rho^A, rho^B, u_x, u_y as double
// [ny][nx] arrays), in FP64 and a fixed order.
#pragma once

#include "lbm_common.cuh"

namespace lbm {

constexpr int DIAG_BLOCKS = 256;  // at most
constexpr int DIAG_THREADS = 512; // at most
// Blocks of 256 threads with a node each while one per SM is enough (a block's
// reduction costs as much FP64 time as a few nodes per thread), then one of
// 512 threads on each SM.
inline int diag_blocks(const Geo& g, int num_sms, int* threads) {
  const int64_t nb = ((int64_t)g.nx * g.ny + 255) / 256, most = num_sms < DIAG_BLOCKS ? num_sms : DIAG_BLOCKS;
  *threads = nb <= most ? 256 : DIAG_THREADS;
  return (int)(nb <= most ? nb : most);
}
// reduced quantities: 0 sum w, 1 sum w x, 2 sum w y, 3 sum w u_x,
// 4 sum w u_y, 5 crossings kept, 6..13 the Kasa sums over kept crossings
// (x, y, xx, yy, xy, x r, y r, r with r = x^2 + y^2, coordinates relative to
// the grid centre), 14 max |u|^2 over finite nodes, 15 fluid nodes whose
// rho^A, rho^B or u is not finite, 16 bridge radius (final kernel only)
constexpr int DIAG_NQ = 17;
constexpr int DIAG_OUT = DIAG_NQ + 1;  // what is read back: these and the error word
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
// FP64 pipe (2 lanes per clock and SM): signs and tests go by the bits, and a
// node without weight adds nothing to the weighted sums. 4096^2 porous, with
// the moments: 1.23 ms; 1.56 with 256 blocks and a tree per quantity.
static __global__ void __launch_bounds__(DIAG_THREADS) k_diag_partial(const double* __restrict__ st,
                                                                      const uint16_t* __restrict__ flags, Geo g,
                                                                      DiagArgs a, double* __restrict__ partial) {
  __shared__ double red[DIAG_THREADS / 32][DIAG_NRED];
  double acc[DIAG_NRED];
#pragma unroll
  for (int q = 0; q < DIAG_NRED; ++q) acc[q] = 0.0;
  long long umax = 0;  // max |u|^2: non-negative values order like their bits
  const int64_t N = (int64_t)g.nx * g.ny;
  pdl_wait();
  for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x) {
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
    umax = max(umax, __double_as_longlong(ux * ux + uy * uy));
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
  for (int o = 16; o > 0; o >>= 1) umax = max(umax, __shfl_xor_sync(0xffffffffu, umax, o));
  // The sums by halving: at each step a lane hands over one half of its
  // quantities and keeps the sums of the other; 16 FP64 additions in all,
  // where a tree per quantity takes 5 each.
#pragma unroll
  for (int w = 8; w >= 1; w >>= 1) {
    const bool hi = lane & (2 * w);
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const double keep = hi ? acc[i + w] : acc[i], give = hi ? acc[i] : acc[i + w];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, 2 * w);
    }
  }
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
  const int mine = lane >> 1;  // the quantity this lane holds now
  if ((lane & 1) == 0) red[wid][mine] = mine == 14 ? __longlong_as_double(umax) : acc[0];
  __syncthreads();
  if (threadIdx.x < DIAG_NRED) {
    const int q = threadIdx.x;
    double v = red[0][q];
    for (int w = 1; w < (int)blockDim.x / 32; ++w) v = q == 14 ? fmax(v, red[w][q]) : v + red[w][q];
    partial[(size_t)blockIdx.x * DIAG_NRED + q] = v;
  }
}

// One warp per quantity: blocks in a fixed order (a lane takes every 32nd,
// then a tree), and the bridge radius by a scan of one column, 32 rows at a
// time (one thread's dependent loads and FP64 additions took 27 us).
static __global__ void __launch_bounds__(32 * DIAG_NQ) k_diag_final(const double* __restrict__ partial, int nblocks,
                                                                    const double* __restrict__ st,
                                                                    const uint16_t* __restrict__ flags, Geo g,
                                                                    DiagArgs a, const volatile int* err,
                                                                    double* __restrict__ out) {
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();
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
  const int e = *err;
  double br = 0.0;
  if (a.bridge_x >= 0) {
    // rho^A on the column, 0 at solid nodes
    auto col = [&](int y) {
      return (flags[g.idx(a.bridge_x, y)] & F_SOLID) ? 0.0 : st[(int64_t)y * g.nx + a.bridge_x];
    };
    // first row from bridge_y0 on below the level (or ny)
    int y1 = g.ny;
    for (int y = a.bridge_y0; y < g.ny; y += 32) {
      const bool below = y + lane < g.ny && !(col(y + lane) >= a.level);
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
      const double c0 = col(y), c1 = col(y1);
      br = y + (c0 - a.level) / (c0 - c1) - (a.bridge_y0 - 0.5);
    }
  }
  if (lane == 0) {
    out[16] = br;
    out[DIAG_NQ] = e;
  }
}

}  // namespace lbm
