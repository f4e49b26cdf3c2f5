// Shared device-side definitions of the GB300 lattice-Boltzmann library:
// D2Q9 tables, the padded grid geometry, population storage formats and the
// per-node physics of one time step (Eqs. 2-5, 7 of arXiv:2009.12584).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace lbm {

// ---------------------------------------------------------------------------
// D2Q9 lattice (Sec. 2): 0 rest, 1 E, 2 N, 3 W, 4 S, 5 NE, 6 NW, 7 SW, 8 SE.
// constexpr functions so that fully unrolled loops fold them to immediates.
__host__ __device__ constexpr int cx_of(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
}
__host__ __device__ constexpr int cy_of(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
}
__host__ __device__ constexpr int opp_of(int i) {
  return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4) + 1 : ((i - 3) % 4) + 5);
}
template <typename C>
__host__ __device__ constexpr C w_of(int i) {
  return i == 0 ? C(4) / C(9) : (i <= 4 ? C(1) / C(9) : C(1) / C(36));
}

// Programmatic dependent launch: a kernel of a step may start (and load what no
// kernel of a step writes: lists, flags, tables) while the one before it in
// the stream drains. pdl_wait returns when all work before the launch is
// complete and visible; only then may the next kernel start (so that its
// first part can rely on everything before this one). Both do nothing in a
// launch without the attribute.
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Ghost layer width around the owned nx * ny nodes. Periodic axes hold
// copies of the opposite border there; walled axes hold solid cells. Four
// layers cover the widest stencil of the step (Eq. 8's D2Q25 reach of 2 plus
// the force's reach of 1, plus one for streaming).
constexpr int GH = 4;
// Columns of padding left of column 0: more than the ghost layers so that
// column 0 starts on a 128-byte boundary for 4-byte types (aligned stores of
// whole rows); the columns beyond the ghost layers count as solid.
constexpr int LP = 32;

// Per-node flag bits (uint16): bit 0 the node is solid; bit i (1..8) the
// neighbour x + c_i is solid; bit 9 interface-solid (a solid node with a
// fluid D2Q9 neighbour).
constexpr uint16_t F_SOLID = 1u;
constexpr uint16_t F_IFACE = 1u << 9;
constexpr uint16_t NB_ANY = 0x1FEu;  // any of the eight neighbours solid
__host__ __device__ constexpr uint16_t nb_bit(int i) { return uint16_t(1u << i); }

struct Geo {
  int nx, ny;      // owned nodes
  int px, py;      // padded pitch and rows
  int64_t plane;   // px * py
  int per_x, per_y;
  __host__ __device__ int idx(int x, int y) const { return (y + GH) * px + (x + LP); }
};

// Call fn(k) for every padded index k that holds a periodic image of owned
// node (x, y) (up to three: one per periodic axis plus the corner). A node
// may have images on both sides of an axis when that axis is shorter than
// twice the ghost width.
template <typename Fn>
__device__ __forceinline__ void for_ghost_images(const Geo& g, int x, int y, Fn&& fn) {
  const bool xa = g.per_x && x < GH, xb = g.per_x && x >= g.nx - GH;
  const bool ya = g.per_y && y < GH, yb = g.per_y && y >= g.ny - GH;
  if (!(xa | xb | ya | yb)) return;
  const int x1 = x + g.nx, x2 = x - g.nx, y1 = y + g.ny, y2 = y - g.ny;
  if (xa) fn(g.idx(x1, y));
  if (xb) fn(g.idx(x2, y));
  if (ya) {
    fn(g.idx(x, y1));
    if (xa) fn(g.idx(x1, y1));
    if (xb) fn(g.idx(x2, y1));
  }
  if (yb) {
    fn(g.idx(x, y2));
    if (xa) fn(g.idx(x1, y2));
    if (xb) fn(g.idx(x2, y2));
  }
}

// Store v at owned node (x, y) of a plane and at its periodic images.
template <typename V>
__device__ __forceinline__ void put_with_ghosts(V* plane, const Geo& g, int x, int y, V v) {
  plane[g.idx(x, y)] = v;
  for_ghost_images(g, x, y, [&](int k) { plane[k] = v; });
}

// ---------------------------------------------------------------------------
// Density planes (rho, rho~ at interface-solid cells, and the encoding
// references of 16-bit storage) hold (component A, component B) pairs: the
// value of component s at padded index k is element 2 k + s.
template <typename C>
struct CPair;
template <>
struct CPair<float> {
  using V = float2;
};
template <>
struct CPair<double> {
  using V = double2;
};

template <typename C>
__device__ __forceinline__ void ldP(const C* __restrict__ P, int64_t k, C& a, C& b) {
  const typename CPair<C>::V v = __ldg(reinterpret_cast<const typename CPair<C>::V*>(P) + k);
  a = v.x;
  b = v.y;
}
template <typename C>
__device__ __forceinline__ void stP(C* __restrict__ P, int64_t k, C a, C b) {
  typename CPair<C>::V v;
  v.x = a;
  v.y = b;
  reinterpret_cast<typename CPair<C>::V*>(P)[k] = v;
}
// Store the pair at owned node (x, y) and at its periodic images.
template <typename C>
__device__ __forceinline__ void stP_ghosts(C* __restrict__ P, const Geo& g, int x, int y, C a, C b) {
  stP(P, g.idx(x, y), a, b);
  for_ghost_images(g, x, y, [&](int k) { stP(P, k, a, b); });
}

// ---------------------------------------------------------------------------
// Population storage. FP32/FP64 store f itself. FP16/BF16 store the
// deviation of f from a reference its writer and reader both know (see
// pull_refs), which keeps the rest-state part exact and spends the 11/8
// significand bits on what varies.
//
// Layout: nine planes of component pairs. The populations of components A
// and B for direction i at padded index k are adjacent, at element
// pslot(g, i, k) + s, so that one vector access (8 bytes for FP32) moves
// both and each plane streams as a single sequence.
__host__ __device__ __forceinline__ int64_t pslot(const Geo& g, int i, int64_t k) {
  return ((int64_t)i * g.plane + k) * 2;
}

template <typename T>
struct Pop;
template <>
struct Pop<float> {
  using C = float;
  using V = float2;  // both components as stored
  static __device__ __forceinline__ float2 unpack(float2 v, float, float) { return v; }
  static __device__ __forceinline__ float2 pack(float a, float b, float, float) { return make_float2(a, b); }
  static __device__ __forceinline__ float ld(const float* p, int64_t k, float) { return p[k]; }
  static __device__ __forceinline__ void st(float* p, int64_t k, float v, float) { p[k] = v; }
  static __device__ __forceinline__ float enc(float v, float) { return v; }
  static __device__ __forceinline__ float dec(float v, float) { return v; }
  static __device__ __forceinline__ void ld2(const float* p, int64_t j, float, float, float& a, float& b) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(p + j));
    a = v.x;
    b = v.y;
  }
  static __device__ __forceinline__ void st2(float* p, int64_t j, float a, float b, float, float) {
    *reinterpret_cast<float2*>(p + j) = make_float2(a, b);
  }
};
template <>
struct Pop<double> {
  using C = double;
  using V = double2;
  static __device__ __forceinline__ double2 unpack(double2 v, double, double) { return v; }
  static __device__ __forceinline__ double2 pack(double a, double b, double, double) { return make_double2(a, b); }
  static __device__ __forceinline__ double ld(const double* p, int64_t k, double) { return p[k]; }
  static __device__ __forceinline__ void st(double* p, int64_t k, double v, double) { p[k] = v; }
  static __device__ __forceinline__ double enc(double v, double) { return v; }
  static __device__ __forceinline__ double dec(double v, double) { return v; }
  static __device__ __forceinline__ void ld2(const double* p, int64_t j, double, double, double& a, double& b) {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p + j));
    a = v.x;
    b = v.y;
  }
  static __device__ __forceinline__ void st2(double* p, int64_t j, double a, double b, double, double) {
    *reinterpret_cast<double2*>(p + j) = make_double2(a, b);
  }
};
// FP16 keeps the deviation times 2^12 (exact: a power of two), so that the
// small deviations left by the references stay out of FP16's subnormal range
// (below 2^-14), where precision would be absolute instead of relative;
// deviations up to 16 in magnitude fit.
// The difference from and the sum with the reference are explicitly rounded
// operations (__fsub_rn, __fadd_rn), which the compiler never fuses with the
// multiply that formed the reference (w_i rho): every kernel encodes and
// decodes with the same roundings, whatever it inlined around them.
constexpr float HALF_SCALE = 4096.0f, HALF_UNSCALE = 1.0f / 4096.0f;
template <>
struct Pop<__half> {
  using C = float;
  using V = __half2;
  static __device__ __forceinline__ float2 unpack(__half2 v, float ra, float rb) {
    return make_float2(fmaf(__low2float(v), HALF_UNSCALE, ra), fmaf(__high2float(v), HALF_UNSCALE, rb));
  }
  static __device__ __forceinline__ __half2 pack(float a, float b, float ra, float rb) {
    return __floats2half2_rn(__fsub_rn(a, ra) * HALF_SCALE, __fsub_rn(b, rb) * HALF_SCALE);
  }
  static __device__ __forceinline__ float ld(const __half* p, int64_t k, float ref) {
    return fmaf(__half2float(p[k]), HALF_UNSCALE, ref);
  }
  static __device__ __forceinline__ void st(__half* p, int64_t k, float v, float ref) {
    p[k] = __float2half_rn(__fsub_rn(v, ref) * HALF_SCALE);
  }
  static __device__ __forceinline__ __half enc(float v, float ref) { return __float2half_rn(__fsub_rn(v, ref) * HALF_SCALE); }
  static __device__ __forceinline__ float dec(__half v, float ref) { return fmaf(__half2float(v), HALF_UNSCALE, ref); }
  static __device__ __forceinline__ void ld2(const __half* p, int64_t j, float ra, float rb, float& a, float& b) {
    const __half2 v = __ldg(reinterpret_cast<const __half2*>(p + j));
    a = fmaf(__low2float(v), HALF_UNSCALE, ra);
    b = fmaf(__high2float(v), HALF_UNSCALE, rb);
  }
  static __device__ __forceinline__ void st2(__half* p, int64_t j, float a, float b, float ra, float rb) {
    *reinterpret_cast<__half2*>(p + j) = __floats2half2_rn(__fsub_rn(a, ra) * HALF_SCALE, __fsub_rn(b, rb) * HALF_SCALE);
  }
};
template <>
struct Pop<__nv_bfloat16> {
  using C = float;
  using V = __nv_bfloat162;
  static __device__ __forceinline__ float2 unpack(__nv_bfloat162 v, float ra, float rb) {
    return make_float2(__fadd_rn(__low2float(v), ra), __fadd_rn(__high2float(v), rb));
  }
  static __device__ __forceinline__ __nv_bfloat162 pack(float a, float b, float ra, float rb) {
    return __floats2bfloat162_rn(__fsub_rn(a, ra), __fsub_rn(b, rb));
  }
  static __device__ __forceinline__ float ld(const __nv_bfloat16* p, int64_t k, float ref) {
    return __fadd_rn(__bfloat162float(p[k]), ref);
  }
  static __device__ __forceinline__ void st(__nv_bfloat16* p, int64_t k, float v, float ref) {
    p[k] = __float2bfloat16_rn(__fsub_rn(v, ref));
  }
  static __device__ __forceinline__ __nv_bfloat16 enc(float v, float ref) { return __float2bfloat16_rn(__fsub_rn(v, ref)); }
  static __device__ __forceinline__ float dec(__nv_bfloat16 v, float ref) { return __fadd_rn(__bfloat162float(v), ref); }
  static __device__ __forceinline__ void ld2(const __nv_bfloat16* p, int64_t j, float ra, float rb, float& a,
                                             float& b) {
    const __nv_bfloat162 v = __ldg(reinterpret_cast<const __nv_bfloat162*>(p + j));
    a = __fadd_rn(__low2float(v), ra);
    b = __fadd_rn(__high2float(v), rb);
  }
  static __device__ __forceinline__ void st2(__nv_bfloat16* p, int64_t j, float a, float b, float ra, float rb) {
    *reinterpret_cast<__nv_bfloat162*>(p + j) = __floats2bfloat162_rn(__fsub_rn(a, ra), __fsub_rn(b, rb));
  }
};

// Where a step stores: the nine planes' base addresses, and those of the slots
// x - c_i, formed on the host. As kernel parameters they sit in constant
// memory, so that a store's address is one multiply-add of the node's padded
// index k.
template <typename T>
struct StorePtrs {
  char *own[9], *bounce[9];
  StorePtrs() = default;
  StorePtrs(T* f, const Geo& g) {
    for (int i = 0; i < 9; ++i) {
      own[i] = (char*)(f + pslot(g, i, 0));
      bounce[i] = (char*)(f + pslot(g, i, 0)) - (int64_t)(cx_of(i) + cy_of(i) * g.px) * 2 * (int64_t)sizeof(T);
    }
  }
  static __device__ __forceinline__ void st(char* base, uint32_t k, typename Pop<T>::V v) {
    *(typename Pop<T>::V*)(base + (uint64_t)k * (2 * sizeof(T))) = v;
  }
};

// ---------------------------------------------------------------------------
// Per-step constants.
enum { BC_MC = 0, BC_LLKC = 1, BC_VAVG = 2, BC_CONST = 3 };

struct Phys {
  double omega[2];   // 1 / tau
  double kF[2];      // 1 - 1 / (2 tau), the Guo prefactor of Eq. 4
  double G_AB;       // Eq. 5
  double G_s[2];     // Eq. 7
  double chi[2];     // Eq. 8
  double rho_s[2];   // constant solid densities
  double rho_ref[2]; // FP16/BF16 storage reference densities
  int bc, pairing, avg9;
  // Eq. 7 with the improved scheme's virtual densities, cross pairing and
  // G_As = G_Bs = G_AB: the solid neighbours then enter exactly like fluid
  // ones (the density plane holds rho~ there), so every node can take the
  // one-sum formula of a node without solid neighbours
  int uniform;
};

// The same constants in the arithmetic type of a kernel, converted once on
// the host (an FP32 kernel then does no FP64 conversions).
template <typename C>
struct PhysK {
  C omega[2];
  C kF[2];   // 1 - 1 / (2 tau)
  C k3[2];   // kF / 3
  C G_AB, G_s[2], chi[2], rho_s[2];
  int bc, pairing, avg9, uniform;
};

template <typename C>
inline PhysK<C> kphys(const Phys& p) {
  PhysK<C> k;
  for (int s = 0; s < 2; ++s) {
    k.omega[s] = C(p.omega[s]);
    k.kF[s] = C(p.kF[s]);
    k.k3[s] = C(p.kF[s] / 3.0);
    k.G_s[s] = C(p.G_s[s]);
    k.chi[s] = C(p.chi[s]);
    k.rho_s[s] = C(p.rho_s[s]);
  }
  k.G_AB = C(p.G_AB);
  k.bc = p.bc;
  k.pairing = p.pairing;
  k.avg9 = p.avg9;
  k.uniform = p.uniform;
  return k;
}

// sum_i w_i c_i phi(x + c_i) for the eight neighbour bits of a node's flags,
// in FP32 as the paired arithmetic forms it (a multiple of fl(1/9) plus one
// of fl(1/36), rounded once) and as the integer 36 sum_i w_i c_i phi. One
// 8-byte load (2 KB tables, resident in L1) in place of eight selects and a
// weighted sum.
struct WallPush {
  float2 w[256], w36[256];
  constexpr WallPush() : w(), w36() {
    constexpr double A = (double)(1.0f / 9.0f), D = (double)(1.0f / 36.0f);
    for (int m = 0; m < 256; ++m) {
      int ax = 0, ay = 0, dx = 0, dy = 0;
      for (int i = 1; i < 9; ++i)
        if (m >> (i - 1) & 1) {
          (i <= 4 ? ax : dx) += cx_of(i);
          (i <= 4 ? ay : dy) += cy_of(i);
        }
      w[m].x = (float)(ax * A + dx * D);
      w[m].y = (float)(ay * A + dy * D);
      w36[m].x = (float)(4 * ax + dx);
      w36[m].y = (float)(4 * ay + dy);
    }
  }
};
static __device__ const WallPush WALL_PUSH = WallPush();
__device__ __forceinline__ float2 wall_push(uint16_t fl) { return __ldg(&WALL_PUSH.w[(fl >> 1) & 0xFF]); }
__device__ __forceinline__ float2 wall_push36(uint16_t fl) { return __ldg(&WALL_PUSH.w36[(fl >> 1) & 0xFF]); }

// sum_i w_i c_i q_i over the eight moving directions (q[0] unused).
template <typename C>
__device__ __forceinline__ void weighted_sum(const C q[9], C& sx, C& sy) {
  const C d57 = q[5] - q[7], d86 = q[8] - q[6];
  sx = fma(q[1] - q[3], C(1.0 / 9.0), (d57 + d86) * C(1.0 / 36.0));
  sy = fma(q[2] - q[4], C(1.0 / 9.0), (d57 - d86) * C(1.0 / 36.0));
}

// Interaction force on both components at a fluid node (Eq. 5 restricted to
// fluid neighbours plus Eq. 7). nbP[s][i] is the value of the density plane
// of component s at x + c_i: the density at fluid nodes, rho~ at interface-
// solid nodes under the improved scheme, 0 at every other solid node; fl
// holds the neighbour bits (unused when !walls: no neighbour is solid). The
// zeros make the sum of Eq. 5 the same weighted sum at every node; with
// ph.uniform (see Phys) that sum also holds the solid part of Eq. 7. A node
// without solid neighbours gets the same bits whatever `walls` says.
template <typename C>
__device__ __forceinline__ void interaction_force(const PhysK<C>& ph, uint16_t fl, bool walls, const C rho[2],
                                                  const C nbP[2][9], C F[2][2]) {
  C ax[2], ay[2], bx[2], by[2];
  const C G = ph.G_AB;
  if (ph.bc != BC_VAVG || ph.uniform || !walls) {
#pragma unroll
    for (int s = 0; s < 2; ++s) weighted_sum(nbP[s], ax[s], ay[s]);
    if (ph.bc == BC_VAVG || !walls) {
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        F[s][0] = -rho[s] * (G * ax[1 - s]);
        F[s][1] = -rho[s] * (G * ay[1 - s]);
      }
      return;
    }
    const float2 v = wall_push36(fl);
    const C vx = C(v.x) * C(1.0 / 36.0), vy = C(v.y) * C(1.0 / 36.0);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      // the component whose solid pseudopotential enters Eq. 7
      const C rho_c = ph.pairing != 0 ? rho[s] : rho[1 - s];
      const C rs_c = ph.pairing != 0 ? ph.rho_s[s] : ph.rho_s[1 - s];
      const C c = ph.bc == BC_LLKC ? rho_c : rs_c;
      bx[s] = ph.bc == BC_MC ? vx : c * vx;
      by[s] = ph.bc == BC_MC ? vy : c * vy;
    }
  } else {
    // the improved scheme with other strengths or the self pairing: the fluid
    // and the solid part are summed apart
    C sx[2], sy[2], qf[9], qs[9];
    qf[0] = qs[0] = C(0);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        const bool solid = fl & nb_bit(i);
        qf[i] = solid ? C(0) : nbP[s][i];
        qs[i] = solid ? nbP[s][i] : C(0);
      }
      weighted_sum(qf, ax[s], ay[s]);
      weighted_sum(qs, sx[s], sy[s]);
    }
    const bool self = ph.pairing != 0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      bx[s] = self ? sx[s] : sx[1 - s];
      by[s] = self ? sy[s] : sy[1 - s];
    }
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    F[s][0] = -rho[s] * fma(G, ax[1 - s], ph.G_s[s] * bx[s]);
    F[s][1] = -rho[s] * fma(G, ay[1 - s], ph.G_s[s] * by[s]);
  }
}

// Momentum sum_i f_i c_i of one component, as paired differences.
template <typename C>
__device__ __forceinline__ void momentum(const C f[9], C& jx, C& jy) {
  jx = (f[1] - f[3]) + ((f[5] - f[7]) + (f[8] - f[6]));
  jy = (f[2] - f[4]) + ((f[5] - f[7]) + (f[6] - f[8]));
}

// rho = sum_i f_i (Eq. 3) as a balanced tree. The collision does not rely
// on rho being correctly rounded: it conserves mass through the rest
// population (see collide).
template <typename C>
__device__ __forceinline__ C density(const C f[9]) {
  return ((f[0] + (f[1] + f[3])) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8]));
}

// rho / 9 with one rounding: the product with the two-term split of 1/9. The
// rounded 1/9 alone makes every weight w_i too large by the same 2^-54.
__device__ __forceinline__ double rho_over_9(double rho) {
  constexpr double HI = 1.0 / 9.0;
  constexpr double LO = HI * 0x1p-54;  // 9 HI = 1 - 2^-54
  return fma(rho, HI, rho * LO);
}

// Force, velocity u of Eq. 3, BGK relaxation towards Eq. 2 and the Guo
// source of Eq. 4 at one fluid node in the FP64 compute type, in place
// (f: pulled populations on entry, f* on exit), each population's increment as
// collide2 forms it:
//   Delta_i = omega ((r - f_i) + r p_i) + S_i, r = w_i rho, with
//   p_+- = e +- 3 c.u, e = 4.5 (c.u)^2 - 1.5 u^2, and S_+- = E +- g,
//   g = 3 w_i (1 - 1/(2 tau)) c.F, E = 3 c.u g - 3 w_i (1 - 1/(2 tau)) u.F
// along c and -c, which share e, g and E. FP64 instructions run at 1/32 of the
// FP32 rate on this GPU and bound every FP64 pass: about 230 per node, where
// one direction at a time took 366 (45 simulations of 400 x 200 by two passes:
// 1290 -> 1005 us per step). Relaxing the sum and the difference of a pair
// instead (180; 839 us) rounds the O(1) part of each increment: against long
// double, after 300 steps of 160 droplets each, 0.76 to 1.7 times the error in
// rho (tau 1.6 to 0.6) and 1.25 to 1.37 times in the momentum; this form 0.68 to
// 1.005 and 0.94 to 1.005 times.
template <typename C>
__device__ __forceinline__ void update_node(C f[2][9], const C nbP[2][9], uint16_t fl, bool walls,
                                            const PhysK<C>& ph, C rho[2], C u[2]) {
  C jx[2], jy[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    rho[s] = density(f[s]);
    momentum(f[s], jx[s], jy[s]);
  }
  C F[2][2];
  interaction_force<C>(ph, fl, walls, rho, nbP, F);
  const C inv = C(1) / (rho[0] + rho[1]);
  const C ux = fma(C(0.5), F[0][0] + F[1][0], jx[0] + jx[1]) * inv;
  const C uy = fma(C(0.5), F[0][1] + F[1][1], jy[0] + jy[1]) * inv;
  const C cx3 = C(3) * ux, cy3 = C(3) * uy;
  const C c3[4] = {cx3, cy3, cx3 + cy3, cy3 - cx3};  // 3 c.u along 1, 2, 5, 6
  const C nusq3 = C(-3) * fma(ux, ux, uy * uy);
  C pp[4], pm[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const C e = C(0.5) * fma(c3[a], c3[a], nusq3);
    pp[a] = e + c3[a];
    pm[a] = e - c3[a];
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const C r9 = rho_over_9(rho[s]), r36 = C(0.25) * r9, om = ph.omega[s];
    const C gx = ph.k3[s] * F[s][0], gy = ph.k3[s] * F[s][1];
    const C uF = fma(ux, gx, uy * gy), uF4 = C(0.25) * uF, gx4 = C(0.25) * gx, gy4 = C(0.25) * gy;
    const C g[4] = {gx, gy, gx4 + gy4, gy4 - gx4};
    C acc = C(0);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int i = a < 2 ? a + 1 : a + 3, o = opp_of(i);
      const C r = a < 2 ? r9 : r36;
      const C E = fma(c3[a], g[a], a < 2 ? -uF : -uF4);
      const C dp = fma(om, fma(r, pp[a], r - f[s][i]), E + g[a]);
      const C dm = fma(om, fma(r, pm[a], r - f[s][o]), E - g[a]);
      acc = a == 0 ? dp : acc + dp;
      acc += dm;
      f[s][i] += dp;
      f[s][o] += dm;
    }
    f[s][0] -= acc;
  }
  u[0] = ux;
  u[1] = uy;
}

// Halfway bounce-back done by the writer. When the upstream node x - c_i of
// fluid node x is solid, what x receives along c_i at the next step is its
// own post-collision f*_opp(i) (Sec. 2); it is stored in slot i of that solid
// node (and its periodic images), which no other node writes, so that every
// pull reads f*_i(x - c_i) without a test. ref[s][d] is the encoding
// reference of the node's value along c_d, so slot i takes ref[s][opp(i)].
template <typename T, typename C>
__device__ __forceinline__ void store_bounced(T* __restrict__ fo, const Geo& g, int x, int y, uint16_t fl,
                                              const C fv[2][9], const C ref[2][9]) {
  if (!(fl & NB_ANY)) return;
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    if (!(fl & nb_bit(opp_of(i)))) continue;
    int sx = x - cx_of(i), sy = y - cy_of(i);
    if (g.per_x) sx = (sx + g.nx) % g.nx;
    if (g.per_y) sy = (sy + g.ny) % g.ny;
    const int ks = g.idx(sx, sy);
    const C a = fv[0][opp_of(i)], b = fv[1][opp_of(i)], ra = ref[0][opp_of(i)], rb = ref[1][opp_of(i)];
    Pop<T>::st2(fo, pslot(g, i, ks), a, b, ra, rb);
    for_ghost_images(g, sx, sy, [&](int kk) { Pop<T>::st2(fo, pslot(g, i, kk), a, b, ra, rb); });
  }
}

// store_bounced for a node that is not within GH + 1 of a periodic border:
// its solid neighbours are owned nodes without images, at padded index
// k - c_i.
template <typename T, typename C>
__device__ __forceinline__ void store_bounced_near(T* __restrict__ fo, const Geo& g, int k, uint16_t fl,
                                                   const C fv[2][9], const C ref[2][9]) {
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    if (!(fl & nb_bit(opp_of(i)))) continue;
    const int ks = k - cx_of(i) - cy_of(i) * g.px;
    Pop<T>::st2(fo, pslot(g, i, ks), fv[0][opp_of(i)], fv[1][opp_of(i)], ref[0][opp_of(i)], ref[1][opp_of(i)]);
  }
}

// Store the 18 post-collision populations of owned node (x, y) at padded
// index k, and at its periodic images.
template <typename T, typename C>
__device__ __forceinline__ void store_node(T* __restrict__ fo, const Geo& g, int x, int y, int k,
                                           const C fv[2][9], const C ref[2][9]) {
#pragma unroll
  for (int i = 0; i < 9; ++i) Pop<T>::st2(fo, pslot(g, i, k), fv[0][i], fv[1][i], ref[0][i], ref[1][i]);
  const bool img = (g.per_x && (x < GH || x >= g.nx - GH)) || (g.per_y && (y < GH || y >= g.ny - GH));
  if (img) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const C a = fv[0][i], b = fv[1][i], ra = ref[0][i], rb = ref[1][i];
      for_ghost_images(g, x, y, [&](int kk) { Pop<T>::st2(fo, pslot(g, i, kk), a, b, ra, rb); });
    }
  }
}

}  // namespace lbm
