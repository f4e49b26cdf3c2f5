// The fluid-node update of the two-pass schedule for the FP32 compute type
// (FP32, FP16 and BF16 storage) with the two components carried as one
// float2 pair (A in .x, B in .y). Components A and B go through the same
// arithmetic with their own rho, F, tau (Eqs. 1-5, 7 of arXiv:2009.12584),
// so each pair of scalar operations becomes one paired FP32 instruction
// (add/mul/fma .f32x2 of sm_100-family GPUs), each lane rounded as its
// scalar operation.
#pragma once

#include "lbm_common.cuh"
#include "lbm_geometry.cuh"

namespace lbm {

// Constants of the paired arithmetic, both lanes alike. A paired instruction
// takes no immediate: out of constant memory they are operands (or uniform
// registers) instead of register pairs that are set up again and again.
struct PairConst {
  float2 neg1, c025, cneg15, c3, cneg3, c45, c9, w9, w36, hi9, lo9;
};
static __constant__ PairConst KC = {
    {-1.0f, -1.0f},
    {0.25f, 0.25f},
    {-1.5f, -1.5f},
    {3.0f, 3.0f},
    {-3.0f, -3.0f},
    {4.5f, 4.5f},
    {9.0f, 9.0f},
    {1.0f / 9.0f, 1.0f / 9.0f},
    {1.0f / 36.0f, 1.0f / 36.0f},
    // 1/9 in two terms
    {(float)(1.0 / 9.0), (float)(1.0 / 9.0)},
    {(float)(1.0 / 9.0 - (double)(float)(1.0 / 9.0)), (float)(1.0 / 9.0 - (double)(float)(1.0 / 9.0))},
};

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b with the one rounding of the difference, as one paired instruction
// (the paired forms take no negated operand).
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, KC.neg1, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return __fmul2_rn(a, KC.neg1); }
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ float2 sel2(bool p, float2 a, float2 b) { return p ? a : b; }

// density() of both components, in the same order.
__device__ __forceinline__ float2 density_pair(const float2 f[9]) {
  return add2(add2(add2(f[0], add2(f[1], f[3])), add2(f[2], f[4])),
              add2(add2(f[5], f[7]), add2(f[6], f[8])));
}
__device__ __forceinline__ double2 density_pair(const double2 f[9]) {
  return make_double2(((f[0].x + (f[1].x + f[3].x)) + (f[2].x + f[4].x)) + ((f[5].x + f[7].x) + (f[6].x + f[8].x)),
                      ((f[0].y + (f[1].y + f[3].y)) + (f[2].y + f[4].y)) + ((f[5].y + f[7].y) + (f[6].y + f[8].y)));
}

// sum_i w_i c_i q_i over the eight moving directions for both components.
__device__ __forceinline__ void weighted_sum2(const float2 q[9], float2& sx, float2& sy) {
  const float2 d57 = sub2(q[5], q[7]), d86 = sub2(q[8], q[6]);
  sx = fma2(sub2(q[1], q[3]), KC.w9, mul2(add2(d57, d86), KC.w36));
  sy = fma2(sub2(q[2], q[4]), KC.w9, mul2(sub2(d57, d86), KC.w36));
}

// Eq. 5 (fluid neighbours) plus Eq. 7 for both components. q[i]: the
// density plane at x + c_i (rho at fluid nodes, rho~ at interface-solid
// nodes under the improved scheme, 0 at every other solid node, so that
// Eq. 5 is the same weighted sum at every node). With ph.uniform (the
// improved scheme with G_As = G_Bs = G_AB and Eq. 7's cross pairing) both
// sums are one weighted sum over the plane, the bulk formula.
template <bool GENERAL>
__device__ __forceinline__ void interaction_force2(const PhysK<float>& ph, uint16_t fl, float2 rho,
                                                   const float2 q[9], float2& Fx, float2& Fy) {
  const float2 G = f2(ph.G_AB);
  const float2 nrho = neg2(rho);
  float2 ax, ay;
  if (!GENERAL || ph.uniform) {
    weighted_sum2(q, ax, ay);
    // component s feels the other component's density
    Fx = mul2(nrho, mul2(G, swap2(ax)));
    Fy = mul2(nrho, mul2(G, swap2(ay)));
    return;
  }
  // the component whose solid pseudopotential enters Eq. 7: the other one
  // (cross pairing) or the same one (self pairing)
  const bool self = ph.pairing != 0;
  float2 bx, by;
  if (ph.bc == BC_VAVG) {
    float2 qf[9], qs[9], sx, sy;
    qf[0] = qs[0] = f2(0.0f);
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      const bool solid = fl & nb_bit(i);
      qf[i] = sel2(solid, f2(0.0f), q[i]);
      qs[i] = sel2(solid, q[i], f2(0.0f));
    }
    weighted_sum2(qf, ax, ay);
    weighted_sum2(qs, sx, sy);
    bx = self ? sx : swap2(sx);
    by = self ? sy : swap2(sy);
  } else {
    weighted_sum2(q, ax, ay);
    const float2 v = wall_push(fl);  // sum_i w_i phi(x + c_i) c_i
    float2 c = f2(1.0f);             // Martys-Chen: S = phi
    if (ph.bc == BC_LLKC) c = self ? rho : swap2(rho);
    if (ph.bc == BC_CONST) c = self ? f2(ph.rho_s[0], ph.rho_s[1]) : f2(ph.rho_s[1], ph.rho_s[0]);
    bx = mul2(c, f2(v.x));
    by = mul2(c, f2(v.y));
  }
  const float2 Gs = f2(ph.G_s[0], ph.G_s[1]);
  Fx = mul2(nrho, fma2(G, swap2(ax), mul2(Gs, bx)));
  Fy = mul2(nrho, fma2(G, swap2(ay), mul2(Gs, by)));
}

// rho / 9 with one rounding per component: the product with the two-term
// split of 1/9. Multiplying by the rounded 1/9 alone makes every weight w_i
// too large by the same 7.5e-9, so sum_i f^eq_i = rho (1 + 7.5e-9) and each
// collision would add that much mass at every node.
__device__ __forceinline__ float2 rho_over_9_2(float2 rho) {
  return fma2(rho, KC.hi9, mul2(rho, KC.lo9));
}

// BGK towards Eq. 2 plus the Guo source of Eq. 4: the moving populations
// take Delta_i = omega (f^eq_i - f_i) + S_i with f^eq_i - f_i = (rho w_i -
// f_i) + rho w_i p_i (p_i = 3 c.u + 4.5 (c.u)^2 - 1.5 u^2, the small part of
// Eq. 2's bracket, so that its O(1) part is never rounded) and S_i = w_i
// (1 - 1/(2 tau)) [3 c.F - 3 u.F + 9 (c.u)(c.F)]; the rest population takes
// minus their sum (sum_i Delta_i = 0 by Eqs. 2 and 4), so that the mass of a
// component changes only by the rounding of the nine final additions.
// Directions go as opposite pairs, which share c.u, c.F and their products;
// u is carried in both lanes, so that every operation is a paired one.
//
// PAIRS false: one direction at a time, u in one register and not in both lanes.
// The same bits, more instructions and fewer registers: for kernels held at 56
// to 64 registers, which spill otherwise (us per step with PAIRS, without:
// tiled batch of 45 x 400 x 200 FP32 144, 135; 4096^2 porous by k_tile_tma 598,
// 568, k_tile FP16 559, 550, k_tile FP32 453, 462; two-pass batch of 45 FP16
// 102.5, 100.7). The halo kernels have 72 and 80.
template <bool PAIRS>
__device__ __forceinline__ void collide2(float2 f[9], float2 rho, float ux, float uy, float2 Fx, float2 Fy,
                                         const PhysK<float>& ph) {
  if constexpr (!PAIRS) {
    const float nusq15 = -1.5f * fmaf(ux, ux, uy * uy);
    const float2 r9 = rho_over_9_2(rho);
    const float2 r36 = mul2(KC.c025, r9);  // exact
    const float2 om = f2(ph.omega[0], ph.omega[1]);
    const float2 k9 = mul2(f2(ph.kF[0], ph.kF[1]), KC.w9);
    const float2 k36 = mul2(f2(ph.kF[0], ph.kF[1]), KC.w36);
    const float2 nuF3 = mul2(KC.cneg3, fma2(f2(ux), Fx, mul2(f2(uy), Fy)));
    float2 acc = f2(0.0f);
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      const float cu = float(cx_of(i)) * ux + float(cy_of(i)) * uy;
      const float p = fmaf(cu, fmaf(4.5f, cu, 3.0f), nusq15);
      const float cu9 = 9.0f * cu;
      float2 cF;  // c_i . F (c_i components are -1, 0, 1)
      if (cx_of(i) == 0)
        cF = cy_of(i) > 0 ? Fy : neg2(Fy);
      else if (cy_of(i) == 0)
        cF = cx_of(i) > 0 ? Fx : neg2(Fx);
      else {
        const float2 a = cx_of(i) > 0 ? Fx : neg2(Fx);
        cF = cy_of(i) > 0 ? add2(a, Fy) : sub2(a, Fy);
      }
      const float2 src = mul2(i <= 4 ? k9 : k36, fma2(f2(cu9), cF, fma2(KC.c3, cF, nuF3)));
      const float2 ri = i <= 4 ? r9 : r36;
      const float2 delta = fma2(om, fma2(ri, f2(p), sub2(ri, f[i])), src);
      acc = add2(acc, delta);
      f[i] = add2(f[i], delta);
    }
    f[0] = sub2(f[0], acc);
    return;
  }
  const float2 ux2 = f2(ux), uy2 = f2(uy);
  const float2 nusq15 = mul2(KC.cneg15, fma2(ux2, ux2, mul2(uy2, uy2)));
  const float2 r9 = rho_over_9_2(rho);
  const float2 r36 = mul2(KC.c025, r9);  // exact
  const float2 om = f2(ph.omega[0], ph.omega[1]);
  const float2 k9 = mul2(f2(ph.kF[0], ph.kF[1]), KC.w9);
  const float2 k36 = mul2(f2(ph.kF[0], ph.kF[1]), KC.w36);
  const float2 nuF3 = mul2(KC.cneg3, fma2(ux2, Fx, mul2(uy2, Fy)));
  float2 acc = f2(0.0f);
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // axis directions 1 ... 4, then diagonal ones 5 ... 8
    float2 d[4];                 // their increments, summed in the order of the directions
    const float2 r = h == 0 ? r9 : r36, k = h == 0 ? k9 : k36;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const int i = 4 * h + a + 1, o = opp_of(i);
      float2 cu, cF;
      if (h == 0) {
        cu = a == 0 ? ux2 : uy2;
        cF = a == 0 ? Fx : Fy;
      } else {
        cu = a == 0 ? add2(ux2, uy2) : sub2(uy2, ux2);
        cF = a == 0 ? add2(Fx, Fy) : sub2(Fy, Fx);
      }
      const float2 pp = fma2(cu, fma2(KC.c45, cu, KC.c3), nusq15);
      const float2 pm = fma2(cu, fma2(KC.c45, cu, KC.cneg3), nusq15);
      const float2 cu9 = mul2(KC.c9, cu);
      const float2 sp = mul2(k, fma2(cu9, cF, fma2(KC.c3, cF, nuF3)));
      const float2 sm = mul2(k, fma2(cu9, cF, fma2(KC.cneg3, cF, nuF3)));
      d[a] = fma2(om, fma2(r, pp, sub2(r, f[i])), sp);
      d[a + 2] = fma2(om, fma2(r, pm, sub2(r, f[o])), sm);
      f[i] = add2(f[i], d[a]);
      f[o] = add2(f[o], d[a + 2]);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) acc = h == 0 && a == 0 ? d[0] : add2(acc, d[a]);
  }
  f[0] = sub2(f[0], acc);
}

// rho, force and velocity u of Eq. 3 of one fluid node; arguments as for
// update_pair.
template <bool GENERAL>
__device__ __forceinline__ float2 moments_pair(const float2 fp[9], const float2 q[9], uint16_t fl,
                                               const PhysK<float>& ph, float2& Fx, float2& Fy, float& ux, float& uy) {
  const float2 rho = density_pair(fp);
  interaction_force2<GENERAL>(ph, fl, rho, q, Fx, Fy);
  // momentum of each component as paired differences, then u of Eq. 3
  const float2 d57 = sub2(fp[5], fp[7]), d86 = sub2(fp[8], fp[6]);
  const float2 jx = add2(sub2(fp[1], fp[3]), add2(d57, d86));
  const float2 jy = add2(sub2(fp[2], fp[4]), sub2(d57, d86));
  const float inv = 1.0f / (rho.x + rho.y);
  ux = ((jx.x + jx.y) + 0.5f * (Fx.x + Fx.y)) * inv;
  uy = ((jy.x + jy.y) + 0.5f * (Fy.x + Fy.y)) * inv;
  return rho;
}

// Force, velocity and collision of one fluid node (Eqs. 1-5, 7): fp holds
// the pulled populations f_i of both components on entry and f*_i on exit;
// q[i] the density plane at x + c_i. GENERAL: the node may have solid
// neighbours (fl holds the neighbour bits); a node without any gets the
// same result on either path. Returns rho of both components and, in
// ux_out, uy_out, the velocity u of Eq. 3 the collision used.
template <bool GENERAL, bool PAIRS>
__device__ __forceinline__ float2 update_pair(float2 fp[9], const float2 q[9], uint16_t fl,
                                              const PhysK<float>& ph, float& ux_out, float& uy_out) {
  float2 Fx, Fy;
  const float2 rho = moments_pair<GENERAL>(fp, q, fl, ph, Fx, Fy, ux_out, uy_out);
  collide2<PAIRS>(fp, rho, ux_out, uy_out, Fx, Fy, ph);
  return rho;
}

}  // namespace lbm
