// Halo-tiled single-pass step: one kernel per time step, every population
// crosses HBM once, and (4- and 8-byte storage) no density plane.
//
// The step needs rho(t) at a fluid node's eight neighbours (Eq. 5) and,
// under the improved scheme, rho~(t) at its solid neighbours, which Eq. 8
// averages from rho(t) up to two nodes further out. Both are recomputed per
// tile from the populations themselves. One CTA takes a HALO_W x HALO_H
// tile. Its inputs arrive by the Tensor Memory Accelerator: the nine
// population planes over the tile's window, R + 1 nodes wider on each side
// (nine 3-D boxes), the encoding references there (16-bit storage: one 2-D
// box) and the tile's node list (one bulk copy), all counted on one
// mbarrier. No load holds registers or is addressed by the threads, and
// three or four CTAs per SM overlap one's copies with the others' updates.
// Out of shared memory,
//   phase A: rho(t) = sum_i f_i (Eq. 3), f_i(x) = f*_i(x - c_i, t), at every
//     fluid node of the tile and of the R rings around it (R = 3 under the
//     improved scheme, 1 otherwise);
//   phase V (improved scheme): Eq. 8 at the interface-solid cells of the
//     tile and its first ring (the other schemes keep 0 there);
//   phase B: each node of the tile evaluates Eqs. 5 and 7, u of Eq. 3 and
//     the collision (Eqs. 1, 2, 4) and stores f*(t+1) to HBM (with bounced
//     slots and periodic images; with 16-bit storage also the references of
//     what it stores).
// Every value is computed with the arithmetic, in the order, of the two-pass
// schedule, so the schedules agree bit for bit.
//
// Lists of a geometry, per tile: its fluid nodes (own nodes, then ring 1,
// then rings 2 and 3, each in row order), an entry holding the node's place
// in the window, its eight solid-neighbour bits and a border tag; and its
// interface-solid cells within ring 1 with their fluid neighbours (Eq. 8's
// 5 x 5 bits).
#pragma once

#include <type_traits>

#include "lbm.h"
#include "lbm_common.cuh"
#include "lbm_fused.cuh"
#include "lbm_geometry.cuh"
#include "lbm_kernels.cuh"
#include "lbm_tma.cuh"

namespace lbm {

constexpr int HALO_W = 32;  // owned columns of a tile
// Owned rows: three windows of three rings, or four of one ring, fill an SM's
// shared memory. Threads: the tile's own nodes of a porous medium (60% fluid)
// take one round or two at 72 to 80 registers each, R = 1 with four CTAs per
// SM, R = 3 with three. 4096^2 porous, us per step, improved scheme / LLKC:
// FP32 with 224 threads 400 / 357, with 256 395 / 367; FP16 375 / 315 and 367 /
// 335, with velocity references 449 and 433 (improved scheme). With 14 (20)
// rows and the window rows of all directions copied for each: FP32 406 / 363,
// FP16 387 / 330. Tiles of 28 x 18 (24) nodes, whose window rows take fewer
// 128-byte lines: FP32 404 / 374, FP16 387 / 338.
constexpr int HALO_H = 16, HALO_H16 = 20;
template <typename T>
constexpr int halo_h = sizeof(T) == 2 ? HALO_H16 : HALO_H;
__host__ __device__ inline int halo_rows(int elem_size) { return elem_size == 2 ? HALO_H16 : HALO_H; }
constexpr int HALO_O = 4;                        // entries count columns and rows from (x0 - 4, y0 - 4)
template <int R>
constexpr int halo_threads = R == 1 ? 224 : 256;
constexpr int HALO_AHEAD = 512;  // CTAs between one and that whose record it asks L2 for
constexpr int HALO_LIST_THREADS = 256;
constexpr int HALO_RW = HALO_W + 6;              // region of the lists: the tile and three rings
static_assert(HALO_W + 2 * HALO_O <= 64 && HALO_H + 2 * HALO_O <= 32 && HALO_H16 + 2 * HALO_O <= 32,
              "entries: 6 column bits, 5 row bits");

// List entry: column (bits 0-5) and row (6-10) from (x0 - 4, y0 - 4),
// solid-neighbour bits 1 ... 8 of the flags (11-18), border tag.
constexpr int HE_NB_SHIFT = 10;
constexpr uint32_t HE_BORDER = 1u << 19;  // own node within GH + 1 of a periodic border

inline int64_t halo_tile_count(const Geo& g, int H) {
  return (int64_t)((g.nx + HALO_W - 1) / HALO_W) * ((g.ny + H - 1) / H);
}
// Rings a step needs for the installed wetting scheme.
inline int halo_reach(const Phys& ph) { return ph.bc == BC_VAVG ? 3 : 1; }

// A tile that owns fluid nodes: its counts (own nodes, + ring 1, + rings 2
// and 3, interface-solid cells), its first entry (a multiple of 4: bulk
// copies start on 16 bytes) and first cell, and its number.
struct alignas(32) HaloTile {
  int4 n;
  int e0, i0, tile, member;  // member: in a batch's list, the simulation it belongs to
};
struct HaloLists {
  const HaloTile* work;  // in tile order
  int n_work;
  const uint32_t* entries;
  const uint2* cells;  // (place in the window as in an entry, 5 x 5 fluid bits)
};

// What a step needs of one simulation besides its tensor maps. P: the density
// plane that takes rho(t), the references of what a 16-bit step stores; Uo:
// with velocity references the velocity plane that does. err: the
// simulation's error word; stop: the word that keeps later CTAs of the step
// from starting (of a batch; err itself otherwise).
template <typename T>
struct HaloArgs {
  using C = typename Pop<T>::C;
  StorePtrs<T> out;
  C* P;
  UPair* Uo;
  const uint32_t* entries;
  const uint2* cells;
  int *err, *stop;
  int ntx;
  Geo g;
  PhysK<C> ph;
};

// Fluid neighbours of the cell at padded index k (k_iface_mask's bits).
__device__ __forceinline__ uint32_t fluid_mask25(const uint16_t* __restrict__ flags, const Geo& g, int k) {
  uint32_t m = 0;
#pragma unroll
  for (int dy = -2; dy <= 2; ++dy)
#pragma unroll
    for (int dx = -2; dx <= 2; ++dx)
      if ((dx != 0 || dy != 0) && !(flags[k + dx + dy * g.px] & F_SOLID)) m |= 1u << ((dy + 2) * 5 + (dx + 2));
  return m;
}

// One CTA per tile, two passes over the same fixed order (a slot per thread and
// chunk, its place by a scan over chunks and warps for each of the four lists:
// own nodes, ring 1, rings 2 and 3, interface-solid cells). Count pass: the
// tile's sizes and whether it owns nodes, which the scans turn into offsets
// and places in the work list. Write pass: work list, entries and cells.
template <bool WRITE>
__global__ void __launch_bounds__(HALO_LIST_THREADS)
    k_halo_lists(const uint16_t* __restrict__ flags, Geo g, int ntx, int H, int* __restrict__ eoff,
                 int* __restrict__ ioff, int* __restrict__ woff, HaloTile* __restrict__ work,
                 uint32_t* __restrict__ entries, uint2* __restrict__ cells) {
  constexpr int CHUNKS = 4, WARPS = HALO_LIST_THREADS / 32;
  static_assert(CHUNKS * HALO_LIST_THREADS >= HALO_RW * (HALO_H + 6) &&
                    CHUNKS * HALO_LIST_THREADS >= HALO_RW * (HALO_H16 + 6) && CHUNKS * WARPS == 32,
                "a region's slots, and one warp's scan over chunks and warps");
  __shared__ int place[4][32];
  __shared__ int total[4];
  const int tile = blockIdx.x;
  const int x0 = (tile % ntx) * HALO_W, y0 = (tile / ntx) * H;
  const int tw = min(HALO_W, g.nx - x0), th = min(H, g.ny - y0), RS = HALO_RW * (H + 6);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint16_t fl[CHUNKS];
  int list[CHUNKS];  // 0 ... 3, or -1
#pragma unroll
  for (int c = 0; c < CHUNKS; ++c) {
    const int slot = c * HALO_LIST_THREADS + threadIdx.x;
    const int row = slot / HALO_RW, col = slot - row * HALO_RW;
    // distance (max norm) from the owned rectangle
    const int dc = col < 3 ? 3 - col : (col >= 3 + tw ? col - (2 + tw) : 0);
    const int dr = row < 3 ? 3 - row : (row >= 3 + th ? row - (2 + th) : 0);
    const int ring = slot < RS ? max(dc, dr) : 99;
    fl[c] = ring <= 3 ? flags[g.idx(x0 - 3 + col, y0 - 3 + row)] : F_SOLID;
    list[c] = !(fl[c] & F_SOLID) ? min(ring, 2) : ring <= 1 && (fl[c] & F_IFACE) ? 3 : -1;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const unsigned ball = __ballot_sync(0xffffffffu, list[c] == l);
      if (lane == 0) place[l][c * WARPS + wid] = __popc(ball);
    }
  }
  __syncthreads();
  if (wid < 4) {
    const int v = place[wid][lane];
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += t;
    }
    place[wid][lane] = x - v;
    if (lane == 31) total[wid] = x;
  }
  __syncthreads();
  const int n0 = total[0], n1 = n0 + total[1], n3 = n1 + total[2];
  if (!WRITE) {
    if (threadIdx.x == 0) {
      eoff[tile] = n0 > 0 ? (n3 + 3) & ~3 : 0;
      ioff[tile] = n0 > 0 ? total[3] : 0;
      woff[tile] = n0 > 0;
    }
    return;
  }
  if (n0 == 0) return;
  const int e0 = eoff[tile], i0 = ioff[tile];
  if (threadIdx.x == 0) work[woff[tile]] = HaloTile{make_int4(n0, n1, n3, total[3]), e0, i0, tile, 0};
#pragma unroll
  for (int c = 0; c < CHUNKS; ++c) {
    const int slot = c * HALO_LIST_THREADS + threadIdx.x;
    const int row = slot / HALO_RW, col = slot - row * HALO_RW;
    const uint32_t at = (uint32_t)(col + 1) | (uint32_t)(row + 1) << 6;
    int pos = 0;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const unsigned ball = __ballot_sync(0xffffffffu, list[c] == l);
      if (list[c] == l)
        pos = place[l][c * WARPS + wid] + __popc(ball & ((1u << lane) - 1u)) + (l == 1 ? n0 : l == 2 ? n1 : 0);
    }
    if (list[c] < 0) continue;
    const int x = x0 - 3 + col, y = y0 - 3 + row;
    if (list[c] == 3)
      cells[i0 + pos] = make_uint2(at, fluid_mask25(flags, g, g.idx(x, y)));
    else
      entries[e0 + pos] = at | (uint32_t)(fl[c] & NB_ANY) << HE_NB_SHIFT |
                          (list[c] == 0 && near_border(g, x, y) ? HE_BORDER : 0u);
  }
}

// Shared memory of a CTA, in bytes from a 128-byte boundary.
template <typename T, int R, bool VR>
struct HaloSmem {
  using C = typename Pop<T>::C;
  // The window: the tile and R rings, R + 1 columns more on each side (four
  // with 16-bit storage, whose copies could not start on 16 bytes otherwise).
  // A plane's rows are those its direction pulls from, y - c_i.y; the
  // references, which every direction reads, have a row more on each side.
  static constexpr int H = halo_h<T>, O = kDev<T> ? 4 : R + 1, P = HALO_W + 2 * O;
  static constexpr int ROWS = H + 2 * R, CELLS = P * ROWS;
  static constexpr int pad(int n) { return (n + 127) / 128 * 128; }
  static constexpr int FBYTES = CELLS * 2 * (int)sizeof(T), FSLOT = pad(FBYTES);
  static constexpr int RBYTES = kDev<T> ? (CELLS + 2 * P) * (VR ? (int)sizeof(UPair) : 2 * (int)sizeof(C)) : 0;
  static constexpr int REF = 9 * FSLOT, RHO = REF + pad(RBYTES), ENT = RHO + pad(CELLS * 2 * (int)sizeof(C));
  static constexpr int BYTES = ENT + pad((HALO_W + 2 * R) * (H + 2 * R) * 4 + 16) + 128;
};

// The copies' barrier of a CTA, initialised while the kernel before it drains (us
// per step, after the wait / before it: 400 x 200 FP32 5.96 / 5.74, 1400 x 1000
// 42.3 / 41.9).
__device__ __forceinline__ void halo_bar_init(uint64_t& bar) {
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
}

// The work of one CTA on a tile with record h. mapf: tensor map of the
// populations (pairs; x in units of Pop<T>::V, FP64 of 8 bytes), with a box of
// one tile's window; mapref: of the references. a: the simulation's arguments,
// and entries its list, which the thread that issues the copies has at hand.
// smem_raw: shared memory of HaloSmem::BYTES; bar: see halo_bar_init. The error
// word is set to 1 when the copies were not seen to complete within the bound;
// extra_tx: see tma_issue. ready(): called once by every thread before the first
// use of a.
// stop: the stop word, as thread 0 read it. A CTA that finds it set does nothing
// (it would wait like the one that set it) and sets its own simulation's error
// word, whose step is missing then (in a batch the words are apart). Another CTA
// of the same launch may be setting the word, so one thread reads it, early, and
// the CTA's first barrier carries the answer: all of its threads go on or none
// does.
// eval: an EvalOut that takes the moments (rho^A, rho^B, u of Eq. 3) of the
// tile's nodes instead of a step, or NoEval; NaN where the wait ran out or the
// CTA stops, so that nothing older is taken for them.
struct NoEval {};
template <typename T, int R, bool VR, typename Ready, typename Eval = NoEval>
__device__ __forceinline__ void halo_tile(const HaloTile& h, const CUtensorMap* mapf, const CUtensorMap* mapref,
                                          const uint32_t* entries, const HaloArgs<T>& a, int stop, int ntx,
                                          unsigned char* smem_raw, uint64_t& bar, uint32_t extra_tx, Ready&& ready,
                                          const Eval& eval = Eval{}) {
  using C = typename Pop<T>::C;
  using V = typename CPair<C>::V;
  using S = HaloSmem<T, R, VR>;
  constexpr int NT = halo_threads<R>;
  constexpr uint32_t FB = 2 * sizeof(T);
  __shared__ int stopped;
  unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
  V* rho = (V*)(sm + S::RHO);
  const uint32_t* ent = (const uint32_t*)(sm + S::ENT);
  const int tid = threadIdx.x;
  const int n_own = h.n.x, n_a = R == 1 ? h.n.y : h.n.z, n_if = h.n.w, i0 = h.i0;
  const int x0 = (h.tile % ntx) * HALO_W, y0 = (h.tile / ntx) * S::H;
  auto give_up = [&] {
    if constexpr (!std::is_same<Eval, NoEval>::value) {
      const float nan = __int_as_float(0x7fffffff);
      for (int t = tid; t < n_own; t += NT) {
        const uint32_t e = __ldg(entries + h.e0 + t);
        const int x = x0 - HALO_O + (int)(e & 63u), y = y0 - HALO_O + (int)(e >> 6 & 31u);
        eval.put((int64_t)y * a.g.nx + x, nan, nan, nan, nan);
      }
    }
  };
  if (tid == 0 && (stopped = stop) == 0) {
    // the window's first node: column x0 - O + LP (a multiple of 4 nodes with
    // 16-bit storage, of 2 otherwise: 16-byte aligned), row y0 - R - c_i.y + GH
    const int xw = x0 - S::O + LP, yw = y0 - R + GH;
    const uint32_t ebytes = (uint32_t)((n_a + 3) & ~3) * 4;
    mbar_expect_tx(&bar, 9u * S::FBYTES + S::RBYTES + ebytes + extra_tx);
#pragma unroll
    for (int i = 0; i < 9; ++i) tma_load_3d(sm + i * S::FSLOT, mapf, sizeof(T) == 8 ? 2 * xw : xw, yw - cy_of(i), i, &bar);
    if (kDev<T>) tma_load_2d(sm + S::REF, mapref, VR ? 2 * xw : xw, yw - 1, &bar);
    bulk_load(sm + S::ENT, entries + h.e0, ebytes, &bar);
  }
  ready();
  __syncthreads();  // the barrier is initialised, or the CTA stops
  if (stopped) {
    if (tid == 0) atomicExch(a.err, 1);
    give_up();
    return;
  }
  const Geo& g = a.g;
  const PhysK<C>& ph = a.ph;
  // this thread's interface-solid cell, needed after phase A
  uint2 cell = make_uint2(0, 0);
  if (tid < n_if) cell = __ldg(a.cells + i0 + tid);
  // An entry's node in the window held in shared memory, and in cells of
  // the padded grid from the entries' node (0, 0).
  auto place = [](uint32_t e) {
    return (int)(e >> 6 & 31u) * S::P + (int)(e & 63u) - ((HALO_O - R) * S::P + HALO_O - S::O);
  };
  auto cells = [&](uint32_t e) { return (e >> 6 & 31u) * (uint32_t)g.px + (e & 63u); };
  // Post-streaming populations of the node at window place w.
  auto gather_node = [&](int w, uint16_t fl, V fp[9]) {
    const typename Pop<T>::V* win = (const typename Pop<T>::V*)sm;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const auto v = win[i * (S::FSLOT / (int)FB) + w - cx_of(i)];  // f*_i(x - c_i)
      C ra = C(0), rb = C(0);
      if constexpr (kDev<T>) {
        // the writer: x - c_i, or the node itself where that is solid (its
        // bounced value, sent along -c_i)
        const bool back = i != 0 && (fl & nb_bit(opp_of(i)));
        const int m = w + S::P - (back ? 0 : cx_of(i) + cy_of(i) * S::P);
        if constexpr (VR) {
          const UVal u = u_unpack(((const UPair*)(sm + S::REF))[m]);
          const float ca = cdot(i, u.v[0]), cb = cdot(i, u.v[1]);
          ra = ref_of(i, u.r[0], back ? -ca : ca);
          rb = ref_of(i, u.r[1], back ? -cb : cb);
        } else {
          const V r = ((const V*)(sm + S::REF))[m];
          ra = w_of<C>(i) * r.x;
          rb = w_of<C>(i) * r.y;
        }
      }
      fp[i] = Pop<T>::unpack(v, ra, rb);
    }
  };

  bool ok = mbar_wait(&bar, 0);
  if (!ok) ok = mbar_wait(&bar, 0);  // the copies in flight, once more

  // phase A; the populations of a thread's first node, which is one of the
  // tile's own or a ring node, stay in registers for phase B (4096^2 porous
  // FP16 387 -> 375 us per step, FP32 402 -> 400)
  V fp[9];
  if (ok) {
    if (tid < n_a) {
      const uint32_t e = ent[tid];
      const int w = place(e);
      gather_node(w, (e >> HE_NB_SHIFT) & NB_ANY, fp);
      rho[w] = density_pair(fp);
    }
    for (int t = tid + NT; t < n_a; t += NT) {
      const uint32_t e = ent[t];
      const int w = place(e);
      V fr[9];
      gather_node(w, (e >> HE_NB_SHIFT) & NB_ANY, fr);
      rho[w] = density_pair(fr);
    }
    if (R == 1)
      for (int t = tid; t < n_if; t += NT) {
        V z;
        z.x = z.y = C(0);
        rho[place(t == tid ? cell.x : __ldg(a.cells + i0 + t).x)] = z;
      }
  }
  if (__syncthreads_or(!ok)) {
    if (tid == 0) {
      atomicExch(a.err, 1);
      atomicExch(a.stop, 1);
    }
    give_up();
    return;
  }

  // phase V
  if (R == 3) {
    for (int t = tid; t < n_if; t += NT) {
      const uint2 cl = t == tid ? cell : __ldg(a.cells + i0 + t);
      const int w = place(cl.x);
      auto load = [&](int dx, int dy, C& a, C& b) {
        const V v = rho[w + dx + dy * S::P];
        a = v.x;
        b = v.y;
      };
      V v;
      if (ph.avg9)
        virtual_density_at<C, true, 1>(cl.y, ph, load, v.x, v.y);
      else
        virtual_density_at<C, false, 1>(cl.y, ph, load, v.x, v.y);
      rho[w] = v;
    }
    __syncthreads();
  }

  // phase B
  const int korg = g.idx(x0 - HALO_O, y0 - HALO_O);  // padded index of the entries' node (0, 0)
  for (int b = 0; b < n_own; b += NT) {
    const bool valid = b + tid < n_own;
    const uint32_t e = valid ? ent[b + tid] : 0u;
    const uint16_t fl = (e >> HE_NB_SHIFT) & NB_ANY;
    const bool warp_edge = __any_sync(0xffffffffu, fl != 0);
    const bool warp_border = __any_sync(0xffffffffu, (e & HE_BORDER) != 0);
    if (!valid) continue;
    const int w = place(e);
    const uint32_t kp = (uint32_t)korg + cells(e);  // padded index
    V q[9];
    if (b > 0) gather_node(w, fl, fp);
    q[0].x = q[0].y = C(0);
#pragma unroll
    for (int i = 1; i < 9; ++i) q[i] = rho[w + cx_of(i) + cy_of(i) * S::P];
    const int x = x0 - HALO_O + (int)(e & 63u), y = y0 - HALO_O + (int)(e >> 6 & 31u);
    if constexpr (!std::is_same<Eval, NoEval>::value) {
      float2 Fx, Fy;
      float ux, uy;
      const float2 r = warp_edge ? moments_pair<true>(fp, q, fl, ph, Fx, Fy, ux, uy)
                                 : moments_pair<false>(fp, q, fl, ph, Fx, Fy, ux, uy);
      eval.put((int64_t)y * g.nx + x, r.x, r.y, ux, uy);
      continue;
    }
    C ref[2][9], rh[2], u[2];
    UVal U{};
    update_pairs<C>(fp, q, fl, warp_edge, ph, rh, u);
    if constexpr (kDev<T>) {
      // the references of what this node stores, for its readers
      const V rv = f2(rh[0], rh[1]);
      UPair up{};
      if constexpr (VR) {
        // momentum of each component's post-collision populations
        const float2 d57 = sub2(fp[5], fp[7]), d86 = sub2(fp[8], fp[6]);
        up = u_pack(add2(sub2(fp[1], fp[3]), add2(d57, d86)), add2(sub2(fp[2], fp[4]), sub2(d57, d86)), rv);
        U = u_unpack(up);
        a.Uo[kp] = up;
      } else {
        stP(a.P, kp, rh[0], rh[1]);
      }
      if (warp_border) {
        for_ghost_images(g, x, y, [&](int kk) {
          if constexpr (VR)
            a.Uo[kk] = up;
          else
            stP(a.P, kk, rh[0], rh[1]);
        });
      }
    }
    write_refs<T>(rh, VR, U, ref);
    if (!warp_border) {
#pragma unroll
      for (int i = 0; i < 9; ++i) StorePtrs<T>::st(a.out.own[i], kp, Pop<T>::pack(fp[i].x, fp[i].y, ref[0][i], ref[1][i]));
      if (warp_edge) {
        // the solid neighbours are owned nodes without images: slot i of x - c_i
#pragma unroll
        for (int i = 1; i < 9; ++i) {
          const int o = opp_of(i);
          if (fl & nb_bit(o)) StorePtrs<T>::st(a.out.bounce[i], kp, Pop<T>::pack(fp[o].x, fp[o].y, ref[0][o], ref[1][o]));
        }
      }
    } else {
      C fv[2][9];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        fv[0][i] = fp[i].x;
        fv[1][i] = fp[i].y;
      }
      T* fo = (T*)a.out.own[0];
      store_node(fo, g, x, y, (int)kp, fv, ref);
      store_bounced(fo, g, x, y, fl, fv, ref);
    }
  }
}

// A step of one simulation, a CTA per tile that owns fluid nodes. FP64 is bound by its arithmetic, not by the one CTA per SM that its
// windows allow.
template <typename T, int R, bool VR>
__global__ void __launch_bounds__(halo_threads<R>, sizeof(T) == 8 ? 1 : R == 1 ? 4 : 3)
    k_halo(const __grid_constant__ CUtensorMap mapf, const __grid_constant__ CUtensorMap mapref,
           const __grid_constant__ HaloArgs<T> a, const HaloTile* __restrict__ work, uint32_t extra_tx) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  halo_bar_init(bar);
  HaloTile h;
  h.n = __ldg(&work[blockIdx.x].n);
  *(int4*)&h.e0 = __ldg((const int4*)&work[blockIdx.x].e0);
  pdl_wait();  // the step before; what is read above, a geometry's lists, it does not write
  const int stop = threadIdx.x == 0 ? *(const volatile int*)a.stop : 0;
  if (threadIdx.x == 32 && blockIdx.x + HALO_AHEAD < gridDim.x)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(work + blockIdx.x + HALO_AHEAD));
  halo_tile<T, R, VR>(h, &mapf, &mapref, a.entries, a, stop, a.ntx, smem_raw, bar, extra_tx, [] {});
}

// The moments of the current state at fluid nodes, one launch where the
// general evaluation takes a density pass, the Eq. 8 pass and its own (1400 x
// 1000, eight steps, the diagnostics and the moments: 481 -> 410 us; 512
// members read one by one: 16.5 -> 7 ms).
template <typename T, int R, bool VR, typename O>
__global__ void __launch_bounds__(halo_threads<R>, R == 1 ? 4 : 3)
    k_halo_moments(const __grid_constant__ CUtensorMap mapf, const __grid_constant__ CUtensorMap mapref,
                   const __grid_constant__ HaloArgs<T> a, const HaloTile* __restrict__ work, uint32_t extra_tx,
                   const __grid_constant__ EvalOut<O> out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  halo_bar_init(bar);
  HaloTile h;
  h.n = __ldg(&work[blockIdx.x].n);
  *(int4*)&h.e0 = __ldg((const int4*)&work[blockIdx.x].e0);
  pdl_wait();
  const int stop = threadIdx.x == 0 ? *(const volatile int*)a.stop : 0;
  halo_tile<T, R, VR>(h, &mapf, &mapref, a.entries, a, stop, a.ntx, smem_raw, bar, extra_tx, [] {}, out);
}

}  // namespace lbm
