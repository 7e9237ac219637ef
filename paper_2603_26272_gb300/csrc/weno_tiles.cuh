// weno_tiles.cuh -- the stage kernels of the central-upwind WENO right-hand
// side and the SSP-RK3 stage update for GB300 (sm_103a), templated on the
// stencil half-width r (scheme of order 2r; r = 3 is WENO-ZA6 of Section 3,
// r = 2, 4, 5 the schemes of the Appendix).  Included by weno_kernels.cu
// (r = 3) and weno_orders.cu (r = 2, 4, 5); everything here has internal
// linkage in each translation unit.
//
// One launch = one Runge-Kutta stage over every problem of the batch
// (Section 4 preamble: third-order TVD Runge-Kutta).  A block owns a tile of
// cells and runs three phases:
//   1. stage the tile and its r-cell halo (the 2r-point stencil of eq. (7))
//      into shared memory, with ghost cells by index clamp or wrap, and form
//      per-cell primitives and physical fluxes once;
//   2. compute every interface flux of the tile exactly once -- in 2D the x-
//      and y-faces of one tile come from the same staged data (dimension by
//      dimension, Section 4.3) -- by characteristic-wise global
//      Lax-Friedrichs splitting (eq. (6), Section 4.2) and the central-upwind
//      WENO flux (Sections 2-3) for the positive and the mirrored negative
//      flux;
//   3. per cell, the conservative difference of eq. (5), the Runge-Kutta
//      combination, and -- for the next stage -- the block's maxima of the
//      characteristic speeds, reduced with warp shuffles and one atomicMax
//      per value and block.
#pragma once
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include <cuda.h>  // CUtensorMap (the type only; the encoder is fetched at run time)

#include "weno_device.cuh"
#include "weno_internal.h"

namespace weno {
namespace {

constexpr int kThreads2D = 256;
constexpr int kTX = 32, kTY = 16;
constexpr int kThreads1D = 128;
constexpr int kT1 = kThreads1D - 1;  // cells per 1D tile: one face per thread

__device__ __forceinline__ long long ghost(long long k, long long n, int bc) {
  if (bc == 1) {
    long long m = k % n;
    return m < 0 ? m + n : m;
  }
  return k < 0 ? 0 : (k >= n ? n - 1 : k);
}

__device__ __forceinline__ double bits2d(unsigned long long u) {
  return __longlong_as_double((long long)u);
}

__device__ void record_status(DevStatus *st, int code, int stage, long long b, long long j,
                              long long i) {
  if (atomicCAS(&st->code, 0, code) == 0) {
    st->stage = stage;
    st->b = b;
    st->j = j;
    st->i = i;
  }
}

// CFL step of problem b from its speed maxima (bit patterns), the rule of
// the oracle: 1D cfl dx / max(|u|+c); 2D cfl / (max(|u|+c)/dx + max(|v|+c)/dy).
// max(|u-c|, |u+c|) = |u| + c exactly (same rounding).
// Scalar systems 2, 3 keep okey(max u) and okey(max -u) in slots 0 and 1.
__device__ __forceinline__ double scalar_alpha_of(int system, double adv, double ustar,
                                                  const unsigned long long *al) {
  if (system == 0) return fabs(adv);
  const double umax = okey_inv(al[0]), umin = -okey_inv(al[1]);
  return scalar_alpha(system, adv, umin, umax, ustar);
}

__device__ double cfl_dt(int system, int ndim, int nc, double cfl, double dx, double dy,
                         double adv, const unsigned long long *al, double ustar = 0.0) {
  if (system == 0) return cfl * dx / fabs(adv);
  if (system >= 2) return cfl * dx / scalar_alpha_of(system, adv, ustar, al);
  const unsigned long long sxb = max(al[0], al[nc == 3 ? 2 : 3]);
  const double sx = bits2d(sxb);
  if (ndim == 1) return cfl * dx / sx;
  const double sy = bits2d(max(al[4], al[7]));
  return cfl / (sx / dx + sy / dy);
}

// Block-level control shared by every stage kernel: clears the slot of the
// stage after next, decides this problem's dt, advances its clock.
// Returns false if the block has nothing to do.
__device__ bool stage_control(const StageArgs &a, long long b, bool first_block_of_b,
                              bool zeroing_block, double &dt_out) {
  __shared__ double s_dt;
  __shared__ int s_go;
  if (a.alpha_zero && zeroing_block)
    for (long long k = threadIdx.x; k < a.nbatch * 8; k += blockDim.x) a.alpha_zero[k] = 0ull;
  if (threadIdx.x == 0) {
    int go = 1;
    double dt = 0.0;
    if (*(volatile int *)&a.status->code != 0) {
      go = 0;
    } else if (a.mode == 0) {
      if (a.stage == 1) {
        const double t = a.t[b];
        if (!(t < a.t_final)) {
          go = 0;
          if (first_block_of_b) a.dt[b] = 0.0;
        } else {
          dt = a.dt_fixed > 0.0 ? a.dt_fixed
                                : cfl_dt(a.system, a.ndim, a.nc, a.cfl, a.dx, a.dy,
                                         a.adv_speed, a.alpha_in + b * 8, a.ustar);
          const double rem = a.t_final - t;
          const bool last = !(dt < rem);
          if (last) dt = rem;
          if (first_block_of_b) {
            a.dt[b] = dt;
            a.tnext[b] = last ? a.t_final : t + dt;
          }
        }
      } else {
        dt = a.dt[b];
        if (dt == 0.0) go = 0;
        if (go && a.stage == 3 && first_block_of_b) {
          a.t[b] = a.tnext[b];
          a.steps[b] += 1;
        }
      }
    }
    s_dt = dt;
    s_go = go;
  }
  __syncthreads();
  dt_out = s_dt;
  return s_go != 0;
}

// The scheme's constants into shared memory (published by the caller's next
// barrier).
__device__ __forceinline__ const SchemeParams &scheme_of(const StageArgs &a) {
  return a.sp_at ? *a.sp_at : a.sp;
}
__device__ __forceinline__ void load_scheme(const StageArgs &a, SchemeParams &s) {
  static_assert(sizeof(SchemeParams) % 8 == 0, "copied as doubles");
  const double *const src = reinterpret_cast<const double *>(&scheme_of(a));
  for (int k = threadIdx.x; k < (int)(sizeof(SchemeParams) / 8); k += blockDim.x)
    reinterpret_cast<double *>(&s)[k] = src[k];
}

// Block reduction of NV maxima (bit patterns) and one atomicMax per value into
// dst[slot[q]], and also into dst[dup[q]] where dup[q] >= 0 (the entropy and
// shear fields share the speed |u|).
template <int NV>
__device__ void block_max_atomic(unsigned long long (&v)[NV], unsigned long long *dst,
                                 const int (&slot)[NV], const int (&dup)[NV]) {
  __shared__ unsigned long long red[32][NV];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] = max(v[q], __shfl_xor_sync(0xffffffffu, v[q], o));
  }
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < NV; ++q) red[warp][q] = v[q];
  __syncthreads();
  if (threadIdx.x < NV) {
    unsigned long long m = 0;
    for (int w = 0; w < nw; ++w) m = max(m, red[w][threadIdx.x]);
    atomicMax(dst + slot[threadIdx.x], m);
    if (dup[threadIdx.x] >= 0) atomicMax(dst + dup[threadIdx.x], m);
  }
}

// ---------------------------------------------------------------------------
// Tensor-memory-accelerator (TMA) staging of a 2D tile: one bulk tensor copy
// brings the conserved variables of the tile and its halo -- a box of
// (TX + 2 XO) x (TY + 2 R) cells of all four planes of the problem -- from
// global into shared memory, completing on an mbarrier.  XO is R rounded up
// to even, so the box starts at x = i0 - XO, a multiple of 2 doubles: the
// 16-byte alignment a tiled copy needs for its innermost coordinate.  Only
// interior tiles (the whole box inside the grid) use it; tiles that need
// ghost cells (clamp, wrap, halo rows) load with plain indexed loads.
// ---------------------------------------------------------------------------
template <int R> struct TmaBox {
  static constexpr int XO = (R + 1) & ~1;
};

template <int TX, int TY, int R>
__host__ __device__ constexpr size_t tma_box_bytes() {
  return sizeof(double) * 4 * (TX + 2 * TmaBox<R>::XO) * (TY + 2 * R);
}

__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}

// Issue the copy (thread 0 only): barrier armed with the byte count first.
__device__ __forceinline__ void tma_issue_box(const CUtensorMap *tm, unsigned bar, void *dst,
                                              int x, int y, int z, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(tm), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// SM clock cycles a TMA wait may take before it gives up (about 1 ms at
// 2 GHz; the copy of one box takes microseconds).  The clock runs on while another
// process has the GPU, so that a poll that was interrupted would use them all up (four
// processes at once saw WENO_ERR_TIMEOUT): no more than kTmaPollCycles of it count
// between two polls.
constexpr long long kTmaWaitCycles = 2000000, kTmaPollCycles = 20000;
__device__ __forceinline__ bool tma_wait(unsigned bar) {
  long long left = kTmaWaitCycles, t = clock64();
  bool done;
  while (!(done = mbar_try_wait(bar, 0)) && left > 0) {
    const long long now = clock64(), dt = now - t;
    left -= dt > 0 && dt < kTmaPollCycles ? dt : kTmaPollCycles;
    t = now;
  }
  return done;
}

// The TMA copy of tile (i0, j0)'s box of problem b into `box` (every thread
// of the block calls this).  Returns false -- after recording
// WENO_ERR_TIMEOUT and a second bounded wait for the copy in flight, which
// writes into this block's shared memory -- when the copy did not complete
// in time; the tile is then left undone.
template <int TX, int TY, int R>
__device__ bool tma_stage_box(const StageArgs &a, const CUtensorMap *tm, double *box, long long b,
                              long long i0, long long j0) {
  __shared__ __align__(8) unsigned long long s_bar;
  const unsigned bar = smem_u32(&s_bar);
  const int tid = threadIdx.x;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  if (tid == 0) {
    if (a.tma_no_copy)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                   "r"((unsigned)tma_box_bytes<TX, TY, R>())
                   : "memory");
    else
      tma_issue_box(tm, bar, box, (int)(i0 - TmaBox<R>::XO), (int)(j0 - R), (int)(b * 4),
                    (unsigned)tma_box_bytes<TX, TY, R>());
  }
  const bool done = tma_wait(bar);
  if (!__syncthreads_and(done)) {
    if (tid == 0) record_status(a.status, 5, a.stage, b, j0, i0);
    tma_wait(bar);
    return false;
  }
  return true;
}

// Where staged cell (r, c) of tile (i0, j0) -- r in [0, TY + 2R), c in
// [0, TX + 2R), the tile's cells at [R, R + TY) x [R, R + TX) -- is read from
// without TMA: the array src with plane stride pst and offset o (the stage
// input, or a neighbour's halo rows of a domain split), after the ghost rule
// of each boundary; (gj, gi) is the cell reported on error.
__device__ __forceinline__ void cell_source(const StageArgs &a, const double *Ub, long long b,
                                            long long i0, long long j0, int R, int r, int c,
                                            const double *&src, long long &o, long long &pst,
                                            long long &gj, long long &gi) {
  gi = ghost(i0 - R + c, a.nx, a.bc_x);
  const long long jj = j0 - R + r;
  src = Ub;
  pst = a.nx * a.ny;
  gj = jj;
  if (jj < 0 && a.halo_lo) {  // a neighbour's rows below this strip
    src = a.halo_lo + b * 4 * (R * a.nx);
    o = (jj + R) * a.nx + gi;
    pst = R * a.nx;
  } else if (jj >= a.ny && a.halo_hi) {  // above it (rows beyond ny+R-1 only
    src = a.halo_hi + b * 4 * (R * a.nx);  // fill a partial tile: any halo row)
    o = min(jj - a.ny, (long long)(R - 1)) * a.nx + gi;
    pst = R * a.nx;
  } else {
    gj = ghost(jj, a.ny, a.bc_y);
    o = gj * a.nx + gi;
  }
}

// The speed maxima of eq. (6) are exact, but most cells are far from setting
// one: a cell whose FP32 estimates stay below what the six maxima have already
// reached needs no FP64 speeds (22 FP64 operations, a tenth of a stage's).
// Floors: the next stage's slot as it stands (any earlier value is a lower
// bound of the final maximum).
__device__ __forceinline__ constexpr int speed_slot(int q) {  // |u-c|, |u|, |u+c|, |v-c|, |v|, |v+c|
  return q == 0 ? 0 : (q == 1 ? 1 : (q == 2 ? 3 : (q == 3 ? 4 : (q == 4 ? 5 : 7))));
}
__device__ __forceinline__ float speed_floor(const unsigned long long *slot, int q) {
  return f32_rn(bits2d(__ldcg(slot + speed_slot(q))));
}
// True where the state is physical and none of its speeds can reach its floor,
// with a margin of 2^-9 of the speeds for the FP32 arithmetic (p above 2^-12 E,
// so the sound speed is good to 2^-11); false (FP64 decides) for anything else,
// NaN and magnitudes near FP32's limits included: c^2 has to be a normal number
// (a cold, dense cell's is flushed to 0, and its c would be missing).
__device__ __forceinline__ bool speeds_below(double rho, double mx, double my, double E, float gg,
                                             const float *floors) {
  const float r = f32_rn(rho), m = f32_rn(mx), n = f32_rn(my), e = f32_rn(E);
  const float ir = fx::rcpf(r), u = m * ir, v = n * ir;
  const float pe = e - 0.5f * (m * u + n * v);
  if (!(r > 1e-18f && r < 1e18f && e > 1e-18f && e < 1e18f && pe > e * 0x1p-12f)) return false;
  const float cc = gg * pe * ir;
  if (!(cc >= 0x1p-126f)) return false;
  float c;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(c) : "f"(cc));
  const float mg = 0x1p-9f * (fmaxf(fabsf(u), fabsf(v)) + c);
  return fabsf(u - c) + mg < floors[0] && fabsf(u) + mg < floors[1] &&
         fabsf(u + c) + mg < floors[2] && fabsf(v - c) + mg < floors[3] &&
         fabsf(v) + mg < floors[4] && fabsf(v + c) + mg < floors[5];
}

// Phase 3 of a 2D tile: per cell the conservative difference of eq. (5)
// from the faces' multiples of F (the factor goes with idx, idy), the
// Runge-Kutta combination with the staged input u_at(r, c, q) of tile cell
// (r, c), the strips' send rows, and the next stage's speed maxima.
template <int TX, int TY, int R, class UAt>
__device__ __forceinline__ void tile2d_update(const StageArgs &a, long long b, long long i0,
                                              long long j0, double dt, const double *fx,
                                              const double *fy, double idx, double idy,
                                              UAt u_at) {
  const long long plane = a.nx * a.ny;
  const double gm1 = a.gamma - 1.0;
  const int tid = threadIdx.x;
  unsigned long long mx6[6] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
  const bool want_alpha = (a.mode == 0) && (a.alpha_out != nullptr);
  const float gg = (float)(a.gamma * gm1);
  const bool filter = want_alpha && a.speed_filter;
  __shared__ float floors[6];
  if (filter) {
    if (tid < 6) floors[tid] = speed_floor(a.alpha_out + b * 8, tid);
    __syncthreads();
  }
  for (int k = tid; k < TX * TY; k += blockDim.x) {
    const int r = k / TX, c = k - r * TX;
    const long long gi = i0 + c, gj = j0 + r;
    if (gi >= a.nx || gj >= a.ny) continue;
    const double *Fl = &fx[(r * (TX + 1) + c) * 4];
    const double *Fr = Fl + 4;
    const double *Gb = &fy[(r * TX + c) * 4];
    const double *Gt = &fy[((r + 1) * TX + c) * 4];
    const long long o = b * 4 * plane + gj * a.nx + gi;
    double uo[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double L = -(Fr[q] - Fl[q]) * idx - (Gt[q] - Gb[q]) * idy;
      if (a.mode == 1) {
        uo[q] = L;
      } else {
        const double base_s = fma(dt, L, u_at(r, c, q));
        uo[q] = (a.a_n != 0.0) ? fma(a.a_n, a.Un[o + q * plane], a.a_s * base_s) : a.a_s * base_s;
      }
      a.Uout[o + q * plane] = uo[q];
    }
    if (a.send_lo && gj < R)  // edge rows of the output for the strips below / above
#pragma unroll
      for (int q = 0; q < 4; ++q) a.send_lo[((b * 4 + q) * R + gj) * a.nx + gi] = uo[q];
    if (a.send_hi && gj >= a.ny - R)
#pragma unroll
      for (int q = 0; q < 4; ++q) a.send_hi[((b * 4 + q) * R + (gj - (a.ny - R))) * a.nx + gi] = uo[q];
    if (want_alpha && !(filter && speeds_below(uo[0], uo[1], uo[2], uo[3], gg, floors))) {
      const double ir = rcp_pos(uo[0]);
      const double u = uo[1] * ir, v = uo[2] * ir;
      const double p = gm1 * (uo[3] - 0.5 * fma(uo[1], u, uo[2] * v));
      if (!(pos_finite(uo[0]) && pos_finite(p))) record_status(a.status, 3, a.stage, b, gj, gi);
      const double cs = sqrt_pos(a.gamma * p * ir);
      mx6[0] = max(mx6[0], abs_bits(u - cs));
      mx6[1] = max(mx6[1], abs_bits(u));
      mx6[2] = max(mx6[2], abs_bits(u + cs));
      mx6[3] = max(mx6[3], abs_bits(v - cs));
      mx6[4] = max(mx6[4], abs_bits(v));
      mx6[5] = max(mx6[5], abs_bits(v + cs));
    }
  }
  if (want_alpha) {
    const int slot[6] = {0, 1, 3, 4, 5, 7};
    const int dup[6] = {-1, 2, -1, -1, 6, -1};
    block_max_atomic<6>(mx6, a.alpha_out + b * 8, slot, dup);
  }
}

// ---------------------------------------------------------------------------
// 2D Euler stage kernel of the orders 4, 8, 10 (R = 2, 4, 5).
// Shared planes per staged cell: 0 rho, 1 rho u, 2 rho v, 3 E, 4 u, 5 v, 6 H,
// 7 sqrt(rho), 8 p (the fluxes are projected from u, v, p: project_flux4).
// ---------------------------------------------------------------------------
constexpr int kPlanes2D = 9;

template <int TX, int TY, int R>
__host__ __device__ constexpr size_t smem_euler2d_gen() {
  return sizeof(double) *
         (kPlanes2D * (TX + 2 * R) * (TY + 2 * R) + 4 * ((TX + 1) * TY + TX * (TY + 1)));
}

// Layout of the sixth-order tile (euler2d_tile6), in doubles, after the
// 128-byte aligned start: box, Roe planes, cell-pair differences, faces.
template <int TX, int TY> struct Tile6 {
  static constexpr int R = 3, XO = TmaBox<3>::XO;
  static constexpr int W = TX + 2 * R, HH = TY + 2 * R, BW = TX + 2 * XO, REG = W * HH;
  static constexpr int NFX = (TX + 1) * TY, NFY = TX * (TY + 1);
  static constexpr int NPX = TY * (W - 1), NPY = TX * (HH - 1);  // cell pairs of each sweep
  static constexpr int ND = NPX > NPY ? NPX : NPY;
  static constexpr int PB = HH * BW;  // plane stride of the box
  static constexpr int kBox = 0, kPl = kBox + 4 * PB, kDd = kPl + 4 * REG, kFx = kDd + 7 * ND,
                       kFy = kFx + 4 * NFX, kEnd = kFy + 4 * NFY;
  static constexpr size_t kBytes = sizeof(double) * kEnd + 128;
};

// Dynamic shared memory of one 2D tile.
template <int TX, int TY, int R = 3>
__host__ __device__ constexpr size_t smem_euler2d() {
  return R == 3 ? Tile6<TX, TY>::kBytes : smem_euler2d_gen<TX, TY, R>();
}

// The same for a tile that may stage by TMA (orders 4, 8, 10: the planes and
// faces, then the box, 128-byte aligned; the sixth-order layout always
// holds the box).
template <int TX, int TY, int R = 3>
__host__ __device__ constexpr size_t smem_euler2d_tma() {
  return R == 3 ? Tile6<TX, TY>::kBytes
                : ((smem_euler2d_gen<TX, TY, R>() + 127) & ~size_t(127)) +
                      tma_box_bytes<TX, TY, R>() + 128;
}

// GLF speed of field m of nc (max|u| + c for every field in the single mode).
__device__ __forceinline__ double field_speed(int alpha_single, const unsigned long long *al, int m,
                                              int nc) {
  unsigned long long v = al[m];
  if (alpha_single)
    for (int q = 0; q < nc; ++q) v = max(v, al[q]);
  return bits2d(v);
}
__device__ __forceinline__ double field_speed(const StageArgs &a, const unsigned long long *al,
                                              int m, int nc) {
  return field_speed(a.alpha_single, al, m, nc);
}

// One tile (tile index `tile` of problem b) of a 2D stage, run by one block.
// R: half-width of the stencil (scheme of order 2R, halo of R cells).
// sm: dynamic shared memory of smem_euler2d_tma<TX, TY, R>() bytes.
// tm: tensor map of the stage input as [nbatch * 4][ny][nx] doubles, or NULL
// (plain loads only; the serving engine and tiles of launches without one).
template <int TX, int TY, int AI, bool P1, int PREC, int R>
__device__ __forceinline__ void euler2d_tile_gen(const StageArgs &a, long long b, long long tile,
                                                 bool zeroing_block, double *sm,
                                                 const CUtensorMap *tm) {
  static_assert(R != 3 && PREC == 0, "orders 4, 8, 10 in FP64");
  constexpr int W = TX + 2 * R, HH = TY + 2 * R, REG = W * HH;
  constexpr int NFX = (TX + 1) * TY, NFY = TX * (TY + 1);
  constexpr int XO = TmaBox<R>::XO, BW = TX + 2 * XO;
  double *const pl = sm;
  double *const fx = sm + kPlanes2D * REG;
  double *const fy = fx + NFX * 4;

  const long long tiles_x = (a.nx + TX - 1) / TX;
  const long long tj = tile / tiles_x, ti = tile - tj * tiles_x;
  const long long i0 = ti * TX, j0 = tj * TY;
  double dt;
  if (!stage_control(a, b, tile == 0, zeroing_block, dt)) return;

  const long long plane = a.nx * a.ny;
  const double *Ub = a.Uin + b * 4 * plane;
  const double gm1 = a.gamma - 1.0;
  const int tid = threadIdx.x;

  // TMA staging of an interior tile: the box of the four conserved planes
  const bool use_tma = tm != nullptr && i0 - XO >= 0 && i0 - XO + BW <= a.nx && j0 - R >= 0 &&
                       j0 + TY + R <= a.ny;
  double *const box = reinterpret_cast<double *>(
      (reinterpret_cast<uintptr_t>(sm) + ((smem_euler2d_gen<TX, TY, R>() + 127) & ~size_t(127)) +
       127) &
      ~uintptr_t(127));
  if (use_tma && !tma_stage_box<TX, TY, R>(a, tm, box, b, i0, j0)) return;

  // Phase 1: stage the cross-shaped region (tile rows with x halo, tile
  // columns with y halo) and per-cell primitives / fluxes.
  for (int k = tid; k < REG; k += blockDim.x) {
    const int r = k / W, c = k - r * W;
    const bool xb = (r >= R) && (r < R + TY), yb = (c >= R) && (c < R + TX);
    if (!(xb || yb)) continue;
    const double *src;
    long long o, pst, gj, gi;
    if (use_tma) {  // the box: x from i0 - XO, y from j0 - R, planes of problem b
      src = box;
      pst = (long long)BW * HH;
      o = (long long)r * BW + (c + XO - R);
      gi = i0 - R + c;
      gj = j0 - R + r;
    } else {
      cell_source(a, Ub, b, i0, j0, R, r, c, src, o, pst, gj, gi);
    }
    const double rho = src[o], mx = src[pst + o], my = src[2 * pst + o], E = src[3 * pst + o];
    const double rs = rsqrt_pos(rho);  // 1/sqrt(rho): gives 1/rho and sqrt(rho)
    const double ir = rs * rs;
    const double u = mx * ir, v = my * ir;
    const double p = gm1 * (E - 0.5 * fma(mx, u, my * v));
    if (!(pos_finite(rho) && pos_finite(p))) record_status(a.status, 3, a.stage, b, gj, gi);
    pl[0 * REG + k] = rho;
    pl[1 * REG + k] = mx;
    pl[2 * REG + k] = my;
    pl[3 * REG + k] = E;
    pl[4 * REG + k] = u;
    pl[5 * REG + k] = v;
    pl[6 * REG + k] = (E + p) * ir;
    pl[7 * REG + k] = rho * rs;
    pl[8 * REG + k] = p;
  }
  __syncthreads();

  // Phase 2: every x- and y-face of the tile once.  Lanes of a warp may mix
  // directions; the code path is the same (only the plane indices differ).
  const unsigned long long *al = a.alpha_in + b * 8;
  const ReconParams rp4 = a.sp.rp[1], rp2 = a.sp.rp[0];
  for (int f = tid; f < NFX + NFY; f += blockDim.x) {
    int base, stride, dir, fr, fc;
    if (f < NFX) {
      fr = f / (TX + 1);
      fc = f - fr * (TX + 1);
      base = (R + fr) * W + fc;
      stride = 1;
      dir = 0;
    } else {
      const int g = f - NFX;
      fr = g / TX;
      fc = g - fr * TX;
      base = fr * W + R + fc;
      stride = W;
      dir = 1;
    }
    const int pmn = 1 + dir, pmt = 2 - dir, pun = 4 + dir, put = 5 - dir;
    const int kL = base + (R - 1) * stride, kR = base + R * stride;
    FaceState fs;
    if (!roe_face(pl[7 * REG + kL], pl[pun * REG + kL], pl[put * REG + kL], pl[6 * REG + kL],
                  pl[7 * REG + kR], pl[pun * REG + kR], pl[put * REG + kR], pl[6 * REG + kR],
                  gm1, fs))
      record_status(a.status, 3, a.stage, b, j0 + (dir ? fr : fr), i0 + fc);
    const double A1 = field_speed(a, al + 4 * dir, 0, 4), A2 = field_speed(a, al + 4 * dir, 1, 4);
    const double A3 = field_speed(a, al + 4 * dir, 2, 4), A4 = field_speed(a, al + 4 * dir, 3, 4);
    double h1, h2, h3, h4;
    {
      // f^+ in stencil order, f^- mirrored (its upwind side is on the right).
      constexpr int N = 2 * R;
      double p1[N], p2[N], p3[N], p4[N], m1[N], m2[N], m3[N], m4[N];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const int k = base + j * stride;
        double w1, w2, w3, w4, g1, g2, g3, g4;
        project4(fs, pl[k], pl[pmn * REG + k], pl[pmt * REG + k], pl[3 * REG + k], w1, w2, w3, w4);
        project_flux4(fs, pl[pun * REG + k], pl[8 * REG + k], w1, w2, w3, w4, g1, g2, g3, g4);
        p1[j] = fma(A1, w1, g1);
        m1[N - 1 - j] = fma(-A1, w1, g1);
        p2[j] = fma(A2, w2, g2);
        m2[N - 1 - j] = fma(-A2, w2, g2);
        p3[j] = fma(A3, w3, g3);
        m3[N - 1 - j] = fma(-A3, w3, g3);
        p4[j] = fma(A4, w4, g4);
        m4[N - 1 - j] = fma(-A4, w4, g4);
      }
      h1 = pair_flux_r<R>(za_r<R, AI, P1>(p1, rp4), za_r<R, AI, P1>(m1, rp4));
      h2 = pair_flux_r<R>(za_r<R, AI, P1>(p2, rp2), za_r<R, AI, P1>(m2, rp2));
      h3 = pair_flux_r<R>(za_r<R, AI, P1>(p3, rp2), za_r<R, AI, P1>(m3, rp2));
      h4 = pair_flux_r<R>(za_r<R, AI, P1>(p4, rp4), za_r<R, AI, P1>(m4, rp4));
    }
    double F0, F1, F2, F3;
    backproject4(fs, h1, h2, h3, h4, F0, F1, F2, F3);
    double *out = dir ? &fy[(fr * TX + fc) * 4] : &fx[(fr * (TX + 1) + fc) * 4];
    out[0] = F0;
    out[1 + dir] = F1;
    out[2 - dir] = F2;
    out[3] = F3;
  }
  __syncthreads();

  tile2d_update<TX, TY, R>(a, b, i0, j0, dt, fx, fy, 0.25 * a.sp.rdx, 0.25 * a.sp.rdy,
                           [&](int r, int c, int q) { return pl[q * REG + (R + r) * W + R + c]; });
}

// ---------------------------------------------------------------------------
// 2D Euler stage kernel of the sixth-order scheme (R = 3).
//
// The reconstruction of a face needs, per characteristic field, only the
// differences of the split fluxes f+- = g +- alpha w over its six stencil
// cells (field_flux), and those are L (F_{j+1} - F_j) +- alpha L (U_{j+1}
// - U_j): the face's left eigenvectors applied to differences of the state
// and of the physical flux between adjacent cells.  Those differences are
// formed once per cell pair and direction and shared by the five faces whose
// stencils hold the pair, so a face projects 10 difference vectors instead
// of 6 states and 6 fluxes and subtracts nothing per field.  The centre
// values g_i + g_{i+1} the reconstruction adds to its differences come back
// through R as the physical 2 (F_i + F_{i+1}) = 2 (2 F_i + dF) (R L = I),
// added after the back-projection.
//
// Phases: 1 stage the conserved variables (TMA or indexed loads) and the Roe
// inputs; then per direction (x, then y) 1d the cell-pair differences and
// 2d the faces; 3 the update (tile2d_update).  Shared memory: Tile6.
// ---------------------------------------------------------------------------

// Components 1..3 of the normal-frame physical flux of a cell (eq. (25)) from
// its state and the staged u_n, H: with p = rho H - E, F1 = m_n u_n + p,
// F2 = m_t u_n, F3 = H m_n (F0 = m_n).
__device__ __forceinline__ void normal_flux(double rho, double mn, double mt, double E, double un,
                                            double H, double &F1, double &F2, double &F3) {
  const double p = fma(rho, H, -E);
  F1 = fma(mn, un, p);
  F2 = mt * un;
  F3 = H * mn;
}

// The GLF speeds of a problem in fixed point, per direction (fx::speed), and
// the exponents above them, ea of the acoustic fields and eb of those that move
// with the flow (u = 0 gives the latter none: 2^-300 of the former stands for
// it); the block's first threads form them once.
struct Speeds {
  fx::Limb ka[2][4];
  int ea[2], eb[2];
};
__device__ __forceinline__ void make_speeds(const StageArgs &a, long long b, int nc, Speeds &s) {
  const int dir = threadIdx.x >> 2, m = threadIdx.x & 3;
  if (dir >= a.ndim || m >= nc) return;
  const unsigned long long *al = a.alpha_in + b * 8 + 4 * dir;
  unsigned long long top = al[0];
  for (int q = 1; q < nc; ++q) top = max(top, al[q]);
  const int ea = fx::exponent(bits2d(top)) - 1022;
  const int eb = max(fx::exponent(field_speed(a, al, 1, nc)) - 1022, ea - 300);
  s.ka[dir][m] = fx::speed(field_speed(a, al, m, nc), m == 0 || m == nc - 1 ? ea : eb);
  if (m == 0) {
    s.ea[dir] = ea;
    s.eb[dir] = eb;
  }
}

// The offsets of face (fr, fc) along dir: its left cell in the box and the
// planes, and the steps to the next cell.
template <int TX, int TY>
struct FaceAt {
  using L = Tile6<TX, TY>;
  int oL, kL, stB, stP;
  __device__ __forceinline__ FaceAt(int dir, int fr, int fc) {
    const int rL = fr + (dir ? L::R - 1 : L::R), cL = fc + (dir ? L::R : L::R - 1);
    oL = rL * L::BW + cL + L::XO - L::R;
    kL = rL * L::W + cL;
    stB = dir ? L::BW : 1;
    stP = dir ? L::W : 1;
  }
};
// The packed differences of a face for the integer path.
template <int ND>
struct PackedFace {
  const fx::u64 *pf;
  int ps;
  __device__ __forceinline__ fx::u64 operator()(int s, int q, int j) const {
    return pf[(s ? (q == 0 ? 1 : 3 + q) : q) * ND + j * ps];
  }
};
// 2 F_hat of a face from its fields' 6 h: F_L + F_R and a twelfth of what
// backproject4 gives.
template <int TX, int TY>
__device__ __forceinline__ void face_flux6(const double *sm, int dir, const FaceAt<TX, TY> &at,
                                           const FaceState &fs, const double (&h)[4], double *out) {
  using L = Tile6<TX, TY>;
  const double *const box = sm + L::kBox, *const pl = sm + L::kPl;
  const double *const bn = box + (1 + dir) * L::PB, *const bt = box + (2 - dir) * L::PB;
  const double *const un = pl + (1 + dir) * L::REG, *const H = pl + 3 * L::REG;
  const int oL = at.oL, oR = oL + at.stB, kL = at.kL, kR = kL + at.stP;
  double F0, F1, F2, F3, FL1, FL2, FL3, FR1, FR2, FR3;
  backproject4(fs, h[0], h[1], h[2], h[3], F0, F1, F2, F3);
  const double mnL = bn[oL], mnR = bn[oR];
  normal_flux(box[oL], mnL, bt[oL], box[3 * L::PB + oL], un[kL], H[kL], FL1, FL2, FL3);
  normal_flux(box[oR], mnR, bt[oR], box[3 * L::PB + oR], un[kR], H[kR], FR1, FR2, FR3);
  out[0] = fma(1.0 / 12.0, F0, mnL + mnR);
  out[1 + dir] = fma(1.0 / 12.0, F1, FL1 + FR1);
  out[2 - dir] = fma(1.0 / 12.0, F2, FL2 + FR2);
  out[3] = fma(1.0 / 12.0, F3, FL3 + FR3);
}
// Face (fr, fc) along dir with all its fields in FP64 from the staged cells: what
// the integer path leaves out.  al: its speed maxima.
template <int TX, int TY, int AI>
__device__ __noinline__ void face_wide(double *sm, int dir, int fr, int fc, FaceState fs,
                                       const unsigned long long *al, int alpha_single,
                                       const SchemeParams &scheme) {
  using L = Tile6<TX, TY>;
  const double *const box = sm + L::kBox, *const pl = sm + L::kPl;
  const double *const un = pl + (1 + dir) * L::REG, *const H = pl + 3 * L::REG;
  const FaceAt<TX, TY> at(dir, fr, fc);
  double U[2][4], F[2][4], dw[4][5], dg[4][5], h[4];
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const int o = at.oL + (j - 2) * at.stB, k = at.kL + (j - 2) * at.stP;
    double *const u = U[j & 1], *const f = F[j & 1];
    u[0] = box[o];
    u[1] = f[0] = box[(1 + dir) * L::PB + o];
    u[2] = box[(2 - dir) * L::PB + o];
    u[3] = box[3 * L::PB + o];
    normal_flux(u[0], u[1], u[2], u[3], un[k], H[k], f[1], f[2], f[3]);
    if (j == 0) continue;
    const double *const u0 = U[(j - 1) & 1], *const f0 = F[(j - 1) & 1];
    project4(fs, u[0] - u0[0], u[1] - u0[1], u[2] - u0[2], u[3] - u0[3], dw[0][j - 1], dw[1][j - 1],
             dw[2][j - 1], dw[3][j - 1]);
    project4(fs, f[0] - f0[0], f[1] - f0[1], f[2] - f0[2], f[3] - f0[3], dg[0][j - 1], dg[1][j - 1],
             dg[2][j - 1], dg[3][j - 1]);
  }
#pragma unroll 1
  for (int m = 0; m < 4; ++m) {
    const double A = field_speed(alpha_single, al, m, 4);
    h[m] = 6.0 * pair_wide<AI, true>(-A * dw[m][2], dw[m], dg[m], A,
                                     scheme.rp[m == 0 || m == 3 ? 1 : 0]);
  }
  double *const out = sm + (dir ? L::kFy + (fr * TX + fc) * 4 : L::kFx + (fr * (TX + 1) + fc) * 4);
  face_flux6<TX, TY>(sm, dir, at, fs, h, out);
}

// One direction (0: x, 1: y) of a tile.  The direction is a run-time value: the
// two sweeps then share their code, which has to stay in the instruction
// cache.
template <int TX, int TY, int AI, bool P1, int PREC>
__device__ __forceinline__ void tile6_sweep(const StageArgs &a, int dir, long long b, long long i0,
                                            long long j0, double gm1, double *sm,
                                            const SchemeParams &scheme, const Speeds &sp) {
  using L = Tile6<TX, TY>;
  constexpr int R = 3, W = L::W, BW = L::BW, XO = L::XO, PB = L::PB, REG = L::REG, ND = L::ND;
  const double *const box = sm + L::kBox;
  const double *const pl = sm + L::kPl;
  double *const dd = sm + L::kDd;
  double *const fo = sm + (dir ? L::kFy : L::kFx);
  // p = 1 in FP64: packed differences, projected on the integer pipes
  constexpr bool kPacked = P1 && PREC == 0;
  fx::u64 *const dp = reinterpret_cast<fx::u64 *>(dd);
  const int tid = threadIdx.x;
  // offsets of staged cell (r, c) in the box and the planes, and to the next
  // cell along the direction; planes of the normal and tangential momentum
  // and velocity
  auto bo = [](int r, int c) { return r * BW + c + XO - R; };
  const int stB = dir ? BW : 1, stP = dir ? W : 1;
  const double *const bn = box + (1 + dir) * PB, *const bt = box + (2 - dir) * PB;
  const double *const un = pl + (1 + dir) * REG, *const ut = pl + (2 - dir) * REG;
  // k / d for the row lengths of pairs and faces (d <= 64, k < 1024)
  auto rows_of = [](int k, int inv) { return (k * inv) >> 16; };
  constexpr auto inv = [](int d) constexpr { return (65536 + d - 1) / d; };

  // 1d: differences of each cell pair along dir (normal frame: m_n = rho u
  // for x, rho v for y), in dd[q * ND + pair]:
  //   x: pair (rr, pc), rr in [0, TY), pc in [0, W - 1): cells (R + rr, pc), (R + rr, pc + 1)
  //   y: pair (pr, cc), pr in [0, HH - 1), cc in [0, TX): cells (pr, R + cc), (pr + 1, R + cc)
  const int NP = dir ? L::NPY : L::NPX, lp = dir ? TX : W - 1, ip = dir ? inv(TX) : inv(W - 1);
  // the x pairs run from the block's last warp down: with phase 1 and the y
  // pairs starting from warp 0, the partial rounds of the three loops fall
  // on different warps (each warp's FP64 work goes to its own sub-partition)
  for (int k = dir ? tid : (int)blockDim.x - 1 - tid; k < NP; k += blockDim.x) {
    const int q0 = rows_of(k, ip), q1 = k - q0 * lp;
    const int rA = q0 + (dir ? 0 : R), cA = q1 + (dir ? R : 0);
    const int oA = bo(rA, cA), oB = oA + stB, kA = rA * W + cA, kB = kA + stP;
    const double rhoA = box[oA], mnA = bn[oA], mtA = bt[oA], EA = box[3 * PB + oA];
    const double rhoB = box[oB], mnB = bn[oB], mtB = bt[oB], EB = box[3 * PB + oB];
    double F1A, F2A, F3A, F1B, F2B, F3B;
    normal_flux(rhoA, mnA, mtA, EA, un[kA], pl[3 * REG + kA], F1A, F2A, F3A);
    normal_flux(rhoB, mnB, mtB, EB, un[kB], pl[3 * REG + kB], F1B, F2B, F3B);
    const double d[7] = {rhoB - rhoA, mnB - mnA /* also dF0 */, mtB - mtA, EB - EA,
                         F1B - F1A,   F2B - F2A,                F3B - F3A};
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      if constexpr (kPacked)
        dp[q * ND + k] = fx::pack(d[q]);
      else
        dd[q * ND + k] = d[q];
    }
  }
  __syncthreads();

  // 2d: the faces along dir.  x-face (fr, fc): between cells (R + fr, R - 1 + fc)
  // and (R + fr, R + fc), stencil pairs fr (W - 1) + fc + j; y-face (fr, fc):
  // between (R - 1 + fr, R + fc) and (R + fr, R + fc), pairs (fr + j) TX + fc.
  const int NF = dir ? L::NFY : L::NFX, lf = dir ? TX : TX + 1, jf = dir ? inv(TX) : inv(TX + 1);
  const int ps = dir ? TX : 1;  // pair stride along the stencil
  const unsigned long long *al = a.alpha_in + b * 8 + 4 * dir;
  const ReconParams &rp2 = scheme.rp[0], &rp4 = scheme.rp[1];
  for (int f = tid; f < NF; f += blockDim.x) {
    const int fr = rows_of(f, jf), fc = f - fr * lf;
    const int p0 = fr * lp + fc;
    const int rL = fr + (dir ? R - 1 : R), cL = fc + (dir ? R : R - 1);
    const int kL = rL * W + cL, kR = kL + stP;
    const int oL = bo(rL, cL);
    FaceState fs;
    if (!roe_face(pl[kL], un[kL], ut[kL], pl[3 * REG + kL], pl[kR], un[kR], ut[kR],
                  pl[3 * REG + kR], gm1, fs))
      record_status(a.status, 3, a.stage, b, j0 + fr, i0 + fc);
    double h[4];
    double *const out = fo + (fr * lf + fc) * 4;
    if constexpr (kPacked) {
      const PackedFace<ND> diff = {dp + p0, ps};
      const bool done = face_fields<4, AI>(
          fs, pl[kL], pl[kR], sp.ka[dir], sp.ea[dir], sp.eb[dir], diff,
          [&](int m) -> const ReconParams & { return (m == 0 || m == 3) ? rp4 : rp2; }, h);
      if (done)
        face_flux6<TX, TY>(sm, dir, FaceAt<TX, TY>(dir, fr, fc), fs, h, out);
      else
        face_wide<TX, TY, AI>(sm, dir, fr, fc, fs, al, a.alpha_single, scheme);
    } else {
      double dw[4][5], dg[4][5];
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        const int pj = p0 + j * ps;
        const double dmn = dd[ND + pj];
        project4(fs, dd[pj], dmn, dd[2 * ND + pj], dd[3 * ND + pj], dw[0][j], dw[1][j], dw[2][j],
                 dw[3][j]);
        project4(fs, dmn, dd[4 * ND + pj], dd[5 * ND + pj], dd[6 * ND + pj], dg[0][j], dg[1][j],
                 dg[2][j], dg[3][j]);
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const double A = field_speed(a, al, m, 4);
        if constexpr (PREC == 1)
          h[m] = field_flux_f32d<P1>(dw[m], dg[m], A, scheme.r32);
        else
          h[m] = field_flux<AI, P1>(dw[m], dg[m], A, (m == 0 || m == 3) ? rp4 : rp2, 0.0);
      }
      // the centre values: 4 F_hat += 2 (F_L + F_R) = 4 F_L + 2 dF of the centre pair
      double F0, F1, F2, F3, FL1, FL2, FL3;
      backproject4(fs, h[0], h[1], h[2], h[3], F0, F1, F2, F3);
      const int pc = p0 + 2 * ps;
      const double mnL = bn[oL];
      normal_flux(box[oL], mnL, bt[oL], box[3 * PB + oL], un[kL], pl[3 * REG + kL], FL1, FL2, FL3);
      out[0] = fma(4.0, mnL, fma(2.0, dd[ND + pc], F0));
      out[1 + dir] = fma(4.0, FL1, fma(2.0, dd[4 * ND + pc], F1));
      out[2 - dir] = fma(4.0, FL2, fma(2.0, dd[5 * ND + pc], F2));
      out[3] = fma(4.0, FL3, fma(2.0, dd[6 * ND + pc], F3));
    }
  }
  __syncthreads();
}

// One tile of a sixth-order 2D stage (see above).  sm: smem_euler2d<TX, TY>()
// bytes; tm: tensor map of the stage input or NULL, as for euler2d_tile_gen.
template <int TX, int TY, int AI, bool P1, int PREC>
__device__ __forceinline__ void euler2d_tile6(const StageArgs &a, long long b, long long tile,
                                              bool zeroing_block, double *sm_in,
                                              const CUtensorMap *tm) {
  using L = Tile6<TX, TY>;
  constexpr int R = 3, W = L::W, BW = L::BW, XO = L::XO, PB = L::PB, REG = L::REG;
  // (an offset, so the compiler keeps seeing shared memory)
  double *const sm = sm_in + (((0u - smem_u32(sm_in)) & 127u) >> 3);
  double *const box = sm + L::kBox;
  double *const pl = sm + L::kPl;

  const long long tiles_x = (a.nx + TX - 1) / TX;
  const long long tj = tile / tiles_x, ti = tile - tj * tiles_x;
  const long long i0 = ti * TX, j0 = tj * TY;
  double dt;
  if (!stage_control(a, b, tile == 0, zeroing_block, dt)) return;

  const double *Ub = a.Uin + b * 4 * (a.nx * a.ny);
  const double gm1 = a.gamma - 1.0;
  const int tid = threadIdx.x;

  // the scheme's constants and speeds (published by the barrier after phase 1)
  __shared__ SchemeParams s_scheme;
  load_scheme(a, s_scheme);
  __shared__ Speeds s_sp;
  if constexpr (P1 && PREC == 0) make_speeds(a, b, 4, s_sp);

  const bool use_tma = tm != nullptr && i0 - XO >= 0 && i0 - XO + BW <= a.nx && j0 - R >= 0 &&
                       j0 + TY + R <= a.ny;
  if (use_tma && !tma_stage_box<TX, TY, R>(a, tm, box, b, i0, j0)) return;

  // Phase 1: the cross-shaped region (tile rows with x halo, tile columns
  // with y halo): the conserved variables into the box where TMA did not
  // bring them, and per cell sqrt(rho), u, v, H.
  for (int k = tid; k < REG; k += blockDim.x) {
    const int r = k / W, c = k - r * W;
    const bool xb = (r >= R) && (r < R + TY), yb = (c >= R) && (c < R + TX);
    if (!(xb || yb)) continue;
    const int ob = r * BW + c + XO - R;
    double rho, mx, my, E;
    long long gj, gi;
    if (use_tma) {
      rho = box[ob];
      mx = box[PB + ob];
      my = box[2 * PB + ob];
      E = box[3 * PB + ob];
      gi = i0 - R + c;
      gj = j0 - R + r;
    } else {
      const double *src;
      long long o, pst;
      cell_source(a, Ub, b, i0, j0, R, r, c, src, o, pst, gj, gi);
      rho = src[o];
      mx = src[pst + o];
      my = src[2 * pst + o];
      E = src[3 * pst + o];
      box[ob] = rho;
      box[PB + ob] = mx;
      box[2 * PB + ob] = my;
      box[3 * PB + ob] = E;
    }
    const double rs = rsqrt_pos(rho);  // 1/sqrt(rho): gives 1/rho and sqrt(rho)
    const double ir = rs * rs;
    const double u = mx * ir, v = my * ir;
    const double p = gm1 * (E - 0.5 * fma(mx, u, my * v));
    if (!(pos_finite(rho) && pos_finite(p))) record_status(a.status, 3, a.stage, b, gj, gi);
    pl[k] = rho * rs;
    pl[REG + k] = u;
    pl[2 * REG + k] = v;
    pl[3 * REG + k] = (E + p) * ir;
  }
  __syncthreads();

#pragma unroll 1
  for (int dir = 0; dir < 2; ++dir)
    tile6_sweep<TX, TY, AI, P1, PREC>(a, dir, b, i0, j0, gm1, sm, s_scheme, s_sp);

  constexpr double f = P1 && PREC == 0 ? 0.5 : 0.25;  // the faces hold 2 F or 4 F
  tile2d_update<TX, TY, R>(a, b, i0, j0, dt, sm + L::kFx, sm + L::kFy, f * s_scheme.rdx,
                           f * s_scheme.rdy,
                           [&](int r, int c, int q) { return box[q * PB + (R + r) * BW + XO + c]; });
}

// One tile of a 2D stage of order 2R (sixth order: euler2d_tile6; 4, 8, 10:
// euler2d_tile_gen).
template <int TX, int TY, int AI, bool P1, int PREC, int R = 3>
__device__ __forceinline__ void euler2d_tile(const StageArgs &a, long long b, long long tile,
                                             bool zeroing_block, double *sm,
                                             const CUtensorMap *tm = nullptr) {
  if constexpr (R == 3)
    euler2d_tile6<TX, TY, AI, P1, PREC>(a, b, tile, zeroing_block, sm, tm);
  else
    euler2d_tile_gen<TX, TY, AI, P1, PREC, R>(a, b, tile, zeroing_block, sm, tm);
}

// Programmatic dependent launch: a stage whose grid is small is bound by its
// length, and 2 to 3 us of that are the launch itself.  Launched with the
// attribute, the next stage's blocks are placed while this one runs (each block
// lets them at its start) and wait, before they read anything, for it to have
// ended with its memory visible; without the attribute both are no-ops.
// Only where the blocks of two stages fit on SMs of their own: a block placed
// early beside a running one shares its SM while others are idle (order 8 of
// 14,000 cells, 111 blocks: 158 us a step plain, 286 chained; FP32 of 96^2, 144
// blocks: 98 and 114; order 6 of 96^2: 123.5 and 144.5).  The lane layout, bound
// by latency and not by the FP64 pipe, gains up to one block per SM (85 blocks,
// shock-density N = 1600: 3.57 -> 2.92 ms for 73 steps; 4 blocks, advection
// N = 200: 2.93 -> 2.00 ms for 100 steps), and so does the engine's persistent
// grid; 20 x 1600 cells, 260 blocks: 79 -> 102 us.
__device__ __forceinline__ void pdl_start() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <class... P, class... A>
cudaError_t launch_chained(bool chain, void (*kern)(P...), dim3 grid, int threads, size_t smem,
                           cudaStream_t s, const A &...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = chain ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// MINB: resident blocks per SM the register allocation must allow.
// tm: tensor map of a.Uin (see euler2d_tile), used when a.use_tma is set.
template <int TX, int TY, int NT, int MINB, int AI, bool P1, int PREC, int R = 3>
__global__ void __launch_bounds__(NT, MINB)
    k_euler2d(const __grid_constant__ StageArgs a, const __grid_constant__ CUtensorMap tm) {
  extern __shared__ __align__(128) double sm[];
  pdl_start();
  euler2d_tile<TX, TY, AI, P1, PREC, R>(a, blockIdx.z, blockIdx.x,
                                        blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0, sm,
                                        a.use_tma ? &tm : nullptr);
}

#include "weno_tiles1d.cuh"

// Multiprocessors of the current device (asked once per process and device).
inline int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  if (cached[dev] == 0) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    cached[dev] = n > 0 ? n : 152;
  }
  return cached[dev];
}

// Whether the blocks of `times` such grids find an SM each.
inline bool fits(dim3 g, int times = 1) {
  return times * (long long)g.x * g.y * g.z <= sm_count();
}

// Shared memory per SM the resident blocks of a launch may take (228 KB,
// less 1 KB the hardware keeps per block).
constexpr size_t kSmemPerSM = 233472;

template <int TX, int TY, int NT, int MINB, int AI, bool P1, int PREC, int R = 3>
cudaError_t launch_2d(const StageArgs &a_in, cudaStream_t s) {
  StageArgs a = a_in;
  // TMA staging when the box fits beside the tile's planes at this
  // occupancy and the input is addressable by a tensor map
  constexpr bool kTmaFits = (smem_euler2d_tma<TX, TY, R>() + 1024) * MINB <= kSmemPerSM;
  CUtensorMap tm;
  std::memset(&tm, 0, sizeof(tm));
  a.use_tma = kTmaFits && encode_state_map(a.Uin, a.nbatch, a.ny, a.nx, TX + 2 * TmaBox<R>::XO,
                                           TY + 2 * R, &tm);
  const char *nc = std::getenv("WENO_TEST_TMA_NO_COPY");
  a.tma_no_copy = (nc && nc[0] == '1') ? 1 : 0;
  const size_t smem = kTmaFits ? smem_euler2d_tma<TX, TY, R>() : smem_euler2d<TX, TY, R>();
  auto kern = k_euler2d<TX, TY, NT, MINB, AI, P1, PREC, R>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long long tiles = ((a.nx + TX - 1) / TX) * ((a.ny + TY - 1) / TY);
  dim3 grid((unsigned)tiles, 1, (unsigned)a.nbatch);
  a.speed_filter = tiles * a.nbatch > (long long)sm_count();
  return launch_chained(fits(grid, 2), kern, grid, NT, smem, s, a, tm);
}

template <int TX, int TY>
inline long long tiles_2d(const StageArgs &a) {
  return ((a.nx + TX - 1) / TX) * ((a.ny + TY - 1) / TY) * a.nbatch;
}

// What a stage of the tiles (TX, TY) costs, orders 4, 8 and 10, with blocks
// that come in rounds of one an SM: `two` for a pair of rounds, `one` for a single
// one.  Measured in 1/40 of a pair of 16x15 (r = 5, right-hand sides of 48 grids
// from 48 to 1024 cells a side): 300 us the first round, 555 a pair, the same on the
// 20x15 tiles 375 and 690, on 16x16 370 and 620, 97 each round of 8x8 tiles, and r = 4
// in the same proportions; r = 2, three blocks an SM, 80 each round of 16x15, 84 of
// 16x16, 100 of 20x15, 26 of 8x8.
template <int TX, int TY, int R>
inline long long tiles_cost(const StageArgs &a) {
  constexpr int two = R == 2 ? (TX == 8 ? 26 : TX == 20 ? 100 : TY == 16 ? 84 : 80)
                             : (TX == 8 ? 14 : TX == 20 ? 50 : TY == 16 ? 45 : 40);
  constexpr int one = R == 2 || TX == 8 ? two / 2 : (TX == 20 || TY == 16 ? 27 : 22);
  const long long rounds = (tiles_2d<TX, TY>(a) + sm_count() - 1) / sm_count();
  return rounds / 2 * two + rounds % 2 * one;
}

template <int AI, bool P1, int PREC, int R>
cudaError_t launch_stage_t(const StageArgs &a, cudaStream_t s) {
  if (a.ndim == 2) {
    // tile variants (cells / threads / blocks per SM the registers allow):
    // 0 = 32x16 / 256 / 1 (fewest halo faces), 1 = 16x16 / 128 / 2,
    // 2 = 16x8 / 64 / 4 (more tiles for small grids), 3 = 16x16 / 128 / 3,
    // 4 = 16x8 / 64 / 6, and two shapes whose face count is a multiple of
    // the block's threads, so every warp computes the same number of faces:
    // 5 = 20x12 / 128 / 3 (512 faces), 6 = 26x14 / 128 / 3 (768 faces).
    // For grids too small to fill the GPU, where a stage lasts as long as one
    // thread's chain of faces, about one face per thread: 7 = 16x8 / 256 / 1
    // (280 faces), 8 = 8x8 / 128 / 2 (144 faces).  The sixth-order tile
    // sweeps the x- and then the y-faces; two shapes give every thread
    // exactly two faces of each sweep (warp i of every block runs on the
    // same SM sub-partition, so an uneven count leaves three of the four
    // FP64 pipes idle at the end of a sweep): 9 = 16x15 / 128 / 3 (255 and
    // 256 faces), 10 = 14x17 / 128 / 3 (255 and 252).
    // Weights other than the default ones (without Ai, with a sensitivity term
    // that counts, p != 1) are built in four of the shapes (2, 7, 8, 9; see
    // tile_shape_built), which keeps the library's build short.
    // The other orders run 3 blocks per SM at r = 2 and 2 at r = 4, 5 (their
    // wider stencils need more registers) in the shape whose rounds cost least
    // (tiles_cost): 16x15 / 128 (511 faces, four a thread), 16x16 / 128 (544: a fifth
    // round for warp 0 alone, but fewer tiles), 20x15 / 128 (635, five a thread), 8x8 /
    // 160 (144, one a thread, for grids where a stage lasts as long as one thread's
    // faces).  Right-hand sides of order 10 in the four, us: 512^2 (1120, 1024, 910,
    // 4096 tiles) 2226 / 2238 / 2089 / 2746; 192x161 319 / 389 / 395 / 400; 100x649 866 /
    // 638 / 707 / 784; 306x140 570 / 635 / 705 / 498; the rule takes the least in all
    // 48 grids at orders 8 and 10, and loses 0.4 % to it at order 4.
    if constexpr (R != 3) {  // r = 2 fits the 168-register cap of 3 blocks per SM
      constexpr int kPerSM = R == 2 ? 3 : 2;
      const long long c15 = tiles_cost<16, 15, R>(a), c16 = tiles_cost<16, 16, R>(a);
      if constexpr (P1) {
        const long long c20 = tiles_cost<20, 15, R>(a), c8 = tiles_cost<8, 8, R>(a);
        const long long large = std::min(c15, std::min(c16, c20));
        if (c8 < large) return launch_2d<8, 8, 160, 1, AI, P1, PREC, R>(a, s);
        if (c20 < std::min(c15, c16)) return launch_2d<20, 15, 128, kPerSM, AI, P1, PREC, R>(a, s);
      }
      if (c16 < c15) return launch_2d<16, 16, 128, kPerSM, AI, P1, PREC, R>(a, s);
      return launch_2d<16, 15, 128, kPerSM, AI, P1, PREC, R>(a, s);
    } else if constexpr (!all_tile_shapes(AI, P1, PREC)) {
      switch (tile_shape_built(false, a.tile_variant)) {
        case 2: return launch_2d<16, 8, 64, 4, AI, P1, PREC>(a, s);
        case 7: return launch_2d<16, 8, 256, 1, AI, P1, PREC>(a, s);
        case 8: return launch_2d<8, 8, 128, 2, AI, P1, PREC>(a, s);
        default: return launch_2d<16, 15, 128, 3, AI, P1, PREC>(a, s);
      }
    } else {
      switch (a.tile_variant) {
        case 1: return launch_2d<16, 16, 128, 2, AI, P1, PREC>(a, s);
        case 2: return launch_2d<16, 8, 64, 4, AI, P1, PREC>(a, s);
        case 3: return launch_2d<16, 16, 128, 3, AI, P1, PREC>(a, s);
        case 4: return launch_2d<16, 8, 64, 6, AI, P1, PREC>(a, s);
        case 5: return launch_2d<20, 12, 128, 3, AI, P1, PREC>(a, s);
        case 6: return launch_2d<26, 14, 128, 3, AI, P1, PREC>(a, s);
        case 7: return launch_2d<16, 8, 256, 1, AI, P1, PREC>(a, s);
        case 8: return launch_2d<8, 8, 128, 2, AI, P1, PREC>(a, s);
        case 9: return launch_2d<16, 15, 128, 3, AI, P1, PREC>(a, s);
        case 10: return launch_2d<14, 17, 128, 3, AI, P1, PREC>(a, s);
        default: return launch_2d<kTX, kTY, kThreads2D, 1, AI, P1, PREC>(a, s);
      }
    }
  }
  const long long tiles = (a.nx + kT1 - 1) / kT1;
  if constexpr (R == 3) {
    // A problem of fewer tiles than the GPU has SMs is bound by the length
    // of one thread's chain of operations: spread each face over several
    // threads (and the problem over more blocks) instead.
    if (tiles * a.nbatch < (long long)sm_count() && (a.nc == 3 || PREC == 0)) {
      constexpr int kL3 = lanes1d(3, P1, PREC);
      const int tl1 = a.nc == 3 ? cells_lanes1d(kL3) : cells_lanes1d(2);
      dim3 g2((unsigned)((a.nx + tl1 - 1) / tl1), (unsigned)a.nbatch, 1);
      if (a.nc == 3)
        return launch_chained(fits(g2), k_line1d_lanes<3, AI, P1, PREC>, g2, kThreads1D,
                              smem_line1d<3, cells_lanes1d(kL3), 3, kL3>(), s, a);
      else if constexpr (PREC == 0)
        return launch_chained(fits(g2), k_line1d_lanes<1, AI, P1, PREC>, g2, kThreads1D,
                              smem_line1d<1, cells_lanes1d(2), 3, 2>(), s, a);
    }
  }
  dim3 grid((unsigned)tiles, (unsigned)a.nbatch, 1);
  if (a.nc == 3)
    return launch_chained(fits(grid, 2), k_line1d<3, AI, P1, PREC, R>, grid, kThreads1D,
                          smem_line1d<3, kT1, R>(), s, a);
  else
    return launch_chained(fits(grid, 2), k_line1d<1, AI, P1, PREC, R>, grid, kThreads1D,
                          smem_line1d<1, kT1, R>(), s, a);
}

}  // namespace
}  // namespace weno
