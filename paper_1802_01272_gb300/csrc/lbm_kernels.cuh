// lbm_kernels.cuh -- device code of the CTU lattice Boltzmann time step for
// GB300 (sm_103a), after arXiv:1802.01272 (Sofonea et al.).
//
// One step, as Sec. II C splits Eq. (eBGK): advection of each f_k over its
// upwind-corner stencil (CTU1, Eq. ctueq; CTU2 with the MC limiter,
// Sec. II C 2), then on the advected f*: rho, u, g (Eq. eder with Eq. evdw,
// 25-point stencils: fourth-order gradient of p^i - p^w, isotropic gradient of
// the 9-point Laplacian), f^eq (Eq. herfeq), F_k (Eq. herforce), BGK
// relaxation (optionally regularised, Eq. ereg), and the density reservoir of
// Sec. III A.
//
// step_stream.cuh has the fused kernel for FP32 arithmetic (FP32 and FP16
// storage), step_split64.cuh the two kernels of the FP64 step, pair_node.cuh the
// per-node operations both use.  Common to them: a strip is TW = 56 output columns
// [56 s, 56 s + 56); a work item is a strip and a block of rows.
#pragma once

#include <cuda.h>  // CUtensorMap (type only)
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ctulbm {

constexpr int REG = 64;         // region columns: output strip plus 4 columns per side
constexpr int TW = REG - 8;     // output columns per strip (56: strips start on 32-byte sectors)
constexpr int XOFF = 4;         // region column of the strip's first output column
constexpr int NT = 256;         // threads per CTA
constexpr int RPI = 4;          // rows per pipeline iteration (a batch)
constexpr int WARM = 2;         // batches of a segment before its first output row

// Per-velocity constants, computed on the host in FP64 and rounded to T.
template <typename T>
struct VelConst {
  T xi_x, xi_y;
  T cx, cy;                 // Courant numbers |xi_x| dt/ds, |xi_y| dt/ds
  T ax;                     // lam |xi_x| (1 - cx): weight of the x-difference of half-limited S^x
  T qy0, qy1;               // FP64: (1 - cy) (1 - cx), (1 - cy) cx: weights of the S^y terms per unit of cy
  T by0, by1;               // FP32: -cy (1 - cy) (1 - cx), -cy (1 - cy) cx: weights of the dS^y terms
  T gbot, gtop;             // wall ghost-row values (storage variable)
};

// Per-class constants of the FP32 collision (velocity groups with the same xi^2):
// w A, A, w B with A = (T - 1)(xi^2 - 2)/2, B = (T - 1)(xi^2 - 4)/2, w = dt/tau.
struct ClassConst {
  float omA, A, omB;
};

template <typename T>
struct StepArgs {
  const void* fin;          // f^n, [16][Ly][Lx] in the storage type (float, double or half)
  void* fout;               // f^{n+1}
  int Lx, Ly;
  long long plane;          // Lx * Ly
  int nstrip;
  int row_block;            // rows per work item
  int sub;                  // FP64 advection: row ranges a work item is split into
  long long items;          // work items: ceil(Ly / row_block) * nstrip, row-block major
  // fused diagnostics of the state after this step (null: off): FP64 mass,
  // bubble sites rho < diag_thr and their exact integer moment sums
  double* diag_mass;
  unsigned long long* diag_sums;  // [6]: nb, sx, sy, sxx, sxy, syy
  T diag_thr;
  int walls, reservoir, regularize;
  T rho_ref, Tt, a, b, omega, one_m_omega;
  // force stencils with dt/ds (and kappa) folded in: g dt/ds = ir * (gradient
  // of p^i - p^w) + kappa * (gradient of the Laplacian)
  T gw1, gw2, gw3, gw4;     // (4/9, 1/9, 1/18, 1/72) dt/ds
  // kappa D_h(9-point Laplacian) composed into one 5x5 stencil: weights of
  // q(+-1, b) - q(-+1, b) for |b| = 0, 1, 2 and of q(+-2, b) - q(-+2, b),
  // (-1, -1/18, 1/18, 1/4, 1/9, 1/72) kappa dt/ds^3
  T kw[6];
  T rho_ext, irho_ext, rbc2, cxc, cyc;
  unsigned int* err;         // bit 0: non-finite or non-positive rho; bit 1: a wait timed out
  int tma_in;               // the tensor maps describe fin (rows are staged by tensor copies)
  T xlo, xhi;               // |xi| components sqrt(3 - sqrt 6), sqrt(3 + sqrt 6)
  T lo2, hi2;               // their squares
  // constants of the collision polynomial, w = dt/tau: s = (T - 1)/2, -2 w s, w - 4 w s,
  // 3 - 2 T, w s, -2 w / 3
  T ps, p00, p10, pg, p20, p30;
  T w[3];                   // weights of the groups (lo,lo), (hi,lo) = (lo,hi), (hi,hi)
  T om2, om6;               // w/2, w/6
  ClassConst cls[3];        // of the same groups
  VelConst<T> v[16];
};

// Tensor maps of f^n.  FP64: as a 3-D tensor (x, plane, row), m[0] loads boxes of
// A64_COLS columns x 1 plane x RPI rows.  FP32 and FP16: as a 4-D tensor (x, sign
// quadrant, group, row), boxes of one quadrant's four planes x SR rows: m[0] all
// columns of a strip's staging, m[1] and m[2] the two runs of the strip at the left
// x seam, m[3] and m[4] of that at the right.
struct RowMaps {
  CUtensorMap m[5];
};

constexpr int MAXB = 12;  // lattices per batched launch (kernel parameter space)

template <typename T>
struct BatchArgs {
  int count;
  long long item_start[MAXB + 1];  // prefix sums of the lattices' work items
  StepArgs<T> L[MAXB];
  RowMaps maps[MAXB];
};

// ---------------------------------------------------------------- helpers
// Storage of f (float, double, or half for FP16 shifted storage) and the
// arithmetic type T: conversions on load and store.
template <typename S, typename T>
__device__ __forceinline__ T from_store(S v) {
  return (T)v;
}
template <>
__device__ __forceinline__ float from_store<__half, float>(__half v) {
  return __half2float(v);
}
template <typename S, typename T>
__device__ __forceinline__ S to_store(T v) {
  return (S)v;
}
template <>
__device__ __forceinline__ __half to_store<__half, float>(float v) {
  return __float2half_rn(v);
}
// Reciprocal in FP32: the hardware approximation (relative error below 2^-22),
// enough for u = (rho u)/rho and the pressure and force terms, which enter the
// update multiplied by dt; FP64 keeps the correctly rounded division.
__device__ __forceinline__ float rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double rcp(double x) { return 1.0 / x; }

// min(|a|, |b|) carrying the sign sgn(a) sgn(b) (one instruction on sm_86+).
__device__ __forceinline__ float min_xorsign_abs(float a, float b) {
  float r;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// Half of the limited jump R Psi(Ru / R) of Sec. II C 2 (Ru the upwind jump).
// For the MC limiter Psi = max(0, min((1 + th)/2, 2, 2 th)) this is the
// three-way minmod of R, Ru and h = (R + Ru)/4: the one of least magnitude when
// all three share a sign, else 0 -- no division, and 0 at R = 0 where the
// limiter's argument is undefined.  FP32: u = minmod(R, Ru) as sgn(R) sgn(Ru)
// min(|R|, |Ru|) clamped at 0, then min(u, |h|) with the sign of h, which is
// sgn(R) whenever u > 0.
template <int LIM>
__device__ __forceinline__ float mc_half(float R, float Ru, float h) {
  if constexpr (LIM == 1) {
    return 0.0f;
  } else if constexpr (LIM == 2) {
    return 0.5f * R;
  } else {
    return min_xorsign_abs(fmaxf(min_xorsign_abs(R, Ru), 0.0f), h);
  }
}

__device__ __forceinline__ int wrapi(int i, int n) {
  int r = i % n;
  return r < 0 ? r + n : r;
}

// Row of the lattice that row r of the periodic (or walled) lattice stands for.
__device__ __forceinline__ int wrap_row(int r, int Ly) {
  r = r < 0 ? r + Ly : (r >= Ly ? r - Ly : r);
  return (unsigned)r < (unsigned)Ly ? r : wrapi(r, Ly);  // (lattices lower than a batch)
}

__device__ __forceinline__ float shfl_up1(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float shfl_dn1(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double shfl_up1(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double shfl_dn1(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// ------------------------------------------------------- pairs of values
// Two neighbouring columns or nodes as one value: in FP32 every operation on
// whole pairs is one packed FP32x2 instruction (sm_100+, round to nearest),
// which issues once for two lanes' worth of work.  A product that only feeds a sum
// is written as one fma2: left apart, the two are contracted in some kernels and
// not in others (also where both are marked .rn), and a node would step
// differently in each.
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// (a sum as an intrinsic: 6144^2 1111 us per step against 1107, 4096^2 FP16 537 against 530)
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(r)
      : "l"(*reinterpret_cast<const unsigned long long*>(&a)),
        "l"(*reinterpret_cast<const unsigned long long*>(&b)));
  return *reinterpret_cast<const float2*>(&r);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;"
      : "=l"(r)
      : "l"(*reinterpret_cast<const unsigned long long*>(&a)),
        "l"(*reinterpret_cast<const unsigned long long*>(&b)));
  return *reinterpret_cast<const float2*>(&r);
}
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
// the same operations on one FP64 value
__device__ __forceinline__ double add2(double a, double b) { return a + b; }
__device__ __forceinline__ double sub2(double a, double b) { return a - b; }
__device__ __forceinline__ double mul2(double a, double b) { return a * b; }
__device__ __forceinline__ double fma2(double a, double b, double c) { return fma(a, b, c); }

template <typename ST>
__device__ __forceinline__ void sload4p(const ST* p, float2& a, float2& b) {
  if constexpr (sizeof(ST) == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    a = make_float2(t.x, t.y);
    b = make_float2(t.z, t.w);
  } else {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
    b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
  }
}

// ------------------------------------- mbarriers, proxies, tensor copies
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Wait for the phase `parity` of `bar` to complete, for at most `ns`
// nanoseconds; false on timeout.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, unsigned parity,
                                                  unsigned long long ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (global_ns() - t0 > ns) return false;
  }
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
// Steps are launched with programmatic dependence (launch_dependent): a step's CTAs
// come up, set up their barriers and fetch parameters and tensor maps while the last
// of the step before end; they touch nothing that a launch before them writes or
// reads until those have completed.  (Also correct after any other launch.)  The
// launch is not let go earlier, by griddepcontrol.launch_dependents: CTAs that wait
// on an SM displace and unbalance those still to come (256^2 10.3 -> 11.8 us per step,
// 1024^2 FP64 970 -> 1160); without programmatic dependence 256^2 takes 10.8, 128^2
// FP64 25.6 against 25.1.
__device__ __forceinline__ void previous_step_done() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];\n" ::"l"(map) : "memory");
}
// One tensor copy from row y.. of plane k of the (x, plane, row) tensor into `dst`.
__device__ __forceinline__ void tma_load_tile(void* dst, const CUtensorMap* map, int x, int k, int y,
                                              unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(smem_u32(dst)),
      "l"(map), "r"(x), "r"(k), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

#include "pair_node.cuh"

__device__ __forceinline__ void store_pair(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
__device__ __forceinline__ void store_pair(__half* p, float2 v) {
  *reinterpret_cast<__half2*>(p) = __floats2half2_rn(v.x, v.y);
}

#include "step_stream.cuh"

}  // namespace ctulbm
