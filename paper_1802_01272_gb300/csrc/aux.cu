// aux.cu -- per-node kernels around the fused step: initialisation to f^eq
// (Eq. herfeq), FP64 <-> storage conversion, moments (Sec. II A) and the
// diagnostics of Sec. III B-C (mass, bubble-site sums of Eq. gyr, probe
// densities, density histogram).
#include <type_traits>

#include "lbm_internal.h"

namespace ctulbm {

namespace {

constexpr int BS = 256;

// Arithmetic type of a storage type: double for double, float for float and half.
template <typename S>
struct Comp {
  using type = float;
};
template <>
struct Comp<double> {
  using type = double;
};

// Velocity table in the arithmetic precision, loaded once per thread.  The
// float table comes rounded from the host, so the one-node-per-thread kernels
// do no double -> float conversions (GB300's FP64 path is narrow).
template <typename T>
struct Vel {
  T x[16], y[16], w[16];
  __device__ explicit Vel(const AuxArgs& a) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      x[k] = a.xi[k][0];
      y[k] = a.xi[k][1];
      w[k] = a.w[k];
    }
  }
};
template <>
struct Vel<float> {
  float x[16], y[16], w[16];
  __device__ explicit Vel(const AuxArgs& a) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      x[k] = a.xif[k][0];
      y[k] = a.xif[k][1];
      w[k] = a.wf[k];
    }
  }
};

// W consecutive stored values of a plane in one access (W = 2 wants an even plane).
template <typename S, int W>
struct __align__(W * sizeof(S)) Run {
  S v[W];
};

// A product that stays one (the compiler would contract it with a sum, and not in the
// same way in each instantiation: the results must not depend on which one runs).
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// Eq. (herfeq) with the storage shift w_k rho_ref removed:
// f^eq - w rho_ref = w [ (rho - rho_ref) + rho (P_k - 1) ],
// P_k - 1 = xi.u + [(xi.u)^2 - u^2 + (T-1)(xi^2-2)]/2 + xi.u [(xi.u)^2 - 3u^2 + 3(T-1)(xi^2-4)]/6
// W neighbouring nodes per thread: bound by HBM, and two nodes make every access of a
// warp whole 128-byte lines (16 of 64 B written, 24 read per node in FP32).
template <typename S, int W>
__global__ void init_feq_kernel(const AuxArgs a, S* f, const double* rho, const double* ux,
                                const double* uy) {
  using T = typename Comp<S>::type;
  const long long q = W * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  if (q >= a.plane) return;
  const Vel<T> v(a);
  const Run<double, W> in[3] = {*reinterpret_cast<const Run<double, W>*>(rho + q),
                                *reinterpret_cast<const Run<double, W>*>(ux + q),
                                *reinterpret_cast<const Run<double, W>*>(uy + q)};
  T r[W], dr[W], u[W], w[W], u2[W];
  const T Tm1 = (T)(a.Tt - 1.0);
#pragma unroll
  for (int e = 0; e < W; ++e) {
    r[e] = (T)in[0].v[e];
    dr[e] = (T)(in[0].v[e] - a.rho_ref);
    u[e] = (T)in[1].v[e];
    w[e] = (T)in[2].v[e];
    u2[e] = fma(u[e], u[e], mul_rn(w[e], w[e]));
  }
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const T x2 = fma(v.y[k], v.y[k], mul_rn(v.x[k], v.x[k]));
    Run<S, W> o;
#pragma unroll
    for (int e = 0; e < W; ++e) {
      const T cu = fma(v.x[k], u[e], mul_rn(v.y[k], w[e])), c2 = mul_rn(cu, cu);
      const T a2 = fma(Tm1, x2 - T(2), c2 - u2[e]);
      const T a3 = fma(T(3) * Tm1, x2 - T(4), fma(T(-3), u2[e], c2));
      const T pm1 = fma(cu / T(6), a3, fma(T(0.5), a2, cu));
      o.v[e] = to_store<S, T>(v.w[k] * fma(r[e], pm1, dr[e]));
    }
    *reinterpret_cast<Run<S, W>*>(f + k * a.plane + q) = o;
  }
}

template <typename S>
__global__ void set_f_kernel(const AuxArgs a, S* f, const double* src) {
  using T = typename Comp<S>::type;
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= a.plane) return;
  for (int k = 0; k < 16; ++k)
    f[k * a.plane + q] = to_store<S, T>((T)(src[k * a.plane + q] - a.w[k] * a.rho_ref));
}

template <typename S>
__global__ void get_f_kernel(const AuxArgs a, const S* f, double* dst) {
  using T = typename Comp<S>::type;
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= a.plane) return;
  for (int k = 0; k < 16; ++k)
    dst[k * a.plane + q] = (double)from_store<S, T>(f[k * a.plane + q]) + a.w[k] * a.rho_ref;
}

// rho - rho_ref = sum_k f_k and rho u = sum_k f_k xi_k of a node's stored (shifted) f, in
// velocity order (the order is part of the results: the same f gives the same moments).
template <typename T>
__device__ __forceinline__ void node_moments(const AuxArgs& a, const Vel<T>& v, const T (&f)[16],
                                             T& drho, T& mx, T& my) {
  drho = mx = my = T(0);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    drho += f[k];
    mx += f[k] * v.x[k];
    my += f[k] * v.y[k];
  }
}
template <typename S, typename T>
__device__ __forceinline__ void node_moments_at(const AuxArgs& a, const Vel<T>& v, const S* f,
                                                long long q, T& drho, T& mx, T& my) {
  T x[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) x[k] = from_store<S, T>(f[k * a.plane + q]);
  node_moments<T>(a, v, x, drho, mx, my);
}

template <typename S, int W>
__global__ void moments_kernel(const AuxArgs a, const S* f, double* rho, double* ux, double* uy) {
  using T = typename Comp<S>::type;
  const long long q = W * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  if (q >= a.plane) return;
  const Vel<T> v(a);
  Run<S, W> in[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) in[k] = *reinterpret_cast<const Run<S, W>*>(f + k * a.plane + q);
  Run<double, W> o[3];
#pragma unroll
  for (int e = 0; e < W; ++e) {
    T x[16], d, mx, my;
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = from_store<S, T>(in[k].v[e]);
    node_moments<T>(a, v, x, d, mx, my);
    const T r = (T)a.rho_ref + d;
    o[0].v[e] = (double)r;
    o[1].v[e] = (double)(mx / r);
    o[2].v[e] = (double)(my / r);
  }
  *reinterpret_cast<Run<double, W>*>(rho + q) = o[0];
  *reinterpret_cast<Run<double, W>*>(ux + q) = o[1];
  *reinterpret_cast<Run<double, W>*>(uy + q) = o[2];
}

// order-preserving 64-bit key of a double
__device__ __forceinline__ unsigned long long dkey(double v) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (b & 0x8000000000000000ULL) ? ~b : (b | 0x8000000000000000ULL);
}

template <typename V>
__device__ __forceinline__ V warp_sum(V v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Ring membership |dist - r_ring| < 1/2 tested exactly on integers:
// (2r-1)^2 < (2i - Lx)^2 + (2j - Ly)^2 < (2r+1)^2.
template <typename S>
__global__ void diag_kernel(const AuxArgs a, const S* f, double thr, double r_ring, DiagAcc* acc) {
  using T = typename Comp<S>::type;
  const Vel<T> v(a);
  double mass = 0.0, ring = 0.0;
  unsigned long long nring = 0, nb = 0, sx = 0, sy = 0, sxx = 0, sxy = 0, syy = 0;
  unsigned long long kmin = ~0ULL, kmax = 0ULL;
  const double rin = fmax(2.0 * r_ring - 1.0, 0.0), rout = 2.0 * r_ring + 1.0;
  const double rin2 = 2.0 * r_ring - 1.0 > 0.0 ? rin * rin : -1.0, rout2 = rout * rout;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < a.plane;
       q += (long long)gridDim.x * blockDim.x) {
    T d, mx, my;
    node_moments_at<S, T>(a, v, f, q, d, mx, my);
    const double rho = a.rho_ref + (double)d;
    const long long i = q % a.Lx, j = q / a.Lx;
    mass += rho;
    const unsigned long long key = dkey(rho);
    kmin = min(kmin, key);
    kmax = max(kmax, key);
    if (rho < thr) {
      nb += 1;
      sx += i;
      sy += j;
      sxx += i * i;
      sxy += i * j;
      syy += j * j;
    }
    const long long di = 2 * i - a.Lx, dj = 2 * j - a.Ly;
    const double d2 = (double)(di * di + dj * dj);
    if (d2 > rin2 && d2 < rout2) {
      ring += rho;
      nring += 1;
    }
    if (i == a.Lx / 2 && j == a.Ly / 2) acc->rho_center = rho;
  }
  mass = warp_sum(mass);
  ring = warp_sum(ring);
  nring = warp_sum(nring);
  nb = warp_sum(nb);
  sx = warp_sum(sx);
  sy = warp_sum(sy);
  sxx = warp_sum(sxx);
  sxy = warp_sum(sxy);
  syy = warp_sum(syy);
  for (int o = 16; o > 0; o >>= 1) {
    kmin = min(kmin, __shfl_down_sync(0xffffffffu, kmin, o));
    kmax = max(kmax, __shfl_down_sync(0xffffffffu, kmax, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&acc->mass, mass);
    atomicAdd(&acc->ring_sum, ring);
    atomicAdd(&acc->ring_n, nring);
    atomicAdd(&acc->nb, nb);
    atomicAdd(&acc->sx, sx);
    atomicAdd(&acc->sy, sy);
    atomicAdd(&acc->sxx, sxx);
    atomicAdd(&acc->sxy, sxy);
    atomicAdd(&acc->syy, syy);
    atomicMin(&acc->rmin_key, kmin);
    atomicMax(&acc->rmax_key, kmax);
  }
}

template <typename S>
__global__ void hist_kernel(const AuxArgs a, const S* f, int nbins, double lo, double hi,
                            unsigned long long* counts) {
  using T = typename Comp<S>::type;
  extern __shared__ unsigned int sh[];
  const bool priv = nbins <= 8192;
  if (priv)
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < a.plane;
       q += (long long)gridDim.x * blockDim.x) {
    T d = T(0);  // in velocity order: counts of the same f stay the same
#pragma unroll
    for (int k = 0; k < 16; ++k) d += from_store<S, T>(f[k * a.plane + q]);
    const double rho = a.rho_ref + (double)d;
    const double t = (rho - lo) / (hi - lo) * nbins;
    if (t >= 0.0 && t < (double)nbins) {
      const int b = (int)t;
      if (priv)
        atomicAdd(&sh[b], 1u);
      else
        atomicAdd(&counts[b], 1ULL);
    }
  }
  __syncthreads();
  if (priv)
    for (int b = threadIdx.x; b < nbins; b += blockDim.x)
      if (sh[b]) atomicAdd(&counts[b], (unsigned long long)sh[b]);
}

unsigned grid_for(long long n) { return (unsigned)((n + BS - 1) / BS); }

// Whether nodes can be taken two at a time: an even number of them, and the caller's
// fields (whose alignment is only that of a double) on 16-byte boundaries.
bool two_nodes(const AuxArgs& a, const void* x, const void* y, const void* z) {
  return a.plane % 2 == 0 &&
         (((uintptr_t)x | (uintptr_t)y | (uintptr_t)z) & 15) == 0;
}

// Calls fn(typed f) with f cast to the storage type of a.storage.
template <typename F>
cudaError_t by_storage(const AuxArgs& a, const void* f, F fn) {
  switch (a.storage) {
    case STORE_F64: fn(static_cast<const double*>(f)); break;
    case STORE_F16: fn(static_cast<const __half*>(f)); break;
    default: fn(static_cast<const float*>(f)); break;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_init_feq(const AuxArgs& a, void* f, const double* rho, const double* ux,
                            const double* uy, cudaStream_t s) {
  return by_storage(a, f, [&](auto p) {
    using S = std::remove_const_t<std::remove_pointer_t<decltype(p)>>;
    if (two_nodes(a, rho, ux, uy))
      init_feq_kernel<S, 2><<<grid_for(a.plane / 2), BS, 0, s>>>(a, const_cast<S*>(p), rho, ux, uy);
    else
      init_feq_kernel<S, 1><<<grid_for(a.plane), BS, 0, s>>>(a, const_cast<S*>(p), rho, ux, uy);
  });
}

cudaError_t launch_set_f(const AuxArgs& a, void* f, const double* src, cudaStream_t s) {
  return by_storage(a, f, [&](auto p) {
    using S = std::remove_const_t<std::remove_pointer_t<decltype(p)>>;
    set_f_kernel<S><<<grid_for(a.plane), BS, 0, s>>>(a, const_cast<S*>(p), src);
  });
}

cudaError_t launch_get_f(const AuxArgs& a, const void* f, double* dst, cudaStream_t s) {
  return by_storage(a, f, [&](auto p) {
    get_f_kernel<<<grid_for(a.plane), BS, 0, s>>>(a, p, dst);
  });
}

cudaError_t launch_moments(const AuxArgs& a, const void* f, double* rho, double* ux, double* uy,
                           cudaStream_t s) {
  return by_storage(a, f, [&](auto p) {
    using S = std::remove_const_t<std::remove_pointer_t<decltype(p)>>;
    if (two_nodes(a, rho, ux, uy))
      moments_kernel<S, 2><<<grid_for(a.plane / 2), BS, 0, s>>>(a, p, rho, ux, uy);
    else
      moments_kernel<S, 1><<<grid_for(a.plane), BS, 0, s>>>(a, p, rho, ux, uy);
  });
}

cudaError_t launch_diag(const AuxArgs& a, const void* f, double thr, double r_ring, DiagAcc* acc,
                        cudaStream_t s) {
  unsigned g = grid_for(a.plane);
  if (g > 4096) g = 4096;
  return by_storage(a, f, [&](auto p) { diag_kernel<<<g, BS, 0, s>>>(a, p, thr, r_ring, acc); });
}

cudaError_t launch_hist(const AuxArgs& a, const void* f, int nbins, double lo, double hi,
                        unsigned long long* counts, cudaStream_t s) {
  unsigned g = grid_for(a.plane);
  if (g > 2048) g = 2048;
  const size_t sh = nbins <= 8192 ? sizeof(unsigned int) * nbins : 0;
  return by_storage(a, f, [&](auto p) {
    hist_kernel<<<g, BS, sh, s>>>(a, p, nbins, lo, hi, counts);
  });
}

size_t step_smem_bytes(size_t stage_elem) {
  return stage_elem == 2 ? StreamSmem<__half>::bytes() : StreamSmem<float>::bytes();
}

}  // namespace ctulbm
