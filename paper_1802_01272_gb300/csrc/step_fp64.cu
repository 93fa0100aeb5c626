// step_fp64.cu -- the FP64 step: advection and collision kernels.
#include "lbm_internal.h"

namespace ctulbm {

#include "step_split64.cuh"

namespace {

void* advect_fn(int order, int lim) {
  if (order == 1) return reinterpret_cast<void*>(&advect64_kernel<1, 0>);
  switch (lim) {
    case 1: return reinterpret_cast<void*>(&advect64_kernel<2, 1>);
    case 2: return reinterpret_cast<void*>(&advect64_kernel<2, 2>);
    default: return reinterpret_cast<void*>(&advect64_kernel<2, 0>);
  }
}
void* collide_fn(bool diag, bool regu) {
  if (diag)
    return regu ? reinterpret_cast<void*>(&collide64_kernel<true, true>)
                : reinterpret_cast<void*>(&collide64_kernel<true, false>);
  return regu ? reinterpret_cast<void*>(&collide64_kernel<false, true>)
              : reinterpret_cast<void*>(&collide64_kernel<false, false>);
}

}  // namespace

Step64 step64(const StepArgs<double>& a, int order, int lim) {
  Step64 s;
  s.advect = advect_fn(order, lim);
  s.collide_grid = (unsigned)((a.Lx + C64_TX - 1) / C64_TX) * (unsigned)((a.Ly + C64_TY - 1) / C64_TY);
  s.collide = collide_fn(a.diag_mass != nullptr, a.regularize != 0);
  s.collide_threads = C64_NT;
  return s;
}

cudaError_t launch_step_f64(const StepArgs<double>& a, void* f, void* work, const RowMaps& maps,
                            int order, int lim, int grid, cudaStream_t s) {
  const Step64 k = step64(a, order, lim);
  StepArgs<double> in = a, out = a;
  in.fin = out.fout = f;
  in.fout = work;
  out.fin = work;
  void* args[] = {&in, const_cast<RowMaps*>(&maps)};
  const cudaError_t e = launch_dependent(k.advect, grid, NT, 0, s, args);
  if (e != cudaSuccess) return e;
  void* args2[] = {&out};
  return launch_dependent(k.collide, k.collide_grid, k.collide_threads, 0, s, args2);
}

int step_occupancy_f64(int order, int lim) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, advect_fn(order, lim), NT, 0) != cudaSuccess)
    return 0;
  return n;
}

int step64_cols() { return A64_COLS; }

}  // namespace ctulbm
