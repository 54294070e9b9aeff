// Device and launch helpers shared by the kernels that work on the padded
// mirrors of the state (zmarch.cu, heun.cu); layouts in kernels.h.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"
#include "tma.cuh"

namespace lcbp {

__device__ __forceinline__ int wrap(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

// The four values at 16-byte aligned element i (a group of the padded
// scratch), as one vector access: float4, or two double2 for FP64.
template <typename real>
__device__ __forceinline__ void ld4(const real* p, int i, real v[4]) {
  if constexpr (sizeof(real) == 4) {
    const float4 a = *reinterpret_cast<const float4*>(p + i);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
  } else {
    const double2 a = *reinterpret_cast<const double2*>(p + i), c = *reinterpret_cast<const double2*>(p + i + 2);
    v[0] = a.x, v[1] = a.y, v[2] = c.x, v[3] = c.y;
  }
}
template <typename real>
__device__ __forceinline__ void st4(real* p, real a, real b, real c, real d) {
  if constexpr (sizeof(real) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
  } else {
    *reinterpret_cast<double2*>(p) = make_double2(a, b);
    *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
  }
}
// st4 to global memory as a streaming store (evict-first in L2): the
// step's outputs, which no CTA of the kernel reads again, leave L2 to the
// staged halos and pulled populations that neighbouring tiles share
template <typename real>
__device__ __forceinline__ void st4g(real* p, real a, real b, real c, real d) {
  if constexpr (sizeof(real) == 4) {
    __stcs(reinterpret_cast<float4*>(p), make_float4(a, b, c, d));
  } else {
    __stcs(reinterpret_cast<double2*>(p), make_double2(a, b));
    __stcs(reinterpret_cast<double2*>(p + 2), make_double2(c, d));
  }
}
// The positions of a padded mirror (site x at column x + px, y at row y + h)
// that hold the value of site (gx, gy): its own, and each ghost position in
// the h columns and rows next to the lattice whose periodic image it is
// (lattice faces only; nx >= 2h gives a site at most one x image).  put1(X, Y)
// is called for each.
template <typename F>
__device__ __forceinline__ void mirror_positions(int px, int h, int nx, int ny, int gx, int gy, F&& put1) {
  const int X = gx + px, Y = gy + h;
  put1(X, Y);
  if (gx >= h && gx < nx - h && gy >= h && gy < ny - h) return;
  // x = nx + gx (site gx < h) or x = gx - nx (site gx >= nx - h)
  const int xg = gx < h ? nx + px + gx : (gx >= nx - h ? gx - nx + px : -1);
  if (xg >= 0) put1(xg, Y);
  for (int g = 0; g < h; ++g) {  // ghost rows y = g - h and y = ny + g (several when ny < 2h)
    const int ya = wrap(g - h, ny) == gy ? g : -1, yb = wrap(ny + g, ny) == gy ? ny + h + g : -1;
    if (ya >= 0) {
      put1(X, ya);
      if (xg >= 0) put1(xg, ya);
    }
    if (yb >= 0) {
      put1(X, yb);
      if (xg >= 0) put1(xg, yb);
    }
  }
}

// plain (coherent) vector loads: the kernel before may still have been writing
// these buffers when this one was launched
template <typename real>
__device__ __forceinline__ Sym5<real> qmirror_at(const real* Q, int cq4, int o) {
  real v[4];
  ld4(Q, 4 * o, v);
  return {v[0], v[1], v[2], v[3], Q[cq4 + o]};
}

// Launch with the programmatic attribute: the kernel's CTAs start as the
// previous kernel of the stream drains, and wait for it in grid_wait.  It hides
// the launch and the barrier set-up of each kernel: 12.5 -> 10.3 us per FP32 step
// at 32^3, 94.5 -> 93.5 us at 64 x 64 x 256 (two-step graphs).
// The FP32 marching kernels let the next kernel's CTAs in at their start
// (grid_launch_dependents), to set up beside them.  The others leave that to their
// end: CTAs that come in early take the places that happen to be free and stay
// there, so that a small grid ends up unevenly spread, and a kernel bound by its
// busiest SM loses more than the set-up saves.  That holds for every FP64 kernel
// (two FP64 lanes an SM: 32^3 80.1 -> 67.9 us a step, 24^3 49.0 -> 37.0, without
// flow 31.5 -> 17.5 at 32^3 together with CTAs of one warp, Gauss-Seidel 99.9 ->
// 73.6), for k_heun (FP32 without flow: 64^3 9.8 -> 8.5 us, 128^3 57.6 -> 53.1;
// 48^3 5.2 -> 5.4) and for the k_lbq before it (FP32 Gauss-Seidel 128^3 256 -> 235
// us, 96^3 99.6 -> 96.1, 80 x 64 x 48 37.6 -> 37.7), and for k_conv_win (its comment).
// The FP32 marching kernels gain from the early trigger at every even width (32^3 10.1
// -> 9.2 us, 64^3 29.6 -> 28.8); the surrogate's other kernels keep it, within 0.3% either
// way (k_rate_input and k_sur_input 5413 us for eight calls against 5425, k_dw_reduce
// the same).
//
// What such a kernel reads and the kernel before it may still be writing is read
// after grid_wait, and through plain pointers: `const T* __restrict__` and __ldg let
// the compiler take the read-only path, which is defined only for memory that nothing
// writes while the kernel lives, and lets it move the load above the wait.  The
// exceptions (f and Qin of k_lbq, the host's tables and force field) were complete
// before the kernel was launched.
template <typename... Params, typename... Args>
void launch_dependent(void (*kernel)(Params...), int grid, int threads, size_t smem, cudaStream_t s, Args&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, Params(args)...);
}

}  // namespace lcbp
