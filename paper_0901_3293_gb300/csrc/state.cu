// Whole-field operations on device arrays: the count of non-finite values
// (used to refuse uploads), the largest absolute difference of two fields
// (used by the surrogate judge to compare a surrogate call with plain steps),
// both reduced in a fixed order, and the copies between a field and its
// padded mirror with periodic ghosts (the fast step's state layout).
#include <algorithm>
#include <cmath>

#include "kernels.h"
#include "runtime.h"

namespace lcbp {

namespace {

constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 512;

// adds a CTA's count to *total (only where there is something to add: the usual
// field holds none, and no CTA writes)
__device__ __forceinline__ void add_count(unsigned bad, unsigned long long* total) {
  const int any = __syncthreads_count(bad != 0);
  if (any && bad) atomicAdd(total, (unsigned long long)bad);
}

// number of non-finite values, 16 bytes a load (v is 16-byte aligned)
template <typename real>
__global__ void __launch_bounds__(kRedThreads)
    k_count_nonfinite(const real* __restrict__ v, long long n, unsigned long long* total) {
  constexpr int W = 16 / sizeof(real);
  unsigned bad = 0;
  const long long step = (long long)gridDim.x * blockDim.x, t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int4* v4 = reinterpret_cast<const int4*>(v);
#pragma unroll 4
  for (long long i = t0; i < n / W; i += step) {
    const int4 q = v4[i];
    const real* x = reinterpret_cast<const real*>(&q);
#pragma unroll
    for (int k = 0; k < W; ++k) bad += isfinite(x[k]) ? 0u : 1u;
  }
  for (long long i = n / W * W + t0; i < n; i += step) bad += isfinite(v[i]) ? 0u : 1u;
  add_count(bad, total);
}

// Uploaded populations (full values) to the state: deviations from the rest
// weights, their moments, and the number of non-finite values, in one pass.  It
// fills buffers that are not the state's yet, so a refused upload costs nothing
// more (count, shift and moments took a pass over the field each: at 128^3 FP32
// 154 us in four launches, the call 62 us beyond its copy now).
template <typename real>
__global__ void __launch_bounds__(kRedThreads) k_load_f(const real* __restrict__ src, real* __restrict__ f,
                                                        real* __restrict__ rhou, long long n,
                                                        unsigned long long* total) {
  unsigned bad = 0;
  const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s < n) {
    real dr = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const real v = src[i * n + s];
      bad += isfinite(v) ? 0u : 1u;
      const real d = v - (real)rest_weight(i);
      f[i * n + s] = d;
      dr += d;
      jx += real(ex(i)) * d;
      jy += real(ey(i)) * d;
      jz += real(ez(i)) * d;
    }
    const real r = real(1) + dr;
    rhou[s] = dr;
    rhou[n + s] = jx / r;
    rhou[2 * n + s] = jy / r;
    rhou[3 * n + s] = jz / r;
  }
  add_count(bad, total);
}

// max |a - b| over n values, as a double; a NaN anywhere gives NaN
template <typename real>
__global__ void k_max_abs_diff(const real* __restrict__ a, const real* __restrict__ b, long long n,
                               double* __restrict__ partial) {
  double m = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double d = fabs((double)a[i] - (double)b[i]);
    m = (d > m || d != d) ? d : m;
  }
  __shared__ double red[kRedThreads];
  red[threadIdx.x] = m;
  __syncthreads();
  for (int s = kRedThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) {
      const double o = red[threadIdx.x + s];
      if (o > red[threadIdx.x] || o != o) red[threadIdx.x] = o;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

// the largest of nb partials, by one warp; a NaN among them gives NaN
__global__ void k_final_max(const double* __restrict__ partial, int nb, double* __restrict__ out) {
  double m = 0.0;
  for (int i = threadIdx.x; i < nb; i += 32) {
    const double v = partial[i];
    if (v > m || v != v) m = v;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double v = __shfl_down_sync(0xffffffffu, m, o);
    if (v > m || v != v) m = v;
  }
  if (threadIdx.x == 0) *out = m;
}

int blocks_for(long long n) {
  const long long b = (n + kRedThreads - 1) / kRedThreads;
  return (int)(b < kRedBlocks ? (b > 0 ? b : 1) : kRedBlocks);
}

}  // namespace

size_t state_check_scratch_bytes() { return (size_t)(kRedBlocks + 1) * 8; }

template <typename real>
cudaError_t launch_count_nonfinite(const void* v, long long n, unsigned long long* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(*out), s);
  if (e != cudaSuccess) return e;
  const long long want = (n / 16 + kRedThreads - 1) / kRedThreads + 1;  // about four 16-byte loads a thread
  k_count_nonfinite<real><<<(int)std::min<long long>(want, sm_count() * 8), kRedThreads, 0, s>>>(
      static_cast<const real*>(v), n, out);
  return cudaGetLastError();
}

template <typename real>
cudaError_t launch_load_f(const void* src, void* f, void* rhou, long long n, unsigned long long* out,
                          cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(*out), s);
  if (e != cudaSuccess) return e;
  k_load_f<real><<<(unsigned)((n + kRedThreads - 1) / kRedThreads), kRedThreads, 0, s>>>(
      static_cast<const real*>(src), static_cast<real*>(f), static_cast<real*>(rhou), n, out);
  return cudaGetLastError();
}

template <typename real>
cudaError_t launch_max_abs_diff(const void* a, const void* b, long long n, void* scratch, double* out,
                                cudaStream_t s) {
  auto* partial = static_cast<double*>(scratch);
  const int nb = blocks_for(n);
  k_max_abs_diff<real><<<nb, kRedThreads, 0, s>>>(static_cast<const real*>(a), static_cast<const real*>(b), n,
                                                   partial);
  k_final_max<<<1, 32, 0, s>>>(partial, nb, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// The state between its flat fields and its padded mirrors (layouts in
// kernels.h): Q and rho u of a plane's position in one thread, 16-byte vectors on
// the mirrors' side and coalesced rows on the flat side.  One launch moves both
// fields of every replica of a class (blockIdx.z): a lattice's copies took a
// launch per field with a CTA per row, whose 64-bit row arithmetic outweighed
// short rows (128^3 FP32: unpack 40 -> 25 us, pack 55 -> 28 us).
// ---------------------------------------------------------------------------
template <typename real>
__device__ __forceinline__ void put4(real* p, real a, real b, real c, real d) {
  if constexpr (sizeof(real) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
  } else {
    *reinterpret_cast<double2*>(p) = make_double2(a, b);
    *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
  }
}
template <typename real>
__device__ __forceinline__ void get4(const real* p, real v[4]) {
  if constexpr (sizeof(real) == 4) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
  } else {
    const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
  }
}

// flat -> mirrors: every site and, in the two (Q) and one (rho u) columns and
// rows next to the lattice, its periodic images
template <typename real>
__global__ void __launch_bounds__(256) k_pack(MirrorCopy a) {
  const int nx = a.nx, ny = a.ny, nz = a.nz, w = nx + 4;
  const int P = blockIdx.x * 256 + threadIdx.x;
  if (P >= w * (ny + 4)) return;
  const int Y = P / w, X = P - Y * w;  // the site's position with two ghosts on each side
  int x = X - 2, y = (Y - 2) % ny;
  x = x < 0 ? x + nx : (x >= nx ? x - nx : x);  // (nx >= 4)
  y = y < 0 ? y + ny : y;
  const bool in_u = X >= 1 && X <= nx + 2 && Y >= 1 && Y <= ny + 2;
  const long long n = (long long)nx * ny * nz;
  const int nxm = zm_mirror_nx(nx);
  for (int j = blockIdx.z; j < a.count; j += gridDim.z) {
    const real* q = static_cast<const real*>(a.q) + 5 * j * a.flat_stride;
    const real* ru = static_cast<const real*>(a.ru) + 4 * j * a.flat_stride;
    real* qm = static_cast<real*>(a.qm) + j * zm_qmirror_elems(nx, ny, nz);
    real* um = static_cast<real*>(a.um) + j * zm_umirror_elems(nx, ny, nz);
    real* yz = qm + 4LL * nxm * (ny + 4) * nz;
    for (int z = blockIdx.y; z < nz; z += gridDim.y) {
      const long long s = ((long long)z * ny + y) * nx + x;
      const long long o = ((long long)z * (ny + 4) + Y) * nxm + X - 2 + kZmMirX;
      put4(qm + 4 * o, q[s], q[n + s], q[2 * n + s], q[3 * n + s]);
      yz[o] = q[4 * n + s];
      if (in_u) {
        const long long ou = ((long long)z * (ny + 2) + Y - 1) * nxm + X - 2 + kZmMirX;
        put4(um + 4 * ou, ru[s], ru[n + s], ru[2 * n + s], ru[3 * n + s]);
      }
    }
  }
}

// mirrors -> flat; either destination may be null, and of rho u components u0..3
// are written (u0 = 1: the velocity alone, from ru on)
template <typename real>
__global__ void __launch_bounds__(256) k_unpack(MirrorCopy a) {
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int P = blockIdx.x * 256 + threadIdx.x;
  if (P >= nx * ny) return;
  const int y = P / nx, x = P - y * nx;
  const long long n = (long long)nx * ny * nz;
  const int nxm = zm_mirror_nx(nx);
  for (int j = blockIdx.z; j < a.count; j += gridDim.z) {
    real* q = a.q ? static_cast<real*>(a.q) + 5 * j * a.flat_stride : nullptr;
    real* ru = a.ru ? static_cast<real*>(a.ru) + 4 * j * a.flat_stride : nullptr;
    const real* qm = static_cast<const real*>(a.qm) + j * zm_qmirror_elems(nx, ny, nz);
    const real* um = static_cast<const real*>(a.um) + j * zm_umirror_elems(nx, ny, nz);
    const real* yz = qm + 4LL * nxm * (ny + 4) * nz;
    for (int z = blockIdx.y; z < nz; z += gridDim.y) {
      const long long s = (long long)z * ny * nx + P;
      real v[4];
      if (q) {
        const long long o = ((long long)z * (ny + 4) + y + 2) * nxm + x + kZmMirX;
        get4(qm + 4 * o, v);
#pragma unroll
        for (int c = 0; c < 4; ++c) q[c * n + s] = v[c];
        q[4 * n + s] = yz[o];
      }
      if (ru) {
        const long long o = ((long long)z * (ny + 2) + y + 1) * nxm + x + kZmMirX;
        get4(um + 4 * o, v);
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c >= a.u0) ru[(c - a.u0) * n + s] = v[c];
      }
    }
  }
}

// a CTA per 256 positions, then planes and replicas as separate CTAs up to about
// 16 CTAs per SM in all (a CTA walks the others)
dim3 copy_grid(const MirrorCopy& a, int positions) {
  const long long bx = (positions + 255) / 256, bz = std::min(a.count, 65535);
  const long long want = sm_count() * 16LL / (bx * bz) + 1;
  return dim3((unsigned)bx, (unsigned)std::min<long long>({(long long)a.nz, want, 65535LL}), (unsigned)bz);
}

template <typename real>
cudaError_t launch_pack(const MirrorCopy& a, cudaStream_t s) {
  k_pack<real><<<copy_grid(a, (a.nx + 4) * (a.ny + 4)), 256, 0, s>>>(a);
  return cudaGetLastError();
}

template <typename real>
cudaError_t launch_unpack(const MirrorCopy& a, cudaStream_t s) {
  k_unpack<real><<<copy_grid(a, a.nx * a.ny), 256, 0, s>>>(a);
  return cudaGetLastError();
}

template cudaError_t launch_pack<float>(const MirrorCopy&, cudaStream_t);
template cudaError_t launch_pack<double>(const MirrorCopy&, cudaStream_t);
template cudaError_t launch_unpack<float>(const MirrorCopy&, cudaStream_t);
template cudaError_t launch_unpack<double>(const MirrorCopy&, cudaStream_t);

template cudaError_t launch_count_nonfinite<float>(const void*, long long, unsigned long long*, cudaStream_t);
template cudaError_t launch_count_nonfinite<double>(const void*, long long, unsigned long long*, cudaStream_t);
template cudaError_t launch_load_f<float>(const void*, void*, void*, long long, unsigned long long*, cudaStream_t);
template cudaError_t launch_load_f<double>(const void*, void*, void*, long long, unsigned long long*, cudaStream_t);
template cudaError_t launch_max_abs_diff<float>(const void*, const void*, long long, void*, double*, cudaStream_t);
template cudaError_t launch_max_abs_diff<double>(const void*, const void*, long long, void*, double*, cudaStream_t);

}  // namespace lcbp
