// Small complex helpers on float2 / double2 (interleaved re, im) and the
// deterministic block reductions used by every kernel.
#pragma once
#include <cuda_runtime.h>

namespace rsn {

template <typename T> struct cx;
template <> struct cx<float> { using t = float2; };
template <> struct cx<double> { using t = double2; };

__host__ __device__ __forceinline__ float2 mk2(float a, float b) { return make_float2(a, b); }
__host__ __device__ __forceinline__ double2 mk2(double a, double b) { return make_double2(a, b); }

template <typename C> __device__ __forceinline__ C czero() { C z; z.x = 0; z.y = 0; return z; }

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { a.x += b.x; a.y += b.y; return a; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { a.x -= b.x; a.y -= b.y; return a; }
// a * b (complex)
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  C r; r.x = a.x * b.x - a.y * b.y; r.y = a.x * b.y + a.y * b.x; return r;
}
// acc + a * b (complex)
template <typename C> __device__ __forceinline__ C cfma(C a, C b, C acc) {
  acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
  acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
  return acc;
}
// acc + s * a (s real)
template <typename C, typename S> __device__ __forceinline__ C rfma(S s, C a, C acc) {
  acc.x = fma(s, a.x, acc.x); acc.y = fma(s, a.y, acc.y); return acc;
}
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  double den = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / den, (a.y * b.x - a.x * b.y) / den);
}
__device__ __forceinline__ double2 to64(float2 a) { return make_double2(a.x, a.y); }
__device__ __forceinline__ double2 to64(double2 a) { return a; }
template <typename C> __device__ __forceinline__ C from64(double2 a);
template <> __device__ __forceinline__ float2 from64<float2>(double2 a) { return make_float2((float)a.x, (float)a.y); }
template <> __device__ __forceinline__ double2 from64<double2>(double2 a) { return a; }

// Sum V values (a power of two <= 32) over the warp; lane l returns the total
// of value l % V.  At each shuffle a lane gives away half of the sums it holds:
// V - 1 + log2(32 / V) adds instead of 5 V.  On this GPU a warp's FP64 add
// occupies its FP64 pipe for 64 cycles, so reductions count their instructions.
// The lanes meet in the same order for V = 8, 16 and 32.
template <int V, int W, int DONE, typename A>
__device__ __forceinline__ void warp_sum_step(A (&v)[V]) {
  if constexpr (W < V) {
    const bool up = (threadIdx.x & W) != 0;
#pragma unroll
    for (int j = 0; j < V; ++j) {
      if ((j & (DONE | W)) == 0) {
        const A send = up ? v[j] : v[j | W];
        const A keep = up ? v[j | W] : v[j];
        v[j] = keep + __shfl_xor_sync(0xffffffffu, send, W);
      }
    }
  }
}
template <int V, typename A>
__device__ __forceinline__ A warp_sum_many(A (&v)[V]) {
  warp_sum_step<V, 4, 0>(v);
  warp_sum_step<V, 2, 4>(v);
  warp_sum_step<V, 1, 6>(v);
  warp_sum_step<V, 8, 7>(v);
  warp_sum_step<V, 16, 15>(v);
  A t = v[0];
#pragma unroll
  for (int w = V; w < 32; w <<= 1) t += __shfl_xor_sync(0xffffffffu, t, w);
  return t;
}

// a / b on a whole warp (every lane passes the same operands): the two real
// divisions run in different lanes of one instruction stream
__device__ __forceinline__ double2 cdiv_warp(double2 a, double2 b) {
  const bool im = (threadIdx.x & 1) != 0;
  const double den = b.x * b.x + b.y * b.y;
  const double num = im ? a.y * b.x - a.x * b.y : a.x * b.x + a.y * b.y;
  const double q = num / den;
  return make_double2(__shfl_sync(0xffffffffu, q, 0), __shfl_sync(0xffffffffu, q, 1));
}

// Sum NV values over the CTA in a fixed order (warp tree, then the warps' sums
// over the first warp's lanes).  Warp stages run in the accumulator type; the
// cross-warp stage in double.  Result valid in thread 0 (every lane of warp 0).
// `red` must hold 32 * (NV rounded up to a power of two) doubles.
template <int NV, typename A>
__device__ __forceinline__ void block_sum(A (&v)[NV], double* red, double (&out)[NV]) {
  constexpr int V = NV <= 1 ? 1 : NV <= 2 ? 2 : 4;
  static_assert(NV <= 4, "block_sum");
  A w[V];
#pragma unroll
  for (int i = 0; i < V; ++i) w[i] = i < NV ? v[i < NV ? i : 0] : (A)0;
  const A t = warp_sum_many<V>(w);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  A* part = reinterpret_cast<A*>(red);
  if (lane < V) part[warp * V + lane] = t;
  __syncthreads();
  if (warp == 0) {
    const int n = ((blockDim.x + 31) >> 5) * V;
    double s = 0.0;
    for (int e = lane; e < n; e += 32) s += (double)part[e];
#pragma unroll
    for (int o = V; o < 32; o <<= 1)
      if (o < n) s += __shfl_xor_sync(0xffffffffu, s, o);
#pragma unroll
    for (int i = 0; i < NV; ++i) out[i] = __shfl_sync(0xffffffffu, s, i);
  }
  __syncthreads();
}

// Allow `smem` bytes of dynamic shared memory for kernel `kern`: the attribute
// is set to the device's opt-in maximum less the kernel's static shared memory
// (not to this launch's size: contexts on other host threads may launch the
// same kernel with other sizes concurrently).
inline cudaError_t set_max_dynamic_smem(const void* kern, size_t smem) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
  cudaFuncAttributes fa;
  if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
  const long long room = (long long)optin - (long long)fa.sharedSizeBytes;
  if (room < (long long)smem) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room);
}

}  // namespace rsn
