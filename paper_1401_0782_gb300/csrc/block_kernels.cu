// Block COCG kernels: the B right-hand sides e_j of one energy share one block
// Krylov space of A(E) = E - H + i Gamma (Eqs. G, Hop; A = A^T by Eq.
// complex-sym, so the unconjugated bilinear form u^T v replaces the inner
// product of block CG).  The residual block is kept orthonormal:
//
//   R_k = Q_k xi_k,  Q_k = W_k tau_k^{-1}  (Cholesky QR: W_k^H W_k = tau_k^H tau_k)
//   P_k = Q_k + P_{k-1} beta_{k-1}                    (P_0 = Q_0)
//   alpha_k = (P_k^T A P_k)^{-1} (Q_k^T Q_k)
//   D += P_k alpha_k xi_k
//   W_{k+1} = Q_k - A P_k alpha_k,   tau_{k+1} from W_{k+1},   xi_{k+1} = tau_{k+1} xi_k
//   beta_k = (Q_k^T Q_k)^{-1} tau_{k+1}^T (Q_{k+1}^T Q_{k+1})
//
// and ||r_j|| = ||xi[:, j]|| because Q is orthonormal.  One inner iteration:
//   comb_p   P = W tau^{-1} + P beta                     (vectors, FP32)
//   project + operator (the apply kernels)   AP = A P
//   gram 0   partial sums of P^T AP                      (b x b, FP32 products)
//   small 1  alpha, alpha xi                             (b x b, FP64, one CTA per block)
//   comb_w   W = W tau^{-1} - AP alpha,  D += P alpha xi (vectors, FP32)
//   gram 1   partial sums of W^H W and W^T W
//   small 2  tau, tau^{-1}, xi, Q^T Q, beta; convergence
// A restart (start of an inner solve on the normalised FP64 residual block Rh)
// takes its QR in FP64: gram64 (Rh^H Rh, Rh^T Rh), small 0 (tau_0, xi_0 = tau_0,
// Q_0^T Q_0), q0 (W = Q_0 = Rh tau_0^{-1}, rounded once).
// Every kernel skips blocks whose flag is set (converged, breakdown, cap).
#include <cfloat>

#include "cplx.cuh"
#include "rsn_internal.h"

namespace rsn {

namespace {

__device__ __forceinline__ float2 cfma_f(float2 a, float2 b, float2 acc) {
  acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
  return acc;
}
// acc + conj(a) b
__device__ __forceinline__ float2 cjfma_f(float2 a, float2 b, float2 acc) {
  acc.x = fmaf(a.x, b.x, fmaf(a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(-a.y, b.x, acc.y));
  return acc;
}
__device__ __forceinline__ double cabs2(double2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ float2 to32(double2 a) { return make_float2((float)a.x, (float)a.y); }

// Sums of FP32 products to about FP64 accuracy in FP32 arithmetic: each
// product a b is split exactly into p = fl(a b) and its rounding error
// e = fma(a, b, -p) (error-free transformation); the p are summed with Kahan's
// compensation, the e plainly (they are ~1e-7 of the p).  The explicit _rn
// intrinsics keep the compiler from contracting p into a later addition.
struct KSum {
  float s, c, e;
};
__device__ __forceinline__ void ks_add(KSum& k, float a, float b) {
  const float p = __fmul_rn(a, b);
  k.e = __fadd_rn(k.e, __fmaf_rn(a, b, -p));
  const float y = __fsub_rn(p, k.c);
  const float t = __fadd_rn(k.s, y);
  k.c = __fsub_rn(__fsub_rn(t, k.s), y);
  k.s = t;
}
__device__ __forceinline__ double ks_val(const KSum& k) { return (double)k.s - (double)k.c + (double)k.e; }

}  // namespace

// ---------------------------------------------------------------------------
// P = W tau^{-1} + P beta   (P = W tau^{-1} in the first iteration)
// ---------------------------------------------------------------------------
template <int B>
__global__ void __launch_bounds__(kBlkThreads) blk_comb_p_kernel(const BlkDev* __restrict__ dp) {
  const BlkDev& d = *dp;
  const int k = d.blist[blockIdx.y];
  if (d.flag[k] != 0) return;
  __shared__ float2 sT[B * B], sB[B * B];
  const bool first = d.its[k] == 0;
  for (int e = threadIdx.x; e < B * B; e += blockDim.x) {
    sT[e] = d.tinv[(size_t)k * B * B + e];
    sB[e] = first ? make_float2(0.f, 0.f) : d.beta[(size_t)k * B * B + e];
  }
  __syncthreads();
  const long long N = d.N;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const size_t base = (size_t)k * B * N + i;
  float2 w[B], p[B];
#pragma unroll
  for (int a = 0; a < B; ++a) w[a] = d.W[base + (size_t)a * N];
  if (!first) {
#pragma unroll
    for (int a = 0; a < B; ++a) p[a] = d.P[base + (size_t)a * N];
  } else {
#pragma unroll
    for (int a = 0; a < B; ++a) p[a] = make_float2(0.f, 0.f);
  }
#pragma unroll
  for (int c = 0; c < B; ++c) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a <= c; ++a) acc = cfma_f(w[a], sT[a * B + c], acc);  // tau^{-1} upper triangular
    if (!first) {
#pragma unroll
      for (int a = 0; a < B; ++a) acc = cfma_f(p[a], sB[a * B + c], acc);
    }
    d.P[base + (size_t)c * N] = acc;
  }
}

// ---------------------------------------------------------------------------
// W = W tau^{-1} - AP alpha,   D += P (alpha xi)
// ---------------------------------------------------------------------------
template <int B>
__global__ void __launch_bounds__(kBlkThreads) blk_comb_w_kernel(const BlkDev* __restrict__ dp) {
  const BlkDev& d = *dp;
  const int k = d.blist[blockIdx.y];
  if (d.flag[k] != 0) return;
  __shared__ float2 sT[B * B], sA[B * B], sX[B * B];
  for (int e = threadIdx.x; e < B * B; e += blockDim.x) {
    sT[e] = d.tinv[(size_t)k * B * B + e];
    const float2 a = d.alpha[(size_t)k * B * B + e];
    sA[e] = make_float2(-a.x, -a.y);
    sX[e] = d.axi[(size_t)k * B * B + e];
  }
  __syncthreads();
  const long long N = d.N;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const size_t base = (size_t)k * B * N + i;
  {
    float2 w[B], q[B];
#pragma unroll
    for (int a = 0; a < B; ++a) {
      w[a] = d.W[base + (size_t)a * N];
      q[a] = d.AP[base + (size_t)a * N];
    }
#pragma unroll
    for (int c = 0; c < B; ++c) {
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int a = 0; a <= c; ++a) acc = cfma_f(w[a], sT[a * B + c], acc);
#pragma unroll
      for (int a = 0; a < B; ++a) acc = cfma_f(q[a], sA[a * B + c], acc);
      d.W[base + (size_t)c * N] = acc;  // every member of this point was read above
    }
  }
  {
    float2 p[B];
#pragma unroll
    for (int a = 0; a < B; ++a) p[a] = d.P[base + (size_t)a * N];
#pragma unroll
    for (int c = 0; c < B; ++c) {
      float2 acc = d.D[base + (size_t)c * N];
#pragma unroll
      for (int a = 0; a < B; ++a) acc = cfma_f(p[a], sX[a * B + c], acc);
      d.D[base + (size_t)c * N] = acc;
    }
  }
}

// ---------------------------------------------------------------------------
// Gram partial sums over one chunk of points of each listed block.
// MODE 0: U = P, V = AP, out[0] = U^T V.   MODE 1: U = V = W, out[0] = W^H W,
// out[1] = W^T W.  Tiles of kBlkTile points of every member are staged in
// shared memory (row pitch kBlkTile + 1 keeps the members' rows on distinct
// banks); each thread owns a 2 x 2 tile of (a, c) pairs and a slice of the
// tile's points.  The sums reach about FP64 accuracy in FP32 arithmetic
// (error-free products, compensated sums; the point slices and chunks in
// FP64): the block recurrence's b x b systems come from Gram matrices of
// nearly dependent directions once its residual columns share the slowest
// modes of A(E), and FP32 sums of them stall its restarts.
// ---------------------------------------------------------------------------
template <int B, int MODE>
__global__ void __launch_bounds__(kBlkThreads) blk_gram_kernel(const BlkDev* __restrict__ dp) {
  constexpr int H = B / 2;
  constexpr int NT = H * H;                // pair tiles
  constexpr int PG = kBlkThreads / NT;     // point slices
  constexpr int TP = kBlkTile;
  constexpr int LD = TP + 1;
  constexpr int NO = MODE == 0 ? 1 : 2;    // outputs
  static_assert(PG >= 1 && TP % PG == 0, "tile split");
  const BlkDev& d = *dp;
  const int k = d.blist[blockIdx.y];
  if (d.flag[k] != 0) return;
  __shared__ float2 sU[B * LD];
  __shared__ float2 sV[(MODE == 0 ? B : 1) * LD];
  __shared__ double2 red[PG * NT * 4 * NO];
  const long long N = d.N;
  const int chunk = blockIdx.x;
  const long long x0 = (long long)chunk * d.chunk_pts;
  const long long x1 = min(N, x0 + d.chunk_pts);
  const size_t base = (size_t)k * B * N;
  const float2* U = MODE == 0 ? d.P : d.W;
  const float2* V = MODE == 0 ? d.AP : d.W;
  const int tid = threadIdx.x;
  const int t = tid % NT, g = tid / NT;
  const int a0 = 2 * (t / H), c0 = 2 * (t % H);
  // [output][pair][re, im]
  KSum ks[NO][4][2];
#pragma unroll
  for (int o = 0; o < NO; ++o)
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int r = 0; r < 2; ++r) ks[o][m][r] = KSum{0.f, 0.f, 0.f};
  for (long long ts = x0; ts < x1; ts += TP) {
    for (int e = tid; e < B * TP; e += kBlkThreads) {
      const int a = e / TP, ii = e % TP;
      const long long i = ts + ii;
      const bool in = i < x1;
      sU[a * LD + ii] = in ? U[base + (size_t)a * N + i] : make_float2(0.f, 0.f);
      if constexpr (MODE == 0) sV[a * LD + ii] = in ? V[base + (size_t)a * N + i] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const float2* sv = MODE == 0 ? sV : sU;
#pragma unroll 2
    for (int ii = g; ii < TP; ii += PG) {
      const float2 uu[2] = {sU[a0 * LD + ii], sU[(a0 + 1) * LD + ii]};
      const float2 vv[2] = {sv[c0 * LD + ii], sv[(c0 + 1) * LD + ii]};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float2 u = uu[m >> 1], v = vv[m & 1];
        if constexpr (MODE == 0) {
          // u v
          ks_add(ks[0][m][0], u.x, v.x);
          ks_add(ks[0][m][0], -u.y, v.y);
          ks_add(ks[0][m][1], u.x, v.y);
          ks_add(ks[0][m][1], u.y, v.x);
        } else {
          // conj(u) v and u v
          ks_add(ks[0][m][0], u.x, v.x);
          ks_add(ks[0][m][0], u.y, v.y);
          ks_add(ks[0][m][1], u.x, v.y);
          ks_add(ks[0][m][1], -u.y, v.x);
          ks_add(ks[1][m][0], u.x, v.x);
          ks_add(ks[1][m][0], -u.y, v.y);
          ks_add(ks[1][m][1], u.x, v.y);
          ks_add(ks[1][m][1], u.y, v.x);
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int o = 0; o < NO; ++o)
#pragma unroll
    for (int m = 0; m < 4; ++m)
      red[((o * PG + g) * NT + t) * 4 + m] = make_double2(ks_val(ks[o][m][0]), ks_val(ks[o][m][1]));
  __syncthreads();
  // slices summed in a fixed order; entry (a, c) of output o
  double2* out = d.part + ((size_t)k * d.nchunk + chunk) * 2 * B * B;
  for (int e = tid; e < NO * B * B; e += kBlkThreads) {
    const int o = e / (B * B), ac = e % (B * B);
    const int a = ac / B, c = ac % B;
    const int tt = (a / 2) * H + (c / 2), m = (a & 1) * 2 + (c & 1);
    double2 v = make_double2(0.0, 0.0);
    for (int gg = 0; gg < PG; ++gg) {
      const double2 r = red[((o * PG + gg) * NT + tt) * 4 + m];
      v.x += r.x;
      v.y += r.y;
    }
    out[(size_t)o * B * B + ac] = v;
  }
}

// ---------------------------------------------------------------------------
// Restart of an inner solve: partial sums of Rh^H Rh and Rh^T Rh of the
// normalised FP64 residual block Rh = R / ||R|| (in R), products and sums in
// FP64.  The residual columns of a restart share the slowest modes of A(E) and
// are close to dependent; an FP32 Gram would lose the orthogonality of Q_0 to
// rounding (~1e-7 kappa^2), the FP64 one keeps it.  Same layout as the FP32
// Gram: a 2 x 2 tile of (a, c) pairs per thread over a slice of the points.
// ---------------------------------------------------------------------------
template <int B>
__global__ void __launch_bounds__(kBlkThreads) blk_gram64_kernel(const BlkDev* __restrict__ dp) {
  constexpr int H = B / 2;
  constexpr int NT = H * H;
  constexpr int PG = kBlkThreads / NT;
  const BlkDev& d = *dp;
  const int k = d.blist[blockIdx.y];
  if (d.flag[k] != 0) return;
  __shared__ double2 red[PG * NT * 4 * 2];
  const long long N = d.N;
  const int chunk = blockIdx.x;
  const long long x0 = (long long)chunk * d.chunk_pts;
  const long long x1 = min(N, x0 + d.chunk_pts);
  const double2* R = d.R + (size_t)k * B * N;
  const int tid = threadIdx.x;
  const int t = tid % NT, g = tid / NT;
  const int a0 = 2 * (t / H), c0 = 2 * (t % H);
  double2 sh[4], st[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) sh[m] = st[m] = make_double2(0.0, 0.0);
  for (long long i = x0 + g; i < x1; i += PG) {
    const double2 u0 = R[(size_t)a0 * N + i], u1 = R[(size_t)(a0 + 1) * N + i];
    const double2 v0 = R[(size_t)c0 * N + i], v1 = R[(size_t)(c0 + 1) * N + i];
    const double2 uu[2] = {u0, u1}, vv[2] = {v0, v1};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const double2 u = uu[m >> 1], v = vv[m & 1];
      sh[m].x += u.x * v.x + u.y * v.y;  // conj(u) v
      sh[m].y += u.x * v.y - u.y * v.x;
      st[m].x += u.x * v.x - u.y * v.y;  // u v
      st[m].y += u.x * v.y + u.y * v.x;
    }
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    red[((0 * PG + g) * NT + t) * 4 + m] = sh[m];
    red[((1 * PG + g) * NT + t) * 4 + m] = st[m];
  }
  __syncthreads();
  double2* out = d.part + ((size_t)k * d.nchunk + chunk) * 2 * B * B;
  for (int e = tid; e < 2 * B * B; e += kBlkThreads) {
    const int o = e / (B * B), ac = e % (B * B);
    const int a = ac / B, c = ac % B;
    const int tt = (a / 2) * H + (c / 2), m = (a & 1) * 2 + (c & 1);
    double2 v = make_double2(0.0, 0.0);
    for (int gg = 0; gg < PG; ++gg) {
      const double2 r = red[((o * PG + gg) * NT + tt) * 4 + m];
      v.x += r.x;
      v.y += r.y;
    }
    out[(size_t)o * B * B + ac] = v;
  }
}

// Q_0 = Rh tau_0^{-1} in FP64 (tau_0^{-1} from the restart's Cholesky, upper
// triangular), rounded to FP32 into W; D = 0.
template <int B>
__global__ void __launch_bounds__(kBlkThreads) blk_q0_kernel(const BlkDev* __restrict__ dp) {
  const BlkDev& d = *dp;
  const int k = d.blist[blockIdx.y];
  if (d.flag[k] != 0) return;
  __shared__ double2 sT[B * B];
  for (int e = threadIdx.x; e < B * B; e += blockDim.x) sT[e] = d.tinv64[(size_t)k * B * B + e];
  __syncthreads();
  const long long N = d.N;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const size_t base = (size_t)k * B * N + i;
  double2 r[B];
#pragma unroll
  for (int a = 0; a < B; ++a) r[a] = d.R[base + (size_t)a * N];
#pragma unroll
  for (int c = 0; c < B; ++c) {
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll
    for (int a = 0; a <= c; ++a) {
      const double2 t = sT[a * B + c];
      acc.x += r[a].x * t.x - r[a].y * t.y;
      acc.y += r[a].x * t.y + r[a].y * t.x;
    }
    d.W[base + (size_t)c * N] = make_float2((float)acc.x, (float)acc.y);
    d.D[base + (size_t)c * N] = make_float2(0.f, 0.f);
  }
}

// ---------------------------------------------------------------------------
// b x b algebra of each listed block, FP64, one CTA of B * B threads (at least a
// warp): thread t owns entry (t / B, t % B).  A warp's FP64 instruction takes 64
// cycles of its FP64 pipe, so what counts is the number of instructions on the
// longest chain: entries are spread over the four pipes, the divisions of a step over
// the lanes of one warp, and the pivot search compares bits.  At B = 16 a phase-1 call
// takes 32 us and a phase-2 call 73 (one warp per block: 225 and 510; Newton
// reciprocals for the divisions and fused products: 27 and 61, at half again the error).
// ---------------------------------------------------------------------------
namespace {

// acc + a b and acc - a b, the product rounded before it meets acc: in the nearly
// diagonal systems of a block the products are small beside acc, and a chain of fused
// additions rounds twice at the size of acc (median error of alpha over 193 systems of
// three junctions at B = 16: 2.4e-16, fused and with reciprocals 3.6e-16; of the
// Cholesky factor 8.4e-17 against 1.1e-16)
__device__ __forceinline__ double2 cmac64(double2 a, double2 b, double2 acc) {
  return make_double2(acc.x + fma(a.x, b.x, -(a.y * b.y)), acc.y + fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cmsub64(double2 a, double2 b, double2 acc) {
  return make_double2(acc.x - fma(a.x, b.x, -(a.y * b.y)), acc.y - fma(a.x, b.y, a.y * b.x));
}
// acc + a b, fused: for sums of like terms (Q^T Q and the right-hand side of beta, whose
// median errors are 2.27e-16 and 1.68e-16 with it, 2.34e-16 and 1.87e-16 without)
__device__ __forceinline__ double2 cfma64(double2 a, double2 b, double2 acc) {
  acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
  acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
  return acc;
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }

// Both factorisations below take one barrier a step: while the other warps apply step
// kk, warp 0 brings the next step's column (or row) up to date and prepares that step,
// whose divisions are the longest chain.  What a step hands over lies in two buffers,
// by parity: one is written while slower warps still read the other.
//
// The threads that apply a step: all but warp 0 and, of eight warps, the one that
// shares its FP64 pipe; a single warp does both.
template <int B>
__device__ __forceinline__ bool step_worker(int& index, int& count) {
  constexpr int NW = B * B <= 32 ? 1 : B * B / 32, NWK = NW == 1 ? 1 : NW <= 4 ? NW - 1 : NW - NW / 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  count = 32 * NWK;
  index = (NW == 1 ? 0 : NW <= 4 ? warp - 1 : warp - warp / 4 - 1) * 32 + lane;
  return NW == 1 || (warp & 3) != 0;
}

// Shared memory of the factorisations.
template <int B>
struct StepMem {
  double2 fac[2][B];
  double ref[B];
  int piv[B];
  int ok[2];
};

// Solve M X = Y in place for aug = [M | Y] (B rows, 2B columns, leading
// dimension LD): Gauss-Jordan elimination with partial pivoting.  X replaces Y.
// Returns false (in every thread) on a zero or non-finite pivot.  Rows stay where they
// are; step k's pivot row is piv[k].
template <int B, int LD>
__device__ bool gauss_jordan(double2* aug, StepMem<B>& sm) {
  const int tid = threadIdx.x, lane = tid & 31;
  unsigned used = 0;  // warp 0: pivot rows so far
  // warp 0: the pivot row of column kk (largest modulus) and the factors of the others,
  // real and imaginary parts in different lanes
  auto prepare = [&](int kk) {
    long long key = -1;  // positive doubles order like their bits
    if (lane < B && !((used >> lane) & 1u)) {
      const double2 v = aug[lane * LD + kk];
      key = __double_as_longlong(fma(v.x, v.x, v.y * v.y)) & 0x7fffffffffffffffll;
    }
    const int hi = (int)(key >> 32), top = __reduce_max_sync(0xffffffffu, hi);
    const unsigned lo = hi == top ? (unsigned)key : 0u, low = __reduce_max_sync(0xffffffffu, lo);
    const int piv = __ffs(__ballot_sync(0xffffffffu, hi == top && lo == low)) - 1;
    used |= 1u << piv;
    const int r = lane % B, part = lane / B;
    const double2 p = aug[piv * LD + kk], v = aug[r * LD + kk];
    const double num = part ? fma(v.y, p.x, -(v.x * p.y)) : fma(v.x, p.x, v.y * p.y);
    const double q = num / fma(p.x, p.x, p.y * p.y);
    if (part < 2) reinterpret_cast<double*>(sm.fac[kk & 1] + r)[part] = q;
    if (lane == 0) {
      sm.piv[kk] = piv;
      sm.ok[kk & 1] = top < 0x7ff00000 && (top > 0 || low > 0) ? 1 : 0;
    }
  };
  if (tid < 32) prepare(0);
  int w, nwk;
  const bool worker = step_worker<B>(w, nwk);
  for (int kk = 0; kk < B; ++kk) {
    __syncthreads();
    if (!sm.ok[kk & 1]) return false;
    const int p = sm.piv[kk];
    const double2* f = sm.fac[kk & 1];
    if (tid < 32 && kk + 1 < B) {
      const int r = lane % B, part = lane / B;
      if (part < 2 && r != p) {
        const double2 a = f[r], b = aug[p * LD + kk + 1];
        const double t = part ? fma(a.x, b.y, a.y * b.x) : fma(a.x, b.x, -(a.y * b.y));
        reinterpret_cast<double*>(aug + r * LD + kk + 1)[part] -= t;
      }
      __syncwarp();
      prepare(kk + 1);
    }
    if (worker) {
      const int c0 = kk + 1 < B ? kk + 2 : B, nc = 2 * B - c0;
      for (int e = w; e < (B - 1) * nc; e += nwk) {
        int r = e / nc;
        const int c = c0 + e - r * nc;
        r += r >= p ? 1 : 0;
        aug[r * LD + c] = cmsub64(f[r], aug[p * LD + c], aug[r * LD + c]);
      }
    }
  }
  __syncthreads();
  const int er = tid / B, ec = tid % B;
  double2 x = make_double2(0.0, 0.0);
  if (er < B) x = cdiv(aug[sm.piv[er] * LD + B + ec], aug[sm.piv[er] * LD + er]);
  __syncthreads();
  if (er < B) aug[er * LD + B + ec] = x;
  __syncthreads();
  return true;
}

// Cholesky factor of the Hermitian positive definite A (B x B, leading dimension
// B, destroyed above its diagonal blocks) and the inverse of its lower factor:
// A = Lc Lc^H; U = Lc^H (upper), Li = Lc^{-1} (lower).  Fails when a pivot is not
// positive or falls below 1e-12 of its diagonal entry (numerically dependent
// columns).
template <int B>
__device__ bool cholesky_inverse(double2* A, double2* U, double2* Li, StepMem<B>& sm) {
  const int tid = threadIdx.x, er = tid / B, ec = tid % B;
  if (er < B) {
    U[tid] = make_double2(0.0, 0.0);
    Li[tid] = make_double2(er == ec ? 1.0 : 0.0, 0.0);
    if (er == ec) sm.ref[er] = A[tid].x;
  }
  __syncthreads();
  // warp 0: row kk of U (columns >= kk) and of Li (columns <= kk), real and imaginary
  // parts in different lanes
  const int lc = (tid & 31) % B, part = (tid & 31) / B;
  auto prepare = [&](int kk) {
    const double dd = A[kk * B + kk].x;
    const double dk = sqrt(dd);
    if (part < 2) {
      const double v = lc == kk ? (part ? 0.0 : 1.0) : reinterpret_cast<const double*>((lc > kk ? A : Li) + kk * B + lc)[part];
      reinterpret_cast<double*>((lc > kk ? U : Li) + kk * B + lc)[part] = v / dk;
      if (tid == kk) U[kk * B + kk] = make_double2(dk, 0.0);
    }
    if (tid == 0) sm.ok[kk & 1] = dd > 1e-12 * sm.ref[kk] && dd <= DBL_MAX ? 1 : 0;
  };
  if (tid < 32) prepare(0);
  int w, nwk;
  const bool worker = step_worker<B>(w, nwk);
  for (int kk = 0; kk < B; ++kk) {
    __syncthreads();
    if (!sm.ok[kk & 1]) return false;
    if (tid < 32 && kk + 1 < B) {
      const int r = kk + 1;
      if (part < 2) {
        const double2 a = cconj(U[kk * B + r]), b = (lc > kk ? U : Li)[kk * B + lc];
        const double t = part ? fma(a.x, b.y, a.y * b.x) : fma(a.x, b.x, -(a.y * b.y));
        reinterpret_cast<double*>((lc > kk ? A : Li) + r * B + lc)[part] -= t;
      }
      __syncwarp();
      prepare(r);
    }
    if (worker) {
      for (int e = (kk + 2) * B + w; e < B * B; e += nwk) {
        const int r = e / B, c = e % B;
        const double2 f = cconj(U[kk * B + r]);  // Lc[r][kk]
        if (c > kk) A[e] = cmsub64(f, U[kk * B + c], A[e]);
        else Li[e] = cmsub64(f, Li[kk * B + c], Li[e]);
      }
    }
  }
  __syncthreads();
  return true;
}

}  // namespace

// Sums of the Gram partials over the chunks, one warp per entry:
// d.gsum[k][o][e], o < no.
template <int B>
__global__ void __launch_bounds__(256) blk_psum_kernel(const BlkDev* __restrict__ dp, int no) {
  const BlkDev& d = *dp;
  const int k = d.blist[blockIdx.y];
  if (d.flag[k] != 0) return;
  const int lane = threadIdx.x & 31, e = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (e >= no * B * B) return;
  double v[2] = {0.0, 0.0};
  for (int ch = lane; ch < d.nchunk; ch += 32) {
    const double2 r = d.part[((size_t)k * d.nchunk + ch) * 2 * B * B + e];
    v[0] += r.x;
    v[1] += r.y;
  }
  const double t = warp_sum_many<2>(v);
  if (lane < 2) reinterpret_cast<double*>(d.gsum + (size_t)k * 2 * B * B + e)[lane] = t;
}

// PHASE 0: start of an inner solve (W holds the normalised residual block):
//          tau_0, tau_0^{-1}, xi_0 = tau_0, ||xi_0[:, j]||, Q_0^T Q_0.
// PHASE 1: alpha = (P^T AP)^{-1} Q^T Q and alpha xi.
// PHASE 2: tau, tau^{-1} of the new W; xi <- tau xi; Q^T Q of the new Q;
//          beta; iteration count and convergence of every column.
template <int B, int PHASE>
__global__ void __launch_bounds__(B * B < 32 ? 32 : B * B) blk_small_kernel(const BlkDev* __restrict__ dp) {
  constexpr int LD = 2 * B + 1;
  const BlkDev& d = *dp;
  const int k = d.blist[blockIdx.x];
  const int tid = threadIdx.x;
  if (PHASE != 0 && d.flag[k] != 0) return;
  __shared__ double2 aug[B * LD];
  __shared__ double2 M0[B * B], M1[B * B], M2[B * B], M3[B * B];
  __shared__ StepMem<B> sm;
  const size_t ko = (size_t)k * B * B;
  const bool own = tid < B * B;
  const int a = tid / B, j = tid % B;  // the thread's entry
  const double2 zero = make_double2(0.0, 0.0);
  const double2* G = d.gsum + 2 * ko;
  if (PHASE == 1) {
    if (own) {
      aug[a * LD + j] = G[tid];  // P^T A P
      aug[a * LD + B + j] = d.QQ[ko + tid];
      M1[tid] = d.xi[ko + tid];
    }
    __syncthreads();
    if (!gauss_jordan<B, LD>(aug, sm)) {
      if (tid == 0) d.flag[k] = 2;
      return;
    }
    if (own) {
      double2 v = zero;  // alpha xi
#pragma unroll 4
      for (int m = 0; m < B; ++m) v = cmac64(aug[a * LD + B + m], M1[m * B + j], v);
      d.alpha[ko + tid] = to32(aug[a * LD + B + j]);
      d.axi[ko + tid] = to32(v);
    }
    return;
  }
  // PHASE 0 / 2: Cholesky QR of W
  if (own) {
    M0[tid] = G[tid];          // W^H W
    M1[tid] = G[B * B + tid];  // W^T W
  }
  __syncthreads();
  if (!cholesky_inverse<B>(M0, M2, M3, sm)) {  // M2 = tau = Lc^H, M3 = Lc^{-1}, tau^{-1} = M3^H
    if (tid == 0) d.flag[k] = 2;
    return;
  }
  // tau^{-1} for the vector kernels: at a restart (PHASE 0) in FP64 for the
  // Q_0 kernel, which writes Q_0 itself into W, so that the FP32 copy is I
  if (own) {
    const double2 v = cconj(M3[j * B + a]);
    if (PHASE == 0) {
      d.tinv64[ko + tid] = v;
      d.tinv[ko + tid] = make_float2(a == j ? 1.f : 0.f, 0.f);
    } else {
      d.tinv[ko + tid] = to32(v);
    }
  }
  // Q^T Q = tau^{-T} (W^T W) tau^{-1}.  Triangular factors: entries are owned so
  // that a warp's lanes run sums of nearly the same length.
  if (own) {
    double2 v = zero;  // T1[j][a] = sum_{m <= a} (W^T W)[j][m] tau^{-1}[m][a]
    for (int m = 0; m <= a; ++m) v = cfma64(M1[j * B + m], cconj(M3[a * B + m]), v);
    M0[j * B + a] = v;
  }
  __syncthreads();
  if (own) {
    double2 v = zero;  // QQ[a][j] = sum_{m <= a} tau^{-1}[m][a] T1[m][j]
    for (int m = 0; m <= a; ++m) v = cfma64(cconj(M3[a * B + m]), M0[m * B + j], v);
    M1[tid] = v;  // W^T W is no longer needed
  }
  if (PHASE == 0) {
    __syncthreads();
    if (own) {
      d.xi[ko + tid] = M2[tid];
      d.QQ[ko + tid] = M1[tid];
    }
    if (tid < B) {
      double s = 0.0;
      for (int m = 0; m < B; ++m) s += cabs2(M2[m * B + tid]);  // column tid of tau
      d.xi0n[(size_t)k * B + tid] = sqrt(s);
    }
    if (tid == 0) {
      d.flag[k] = 0;
      d.its[k] = 0;
    }
    return;
  }
  // xi_{k+1} = tau xi_k
  if (own) aug[tid] = d.xi[ko + tid];
  __syncthreads();  // M1 and the old xi are complete
  double2 xn = zero, rhs = zero;
  if (own) {
    for (int m = a; m < B; ++m) xn = cmac64(M2[a * B + m], aug[m * B + j], xn);
    // right-hand side of beta: tau^T QQ_{k+1}
    for (int m = 0; m <= a; ++m) rhs = cfma64(M2[m * B + a], M1[m * B + j], rhs);
    d.xi[ko + tid] = xn;
    M0[tid] = make_double2(cabs2(xn), 0.0);
  }
  __syncthreads();
  // every column's residual norm ||xi[:, j]|| against its start
  bool conv = true;
  if (tid < B) {
    double s = 0.0;
    for (int m = 0; m < B; ++m) s += M0[m * B + tid].x;
    conv = sqrt(s) <= d.tol_in * d.xi0n[(size_t)k * B + tid];
  }
  // beta = QQ_k^{-1} (tau^T QQ_{k+1})
  if (own) {
    aug[a * LD + j] = d.QQ[ko + tid];
    aug[a * LD + B + j] = rhs;
  }
  conv = __syncthreads_and(conv);
  const bool ok = gauss_jordan<B, LD>(aug, sm);
  if (own) {
    d.QQ[ko + tid] = M1[tid];
    if (ok) d.beta[ko + tid] = to32(aug[a * LD + B + j]);
  }
  if (tid == 0) {
    const int it = d.its[k] + 1;
    d.its[k] = it;
    d.flag[k] = conv ? 1 : !ok ? 2 : it >= d.icap[k] ? 3 : 0;
  }
}

// ---------------------------------------------------------------------------
// Outer (FP64) steps over the members of the listed blocks: grid.y = listed
// blocks x B, member v = blist[y / B] * B + y % B.
// ---------------------------------------------------------------------------
// R = e_col - A X (A X already in R when have_ax), partial ||R||^2 and
// sum_{i} Gamma_L(i) |X(i)|^2 per chunk of points.
__global__ void __launch_bounds__(kBlkThreads) blk_resid_kernel(const BlkDev* __restrict__ dp, int have_ax) {
  const BlkDev& d = *dp;
  const int B = d.B;
  const int v = d.blist[blockIdx.y / B] * B + (int)(blockIdx.y % B);
  const long long N = d.N;
  const long long x0 = (long long)blockIdx.x * d.chunkR_pts;
  const long long x1 = min(N, x0 + d.chunkR_pts);
  const int col = d.col[v];
  double2* R = d.R + (size_t)v * N;
  const double2* X = d.X + (size_t)v * N;
  double acc[2] = {0.0, 0.0};
  for (long long i = x0 + threadIdx.x; i < x1; i += blockDim.x) {
    double2 r = have_ax ? R[i] : make_double2(0.0, 0.0);
    r.x = (i == col ? 1.0 : 0.0) - r.x;
    r.y = -r.y;
    R[i] = r;
    acc[0] += cabs2(r);
    const double g = d.gl[i];
    if (g > 0.0) acc[1] += g * cabs2(X[i]);
  }
  __shared__ double red[32 * 2];
  double out[2];
  block_sum<2>(acc, red, out);
  if (threadIdx.x == 0) {
    double* p = d.rpart + ((size_t)v * d.nchunkR + blockIdx.x) * 2;
    p[0] = out[0];
    p[1] = out[1];
  }
}

// rn = ||R||, tt = sum Gamma_L |X|^2 per listed member (chunks in order)
__global__ void blk_norm_kernel(const BlkDev* __restrict__ dp, int n_members) {
  const BlkDev& d = *dp;
  const int y = blockIdx.x * blockDim.x + threadIdx.x;
  if (y >= n_members) return;
  const int B = d.B;
  const int v = d.blist[y / B] * B + y % B;
  double s0 = 0.0, s1 = 0.0;
  for (int ch = 0; ch < d.nchunkR; ++ch) {
    s0 += d.rpart[((size_t)v * d.nchunkR + ch) * 2];
    s1 += d.rpart[((size_t)v * d.nchunkR + ch) * 2 + 1];
  }
  d.rn[v] = sqrt(s0);
  d.tt[v] = s1;
}

// R <- R / ||R|| per member (FP64, in place): the right-hand sides of the next
// inner solve, each of unit norm
__global__ void __launch_bounds__(kBlkThreads) blk_scale_kernel(const BlkDev* __restrict__ dp) {
  const BlkDev& d = *dp;
  const int B = d.B;
  const int v = d.blist[blockIdx.y / B] * B + (int)(blockIdx.y % B);
  const long long N = d.N;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double rn = d.rn[v];
  const double s = rn > 0.0 ? 1.0 / rn : 0.0;
  double2 r = d.R[(size_t)v * N + i];
  r.x *= s;
  r.y *= s;
  d.R[(size_t)v * N + i] = r;
}

// X += ||R|| D (the inner solution solves A D = R / ||R|| per column)
__global__ void __launch_bounds__(kBlkThreads) blk_xupd_kernel(const BlkDev* __restrict__ dp) {
  const BlkDev& d = *dp;
  const int B = d.B;
  const int v = d.blist[blockIdx.y / B] * B + (int)(blockIdx.y % B);
  const long long N = d.N;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double rn = d.rn[v];
  const float2 dd = d.D[(size_t)v * N + i];
  double2 x = d.X[(size_t)v * N + i];
  x.x = fma(rn, (double)dd.x, x.x);
  x.y = fma(rn, (double)dd.y, x.y);
  d.X[(size_t)v * N + i] = x;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
#define RSN_BLK_DISPATCH(B, CALL) \
  switch (B) {                    \
    case 4: CALL(4); break;       \
    case 8: CALL(8); break;       \
    case 16: CALL(16); break;     \
    default: return cudaErrorInvalidValue; \
  }

cudaError_t launch_blk_comb_p(int B, int nb, cudaStream_t st, const BlkDev* d, long long N) {
  const dim3 grid((unsigned)((N + kBlkThreads - 1) / kBlkThreads), nb);
#define L_(BB) blk_comb_p_kernel<BB><<<grid, kBlkThreads, 0, st>>>(d)
  RSN_BLK_DISPATCH(B, L_)
#undef L_
  return cudaGetLastError();
}

cudaError_t launch_blk_comb_w(int B, int nb, cudaStream_t st, const BlkDev* d, long long N) {
  const dim3 grid((unsigned)((N + kBlkThreads - 1) / kBlkThreads), nb);
#define L_(BB) blk_comb_w_kernel<BB><<<grid, kBlkThreads, 0, st>>>(d)
  RSN_BLK_DISPATCH(B, L_)
#undef L_
  return cudaGetLastError();
}

cudaError_t launch_blk_gram(int B, int mode, int nb, int nchunk, cudaStream_t st, const BlkDev* d) {
  const dim3 grid(nchunk, nb);
  if (mode == 0) {
#define L_(BB) blk_gram_kernel<BB, 0><<<grid, kBlkThreads, 0, st>>>(d)
    RSN_BLK_DISPATCH(B, L_)
#undef L_
  } else {
#define L_(BB) blk_gram_kernel<BB, 1><<<grid, kBlkThreads, 0, st>>>(d)
    RSN_BLK_DISPATCH(B, L_)
#undef L_
  }
  return cudaGetLastError();
}

cudaError_t launch_blk_gram64(int B, int nb, int nchunk, cudaStream_t st, const BlkDev* d) {
  const dim3 grid(nchunk, nb);
#define L_(BB) blk_gram64_kernel<BB><<<grid, kBlkThreads, 0, st>>>(d)
  RSN_BLK_DISPATCH(B, L_)
#undef L_
  return cudaGetLastError();
}

cudaError_t launch_blk_q0(int B, int nb, cudaStream_t st, const BlkDev* d, long long N) {
  const dim3 grid((unsigned)((N + kBlkThreads - 1) / kBlkThreads), nb);
#define L_(BB) blk_q0_kernel<BB><<<grid, kBlkThreads, 0, st>>>(d)
  RSN_BLK_DISPATCH(B, L_)
#undef L_
  return cudaGetLastError();
}

cudaError_t launch_blk_small(int B, int phase, int nb, cudaStream_t st, const BlkDev* d) {
  const int no = phase == 1 ? 1 : 2, nt = B * B < 32 ? 32 : B * B;
  const dim3 gs((no * B * B + 7) / 8, nb);
#define L_(BB)                                                                 \
  {                                                                            \
    blk_psum_kernel<BB><<<gs, 256, 0, st>>>(d, no);                            \
    if (phase == 0) blk_small_kernel<BB, 0><<<nb, nt, 0, st>>>(d);             \
    else if (phase == 1) blk_small_kernel<BB, 1><<<nb, nt, 0, st>>>(d);        \
    else blk_small_kernel<BB, 2><<<nb, nt, 0, st>>>(d);                        \
  }
  RSN_BLK_DISPATCH(B, L_)
#undef L_
  return cudaGetLastError();
}

cudaError_t launch_blk_resid(int B, int nb, int nchunkR, bool have_ax, cudaStream_t st, const BlkDev* d) {
  blk_resid_kernel<<<dim3(nchunkR, nb * B), kBlkThreads, 0, st>>>(d, have_ax ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_blk_norm(int B, int nb, int nchunkR, cudaStream_t st, const BlkDev* d) {
  (void)nchunkR;
  const int n = nb * B;
  blk_norm_kernel<<<(n + 127) / 128, 128, 0, st>>>(d, n);
  return cudaGetLastError();
}

cudaError_t launch_blk_scale(int B, int nb, cudaStream_t st, const BlkDev* d, long long N) {
  blk_scale_kernel<<<dim3((unsigned)((N + kBlkThreads - 1) / kBlkThreads), nb * B), kBlkThreads, 0, st>>>(d);
  return cudaGetLastError();
}

cudaError_t launch_blk_xupd(int B, int nb, cudaStream_t st, const BlkDev* d, long long N) {
  blk_xupd_kernel<<<dim3((unsigned)((N + kBlkThreads - 1) / kBlkThreads), nb * B), kBlkThreads, 0, st>>>(d);
  return cudaGetLastError();
}

}  // namespace rsn
