// FP32 operator kernel on point pairs with plane streaming: y = A_loc(E) v
// (COCG) or y = A_loc(E) x (apply), A_loc = E - H + i(Gamma_L + Gamma_R) (Eqs. G
// and Hop) with H = -1/2 lap_FD + V_loc (Sec. II.C); the projector term is added
// by the COCG update kernel, or by nonlocal_kernel after an application.
//
// One CTA owns whole x-y planes [z0, z0+Lz) of one slot and marches along z.
//  * The input planes (r and p_old, or x) of planes z0-R .. z0+Lz+R-1 arrive by
//    bulk copies (TMA, cp.async.bulk) in a ring of kPairStages shared-memory
//    stages, issued kPairStages planes ahead of use and completed on one
//    mbarrier per stage, so the bytes in flight cost no registers.
//  * Each thread owns two x-neighbours (x0, x0+1) of one row (nx even), so each
//    shared-memory access moves one 128-bit pair and each global store 16 bytes.
//  * The 2R+1 produced planes around the current one sit in a register ring
//    whose slot for plane z is (z - z0 + R) mod (2R+1); the march is unrolled by
//    2R+1, so every ring index is a compile-time constant and nothing is shifted.
//  * The current plane goes through a double-buffered shared-memory tile for
//    the x and y neighbours (one barrier per plane), with a compile-time row pitch
//    for the common widths (pair_pitch_const); the zero columns and rows around it are the Dirichlet boundary.
// 24x24x120, order 8: 256 systems 158 us, 3.6 TB/s of the 32 B a point (235 us with
// a run-time pitch, whose neighbour addresses spilled, and fixed z chunks); IPC 2.0
// of 4 at 18 warps an SM, waits on shared memory, fixed latencies and the barrier.
//
// FP32 accuracy: the neighbour terms at distances m <= 2, whose weights carry
// the large part of the Laplacian, are summed in difference form,
// w_m sum_nb (v_nb - v_c): near-equal values subtract exactly, so the large
// FD diagonal never meets the small result of smooth fields.  The terms at
// m > 2 (weights below 1/10 of w_1) are summed directly, and their share of
// the diagonal, -6 sum_{m>2} w_m, is folded into E - V_loc.
#pragma once
#include "cplx.cuh"
#include "exact_sum.cuh"
#include "rsn_internal.h"
#include "tma.cuh"

namespace rsn {

// elementwise a + b, a - b, a * b + c on (re, im) pairs (the compiler pairs
// them into Blackwell's two-wide FP32 instructions where that pays; explicit
// f32x2 inline assembly measured slower, its operand packing costs moves)
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
}
// acc + a * b for complex a, b
__device__ __forceinline__ float2 cfma2(float2 a, float2 b, float2 acc) {
  acc = fma2(make_float2(a.x, a.x), b, acc);
  return fma2(make_float2(-a.y, a.y), make_float2(b.y, b.x), acc);
}

// The CTA's tile of its slot: tiles past the 65,535 of a grid's y dimension go on in
// its z dimension (op_grid).
__device__ __forceinline__ int launch_tile() { return (int)(blockIdx.z * gridDim.y + blockIdx.y); }

// Planes per z chunk of a COCG operator launch, by the number of active slots
// (host: choose_tiling), and the operator CTAs of a slot with it.
__device__ __forceinline__ int cocg_lz(const JuncDev& J, const BatchDev& b) {
  const int n = *b.nact;
  return J.lz_act[n <= 1 ? 0 : min(kActBuckets - 1, 32 - __clz(n - 1))];
}
__device__ __forceinline__ int cocg_tiles(const JuncDev& J, const BatchDev& b) {
  const int lz = cocg_lz(J, b);
  return J.ytiles * ((J.nz + lz - 1) / lz);
}
__device__ __forceinline__ int cocg_parts(const JuncDev& J) {
  return J.ytiles * ((J.nz + kMuPlanes - 1) / kMuPlanes);
}

// alpha = rho / mu of slot s, by a warp, once all its mu partials are written: the
// operator's and the J.n_groups projections' partials added, FP64's in fixed point
// (FP32's, which carry their own rounding errors, in a shuffle tree).
template <bool FP64>
__device__ __forceinline__ void mu_alpha(const BatchDev& b, const JuncDev& J, const int s) {
  const int lane = threadIdx.x & 31, n = cocg_parts(J) + J.n_groups;
  const double2* part = b.mu_part + (size_t)s * b.PA;
  double2 mu;
  if constexpr (FP64) {
    mu = warp_sum_parts(part, n);
  } else {
    double v[2] = {0.0, 0.0};
    for (int t = lane; t < n; t += 32) {
      const double2 w = __ldcg(part + t);
      v[0] += w.x;
      v[1] += w.y;
    }
    const double t = warp_sum_many<2>(v);
    mu = make_double2(__shfl_sync(0xffffffffu, t, 0), __shfl_sync(0xffffffffu, t, 1));
  }
  const double2 a = cdiv_warp(b.rho_cur[s], mu);
  if (lane == 0) {
    b.mu_cnt[s] = 0;
    b.alpha[s] = a;
    b.alpha32[s] = make_float2((float)a.x, (float)a.y);
    if (b.n_shift > 0) b.salpha[(size_t)(b.iters[s] & 1) * b.nslots + s] = a;
  }
}

// One lane, once the CTA's mu partials of slot s are written (and seen by it):
// counts the CTA in; true for the last of the operator and projection CTAs, whose
// warp then forms alpha, once per system instead of in every update CTA.
__device__ __forceinline__ bool mu_arrive(const BatchDev& b, const JuncDev& J, const int s) {
  __threadfence();
  const bool last = atomicAdd(b.mu_cnt + s, 1) == cocg_tiles(J, b) + J.n_groups - 1;
  if (last) __threadfence();
  return last;
}

// sum over w < nw of part[w * ld] (see the callers): FP64, or for FP32 parts an
// error-free FP32 sum (hi + lo) rounded to FP64 at the end, which leaves the FP64
// pipe with three operations
__device__ __forceinline__ double sum_strided(const double* part, int nw, int ld) {
  double o = part[0];
  for (int w = 1; w < nw; ++w) o += part[w * ld];
  return o;
}
__device__ __forceinline__ double sum_strided(const float* part, int nw, int ld) {
  float hi = part[0], lo = 0.f;
  for (int w = 1; w < nw; ++w) {
    const float a = part[w * ld];
    const float s = __fadd_rn(hi, a), bb = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(a, bb)));
    hi = s;
  }
  // (an infinite part makes the error inf - inf; hi is the plain sum)
  return isfinite(lo) ? (double)hi + (double)lo : (double)hi;
}

// A running sum that a thread keeps over kMuPlanes planes: FP64 plain, FP32
// Kahan-compensated (the sum is hi - carry).  In FP64 the sums over a warp and over the
// partials are rounded once each (exact_sum.cuh), which pays for the compensation that
// a thread's sum does without.  Rms error relative to sum |p q| in a model with FP32 in
// place of FP64, 400 vectors: 24x24x120 2.9e-10 (compensated sums of whole chunks and
// plain trees 5.1e-10 at 10 planes, 4.0e-10 at 40, 3.6e-10 at 120; plain trees here
// 4.3e-10), 16x16x64 6.3e-10 (8.1e-10 at 11, 6.7e-10 at 64; 8.3e-10), 8x8x48 1.20e-9
// (1.47e-9 at 24, 1.34e-9 at 48; 1.67e-9).
struct MuSum64 {
  double re = 0.0, im = 0.0;
  __device__ __forceinline__ void reset() { re = im = 0.0; }
};
struct MuSum32 {
  float re = 0.f, im = 0.f, cre = 0.f, cim = 0.f;
  __device__ __forceinline__ void add(float tre, float tim) {
    const float yr = __fsub_rn(tre, cre), yi = __fsub_rn(tim, cim);
    const float sr = __fadd_rn(re, yr), si = __fadd_rn(im, yi);
    cre = __fsub_rn(__fsub_rn(sr, re), yr);
    cim = __fsub_rn(__fsub_rn(si, im), yi);
    re = sr;
    im = si;
  }
  __device__ __forceinline__ void reset() { re = im = cre = cim = 0.f; }
};

// mu partials of an operator CTA: each warp leaves its sum of every kMuPlanes
// planes in s_mu[block][warp][re, im], FP32 ones as hi + lo pairs ([..][re, im][hi,
// lo]: the shuffle tree carries the rounding errors along, so the sums of four
// planes lose nothing against longer compensated ones: 2.5e-10 of sum |p q| rms on
// 24x24x120 vectors, 3.6e-10 with 24-plane sums and plain trees); at the end the
// first warp's lanes (block, component) add the warps' sums and write mu_part, and
// the CTA arrives.
constexpr int kMuSlots32 = 4, kMuSlots64 = 2;  // values per (block, warp)
__device__ __forceinline__ void mu_flush(double* s_mu, int block, MuSum64& m) {
  const double t = warp_sum2_exact(m.re, m.im);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane < 2) s_mu[(block * nw + warp) * kMuSlots64 + lane] = t;
  m.reset();
}
__device__ __forceinline__ void mu_flush(float* s_mu, int block, MuSum32& m) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const bool odd = (lane & 1) != 0;  // odd lanes keep the imaginary part
  float hi = odd ? m.im : m.re, lo = odd ? -m.cim : -m.cre;
  float ohi = __shfl_xor_sync(0xffffffffu, odd ? m.re : m.im, 1);
  float olo = __shfl_xor_sync(0xffffffffu, odd ? -m.cre : -m.cim, 1);
#pragma unroll
  for (int w = 2; w <= 32; w <<= 1) {
    const float s = __fadd_rn(hi, ohi), bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(ohi, bb));
    lo = __fadd_rn(__fadd_rn(lo, olo), e);
    hi = s;
    if (w < 32) {
      ohi = __shfl_xor_sync(0xffffffffu, hi, w);
      olo = __shfl_xor_sync(0xffffffffu, lo, w);
    }
  }
  if (lane < 2) *reinterpret_cast<float2*>(s_mu + (block * nw + warp) * kMuSlots32 + 2 * lane) = make_float2(hi, lo);
  m.reset();
}
__device__ __forceinline__ double mu_warps(const double* s_mu, int block, int c, int nw) {
  return sum_strided(s_mu + block * nw * kMuSlots64 + c, nw, kMuSlots64);
}
__device__ __forceinline__ double mu_warps(const float* s_mu, int block, int c, int nw) {
  // error-free FP32 sum of the hi parts, the lo parts beside it
  const float* p = s_mu + block * nw * kMuSlots32 + 2 * c;
  float hi = p[0], lo = p[1];
  for (int w = 1; w < nw; ++w) {
    const float2 a = *reinterpret_cast<const float2*>(p + w * kMuSlots32);
    const float s = __fadd_rn(hi, a.x), bb = __fsub_rn(s, hi);
    lo = __fadd_rn(__fadd_rn(lo, a.y), __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(a.x, bb)));
    hi = s;
  }
  return (double)hi + (double)lo;
}
template <typename A>
__device__ __forceinline__ void mu_finish(const BatchDev& b, const JuncDev& J, int s, const A* s_mu, int yt, int z0,
                                          int z1) {
  const int nw = blockDim.x >> 5, nb = (z1 - z0 + kMuPlanes - 1) / kMuPlanes;
  __syncthreads();
  if (threadIdx.x >= 32) return;
  double* out = reinterpret_cast<double*>(b.mu_part + (size_t)s * b.PA +
                                          (size_t)yt * ((J.nz + kMuPlanes - 1) / kMuPlanes) + z0 / kMuPlanes);
  for (int e = threadIdx.x; e < 2 * nb; e += 32) out[e] = mu_warps(s_mu, e >> 1, e & 1, nw);
  __threadfence();
  __syncwarp();
  const bool last = threadIdx.x == 0 && mu_arrive(b, J, s);
  if (__any_sync(0xffffffffu, last)) mu_alpha<sizeof(A) == 8>(b, J, s);
}

struct Pair {
  float2 a, b;  // values at x0 and x0 + 1
};

__device__ __forceinline__ Pair zero_pair() { return Pair{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }

__device__ __forceinline__ Pair lds_pair(const float2* s) {
  const float4 v = *reinterpret_cast<const float4*>(s);
  return Pair{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ void sts_pair(float2* s, const Pair& v) {
  *reinterpret_cast<float4*>(s) = make_float4(v.a.x, v.a.y, v.b.x, v.b.y);
}


template <int R, int MODE, int PITCH>
__global__ void __maxnreg__(96)
op_pair_kernel(const JuncDev* __restrict__ jt, const BatchDev* __restrict__ bp, const void* __restrict__ x_in,
               void* __restrict__ y_out) {
  constexpr int Q = 2 * R + 1;
  constexpr int MD = R < 2 ? R : 2;  // distances summed in difference form
  constexpr int KX = (R + 1) / 2;    // neighbour pairs left / right in x
  constexpr int NIN = (MODE == OP_COCG) ? 2 : 1;
  const BatchDev& b = *bp;
  const int s = blockIdx.x;
  if constexpr (MODE == OP_COCG) {
    if (b.state[s] != SL_ACTIVE) return;
  }
  const JuncDev& J = jt[b.junc[s]];
  const int tile = launch_tile();
  if (tile >= J.nA || J.kind != kOpPair) return;

  const int nx = J.nx, ny = J.ny, nz = J.nz, plane = J.plane;
  const int hx = nx >> 1;  // pairs per row
  const int Lz = MODE == OP_COCG ? cocg_lz(J, b) : J.Lz;
  const int z0 = tile * Lz, z1 = min(z0 + Lz, nz);
  if (z0 >= nz) return;
  const int pitch = PITCH > 0 ? PITCH : nx + 2 * kPairXO;
  const int rows = ny + 2 * R;
  const int tid = threadIdx.x, nt = blockDim.x;
  const long long vo = b.voff[s];

  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* stage = reinterpret_cast<float2*>(smem_raw);  // [kPairStages][NIN][plane]
  float2* exch = stage + kPairStages * NIN * plane;    // [2][rows][pitch]
  uint64_t* bars = reinterpret_cast<uint64_t*>(
      (reinterpret_cast<uintptr_t>(exch + 2 * rows * pitch) + 15) & ~static_cast<uintptr_t>(15));
  // mu partials (COCG): [block of planes][warp][re, im][hi, lo]
  __shared__ __align__(8) float s_mu[MODE == OP_COCG ? kMaxLz / kMuPlanes * (kPairThreadsBig / 32) * kMuSlots32 : 1];
  __shared__ int s_bad;

  for (int i = tid; i < 2 * rows * pitch; i += nt) exch[i] = make_float2(0.f, 0.f);
  if (tid == 0) {
    for (int k = 0; k < kPairStages; ++k) mbar_init(bars + k, 1);
    s_bad = 0;
  }

  // ---- per-system scalars and vectors --------------------------------------
  const int k = (MODE == OP_COCG) ? b.iters[s] : 0;
  const bool first = (MODE == OP_COCG) && (k == 0);
  float2 beta = make_float2(0.f, 0.f);
  if (MODE == OP_COCG && !first) beta = make_float2((float)b.beta_cur[s].x, (float)b.beta_cur[s].y);
  const float2* src0;
  const float2* src1 = nullptr;
  float2* pnew = nullptr;
  float2* yv;
  if constexpr (MODE == OP_COCG) {
    src0 = reinterpret_cast<const float2*>(b.r) + vo;
    if (!first) src1 = reinterpret_cast<const float2*>((k & 1) ? b.p1 : b.p0) + vo;
    pnew = reinterpret_cast<float2*>((k & 1) ? b.p0 : b.p1) + vo;
    yv = reinterpret_cast<float2*>(b.q) + vo;
  } else {
    src0 = reinterpret_cast<const float2*>(x_in) + vo;
    yv = reinterpret_cast<float2*>(y_out) + vo;
  }
  __syncthreads();

  // planes [zb, ze) stream through the ring; plane zl uses stage (zl - zb) % kPairStages
  const int zb = z0 - R, ze = z1 + R;
  const uint32_t pbytes = (uint32_t)(plane * sizeof(float2));
  auto issue = [&](int zl) {
    const int st = (zl - zb) % kPairStages;
    uint64_t* bar = bars + st;
    if (zl >= 0 && zl < nz) {
      mbar_arrive_expect_tx(bar, src1 ? 2 * pbytes : pbytes);
      bulk_g2s(stage + (st * NIN) * plane, src0 + (size_t)zl * plane, pbytes, bar);
      if (src1) bulk_g2s(stage + (st * NIN + 1) * plane, src1 + (size_t)zl * plane, pbytes, bar);
    } else {
      mbar_arrive(bar);  // nothing to copy outside the box: complete the phase
    }
  };
  if (tid == 0) {
    fence_proxy_async();
    for (int f = 0; f < kPairStages && zb + f < ze; ++f) issue(zb + f);
  }

  // ---- owned pair ------------------------------------------------------------
  const bool own = tid < ny * hx;
  const int yl = own ? tid / hx : 0;
  const int x0 = own ? 2 * (tid - yl * hx) : 0;
  const int po = x0 + yl * nx;                     // offset within a plane (even)
  const int so = (yl + R) * pitch + x0 + kPairXO;  // exchange-tile index of the pair (even)

  // FD weights and E - 6 sum_{m > MD} w_m (the direct terms' share of the
  // diagonal) in shared memory: broadcast reads instead of live registers
  __shared__ float s_w[R + 2];
  if (tid == 0) {
    float dshift = 0.f;
    for (int m = 1; m <= R; ++m) {
      s_w[m] = J.w32[m];
      if (m > MD) dshift -= 6.f * J.w32[m];
    }
    s_w[0] = (float)b.E[s] + dshift;
  }
  __syncthreads();
  const float4* dg4 = reinterpret_cast<const float4*>(J.dg32);

  Pair zq[Q];
#pragma unroll
  for (int m = 0; m < Q; ++m) zq[m] = zero_pair();
  MuSum32 mu;                                        // mu = v^T A_loc v over kMuPlanes planes
  int sidx = 0;                                      // stage of the plane entering the ring
  uint32_t sph = 0;                                  // its mbarrier phase parity

  for (int zr = z0 - 2 * R; zr < z1; zr += Q) {
#pragma unroll
    for (int u = 0; u < Q; ++u) {
      const int zc = zr + u;
      if (zc < z1) {
        // plane zl = zc + R arrives in stage sidx and enters ring slot u
        const int zl = zc + R;
        float4 dgc = make_float4(0.f, 0.f, 0.f, 0.f);  // (-V_loc, Gamma) of both points of plane zc
        if (own && zc >= z0) dgc = __ldg(dg4 + ((zc * plane + po) >> 1));
        Pair v = zero_pair();
        if (!mbar_wait(bars + sidx, sph)) {
          s_bad = 1;
        } else if (own && zl >= 0 && zl < nz) {
          v = lds_pair(stage + (sidx * NIN) * plane + po);
          if constexpr (MODE == OP_COCG) {
            if (src1) {
              const Pair pp = lds_pair(stage + (sidx * NIN + 1) * plane + po);
              v.a = cfma2(beta, pp.a, v.a);
              v.b = cfma2(beta, pp.b, v.b);
            }
          }
        }
        zq[u] = v;
        const int C = (u + R + 1) % Q;  // ring slot of plane zc (a constant once unrolled)
        float2* smb = exch + (((zc - z0) & 1) ? rows * pitch : 0);
        if (zc >= z0 && own) sts_pair(smb + so, zq[C]);
        __syncthreads();
        if (s_bad) {
          // a copy never arrived: report, let in-flight copies land (bounded), leave
          if (tid == 0) {
            if (b.sched) atomicExch(b.sched + 2, 1);
            for (int f = 0; f < kPairStages; ++f) {
              const int zq2 = zl + f;
              if (zq2 < ze) mbar_wait(bars + (zq2 - zb) % kPairStages, (uint32_t)(((zq2 - zb) / kPairStages) & 1));
            }
          }
          return;
        }
        // every thread has read stage sidx: refill it with plane zl + kPairStages
        if (tid == 0 && zl + kPairStages < ze) {
          fence_proxy_async();
          issue(zl + kPairStages);
        }
        if (++sidx == kPairStages) {
          sidx = 0;
          sph ^= 1u;
        }
        if (zc >= z0 && own) {
          // x neighbours at offsets -2KX .. 2KX+1 from x0
          float2 X[4 * KX + 2];
#pragma unroll
          for (int kk = 0; kk < 2 * KX + 1; ++kk) {
            const Pair pr = (kk == KX) ? zq[C] : lds_pair(smb + so + 2 * (kk - KX));
            X[2 * kk] = pr.a;
            X[2 * kk + 1] = pr.b;
          }
          float2 lap0 = make_float2(0.f, 0.f), lap1 = lap0;
          const float2 c0 = zq[C].a, c1 = zq[C].b;
#pragma unroll
          for (int m = 1; m <= R; ++m) {
            const Pair zm = zq[(C + Q - m) % Q], zp = zq[(C + m) % Q];
            const Pair ym = lds_pair(smb + so - m * pitch), yp = lds_pair(smb + so + m * pitch);
            const float2 xm0 = X[2 * KX - m], xp0 = X[2 * KX + m];
            const float2 xm1 = X[2 * KX + 1 - m], xp1 = X[2 * KX + 1 + m];
            const float2 w = make_float2(s_w[m], s_w[m]);
            float2 s0, s1;
            if (m <= MD) {
              s0 = add2(add2(add2(sub2(zm.a, c0), sub2(zp.a, c0)), add2(sub2(ym.a, c0), sub2(yp.a, c0))),
                        add2(sub2(xm0, c0), sub2(xp0, c0)));
              s1 = add2(add2(add2(sub2(zm.b, c1), sub2(zp.b, c1)), add2(sub2(ym.b, c1), sub2(yp.b, c1))),
                        add2(sub2(xm1, c1), sub2(xp1, c1)));
            } else {
              s0 = add2(add2(add2(zm.a, zp.a), add2(ym.a, yp.a)), add2(xm0, xp0));
              s1 = add2(add2(add2(zm.b, zp.b), add2(ym.b, yp.b)), add2(xm1, xp1));
            }
            lap0 = fma2(w, s0, lap0);
            lap1 = fma2(w, s1, lap1);
          }
          // + (E - V_loc + dshift + i Gamma) v
          const float Ef = s_w[0];
          float2 y0v = cfma2(make_float2(Ef + dgc.x, dgc.y), c0, lap0);
          float2 y1v = cfma2(make_float2(Ef + dgc.z, dgc.w), c1, lap1);
          const int gi = zc * plane + po;
          if constexpr (MODE == OP_COCG) {
            *reinterpret_cast<float4*>(pnew + gi) = make_float4(c0.x, c0.y, c1.x, c1.y);
            // mu partial v^T y (unconjugated) of both points
            const float2 t = cfma2(c1, y1v, cfma2(c0, y0v, make_float2(0.f, 0.f)));
            mu.add(t.x, t.y);
          }
          *reinterpret_cast<float4*>(yv + gi) = make_float4(y0v.x, y0v.y, y1v.x, y1v.y);
        }
        if constexpr (MODE == OP_COCG) {
          // every kMuPlanes planes and at the chunk's end: the warp's sum so far
          if (zc >= z0 && ((zc - z0) % kMuPlanes == kMuPlanes - 1 || zc == z1 - 1)) {
            mu_flush(s_mu, (zc - z0) / kMuPlanes, mu);
          }
        }
      }
    }
  }
  if constexpr (MODE == OP_COCG) mu_finish(b, J, s, s_mu, 0, z0, z1);
}

// ---------------------------------------------------------------------------
// One point per thread, whole planes streamed by bulk copies: the same march
// as op_pair_kernel (bulk-copied input planes, register ring of 2R+1 produced
// planes unrolled by 2R+1, double-buffered exchange tile, hybrid difference
// form) with one grid point per thread, so that the z ring takes 2R+1 complex
// values and two CTAs of up to kPlaneThreads threads fit one SM.  Any nx; the
// plane size must be even (16-byte bulk copies).
// ---------------------------------------------------------------------------
template <int R, int MODE>
__global__ void __launch_bounds__(kPlaneThreads, 2)
op_plane_kernel(const JuncDev* __restrict__ jt, const BatchDev* __restrict__ bp, const void* __restrict__ x_in,
                void* __restrict__ y_out) {
  constexpr int Q = 2 * R + 1;
  constexpr int MD = R < 2 ? R : 2;  // distances summed in difference form
  constexpr int NIN = (MODE == OP_COCG) ? 2 : 1;
  const BatchDev& b = *bp;
  const int s = blockIdx.x;
  if constexpr (MODE == OP_COCG) {
    if (b.state[s] != SL_ACTIVE) return;
  }
  const JuncDev& J = jt[b.junc[s]];
  const int tile = launch_tile();
  if (tile >= J.nA || J.kind != kOpPlane) return;

  const int nx = J.nx, ny = J.ny, nz = J.nz, plane = J.plane;
  const int Lz = MODE == OP_COCG ? cocg_lz(J, b) : J.Lz;
  const int z0 = tile * Lz, z1 = min(z0 + Lz, nz);
  if (z0 >= nz) return;
  const int pitch = nx + 2 * kPairXO;
  const int rows = ny + 2 * R;
  const int tid = threadIdx.x, nt = blockDim.x;
  const long long vo = b.voff[s];

  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* stage = reinterpret_cast<float2*>(smem_raw);  // [kPairStages][NIN][plane]
  float2* exch = stage + kPairStages * NIN * plane;    // [2][rows][pitch]
  uint64_t* bars = reinterpret_cast<uint64_t*>(
      (reinterpret_cast<uintptr_t>(exch + 2 * rows * pitch) + 15) & ~static_cast<uintptr_t>(15));
  __shared__ __align__(8) float s_mu[MODE == OP_COCG ? kMaxLz / kMuPlanes * (kPlaneThreads / 32) * kMuSlots32 : 1];
  __shared__ int s_bad;
  __shared__ float s_w[R + 2];

  for (int i = tid; i < 2 * rows * pitch; i += nt) exch[i] = make_float2(0.f, 0.f);
  if (tid == 0) {
    for (int k = 0; k < kPairStages; ++k) mbar_init(bars + k, 1);
    s_bad = 0;
    // FD weights and E - 6 sum_{m > MD} w_m (the direct terms' share of the diagonal)
    float dshift = 0.f;
    for (int m = 1; m <= R; ++m) {
      s_w[m] = J.w32[m];
      if (m > MD) dshift -= 6.f * J.w32[m];
    }
    s_w[0] = (float)b.E[s] + dshift;
  }

  const int k = (MODE == OP_COCG) ? b.iters[s] : 0;
  const bool first = (MODE == OP_COCG) && (k == 0);
  float2 beta = make_float2(0.f, 0.f);
  if (MODE == OP_COCG && !first) beta = make_float2((float)b.beta_cur[s].x, (float)b.beta_cur[s].y);
  const float2* src0;
  const float2* src1 = nullptr;
  float2* pnew = nullptr;
  float2* yv;
  if constexpr (MODE == OP_COCG) {
    src0 = reinterpret_cast<const float2*>(b.r) + vo;
    if (!first) src1 = reinterpret_cast<const float2*>((k & 1) ? b.p1 : b.p0) + vo;
    pnew = reinterpret_cast<float2*>((k & 1) ? b.p0 : b.p1) + vo;
    yv = reinterpret_cast<float2*>(b.q) + vo;
  } else {
    src0 = reinterpret_cast<const float2*>(x_in) + vo;
    yv = reinterpret_cast<float2*>(y_out) + vo;
  }
  __syncthreads();

  const int zb = z0 - R, ze = z1 + R;
  const uint32_t pbytes = (uint32_t)(plane * sizeof(float2));
  auto issue = [&](int zl) {
    const int st = (zl - zb) % kPairStages;
    uint64_t* bar = bars + st;
    if (zl >= 0 && zl < nz) {
      mbar_arrive_expect_tx(bar, src1 ? 2 * pbytes : pbytes);
      bulk_g2s(stage + (st * NIN) * plane, src0 + (size_t)zl * plane, pbytes, bar);
      if (src1) bulk_g2s(stage + (st * NIN + 1) * plane, src1 + (size_t)zl * plane, pbytes, bar);
    } else {
      mbar_arrive(bar);
    }
  };
  if (tid == 0) {
    fence_proxy_async();
    for (int f = 0; f < kPairStages && zb + f < ze; ++f) issue(zb + f);
  }

  const bool own = tid < plane;
  const int yl = own ? tid / nx : 0;
  const int xl = own ? tid - yl * nx : 0;
  const int so = (yl + R) * pitch + xl + kPairXO;  // exchange-tile index of the point

  float2 dgn = make_float2(0.f, 0.f);  // (-V_loc, Gamma) of the next plane to compute
  if (own && z0 < z1) dgn = __ldg(J.dg32 + (z0 * plane + tid));

  float2 zq[Q];
#pragma unroll
  for (int m = 0; m < Q; ++m) zq[m] = make_float2(0.f, 0.f);
  MuSum32 mu;  // mu = v^T A_loc v over kMuPlanes planes
  int sidx = 0;
  uint32_t sph = 0;

  for (int zr = z0 - 2 * R; zr < z1; zr += Q) {
#pragma unroll
    for (int u = 0; u < Q; ++u) {
      const int zc = zr + u;
      if (zc < z1) {
        const int zl = zc + R;
        float2 v = make_float2(0.f, 0.f);
        if (!mbar_wait(bars + sidx, sph)) {
          s_bad = 1;
        } else if (own && zl >= 0 && zl < nz) {
          v = stage[(sidx * NIN) * plane + tid];
          if constexpr (MODE == OP_COCG) {
            if (src1) {
              const float2 pp = stage[(sidx * NIN + 1) * plane + tid];
              v.x = fmaf(beta.x, pp.x, fmaf(-beta.y, pp.y, v.x));
              v.y = fmaf(beta.x, pp.y, fmaf(beta.y, pp.x, v.y));
            }
          }
        }
        zq[u] = v;
        const int C = (u + R + 1) % Q;  // ring slot of plane zc (a constant once unrolled)
        float2* smb = exch + (((zc - z0) & 1) ? rows * pitch : 0);
        if (zc >= z0 && own) smb[so] = zq[C];
        __syncthreads();
        if (s_bad) {
          if (tid == 0) {
            if (b.sched) atomicExch(b.sched + 2, 1);
            for (int f = 0; f < kPairStages; ++f) {
              const int zq2 = zl + f;
              if (zq2 < ze) mbar_wait(bars + (zq2 - zb) % kPairStages, (uint32_t)(((zq2 - zb) / kPairStages) & 1));
            }
          }
          return;
        }
        if (tid == 0 && zl + kPairStages < ze) {
          fence_proxy_async();
          issue(zl + kPairStages);
        }
        if (++sidx == kPairStages) {
          sidx = 0;
          sph ^= 1u;
        }
        if (zc >= z0 && own) {
          const float2 dgc = dgn;
          if (zc + 1 < z1) dgn = __ldg(J.dg32 + ((zc + 1) * plane + tid));
          const float2 c = zq[C];
          float lx = 0.f, ly = 0.f;
#pragma unroll
          for (int m = 1; m <= R; ++m) {
            const float2 zm = zq[(C + Q - m) % Q], zp = zq[(C + m) % Q];
            const float2 ym = smb[so - m * pitch], yp = smb[so + m * pitch];
            const float2 xm = smb[so - m], xp = smb[so + m];
            const float w = s_w[m];
            float sx, sy;
            if (m <= MD) {
              sx = ((zm.x - c.x) + (zp.x - c.x)) + ((ym.x - c.x) + (yp.x - c.x)) + ((xm.x - c.x) + (xp.x - c.x));
              sy = ((zm.y - c.y) + (zp.y - c.y)) + ((ym.y - c.y) + (yp.y - c.y)) + ((xm.y - c.y) + (xp.y - c.y));
            } else {
              sx = ((zm.x + zp.x) + (ym.x + yp.x)) + (xm.x + xp.x);
              sy = ((zm.y + zp.y) + (ym.y + yp.y)) + (xm.y + xp.y);
            }
            lx = fmaf(w, sx, lx);
            ly = fmaf(w, sy, ly);
          }
          // + (E - V_loc + dshift + i Gamma) v
          const float dr = s_w[0] + dgc.x, di = dgc.y;
          float2 y = make_float2(fmaf(dr, c.x, fmaf(-di, c.y, lx)), fmaf(dr, c.y, fmaf(di, c.x, ly)));
          const int gi = zc * plane + tid;
          if constexpr (MODE == OP_COCG) {
            pnew[gi] = c;
            // mu partial v^T y (unconjugated)
            mu.add(fmaf(c.x, y.x, -c.y * y.y), fmaf(c.x, y.y, c.y * y.x));
          }
          yv[gi] = y;
        }
        if constexpr (MODE == OP_COCG) {
          if (zc >= z0 && ((zc - z0) % kMuPlanes == kMuPlanes - 1 || zc == z1 - 1)) {
            mu_flush(s_mu, (zc - z0) / kMuPlanes, mu);
          }
        }
      }
    }
  }
  if constexpr (MODE == OP_COCG) mu_finish(b, J, s, s_mu, 0, z0, z1);
}

template <int R>
cudaError_t launch_op_plane_r(int mode, dim3 grid, int threads, size_t smem, cudaStream_t st, const JuncDev* jt,
                              const BatchDev* b, const void* x_in, void* y_out) {
  void (*kern)(const JuncDev*, const BatchDev*, const void*, void*) = nullptr;
  if (mode == OP_COCG) kern = op_plane_kernel<R, OP_COCG>;
  else if (mode == OP_APPLY) kern = op_plane_kernel<R, OP_APPLY>;
  else return cudaErrorInvalidValue;
  if (threads > kPlaneThreads) return cudaErrorInvalidValue;
  if (smem > 16 * 1024) {  // beside the static arrays
    cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
  }
  cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  kern<<<grid, threads, smem, st>>>(jt, b, x_in, y_out);
  return cudaGetLastError();
}

template <int R>
cudaError_t launch_op_pair_r(int mode, bool big, int pitch, dim3 grid, int threads, size_t smem, cudaStream_t st,
                             const JuncDev* jt, const BatchDev* b, const void* x_in, void* y_out) {
  void (*kern)(const JuncDev*, const BatchDev*, const void*, void*) = nullptr;
#define RSN_PAIR(M) \
  kern = pitch == 40 ? op_pair_kernel<R, M, 40> : pitch == 56 ? op_pair_kernel<R, M, 56> : op_pair_kernel<R, M, 0>;
  if (mode == OP_COCG) {
    RSN_PAIR(OP_COCG)
  } else if (mode == OP_APPLY) {
    RSN_PAIR(OP_APPLY)
  } else {
    return cudaErrorInvalidValue;
  }
#undef RSN_PAIR
  if (threads > (big ? kPairThreadsBig : kPairThreads)) return cudaErrorInvalidValue;
  if (smem > 16 * 1024) {  // beside the static arrays
    cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
  }
  cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  kern<<<grid, threads, smem, st>>>(jt, b, x_in, y_out);
  return cudaGetLastError();
}

}  // namespace rsn
