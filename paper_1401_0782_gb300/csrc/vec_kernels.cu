// Streaming, reduction and scheduling kernels of the batched COCG solver,
// the T(E) reduction (Eq. T-realspace) and the adjoint gradient.
//
// Per iteration of the streaming solver (all kernels skip slots in other states):
//   zero      (NEW)            x = 0, d = 0
//   project   (NEW|CHECK)      c_x = v_p . (x + d)                       [projectors]
//   op RESID  (NEW|CHECK)      r = b - A (x + d) in FP64, ||r||^2, r^T r
//   x_update  (NEW|CHECK)      x += d, d = 0
//   emit      (DRAIN)          T partial of the finished system
//   project   (ACTIVE)         c_r = v_p . r                             [projectors]
//   op COCG   (ACTIVE)         p = r + beta p, q = A p, p^T q; alpha = rho/mu
//   update    (ACTIVE)         r -= alpha q, d += alpha p, r^T r, ||r||^2, then the slot's
//                              iteration counts; recurrence target reached -> CHECK
//   sched     (all, 1 CTA)     converged? -> DRAIN; else reliable update -> ACTIVE;
//                              DRAIN -> FREE; FREE slots take queued systems; list
#include <algorithm>
#include <type_traits>

#include "cplx.cuh"
#include "ops_kernel.cuh"
#include "rsn_internal.h"

namespace rsn {

// ---------------------------------------------------------------------------
// List of the slots that need a true residual in the next iteration (NEW and
// CHECK), in slot order: one CTA, ballot + warp-count prefix per 1024 slots.
// Built at the end of the scheduler (a kernel of its own for the micro-benchmark).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void build_list(const BatchDev& b, int* warp_cnt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int total = 0;
  for (int base = 0; base < b.nslots; base += blockDim.x) {
    const int s = base + threadIdx.x;
    int st = SL_FREE;
    if (s < b.nslots) st = b.state[s];
    const bool in = st == SL_NEW || st == SL_CHECK || st == SL_CHECKT;
    if (s < b.nslots) b.inlist[s] = in ? 1 : 0;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (lane == 0) warp_cnt[warp] = __popc(m);
    __syncthreads();
    int before = 0, sum = 0;
    for (int w = 0; w < nw; ++w) {
      if (w < warp) before += warp_cnt[w];
      sum += warp_cnt[w];
    }
    if (in) b.lst[total + before + __popc(m & ((1u << lane) - 1u))] = s;
    total += sum;
    __syncthreads();
  }
  if (threadIdx.x == 0) *b.lst_n = total;
}

__global__ void __launch_bounds__(kSchedThreads) list_kernel(const BatchDev* __restrict__ bp) {
  __shared__ int warp_cnt[kSchedThreads / 32];
  build_list(*bp, warp_cnt);
}

// ---------------------------------------------------------------------------
// zero x and d of newly assigned systems (CTA rows over the NEW / CHECK list)
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kVecThreads) zero_kernel(const JuncDev* __restrict__ jt,
                                                           const BatchDev* __restrict__ bp) {
  using C = typename cx<T>::t;
  const BatchDev& b = *bp;
  const int n = *b.lst_n;
  for (int li = blockIdx.y; li < n; li += gridDim.y) {
    const int s = b.lst[li];
    if (b.state[s] != SL_NEW) continue;
    const JuncDev& J = jt[b.junc[s]];
    if ((int)blockIdx.x >= J.nB) continue;
    const long long vo = b.voff[s], xo = b.xo[s];
    const long long i0 = (long long)blockIdx.x * kVecPts, i1 = min(i0 + (long long)kVecPts, J.N);
    C* dv = reinterpret_cast<C*>(b.d);
    const bool keep_x = b.warm[s] != 0;
    for (long long i = i0 + threadIdx.x; i < i1; i += kVecThreads) {
      if (!keep_x) b.x64[xo + i] = make_double2(0.0, 0.0);
      dv[vo + i] = czero<C>();
    }
  }
}

// ---------------------------------------------------------------------------
// COCG update (after the operator and projection kernels of the same iteration):
//   r -= alpha q,  d += alpha p_new,
//   partial sums of rho_{k+1} = r^T r and ||r||^2,
// then, in the CTA that finishes its slot's last chunk, the bookkeeping of the
// iteration (book_slot).  alpha = rho_k / mu_k was formed by whichever operator
// or projection CTA of the slot finished last (mu_arrive).
// q arrives without the projector term (the operator kernel leaves it out); it
// is formed here, from e_kb c_p of the new direction (projection kernel), for
// the blocks of points that hold support points, so q is never written back.
// Each warp covers one block of one system.  A non-finite alpha leaves r and d
// untouched and flags the slot through a NaN norm.
// FP32 is bound by HBM (48 B a point), FP64 by the FP64 pipe (2 operations a
// cycle and SM; 12 a point and 8 a projector value quad).  24x24x120 with 20 atoms:
// 144 FP32 systems 117 us (4.1 TB/s; 165 with per-point lookups and 4,096-point
// CTAs, 101 without projectors), 512 systems 4.5 TB/s; 1 system 16 us (37); FP64,
// 16 systems 70 us (132), 144 systems 433.
// ---------------------------------------------------------------------------
// Bookkeeping after a COCG iteration, by the first warp of the slot's last
// update CTA: rho_{k+1} and ||r||^2 from the partials (fixed-order warp tree),
// beta_{k+1} = rho_{k+1} / rho_k, iteration counts, the recurrence target of
// the current cycle, breakdown detection (NaN partial).
__device__ __forceinline__ void book_slot(const BatchDev& b, const int s, const int nU, const int slot_it) {
  const int lane = threadIdx.x & 31;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (int t = lane; t < nU; t += 32) {
    v[0] += __ldcg(b.nrm_part + (size_t)s * b.PB + t);
    const double2 w = __ldcg(b.rho_part + (size_t)s * b.PB + t);
    v[1] += w.x;
    v[2] += w.y;
  }
  const double sum = warp_sum_many<4>(v);
  const double nrm = __shfl_sync(0xffffffffu, sum, 0);
  const double2 rho = make_double2(__shfl_sync(0xffffffffu, sum, 1), __shfl_sync(0xffffffffu, sum, 2));
  const double2 beta = cdiv_warp(rho, b.rho_cur[s]);
  if (lane != 0) return;
  const int k = b.iters[s] + 1;
  b.iters[s] = k;
  const int tot = b.total_iters[s] + 1;
  b.total_iters[s] = tot;
  const int cyc = b.cyc_iters[s] + 1;
  b.cyc_iters[s] = cyc;
  atomicAdd(b.counters, 1ull);
  atomicAdd(b.sched + 3 + kMaxGraphIters + slot_it, 1);
  if (b.n_shift > 0) {
    b.rn2[s] = nrm;
    b.stamp[s] = *b.iter_no;  // the shifted update of this iteration takes the slot
  }
  b.beta_cur[s] = beta;
  b.rho_cur[s] = rho;
  // (the mixed mode has its cycle cap; shifted systems must keep their one Krylov space)
  const bool thrown = watch_step(b.rmin2[s], b.rmin_it[s], nrm, tot) && !b.handback && b.n_shift == 0;
  if (!isfinite(nrm) || thrown) {
    b.restart[s] = 1;
    b.rrec2[s] = thrown ? nrm : 0.0;
    b.state[s] = SL_CHECK;
  } else if (nrm <= b.tol2[s] || tot >= b.max_iter || cyc >= b.cycle_cap) {
    b.rrec2[s] = nrm;
    b.state[s] = b.gphase[s] ? SL_CHECKT : SL_CHECK;
  }
}

// The projector term of one block of kBlkPts points, by one warp:
// acc[l] = -sum over the block's projector rows of value * ce, acc and ce in
// shared memory.  A row holds up to 32 entries (support point, atom) of different
// points, so its lanes never meet: the rows of layer k hold the k-th atom of every
// point that has one, which fixes the order of a point's sum and fills the lanes
// (rows of one atom each left a third of them empty).  The loads of up to four
// rows are in flight together (NQ: value quads per entry).  SPV vectors at once:
// vector v has its coefficients at ce + v * ces, its sums at acc + v * kBlkPts.
template <typename T, int NQ, int SPV>
__device__ __forceinline__ void block_nonlocal_nq(const JuncDev& J, const typename cx<T>::t* ce, const int ces,
                                                  const int row0, const int row1, typename cx<T>::t* acc) {
  using C = typename cx<T>::t;
  constexpr int D = NQ == 1 ? 4 : NQ == 2 ? 2 : 1;
  const int lane = threadIdx.x & 31;
  for (int row = row0; row < row1; row += D) {
    int m[D];  // first projector * kBlkPts + point, -1: no entry
    T a[D][4 * NQ];
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const int rr = min(row + j, row1 - 1);
      m[j] = __ldg(J.row_ent + (size_t)rr * 32 + lane);
      if (row + j >= row1) m[j] = -1;
#pragma unroll
      for (int qd = 0; qd < NQ; ++qd) {
        const size_t at = ((size_t)rr * NQ + qd) * 32 + lane;
        if constexpr (sizeof(T) == 8) {
          const double2 a01 = __ldg(J.row_q64 + 2 * at), a23 = __ldg(J.row_q64 + 2 * at + 1);
          a[j][4 * qd] = a01.x, a[j][4 * qd + 1] = a01.y, a[j][4 * qd + 2] = a23.x, a[j][4 * qd + 3] = a23.y;
        } else {
          const float4 v = __ldg(J.row_q32 + at);
          a[j][4 * qd] = v.x, a[j][4 * qd + 1] = v.y, a[j][4 * qd + 2] = v.z, a[j][4 * qd + 3] = v.w;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < D; ++j) {
      if (m[j] >= 0) {
        const int l = m[j] % kBlkPts;
        const C* cp = ce + m[j] / kBlkPts;
#pragma unroll
        for (int v = 0; v < SPV; ++v) {
          C y = acc[v * kBlkPts + l];
#pragma unroll
          for (int i = 0; i < 4 * NQ; ++i) y = rfma(-a[j][i], cp[v * ces + i], y);
          acc[v * kBlkPts + l] = y;
        }
      }
      __syncwarp();
    }
  }
}

template <typename T, int SPV>
__device__ __forceinline__ void block_nonlocal(const JuncDev& J, const typename cx<T>::t* ce, const int ces,
                                               const int row0, const int row1, typename cx<T>::t* acc) {
  for (int l = threadIdx.x & 31; l < SPV * kBlkPts; l += 32) acc[l] = czero<typename cx<T>::t>();
  __syncwarp();
  switch (J.inv_nq) {
    case 1: block_nonlocal_nq<T, 1, SPV>(J, ce, ces, row0, row1, acc); break;
    case 2: block_nonlocal_nq<T, 2, SPV>(J, ce, ces, row0, row1, acc); break;
    case 3: block_nonlocal_nq<T, 3, SPV>(J, ce, ces, row0, row1, acc); break;
    default: block_nonlocal_nq<T, 4, SPV>(J, ce, ces, row0, row1, acc); break;
  }
}

// vectors of a thread's U points, in 16-byte pairs where `pairs` (at[u], at[u + 1]
// neighbours, U even), else one at a time; points at or past `end` read as zero
// and are not stored
template <typename C, int U>
__device__ __forceinline__ void load_pts(const C* src, const int (&at)[U], int end, bool pairs, C (&v)[U]) {
  if constexpr (sizeof(C) == 8) {
    if (pairs) {
#pragma unroll
      for (int u = 0; u < U; u += 2) {
        float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
        if (at[u] < end) w = *reinterpret_cast<const float4*>(src + at[u]);
        v[u] = mk2(w.x, w.y);
        v[u + 1] = mk2(w.z, w.w);
      }
      return;
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) v[u] = at[u] < end ? src[at[u]] : czero<C>();
}
template <typename C, int U>
__device__ __forceinline__ void store_pts(C* dst, const int (&at)[U], int end, bool pairs, const C (&v)[U]) {
  if constexpr (sizeof(C) == 8) {
    if (pairs) {
#pragma unroll
      for (int u = 0; u < U; u += 2)
        if (at[u] < end) *reinterpret_cast<float4*>(dst + at[u]) = make_float4(v[u].x, v[u].y, v[u + 1].x, v[u + 1].y);
      return;
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (at[u] < end) dst[at[u]] = v[u];
}

// EARLY: the vectors are requested before the projector term is formed, which
// takes 90 registers; for launches whose latency counts (upd_early).  STAGED: the
// coefficients are copied to shared memory, as long as they fit (more than about
// 13,900 projectors in FP64 do not; they are read where they lie).
template <typename T, bool EARLY, bool STAGED = true>
__global__ void __launch_bounds__(kUpdThreads, EARLY ? 4 : sizeof(T) == 4 ? 8 : 6)
cocg_update_kernel(const JuncDev* __restrict__ jt, const BatchDev* __restrict__ bp, int slot_it) {
  using C = typename cx<T>::t;
  constexpr int U = sizeof(T) == 4 ? 4 : 2;  // points in flight per thread
  constexpr int NL = kBlkPts / (32 * U);
  const BatchDev& b = *bp;
  const int s = blockIdx.y;
  if (b.state[s] != SL_ACTIVE) return;
  const JuncDev& J = jt[b.junc[s]];
  const int N = (int)J.N;  // < 2^31
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int nU = upd_ctas(N);
  if ((int)blockIdx.x >= nU) return;
  const int blk = blockIdx.x * nw + warp;
  const int n = blk_len(blk, N);  // points of the warp's block
  const long long vo = b.voff[s], bo = vo + blk_first(blk, N);
  const int k = b.iters[s];
  C al;  // (FP32: rounded once by mu_alpha, which keeps conversions off the FP64 pipe here)
  if constexpr (sizeof(T) == 4) al = b.alpha32[s];
  else al = b.alpha[s];
  const bool fin = isfinite(al.x) && isfinite(al.y);
  extern __shared__ __align__(16) unsigned char upd_smem[];
  C* s_ce = reinterpret_cast<C*>(upd_smem);         // e_kb c_p of the new direction, ce_stride entries
  C* s_nl = s_ce + (STAGED ? b.ce_stride : 0) + warp * kBlkPts;  // projector term of the warp's block
  __shared__ double red[4 * (kUpdThreads / 32)];
  __shared__ int s_last;
  T re = 0, sy = 0, sxy = 0;  // sums of r.x^2 - r.y^2 (cancelling inside the sum), r.y^2, r.x r.y
  if (fin) {  // uniform across the CTA
    const C* pn = reinterpret_cast<const C*>((k & 1) ? b.p0 : b.p1) + bo;
    const C* qv = reinterpret_cast<const C*>(b.q) + bo;
    C* rv = reinterpret_cast<C*>(b.r) + bo;
    C* dv = reinterpret_cast<C*>(b.d) + bo;
    const T ax = al.x, ay = al.y;
    // FP32: 16-byte pairs where the slot starts on a pair and holds whole
    // pairs; else (and in FP64, 16 bytes a point) one point at a time
    const bool pairs = sizeof(T) == 4 && ((vo | N) & 1) == 0;
    C q[U], r[U], p[U], d[U];
    int at[U];
    auto fetch = [&](int l) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        at[u] = l * 32 * U + (pairs ? 2 * lane + (u >> 1) * 64 + (u & 1) : u * 32 + lane);
      load_pts(qv, at, n, pairs, q);
      load_pts(rv, at, n, pairs, r);
      load_pts(pn, at, n, pairs, p);
      load_pts(dv, at, n, pairs, d);
    };
    if constexpr (EARLY) fetch(0);
    int row0 = 0, row1 = 0;
    if (J.n_proj > 0) {
      const int nblk = blk_count(N);
      const int ra = J.blk_row[blockIdx.x * nw], rb = J.blk_row[min((int)(blockIdx.x + 1) * nw, nblk)];
      if (rb > ra) {  // uniform across the CTA
        const C* cen = reinterpret_cast<const C*>(b.c_e) + (size_t)s * b.ce_stride;
        if constexpr (STAGED)
          for (int e = tid; e < b.ce_stride; e += blockDim.x) s_ce[e] = cen[e];
        if (blk < nblk) {
          row0 = J.blk_row[blk];
          row1 = J.blk_row[blk + 1];
        }
        if constexpr (STAGED) __syncthreads();
        if (row1 > row0) block_nonlocal<T, 1>(J, STAGED ? s_ce : cen, 0, row0, row1, s_nl);
      }
    }
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      if (!EARLY || l > 0) fetch(l);
      if (row1 > row0) {
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = cadd(q[u], s_nl[at[u]]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        // r -= alpha q, d += alpha p (points past the end are zero and not stored)
        r[u].x = fma(-ax, q[u].x, fma(ay, q[u].y, r[u].x));
        r[u].y = fma(-ax, q[u].y, fma(-ay, q[u].x, r[u].y));
        d[u].x = fma(ax, p[u].x, fma(-ay, p[u].y, d[u].x));
        d[u].y = fma(ax, p[u].y, fma(ay, p[u].x, d[u].y));
        const bool in = at[u] < n;  // (a short block's accumulators past its end are not its own)
        const T rx = in ? r[u].x : (T)0, ry = in ? r[u].y : (T)0;
        re = fma(rx, rx, fma(-ry, ry, re));
        sy = fma(ry, ry, sy);
        sxy = fma(rx, ry, sxy);
      }
      store_pts(rv, at, n, pairs, r);
      store_pts(dv, at, n, pairs, d);
    }
  }
  // r^T r = (re, 2 sxy), ||r||^2 = re + 2 sy over the CTA, fixed order
  double o[3];
  if constexpr (sizeof(T) == 4) {
    float v[4] = {re, sy, sxy, 0.f};
    const float t = warp_sum_many<4>(v);
    float* part = reinterpret_cast<float*>(red);
    if (lane < 4) part[warp * 4 + lane] = t;
    __syncthreads();
    if (warp != 0) return;
    const double d = lane < 3 ? sum_strided(part + lane, nw, 4) : 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) o[i] = __shfl_sync(0xffffffffu, d, i);
  } else {
    T v[3] = {re, sy, sxy};
    block_sum<3>(v, red, o);
    if (warp != 0) return;
  }
  if (lane == 0) {
    const size_t at = (size_t)s * b.PB + blockIdx.x;
    b.nrm_part[at] = fin ? fma(2.0, o[1], o[0]) : __longlong_as_double(0x7ff8000000000000ll);
    b.rho_part[at] = fin ? make_double2(o[0], 2.0 * o[2]) : make_double2(0.0, 0.0);
    __threadfence();
    const int done = atomicAdd(b.upd_cnt + s, 1);
    s_last = done == nU - 1 ? 1 : 0;
    if (done == nU - 1) {
      b.upd_cnt[s] = 0;
      __threadfence();
    }
  }
  __syncwarp();
  if (s_last) book_slot(b, s, nU, slot_it);
}

// ---------------------------------------------------------------------------
// Projections c_p = v_p . v for every projector, one CTA per (atom, SPB slots):
// the atom's support is gathered once and dotted with each of its projectors.
//   PJ_R: v = r (inner precision), ACTIVE slots         -> c_r
//   PJ_X: v = x64 + d (FP64), NEW / CHECK slots         -> c_x
//   PJ_IN: v = x_in (apply entry point)                 -> c_out
// Bound by the latency of the gather (about ten support points a thread) and by
// the reduction of its SPB * NP complex sums: a warp reduces all of them
// together, halving the number of sums a lane holds at each shuffle (V - 1
// shuffles and adds for V = 32 sums instead of 5 V), and the warps' results
// meet once in shared memory.  Two slots a CTA: four held 32 sums a thread and two
// CTAs an SM (256 FP32 vectors of 24x24x120, 20 atoms: 96 us with four, 38 with two).
// ---------------------------------------------------------------------------
enum { PJ_R = 0, PJ_X = 1, PJ_IN = 2 };
constexpr int kProjThreads = 256;

template <typename T, int MODE, int NP, int SPB>
__global__ void __launch_bounds__(kProjThreads) project_kernel(const JuncDev* __restrict__ jt,
                                                               const BatchDev* __restrict__ bp,
                                                               const void* __restrict__ x_in,
                                                               void* __restrict__ c_out) {
  // NP: projectors per atom at compile time (>= the junction's largest group);
  // SPB: slots per CTA, so each projector value is loaded once for SPB slots
  using CT = typename std::conditional<MODE == PJ_X, double, T>::type;
  using C = typename cx<CT>::t;
  using CO = typename cx<T>::t;
  constexpr int NV = 2 * NP * SPB;            // real sums per thread: [slot][projector][re, im]
  constexpr int V = NV >= 32 ? 32 : NV > 16 ? 32 : NV > 8 ? 16 : 8;  // reduced together
  constexpr int NR = (NV + V - 1) / V;        // rounds of V
  constexpr int NW = kProjThreads / 32;
  static_assert(NR * V <= 64, "sums per thread");
  const BatchDev& b = *bp;
  const int g = blockIdx.x;
  __shared__ CT part[NW][NR * V];
  __shared__ double s_mu[2 * NP * SPB];
  __shared__ int s_slot[SPB];
  __shared__ int s_any;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // PJ_X takes SPB entries of the NEW / CHECK list per CTA row (rows stride by
  // gridDim.y); PJ_R and PJ_IN take slots blockIdx.y * SPB + u
  int n_ent = b.nslots;
  if constexpr (MODE == PJ_X) n_ent = *b.lst_n;
  for (int base = blockIdx.y * SPB; base < n_ent; base += gridDim.y * SPB) {
    __syncthreads();  // shared memory of the previous entries is consumed
    if (tid == 0) s_any = 0;
    __syncthreads();
    if (tid < SPB) {
      const int e = base + tid;
      int s = e;
      if constexpr (MODE == PJ_X) s = e < n_ent ? b.lst[e] : -1;
      bool use = s >= 0 && s < b.nslots;
      if (use) {
        if constexpr (MODE == PJ_R) {
          use = b.state[s] == SL_ACTIVE;
        } else if constexpr (MODE == PJ_X) {
          const int st = b.state[s];
          use = st == SL_NEW || st == SL_CHECK;
        }
      }
      if (use && g >= jt[b.junc[s]].n_groups) use = false;
      s_slot[tid] = use ? s : -1;
      if (use) atomicOr(&s_any, 1);
    }
    __syncthreads();
    if (!s_any) continue;
    int slot[SPB];
    long long vo[SPB], xo[SPB];
    double sig[SPB];
    // every active slot of this CTA belongs to a junction with this group; the
    // junction of the first active slot supplies the support (batches share it)
    int s0 = 0;
    for (int u = SPB - 1; u >= 0; --u)
      if (s_slot[u] >= 0) s0 = s_slot[u];
#pragma unroll
    for (int u = 0; u < SPB; ++u) {
      slot[u] = s_slot[u];
      const int s = slot[u] >= 0 ? slot[u] : s0;
      vo[u] = b.voff[s];
      xo[u] = (MODE == PJ_X) ? b.xo[s] : 0;
      sig[u] = (MODE == PJ_X) ? b.sigma[s] : 1.0;
    }
    const JuncDev& J = jt[b.junc[s0]];
    const int p0 = J.grp_p0[g], np = J.grp_np[g];
    const int k0 = J.grp_ptr[g], k1 = J.grp_ptr[g + 1], len = k1 - k0;
    const long long vb = J.grp_voff[g];
    CT acc[NR * V];
#pragma unroll
    for (int j = 0; j < NR * V; ++j) acc[j] = 0;
#pragma unroll(NP * SPB <= 8 ? 4 : 2)
    for (int kk = tid; kk < len; kk += kProjThreads) {
      const int gi = J.grp_idx[k0 + kk];
      CT a[NP];
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        // (past the atom's projectors: its last one again, dropped at the end)
        const long long at = vb + kk + (long long)min(p, np - 1) * len;
        if constexpr (sizeof(CT) == 8) a[p] = (CT)J.grp_val64[at];
        else a[p] = (CT)J.grp_val32[at];
      }
      C v[SPB];
#pragma unroll
      for (int u = 0; u < SPB; ++u) {
        // (a slot that sits out reads another one's vector; its sums are dropped)
        if constexpr (MODE == PJ_R) {
          v[u] = reinterpret_cast<const CO*>(b.r)[vo[u] + gi];
        } else if constexpr (MODE == PJ_X) {
          const double2 xx = b.x64[xo[u] + gi];
          const double2 dd = to64(reinterpret_cast<const CO*>(b.d)[vo[u] + gi]);
          v[u] = mk2(fma(sig[u], dd.x, xx.x), fma(sig[u], dd.y, xx.y));
        } else {
          v[u] = reinterpret_cast<const CO*>(x_in)[vo[u] + gi];
        }
      }
#pragma unroll
      for (int u = 0; u < SPB; ++u)
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          acc[2 * (u * NP + p)] = fma(a[p], v[u].x, acc[2 * (u * NP + p)]);
          acc[2 * (u * NP + p) + 1] = fma(a[p], v[u].y, acc[2 * (u * NP + p) + 1]);
        }
    }
#pragma unroll
    for (int rd = 0; rd < NR; ++rd) {
      CT w[V];
#pragma unroll
      for (int j = 0; j < V; ++j) w[j] = acc[rd * V + j];
      const CT t = warp_sum_many<V>(w);
      if (lane < V) part[warp][rd * V + lane] = t;
    }
    __syncthreads();
    // thread t: real sum t of [slot][projector][re, im] over the warps, in warp order
    constexpr int NT = 2 * NP * SPB;
    const bool mine = tid < NT;
    const int u = mine ? tid / (2 * NP) : 0, p = mine ? (tid >> 1) % NP : 0, sl = s_slot[u];
    double mu = 0.0;
    if (tid < (NT + 31) / 32 * 32) {
      const double o = mine ? sum_strided(&part[0][tid], NW, NR * V) : 0.0;
      const double x = __shfl_sync(0xffffffffu, o, lane & ~1), y = __shfl_sync(0xffffffffu, o, lane | 1);
      if (mine && sl >= 0 && p < np) {
        const C cr = mk2((CT)x, (CT)y);
        const bool re = (tid & 1) == 0;
        if (re) reinterpret_cast<C*>(c_out)[(size_t)sl * b.pstride + p0 + p] = cr;
        // PJ_R: the projections of the new direction c_p = c_r + beta c_p_old
        // (c_p = c_r in the first iteration), e_kb c_p for the update kernel, and
        // the projector's share of mu = p^T A p, -e_kb[p] c_p^2
        if constexpr (MODE == PJ_R) {
          const int k = b.iters[sl];
          const C* cpo = reinterpret_cast<const C*>(b.c_p) + ((size_t)(k & 1) * b.nslots + sl) * b.pstride;
          C* cpn = reinterpret_cast<C*>(b.c_p) + ((size_t)((k + 1) & 1) * b.nslots + sl) * b.pstride;
          C* cen = reinterpret_cast<C*>(b.c_e) + (size_t)sl * b.ce_stride;
          C c = cr;
          if (k > 0) c = cfma(from64<C>(b.beta_cur[sl]), cpo[p0 + p], c);
          const double e64 = J.ekb[p0 + p];
          if (re) {
            const CT e = (CT)e64;
            cpn[p0 + p] = c;
            cen[p0 + p] = mk2(e * c.x, e * c.y);
          }
          // lanes of the real part -e (cx cx - cy cy), of the imaginary part -e (2 cx) cy
          const double cx = c.x, cy = c.y;
          mu = -e64 * (re ? fma(cx, cx, -cy * cy) : 2.0 * cx * cy);
        }
      }
    }
    if constexpr (MODE == PJ_R) {
      // the atom's share of mu, one more partial after the operator tiles'
      if (mine) s_mu[tid] = mu;
      __syncthreads();
      if (warp == 0) {
        const int nP = cocg_parts(J);
        double m = 0.0;
        if (lane < 2 * SPB) {
#pragma unroll
          for (int q = 0; q < NP; ++q) m += s_mu[(lane >> 1) * 2 * NP + 2 * q + (lane & 1)];
          const int sm = s_slot[lane >> 1];
          if (sm >= 0) reinterpret_cast<double*>(b.mu_part + (size_t)sm * b.PA + nP + g)[lane & 1] = m;
        }
        __threadfence();
        __syncwarp();
        // the slots' arrivals side by side
        const unsigned last = __ballot_sync(0xffffffffu, lane < SPB && s_slot[lane < SPB ? lane : 0] >= 0 &&
                                                             mu_arrive(b, J, s_slot[lane < SPB ? lane : 0]));
        for (int v = 0; v < SPB; ++v)
          if ((last >> v) & 1u) mu_alpha<sizeof(T) == 8>(b, J, s_slot[v]);
      }
    }
  }  // list entries
}

// ---------------------------------------------------------------------------
// Projector term of an operator application: y -= sum_p v_p e_kb[p] c_p over the
// blocks of points that hold support points, one warp per block and SPV vectors
// (the block's rows are read once for all of them).  A kernel of its own: inside
// the operator kernel the lookups stalled every plane of the march (24x24x120,
// 256 FP32 vectors: operator with the term 430 us, without 130 us).
// ---------------------------------------------------------------------------
template <typename T, int SPV>
__global__ void __launch_bounds__(kUpdThreads) nonlocal_kernel(const JuncDev* __restrict__ jt,
                                                               const BatchDev* __restrict__ bp,
                                                               const void* __restrict__ c_in, void* __restrict__ y_out) {
  using C = typename cx<T>::t;
  const BatchDev& b = *bp;
  const int v0 = blockIdx.y * SPV, nv = min(SPV, b.nslots - v0);
  const JuncDev& J = jt[b.junc[v0]];
  const int N = (int)J.N;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int nblk = blk_count(N);
  const int blk0 = blockIdx.x * nw, blk = blk0 + warp;
  if (J.blk_row[min(blk0 + nw, nblk)] == J.blk_row[min(blk0, nblk)]) return;  // uniform across the CTA
  extern __shared__ __align__(16) unsigned char nl_smem[];
  const int np = J.n_proj, ces = np + kCePad;
  C* s_ce = reinterpret_cast<C*>(nl_smem);  // [SPV][ces] e_kb c
  C* s_acc = s_ce + SPV * ces + warp * SPV * kBlkPts;
  for (int e = tid; e < SPV * ces; e += blockDim.x) {
    const int v = e / ces, p = e - v * ces;
    C w = czero<C>();
    if (v < nv && p < np) {
      const T k = (T)J.ekb[p];
      const C c = reinterpret_cast<const C*>(c_in)[(size_t)(v0 + v) * b.pstride + p];
      w = mk2(k * c.x, k * c.y);
    }
    s_ce[e] = w;
  }
  __syncthreads();
  if (blk >= nblk) return;
  const int row0 = J.blk_row[blk], row1 = J.blk_row[blk + 1];
  if (row1 == row0) return;
  block_nonlocal<T, SPV>(J, s_ce, ces, row0, row1, s_acc);
  const int n = blk_len(blk, N);
  for (int v = 0; v < nv; ++v) {
    C* y = reinterpret_cast<C*>(y_out) + b.voff[v0 + v] + blk_first(blk, N);
    C w[kBlkPts / 32];
#pragma unroll
    for (int h = 0; h < kBlkPts / 32; ++h)
      if (h * 32 + lane < n) w[h] = y[h * 32 + lane];
#pragma unroll
    for (int h = 0; h < kBlkPts / 32; ++h)
      if (h * 32 + lane < n) y[h * 32 + lane] = cadd(w[h], s_acc[v * kBlkPts + h * 32 + lane]);
  }
}

// ---------------------------------------------------------------------------
// Scheduler (one CTA, after the true-residual path and the COCG step of the
// same iteration): finishes converged
// systems, performs reliable updates (the true FP64 residual replaces the
// recurrence residual, the search direction is kept), frees drained slots and
// assigns queued systems to free slots in slot order.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kSchedThreads) sched_kernel(const JuncDev* __restrict__ jt,
                                                             const BatchDev* __restrict__ bp, int slot_it) {
  const BatchDev& b = *bp;
  const int S = b.nslots;
  __shared__ int warp_cnt[32];
  int upd = 0, busy = 0;
  if (b.n_shift > 0 && threadIdx.x == 0) *b.iter_no += 1;
  {
    // most iterations change no slot: nothing drained, listed, due for a list or
    // waiting for a slot; the list stays empty and the busy count what it was
    // (the whole kernel takes 7 us, this way out 3; with FP64 reductions it took 11)
    const bool queued = b.sched[0] < b.nsys;
    bool work = false;
    for (int s = threadIdx.x; s < S; s += blockDim.x) {
      const int st = b.state[s];
      work = work || !(st == SL_ACTIVE || (st == SL_FREE && !queued));
    }
    if (!__syncthreads_or(work)) {
      if (threadIdx.x == 0) b.sched[3 + slot_it] = b.sched[1];
      return;
    }
  }
  for (int s = threadIdx.x; s < S; s += blockDim.x) {
    int st = b.state[s];
    // NEW / CHECK / CHECKT slots are handled only if this iteration's list took
    // them (their true residual or goal check ran): the bookkeeping kernel, which
    // runs beside the list path, can move a slot to CHECK after the list was made
    const bool listed = b.inlist[s] != 0;
    if (st == SL_DRAIN) {
      st = SL_FREE;
    } else if (st == SL_CHECKT && listed) {
      // goal phase: compare the T partial of the iterate with the previous check;
      // the recurrence continues untouched towards a tenfold lower residual
      const double tcur = b.tgoal[s], tl = b.tlast[s];
      b.tlast[s] = tcur;
      const int gcnt = b.gcnt[s] + 1;
      b.gcnt[s] = gcnt;
      const bool settled = fabs(tcur - tl) <= b.tol_T * fabs(tcur);
      const bool capped = gcnt >= kMaxGoalChecks || b.total_iters[s] >= b.max_iter;
      if (settled || capped) {
        // a mixed-precision system whose T partial did not settle within the cap
        // is handed back (solved again in FP64); FP64 keeps its iterate
        const bool back = !settled && b.handback;
        const int sy = b.sys[s];
        b.out_iters[sy] = b.total_iters[s];
        b.out_relres[sy] = b.rgoal[s];
        b.out_status[sy] = back ? 3 : 0;
        atomicAdd(b.counters + 2, 1ull);
        if (back) atomicAdd(b.counters + 3, 1ull);
        st = SL_DRAIN;
      } else {
        b.tol2[s] = 0.01 * b.rrec2[s];
        b.cyc_iters[s] = 0;
        st = SL_ACTIVE;
      }
    } else if ((st == SL_NEW || st == SL_CHECK) && listed) {
      const double nrm = b.res_tot[4 * s], tcur = b.res_tot[4 * s + 3];
      const double2 rho = make_double2(b.res_tot[4 * s + 1], b.res_tot[4 * s + 2]);
      if (st == SL_NEW) {
        // cold start: r = b, so ||b||^2 = nrm; warm start: ||b||^2 is given
        const double bn = b.warm[s] ? b.sys_bn2[b.sys[s]] : nrm;
        b.bnorm2[s] = bn > 0.0 ? bn : 1.0;
        b.sigma[s] = bn > 0.0 ? sqrt(bn) : 1.0;
        b.rlast2[s] = 4.0 * nrm;
        b.stall[s] = 0;
        b.iters[s] = 0;
        b.total_iters[s] = 0;
        b.n_upd[s] = 0;
        b.restart[s] = 0;
        b.tlast[s] = -1.0;
        b.gcnt[s] = 0;
        b.gphase[s] = 0;
      }
      const double bn2 = b.bnorm2[s];
      const double rel = sqrt(nrm / bn2);
      const int sy = b.sys[s];
      const double tol = b.col[s] >= 0 ? b.tol : b.tol_adj;
      // a shifted system reaches CHECK only once every shift converged (or at
      // the iteration cap, which its per-shift records show): it is finished
      const bool res_ok = ((st == SL_CHECK || b.warm[s]) && rel <= tol) || nrm == 0.0;
      // goal-oriented finish of forward systems: the transmission reads x only
      // on the Gamma_L support, where x is exponentially small when the lead
      // channels are closed, so a residual of tol relative to the whole column
      // does not fix it; once the residual meets tol, iterations continue until
      // sum Gamma_L |x|^2 changes by at most tol_T of itself between two true
      // residuals (the Krylov iterate keeps converging there after its residual
      // has reached the rounding floor)
      const double tl = b.tlast[s];
      b.tlast[s] = tcur;
      const bool goal = b.tol_T > 0.0 && b.col[s] >= 0 && b.n_shift == 0;
      const bool goal_ok = !goal || nrm == 0.0 || (tl >= 0.0 && fabs(tcur - tl) <= b.tol_T * fabs(tcur));
      const bool goal_phase = res_ok && !goal_ok;  // the residual met tol, the T partial not yet
      // a goal phase that would start at the iteration or update cap keeps its
      // residual-converged iterate
      const bool goal_capped = goal_phase && (b.total_iters[s] >= b.max_iter || b.n_upd[s] >= b.max_upd);
      const bool conv = (res_ok && goal_ok) || goal_capped || (b.n_shift > 0 && st == SL_CHECK);
      // the recurrence has drifted when the true residual is more than 4x the
      // recurrence residual of the cycle that just ended (rounding in the
      // inner-precision Krylov basis): restart it from the true residual.
      // Cycles that did not cut the previous true residual by 4x are counted.
      // Early on such a plateau is ordinary slow Krylov convergence on an
      // indefinite operator, and a restart would throw the Krylov space away;
      // within three decades of the tolerance, two of them in a row mean the
      // recurrence has lost its accuracy (the true residuals that replace it
      // at the cycle cap hide the drift) and it restarts.
      // (in the goal phase the residual sits at its rounding floor: neither applies)
      const bool drift = st == SL_CHECK && !goal_phase && nrm > 16.0 * b.rrec2[s] * bn2;
      const bool no_gain = st == SL_CHECK && !goal_phase && nrm > 0.0625 * b.rlast2[s];
      const int stall = no_gain ? b.stall[s] + 1 : 0;
      // precision-limited systems are handed back early: either the true
      // residual stopped improving, or its rate so far (log rel per
      // iteration) predicts more iterations than the budget allows
      const int tot = b.total_iters[s];
      const bool slow = st == SL_CHECK && !goal_phase && tot >= 500 &&
                        (rel >= 1.0 || (double)tot * log(tol) / log(rel) > 1.5 * (double)b.max_iter);
      const bool stalled = (b.stall_cap > 0 && stall >= b.stall_cap) || (b.handback && slow);
      const bool fail = !isfinite(rel) || b.total_iters[s] >= b.max_iter || b.n_upd[s] >= b.max_upd || stalled;
      if (conv || fail) {
        b.out_iters[sy] = b.total_iters[s];
        b.out_relres[sy] = rel;
        b.out_status[sy] = conv ? 0 : (stalled ? 3 : (b.restart[s] ? 2 : 1));
        atomicAdd(b.counters + 2, 1ull);               // finished systems
        if (!conv) atomicAdd(b.counters + 3, 1ull);    // handed back (precision-limited / failed)
        st = SL_DRAIN;
      } else {
        // a drifted recurrence restarts from the true residual instead of
        // continuing with its direction
        b.stall[s] = stall;
        if (drift || (stall >= 2 && rel < 1e3 * tol)) b.restart[s] = 1;
        const double2 rho_s = make_double2(rho.x / bn2, rho.y / bn2);  // r^T r of r / sigma
        b.rlast2[s] = nrm;
        if (st == SL_NEW || b.restart[s]) {
          // fresh start: p = r at the next iteration
          b.iters[s] = 0;
          b.restart[s] = 0;
        } else {
          // reliable update: the true residual replaces the recurrence residual
          // and the direction update continues with beta_k = rho_new / rho_{k-1}
          // (beta_cur holds rho_k / rho_{k-1}, rho_cur holds rho_k)
          b.beta_cur[s] = cmul(b.beta_cur[s], cdiv(rho_s, b.rho_cur[s]));
        }
        b.rho_cur[s] = rho_s;
        // targets in the inner vectors' units (r / sigma, sigma^2 = ||b||^2)
        const double t_in = b.delta * b.delta * nrm / bn2, t_out = 0.25 * tol * tol;
        // shifted systems: the shift kernel ends the cycle once every shift converged;
        // goal phase: cycles of a tenfold cut of the recurrence residual
        b.tol2[s] = b.n_shift > 0 ? 0.0 : goal_phase ? 0.01 * nrm / bn2 : (t_in > t_out ? t_in : t_out);
        if (goal_phase) {
          // from here on the T partial is checked without true residuals (CHECKT)
          b.gphase[s] = 1;
          b.rgoal[s] = rel;
          b.gcnt[s] = 0;
        } else {
          // (a breakdown or a thrown-off recurrence in the goal phase whose true residual
          // no longer meets tol: the system has to meet it again first)
          b.gphase[s] = 0;
        }
        if (st == SL_CHECK) {
          b.n_upd[s] += 1;
          ++upd;
        }
        b.cyc_iters[s] = 0;
        b.rmin2[s] = nrm / bn2;
        b.rmin_it[s] = tot;
        st = SL_ACTIVE;
      }
    }
    b.state[s] = st;
  }
  __syncthreads();
  // Assign ready systems to FREE slots.  Free slots are taken in slot order,
  // systems in queue order from the first unstarted one, skipping those whose
  // dependency has not finished: an adjoint waits for its forward column but
  // does not hold up the systems queued behind it.  At most kReadyWindow
  // systems past the first unstarted one are examined.
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned below = (1u << lane) - 1u;
  __shared__ int s_nf, s_done, s_first;
  // (1) the free slots, compacted in slot order
  if (threadIdx.x == 0) s_nf = 0;
  __syncthreads();
  const int next0 = b.sched[0];
  for (int base = 0; base < S && next0 < b.nsys; base += blockDim.x) {
    const int s = base + threadIdx.x;
    const bool fr = s < S && b.state[s] == SL_FREE;
    const unsigned m = __ballot_sync(0xffffffffu, fr);
    if (lane == 0) warp_cnt[warp] = __popc(m);
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < nw; ++w) {
      if (w < warp) before += warp_cnt[w];
      total += warp_cnt[w];
    }
    if (fr) b.fslot[s_nf + before + __popc(m & below)] = s;
    __syncthreads();
    if (threadIdx.x == 0) s_nf += total;
    __syncthreads();
  }
  const int nf = s_nf;
  // (2) ready systems, in queue order, to the free slots
  if (threadIdx.x == 0) s_done = 0;
  __syncthreads();
  const int wend = min(b.nsys, next0 + kReadyWindow);
  for (int base = next0; base < wend && nf > 0; base += blockDim.x) {
    if (s_done >= nf) break;  // uniform: written before the last barrier
    const int n = base + threadIdx.x;
    bool ready = false;
    if (n < wend && !b.sys_started[n]) {
      const int dep = b.sys_dep ? b.sys_dep[n] : -1;
      ready = dep < 0 || b.out_status[dep] >= 0;
    }
    const unsigned m = __ballot_sync(0xffffffffu, ready);
    if (lane == 0) warp_cnt[warp] = __popc(m);
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < nw; ++w) {
      if (w < warp) before += warp_cnt[w];
      total += warp_cnt[w];
    }
    const int k = s_done + before + __popc(m & below);
    if (ready && k < nf) {
      const int s = b.fslot[k];
      b.sys[s] = n;
      b.junc[s] = b.sys_junc[n];
      b.E[s] = b.sys_E[n];
      b.col[s] = b.sys_col[n];
      const long long xo = b.sys_xo[n];
      b.xo[s] = xo >= 0 ? xo : b.voff[s];
      b.xfo[s] = b.sys_xfo[n];
      b.warm[s] = (b.sys_bn2 != nullptr && b.sys_bn2[n] > 0.0) ? 1 : 0;
      b.state[s] = SL_NEW;
      b.sys_started[n] = 1;
    }
    __syncthreads();
    if (threadIdx.x == 0) s_done = min(nf, s_done + total);
    __syncthreads();
  }
  // (3) the first unstarted system
  if (threadIdx.x == 0) s_first = b.nsys;
  __syncthreads();
  for (int base = next0; base < b.nsys; base += blockDim.x) {
    const int n = base + threadIdx.x;
    if (n < b.nsys && !b.sys_started[n]) atomicMin(&s_first, n);
    __syncthreads();
    const bool found = s_first < b.nsys;
    __syncthreads();
    if (found) break;
  }
  for (int s = threadIdx.x; s < S; s += blockDim.x) busy += (b.state[s] != SL_FREE) ? 1 : 0;
  build_list(b, warp_cnt);
  busy = __reduce_add_sync(0xffffffffu, busy);
  upd = __reduce_add_sync(0xffffffffu, upd);
  if (threadIdx.x == 0) s_nf = s_done = 0;  // reused: the CTA's totals
  __syncthreads();
  if (lane == 0) {
    if (busy) atomicAdd(&s_nf, busy);
    if (upd) atomicAdd(&s_done, upd);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    b.sched[0] = s_first;
    b.sched[1] = s_nf;
    b.sched[3 + slot_it] = s_nf;
    b.counters[1] += (unsigned long long)s_done;
  }
}

// After a true residual (NEW or CHECK slots): x64 += sigma d, d = 0, and the
// inner-precision residual is rescaled to r / sigma, sigma = ||b||, so the
// inner recurrence works on O(1) numbers whatever the size of b (an adjoint
// right-hand side Gamma_L o conj(x) can be ~1e-6 or smaller, whose squares
// would leave the FP32 range).  For a NEW slot sigma comes from the residual
// kernel's sum (r = b from a cold start; a warm start, whose r is smaller, brings
// ||b||^2 along); each thread touches only its own points.
template <typename T>
__global__ void __launch_bounds__(kVecThreads) x_update_kernel(const JuncDev* __restrict__ jt,
                                                               const BatchDev* __restrict__ bp) {
  using C = typename cx<T>::t;
  const BatchDev& b = *bp;
  __shared__ double s_sig;
  const int n = *b.lst_n;
  for (int li = blockIdx.y; li < n; li += gridDim.y) {
    const int s = b.lst[li];
    const int st = b.state[s];
    if (st != SL_NEW && st != SL_CHECK && st != SL_CHECKT) continue;
    const JuncDev& J = jt[b.junc[s]];
    if ((int)blockIdx.x >= J.nB) continue;
    __syncthreads();  // s_sig of the previous entry are consumed
    if (threadIdx.x == 0) {
      double sg = b.sigma[s];
      if (st == SL_NEW) {  // ||b||^2, as the scheduler takes it
        const double n2 = b.warm[s] ? b.sys_bn2[b.sys[s]] : b.res_tot[4 * s];
        sg = n2 > 0.0 ? sqrt(n2) : 1.0;
        if (blockIdx.x == 0) b.sigma[s] = sg;
      }
      s_sig = sg;
    }
    __syncthreads();
    const double sig = s_sig;
    // a goal-phase check keeps the recurrence (r is not a fresh true residual)
    const T isig = st == SL_CHECKT ? (T)1 : (T)(1.0 / sig);
    const long long vo = b.voff[s], xo = b.xo[s];
    const long long i0 = (long long)blockIdx.x * kVecPts;
    const long long i1 = min(i0 + (long long)kVecPts, J.N);
    C* dv = reinterpret_cast<C*>(b.d);
    C* rv = reinterpret_cast<C*>(b.r);
    for (long long i = i0 + threadIdx.x; i < i1; i += kVecThreads) {
      const double2 d = to64(dv[vo + i]);
      double2 x = b.x64[xo + i];
      x.x = fma(sig, d.x, x.x);
      x.y = fma(sig, d.y, x.y);
      b.x64[xo + i] = x;
      dv[vo + i] = czero<C>();
      C r = rv[vo + i];
      r.x *= isig;
      r.y *= isig;
      rv[vo + i] = r;
    }
  }
}

// Goal-phase checks (CHECKT slots of the list, after x_update moved d into x):
// tgoal[s] = sum_{i in L} Gamma_L,i |x(i)|^2, one CTA per list entry.
__global__ void __launch_bounds__(256) tgoal_kernel(const JuncDev* __restrict__ jt, const BatchDev* __restrict__ bp) {
  const BatchDev& b = *bp;
  __shared__ double red[32];
  const int n = *b.lst_n;
  for (int li = blockIdx.x; li < n; li += gridDim.x) {
    const int s = b.lst[li];
    if (b.state[s] != SL_CHECKT) continue;  // uniform across the CTA
    const JuncDev& J = jt[b.junc[s]];
    const long long xo = b.xo[s];
    double acc = 0.0;
    for (int l = threadIdx.x; l < J.nL; l += blockDim.x) {
      const double2 x = b.x64[xo + J.L_idx[l]];
      acc += J.L_gam[l] * (x.x * x.x + x.y * x.y);
    }
    double v[1] = {acc};
    double out[1];
    block_sum<1>(v, red, out);
    if (threadIdx.x == 0) b.tgoal[s] = out[0];
  }
}

// T partial of finished forward systems: out_t[sys] = sum_{i in L} Gamma_L,i |x(i)|^2.
__global__ void __launch_bounds__(256) emit_kernel(const JuncDev* __restrict__ jt, const BatchDev* __restrict__ bp) {
  const BatchDev& b = *bp;
  const int s = blockIdx.x;
  if (b.state[s] != SL_DRAIN || b.out_t == nullptr || b.col[s] < 0) return;
  const JuncDev& J = jt[b.junc[s]];
  __shared__ double red[32];
  const long long xo = b.xo[s];
  double acc = 0.0;
  for (int l = threadIdx.x; l < J.nL; l += blockDim.x) {
    const double2 x = b.x64[xo + J.L_idx[l]];
    acc += J.L_gam[l] * (x.x * x.x + x.y * x.y);
  }
  double v[1] = {acc};
  double out[1];
  block_sum<1>(v, red, out);
  if (threadIdx.x == 0) b.out_t[b.sys[s]] = out[0];
}

// T[e] = 4 sum_c Gamma_R[cols[c]] t[e][c]   (one warp per energy, fixed order).
__global__ void t_final_kernel(int n_e, int n_cols, const double* __restrict__ t_all,
                               const double* __restrict__ gr_cols, double* __restrict__ T) {
  const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (e >= n_e) return;
  double acc = 0.0;
  for (int c = lane; c < n_cols; c += 32) acc += gr_cols[c] * t_all[(size_t)e * n_cols + c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) T[e] = 4.0 * acc;
}

// g[i] += sum_k wt[k] Re(lambda_k(i) x_k(i)) over systems k in index order
// (lambda_k = lam + k N, x_k = x + k N).
__global__ void __launch_bounds__(256) grad_sys_kernel(int nsys, long long N, const double2* __restrict__ lam,
                                                       const double2* __restrict__ x, const double* __restrict__ wt,
                                                       double* __restrict__ g) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  double acc = 0.0;
  for (int k = 0; k < nsys; ++k) {
    const double w = wt[k];
    if (w == 0.0) continue;
    const double2 l = lam[(long long)k * N + i];
    const double2 v = x[(long long)k * N + i];
    acc += w * (l.x * v.x - l.y * v.y);
  }
  g[i] += acc;
}

// ---------------------------------------------------------------------------
// Shifted COCG (one seed Krylov space for every energy of a window).
//
// A(E_e) = A(E_s) + sigma_e 1 with sigma_e = E_e - E_s (Eq. G: E enters A only
// on the diagonal), so the seed recurrence's residual r_k = R_k(A_s) b serves
// every shifted system: its residual is collinear, r_{e,k} = r_k / pi_{e,k},
// with pi_{e,k} = R_k(-sigma_e) from the three-term recurrence of R_k:
//   pi_{k+1} = (1 + alpha_k sigma) pi_k + (alpha_k beta_{k-1} / alpha_{k-1}) (pi_k - pi_{k-1}),
//   alpha_e = alpha_k pi_k / pi_{k+1},  beta_e = beta_k (pi_k / pi_{k+1})^2,
//   x_e += alpha_e p_e,  p_e = r_{k+1} / pi_{k+1} + beta_e p_e
// (alpha_{-1} = 1, beta_{-1} = 0, pi_{-1} = pi_0 = 1, p_{e,0} = b).  What is kept
// is the scaled direction g_e = pi_{e,k} p_e, which needs no product with r:
//   x_e += (alpha_k / pi_{k+1}) g_e,  g_e = r_{k+1} + (beta_k pi_k / pi_{k+1}) g_e
// (products with conj(pi) / |pi|^2 instead of quotients; in a model of 288 shifted
// systems of three junctions on the same seed scalars, the iterates' median error
// against extended precision is 3.1e-15, 3.2e-15 with quotients and p_e, the rms 1.3e-11
// both ways;
// 8 instead of 12 operations of the FP64 pipe per shift and tracked point; the
// loads of four shifts are in flight together; 16 systems x 16 shifts x 4,608
// points: 43 -> 37 us in one CTA row, against 16 of FP64 work).  The seed
// runs the FP64 slot solver unchanged; the shifted iterates live only on the
// tracked points (the Gamma_L support for T, every point for full columns).
// A shift is frozen once ||r_{k+1}|| / |pi_{e,k+1}| <= tol ||b||.
// ---------------------------------------------------------------------------

// x_e = 0, p_e = b on the tracked points, pi = 1, no shift converged; NEW slots
// (rows over the NEW / CHECK list, like the zero kernel)
__global__ void __launch_bounds__(kVecThreads) shift_init_kernel(const JuncDev* __restrict__ jt,
                                                                 const BatchDev* __restrict__ bp) {
  const BatchDev& b = *bp;
  const int n = *b.lst_n, ns = b.n_shift, nT = b.nT;
  for (int li = blockIdx.y; li < n; li += gridDim.y) {
    const int s = b.lst[li];
    if (b.state[s] != SL_NEW) continue;
    const int col = b.col[s];
    double2* xb = b.xs + (long long)(b.xs_by_sys ? b.sys[s] : s) * b.xs_sstride;
    double2* pb = b.ps + (size_t)s * ns * nT;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nT; i += (long long)gridDim.x * blockDim.x) {
      const double one = b.T_idx[i] == col ? 1.0 : 0.0;
      for (int e = 0; e < ns; ++e) {
        xb[(long long)e * b.xs_estride + i] = make_double2(0.0, 0.0);
        pb[(size_t)e * nT + i] = make_double2(one, 0.0);
      }
    }
    if (blockIdx.x == 0) {
      const size_t S = (size_t)b.nslots;
      for (int e = threadIdx.x; e < ns; e += blockDim.x) {
        b.spi[(0 * S + s) * ns + e] = make_double2(1.0, 0.0);  // pi_0
        b.spi[(2 * S + s) * ns + e] = make_double2(1.0, 0.0);  // pi_{-1}
        b.sconv_it[(size_t)s * ns + e] = 0x7fffffff;
      }
      if (threadIdx.x == 0) {
        b.salpha[1 * S + s] = make_double2(1.0, 0.0);  // alpha_{-1}
        b.sbeta[1 * S + s] = make_double2(0.0, 0.0);   // beta_{-1}
      }
    }
  }
}

// One shifted step after iteration k of the seed (the slots that did it: ACTIVE
// ones, and those whose bookkeeping just moved them to CHECK).  CTA rows z take
// the shifts z * 8 .. + 7.  Every CTA of a slot derives the
// same scalars; CTA 0 records them (pi in a ring of three, so no CTA reads a
// value that is being overwritten) and ends the cycle once every shift converged.
__global__ void __launch_bounds__(kVecThreads) shift_update_kernel(const JuncDev* __restrict__ jt,
                                                                   const BatchDev* __restrict__ bp) {
  const BatchDev& b = *bp;
  const int s = blockIdx.y;
  if (b.stamp[s] != *b.iter_no) return;  // no COCG iteration just now
  const int ns = b.n_shift, nT = b.nT;
  const size_t S = (size_t)b.nslots;
  const int k = b.iters[s] - 1;  // the iteration just completed
  extern __shared__ double2 sh[];  // [ns] alpha_k / pi_{k+1}, [ns] beta_k pi_k / pi_{k+1}
  __shared__ int s_left;
  double2* sa = sh;
  double2* sb = sh + ns;
  if (threadIdx.x == 0) s_left = 0;
  __syncthreads();
  const double2 be = b.beta_cur[s];
  int* cit = b.sconv_it + (size_t)s * ns;
  if (threadIdx.x < 32 || ns > 32) {
    const double2 al = b.salpha[(size_t)(k & 1) * S + s];
    const double2 al_m = b.salpha[(size_t)((k + 1) & 1) * S + s];
    const double2 be_m = b.sbeta[(size_t)((k + 1) & 1) * S + s];
    const double rn2 = b.rn2[s], bn2 = b.bnorm2[s];
    const double2 cc = cmul(al, cdiv(be_m, al_m));  // alpha_k beta_{k-1} / alpha_{k-1}
    const double2* pi_k = b.spi + ((size_t)(k % 3) * S + s) * ns;
    const double2* pi_m = b.spi + ((size_t)((k + 2) % 3) * S + s) * ns;
    double2* pi_n = b.spi + ((size_t)((k + 1) % 3) * S + s) * ns;
    for (int e = threadIdx.x; e < ns; e += blockDim.x) {
      if (cit[e] < k) {  // frozen at an earlier iteration
        sa[e] = sb[e] = make_double2(0.0, 0.0);
        continue;
      }
      const double sg = b.shift_sig[e];
      const double2 p0 = pi_k[e], pm = pi_m[e];
      // pi_{k+1} = (1 + alpha sigma) pi_k + c (pi_k - pi_{k-1})
      const double2 f = make_double2(1.0 + al.x * sg, al.y * sg);
      const double2 pn = cadd(cmul(f, p0), cmul(cc, csub(p0, pm)));
      const double apn2 = pn.x * pn.x + pn.y * pn.y;
      const double inv2 = 1.0 / apn2;
      const double2 inv = make_double2(pn.x * inv2, -pn.y * inv2);  // 1 / pi_{k+1}
      sa[e] = cmul(al, inv);
      sb[e] = cmul(be, cmul(p0, inv));
      const double est2 = rn2 / (apn2 * bn2);
      const bool conv = est2 <= b.tol * b.tol;
      if (!isfinite(est2)) sa[e] = sb[e] = make_double2(0.0, 0.0);
      if (blockIdx.x == 0 && blockIdx.z == 0) {
        pi_n[e] = pn;
        const int sy = b.sys[s];
        b.out_srel[(size_t)e * b.nsys + sy] = sqrt(est2);
        if (conv) {
          cit[e] = k;
          b.out_sit[(size_t)e * b.nsys + sy] = k + 1;
        } else {
          atomicAdd(&s_left, 1);
        }
      }
    }
  }
  __syncthreads();
  if (blockIdx.x == 0 && blockIdx.z == 0 && threadIdx.x == 0) {
    b.sbeta[(size_t)(k & 1) * S + s] = be;
    if (s_left == 0) b.state[s] = SL_CHECK;  // every shift converged: end of the seed's cycle
  }
  double2* xb = b.xs + (long long)(b.xs_by_sys ? b.sys[s] : s) * b.xs_sstride;
  double2* pb = b.ps + (size_t)s * ns * nT;
  const double2* rv = reinterpret_cast<const double2*>(b.r) + b.voff[s];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nT; i += (long long)gridDim.x * blockDim.x) {
    const double2 r = rv[b.T_idx[i]];
    for (int e0 = 8 * blockIdx.z; e0 < min(ns, 8 * ((int)blockIdx.z + 1)); e0 += 4) {
      double2 g[4], x[4];
      bool on[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u;
        on[u] = false;
        if (e < ns) {  // (e0 + 4 <= 8 (z + 1)) frozen shifts are skipped (uniform across the CTA)
          const double2 a = sa[e], c = sb[e];
          on[u] = a.x != 0.0 || a.y != 0.0 || c.x != 0.0 || c.y != 0.0;
        }
        if (on[u]) {
          g[u] = pb[(size_t)e * nT + i];
          x[u] = xb[(long long)e * b.xs_estride + i];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u;
        if (!on[u]) continue;
        xb[(long long)e * b.xs_estride + i] = cfma(sa[e], g[u], x[u]);
        pb[(size_t)e * nT + i] = cfma(sb[e], g[u], r);
      }
    }
  }
}

// T partials of finished shifted systems: out_ts[e][sys] = sum over the tracked
// points of Gamma_L |x_e|^2 (one CTA per (shift, slot), fixed-order sums).
__global__ void __launch_bounds__(256) shift_emit_kernel(const JuncDev* __restrict__ jt,
                                                         const BatchDev* __restrict__ bp) {
  const BatchDev& b = *bp;
  const int s = blockIdx.y, e = blockIdx.x;
  if (b.state[s] != SL_DRAIN || e >= b.n_shift) return;
  const JuncDev& J = jt[b.junc[s]];
  __shared__ double red[32];
  const double2* xb = b.xs + (long long)(b.xs_by_sys ? b.sys[s] : s) * b.xs_sstride + (long long)e * b.xs_estride;
  double acc = 0.0;
  for (int i = threadIdx.x; i < b.nT; i += blockDim.x) {
    const double g = J.gl[b.T_idx[i]];
    if (g > 0.0) {
      const double2 x = xb[i];
      acc += g * (x.x * x.x + x.y * x.y);
    }
  }
  double v[1] = {acc};
  double out[1];
  block_sum<1>(v, red, out);
  if (threadIdx.x == 0) b.out_ts[(size_t)e * b.nsys + b.sys[s]] = out[0];
}

// ---------------------------------------------------------------------------
// Landauer current (Eq. Landauer): I(V_k) = (2e/h) int T(E) [f(E - mu_L) -
// f(E - mu_R)] dE with mu_{L,R} = E_F +- V_k / 2, atomic units (2e/h = 1/pi),
// by the trapezoidal rule on the given ascending energy grid; one CTA per
// bias, fixed-order sums.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double fermi_dev(double x, double kT) {
  if (kT == 0.0) return x < 0.0 ? 1.0 : (x > 0.0 ? 0.0 : 0.5);
  return 0.5 * (1.0 - tanh(x / (2.0 * kT)));
}

__global__ void __launch_bounds__(256) landauer_kernel(int n_e, const double* __restrict__ E,
                                                       const double* __restrict__ T, const double* __restrict__ V,
                                                       double E_F, double kT, double* __restrict__ I) {
  __shared__ double red[32];
  const double v = V[blockIdx.x];
  const double muL = E_F + 0.5 * v, muR = E_F - 0.5 * v;
  double acc = 0.0;
  for (int e = threadIdx.x; e + 1 < n_e; e += blockDim.x) {
    const double g0 = T[e] * (fermi_dev(E[e] - muL, kT) - fermi_dev(E[e] - muR, kT));
    const double g1 = T[e + 1] * (fermi_dev(E[e + 1] - muL, kT) - fermi_dev(E[e + 1] - muR, kT));
    acc += 0.5 * (E[e + 1] - E[e]) * (g0 + g1);
  }
  double vv[1] = {acc};
  double out[1];
  block_sum<1>(vv, red, out);
  if (threadIdx.x == 0) I[blockIdx.x] = out[0] / 3.14159265358979323846;
}

// Value quads of the row tables, [row][quad][lane], gathered from the per-point
// entries (setup).
__global__ void row_values_kernel(long long n, int nq, const int* __restrict__ src, const double* __restrict__ inv_q64,
                                  double* __restrict__ q64, float* __restrict__ q32) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * 4 * nq) return;
  const long long i = t / (4 * nq);  // entry: row * 32 + lane
  const int j = (int)(t - i * 4 * nq), e = src[i];
  const double v = e >= 0 ? inv_q64[(size_t)e * 4 * nq + j] : 0.0;
  const long long at = (((i / 32) * nq + j / 4) * 32 + i % 32) * 4 + j % 4;
  q64[at] = v;
  q32[at] = (float)v;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
#define RSN_DECL_OP(R)                                                                                        \
  cudaError_t launch_op_R##R(int, bool, int, dim3, int, size_t, cudaStream_t, const JuncDev*, const BatchDev*, \
                             const void*, void*);                                                 \
  cudaError_t launch_op_tma_R##R(int, bool, dim3, int, size_t, cudaStream_t, const JuncDev*, const BatchDev*,  \
                                 const void*, void*);                                             \
  cudaError_t launch_op_pair_R##R(int, bool, int, dim3, int, size_t, cudaStream_t, const JuncDev*, const BatchDev*, \
                                  const void*, void*);                                            \
  cudaError_t launch_op_plane_R##R(int, dim3, int, size_t, cudaStream_t, const JuncDev*, const BatchDev*,      \
                                   const void*, void*);
RSN_DECL_OP(1)
RSN_DECL_OP(2)
RSN_DECL_OP(3)
RSN_DECL_OP(4)
RSN_DECL_OP(5)
RSN_DECL_OP(6)
#undef RSN_DECL_OP

cudaError_t launch_op(int mode, bool fp32, int R, int ppt, dim3 grid, int threads, size_t smem, cudaStream_t st,
                      const JuncDev* jt, const BatchDev* b, const void* x_in, void* y_out) {
  switch (R) {
    case 1: return launch_op_R1(mode, fp32, ppt, grid, threads, smem, st, jt, b, x_in, y_out);
    case 2: return launch_op_R2(mode, fp32, ppt, grid, threads, smem, st, jt, b, x_in, y_out);
    case 3: return launch_op_R3(mode, fp32, ppt, grid, threads, smem, st, jt, b, x_in, y_out);
    case 4: return launch_op_R4(mode, fp32, ppt, grid, threads, smem, st, jt, b, x_in, y_out);
    case 5: return launch_op_R5(mode, fp32, ppt, grid, threads, smem, st, jt, b, x_in, y_out);
    case 6: return launch_op_R6(mode, fp32, ppt, grid, threads, smem, st, jt, b, x_in, y_out);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_op_tma(int mode, bool fp32, int R, dim3 grid, int threads, size_t smem, cudaStream_t st,
                          const JuncDev* jt, const BatchDev* b, const void* x_in, void* y_out) {
  switch (R) {
    case 1: return launch_op_tma_R1(mode, fp32, grid, threads, smem, st, jt, b, x_in, y_out);
    case 2: return launch_op_tma_R2(mode, fp32, grid, threads, smem, st, jt, b, x_in, y_out);
    case 3: return launch_op_tma_R3(mode, fp32, grid, threads, smem, st, jt, b, x_in, y_out);
    case 4: return launch_op_tma_R4(mode, fp32, grid, threads, smem, st, jt, b, x_in, y_out);
    case 5: return launch_op_tma_R5(mode, fp32, grid, threads, smem, st, jt, b, x_in, y_out);
    case 6: return launch_op_tma_R6(mode, fp32, grid, threads, smem, st, jt, b, x_in, y_out);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_op_pair(int mode, int R, bool big, int pitch, dim3 grid, int threads, size_t smem, cudaStream_t st,
                           const JuncDev* jt, const BatchDev* b, const void* x_in, void* y_out) {
  switch (R) {
    case 1: return launch_op_pair_R1(mode, big, pitch, grid, threads, smem, st, jt, b, x_in, y_out);
    case 2: return launch_op_pair_R2(mode, big, pitch, grid, threads, smem, st, jt, b, x_in, y_out);
    case 3: return launch_op_pair_R3(mode, big, pitch, grid, threads, smem, st, jt, b, x_in, y_out);
    case 4: return launch_op_pair_R4(mode, big, pitch, grid, threads, smem, st, jt, b, x_in, y_out);
    case 5: return launch_op_pair_R5(mode, big, pitch, grid, threads, smem, st, jt, b, x_in, y_out);
    case 6: return launch_op_pair_R6(mode, big, pitch, grid, threads, smem, st, jt, b, x_in, y_out);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_op_plane(int mode, int R, dim3 grid, int threads, size_t smem, cudaStream_t st, const JuncDev* jt,
                            const BatchDev* b, const void* x_in, void* y_out) {
  switch (R) {
    case 1: return launch_op_plane_R1(mode, grid, threads, smem, st, jt, b, x_in, y_out);
    case 2: return launch_op_plane_R2(mode, grid, threads, smem, st, jt, b, x_in, y_out);
    case 3: return launch_op_plane_R3(mode, grid, threads, smem, st, jt, b, x_in, y_out);
    case 4: return launch_op_plane_R4(mode, grid, threads, smem, st, jt, b, x_in, y_out);
    case 5: return launch_op_plane_R5(mode, grid, threads, smem, st, jt, b, x_in, y_out);
    case 6: return launch_op_plane_R6(mode, grid, threads, smem, st, jt, b, x_in, y_out);
    default: return cudaErrorInvalidValue;
  }
}

size_t op_pair_smem_bytes(int mode, int R, int nx, int ny) {
  const size_t nin = mode == OP_COCG ? 2 : 1;
  const size_t pitch = (size_t)std::max(pair_pitch_const(nx), nx + 2 * kPairXO);
  return sizeof(float2) * (kPairStages * nin * (size_t)nx * ny + 2 * (size_t)(ny + 2 * R) * pitch) + 16 +
         8 * kPairStages;
}

size_t op_tma_smem_bytes(int mode, int R, int nx, int ny) {
  const size_t el = sizeof(float2);
  const size_t nin = mode == OP_COCG ? 2 : 1;
  return el * (kStages * nin * (size_t)nx * ny + 2 * (size_t)(nx + 2 * R) * (ny + 2 * R)) + 16 + 8 * kStages;
}

size_t op_smem_bytes(bool fp32, int mode, int R, int TY, int nx, int n_proj, int lz) {
  static_assert(kMuSlots64 * sizeof(double) == kMuSlots32 * sizeof(float) &&
                kMuBlockBytes == kOpThreads / 32 * kMuSlots64 * sizeof(double), "mu partials of a block of planes");
  const size_t el = (mode == OP_RESID || !fp32) ? sizeof(double2) : sizeof(float2);
  const size_t cep = mode == OP_RESID ? (size_t)n_proj + kCePad : 0;
  const size_t mu = mode == OP_COCG ? (size_t)((lz + kMuPlanes - 1) / kMuPlanes) * kMuBlockBytes : 0;
  return el * (2 * (size_t)(TY + 2 * R) * (nx + 2 * R) + cep) + mu;
}

cudaError_t launch_zero(bool fp32, int nslots, int nB, cudaStream_t st, const JuncDev* jt, const BatchDev* b) {
  dim3 grid(nB, nslots);
  if (fp32) zero_kernel<float><<<grid, kVecThreads, 0, st>>>(jt, b);
  else zero_kernel<double><<<grid, kVecThreads, 0, st>>>(jt, b);
  return cudaGetLastError();
}

cudaError_t launch_cocg_update(bool fp32, int nslots, long long N_max, bool proj, int ce_stride, int slot_it,
                               cudaStream_t st, const JuncDev* jt, const BatchDev* b) {
  constexpr int nw = kUpdThreads / 32;
  const dim3 grid(upd_ctas(N_max), nslots);
  const size_t el = fp32 ? sizeof(float2) : sizeof(double2);
  size_t smem = proj ? ((size_t)ce_stride + nw * kBlkPts) * el : 0;
  const bool early = upd_early(N_max, nslots);
  void (*kern)(const JuncDev*, const BatchDev*, int) =
      fp32 ? (early ? cocg_update_kernel<float, true> : cocg_update_kernel<float, false>)
           : (early ? cocg_update_kernel<double, true> : cocg_update_kernel<double, false>);
  if (!fp32 && smem + 256 > (size_t)kMaxSmem) {  // (FP32: the true residual's limit comes first)
    kern = cocg_update_kernel<double, false, false>;
    smem = nw * kBlkPts * el;
  }
  if (smem > 32 * 1024) {
    cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<grid, 32 * nw, smem, st>>>(jt, b, slot_it);
  return cudaGetLastError();
}

template <int NP, int SPB>
static void launch_project_np(int mode, bool fp32, dim3 grid, cudaStream_t st, const JuncDev* jt, const BatchDev* b,
                              const void* x_in, void* c_out) {
  if (mode == PJ_R) {
    if (fp32) project_kernel<float, PJ_R, NP, SPB><<<grid, kProjThreads, 0, st>>>(jt, b, x_in, c_out);
    else project_kernel<double, PJ_R, NP, SPB><<<grid, kProjThreads, 0, st>>>(jt, b, x_in, c_out);
  } else if (mode == PJ_X) {
    if (fp32) project_kernel<float, PJ_X, NP, SPB><<<grid, kProjThreads, 0, st>>>(jt, b, x_in, c_out);
    else project_kernel<double, PJ_X, NP, SPB><<<grid, kProjThreads, 0, st>>>(jt, b, x_in, c_out);
  } else {
    if (fp32) project_kernel<float, PJ_IN, NP, SPB><<<grid, kProjThreads, 0, st>>>(jt, b, x_in, c_out);
    else project_kernel<double, PJ_IN, NP, SPB><<<grid, kProjThreads, 0, st>>>(jt, b, x_in, c_out);
  }
}

cudaError_t launch_project(int mode, bool fp32, int nslots, int n_groups, int max_np, cudaStream_t st,
                           const JuncDev* jt, const BatchDev* b, const void* x_in, void* c_out,
                           bool one_slot_per_cta) {
  // slots per CTA: the projector values of an atom are loaded once for all of
  // them; a pool over several junctions takes one slot per CTA (atom g differs
  // between junctions), and so does a launch that would leave SMs idle
  const bool one = one_slot_per_cta || (long long)n_groups * ((nslots + 1) / 2) < 2 * 152;
  if (max_np <= 4) {
    if (one) launch_project_np<4, 1>(mode, fp32, dim3(n_groups, nslots), st, jt, b, x_in, c_out);
    else launch_project_np<4, 2>(mode, fp32, dim3(n_groups, (nslots + 1) / 2), st, jt, b, x_in, c_out);
  } else if (max_np <= 9) {
    if (one) launch_project_np<9, 1>(mode, fp32, dim3(n_groups, nslots), st, jt, b, x_in, c_out);
    else launch_project_np<9, 2>(mode, fp32, dim3(n_groups, (nslots + 1) / 2), st, jt, b, x_in, c_out);
  } else if (max_np <= kMaxGroupNp) {
    launch_project_np<kMaxGroupNp, 1>(mode, fp32, dim3(n_groups, nslots), st, jt, b, x_in, c_out);
  } else {
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_nonlocal(bool fp32, int n_rhs, long long N, int n_proj, cudaStream_t st, const JuncDev* jt,
                            const BatchDev* b, const void* c, void* y) {
  const size_t el = fp32 ? sizeof(float2) : sizeof(double2);
  // four blocks a CTA, one where the coefficients leave no room for the sums of more
  const int nw = ((size_t)n_proj + kCePad + kUpdThreads / 32 * kBlkPts) * el > (size_t)kMaxSmem ? 1 : kUpdThreads / 32;
  // several vectors a warp where that still leaves every SM a few CTAs and the
  // coefficients fit beside the sums
  const int gx = (blk_count((int)N) + nw - 1) / nw, many = fp32 ? 4 : 2;
  const bool one = (long long)gx * ((n_rhs + many - 1) / many) < 4 * 152 ||
                   many * ((size_t)n_proj + kCePad) * el > 24 * 1024;
  const int spv = one ? 1 : many;
  const size_t smem = spv * ((size_t)n_proj + kCePad + nw * kBlkPts) * el;
  void (*kern)(const JuncDev*, const BatchDev*, const void*, void*) =
      fp32 ? (one ? nonlocal_kernel<float, 1> : nonlocal_kernel<float, 4>)
           : (one ? nonlocal_kernel<double, 1> : nonlocal_kernel<double, 2>);
  if (smem > 48 * 1024) {
    cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<dim3(gx, (n_rhs + spv - 1) / spv), 32 * nw, smem, st>>>(jt, b, c, y);
  return cudaGetLastError();
}

cudaError_t launch_sched(int slot_it, cudaStream_t st, const JuncDev* jt, const BatchDev* b) {
  sched_kernel<<<1, kSchedThreads, 0, st>>>(jt, b, slot_it);
  return cudaGetLastError();
}

cudaError_t launch_x_update(bool fp32, int nslots, int nB, cudaStream_t st, const JuncDev* jt, const BatchDev* b) {
  dim3 grid(nB, nslots);
  if (fp32) x_update_kernel<float><<<grid, kVecThreads, 0, st>>>(jt, b);
  else x_update_kernel<double><<<grid, kVecThreads, 0, st>>>(jt, b);
  return cudaGetLastError();
}

cudaError_t launch_shift_init(int nT, cudaStream_t st, const JuncDev* jt, const BatchDev* b) {
  const int bx = std::max(1, std::min(64, (nT + kVecThreads - 1) / kVecThreads));
  shift_init_kernel<<<dim3(bx, kListRows), kVecThreads, 0, st>>>(jt, b);
  return cudaGetLastError();
}

cudaError_t launch_shift_update(int nslots, int nT, int n_shift, cudaStream_t st, const JuncDev* jt,
                                const BatchDev* b) {
  const int bx = std::max(1, (nT + kVecThreads - 1) / kVecThreads);
  shift_update_kernel<<<dim3(bx, nslots, (n_shift + 7) / 8), kVecThreads, 2 * n_shift * sizeof(double2), st>>>(jt, b);
  return cudaGetLastError();
}

cudaError_t launch_shift_emit(int nslots, int n_shift, cudaStream_t st, const JuncDev* jt, const BatchDev* b) {
  shift_emit_kernel<<<dim3(n_shift, nslots), 256, 0, st>>>(jt, b);
  return cudaGetLastError();
}

cudaError_t launch_tgoal(int rows, cudaStream_t st, const JuncDev* jt, const BatchDev* b) {
  tgoal_kernel<<<rows, 256, 0, st>>>(jt, b);
  return cudaGetLastError();
}

cudaError_t launch_landauer(int n_e, const double* E, const double* T, int n_v, const double* V, double E_F,
                            double kT, double* I, cudaStream_t st) {
  landauer_kernel<<<n_v, 256, 0, st>>>(n_e, E, T, V, E_F, kT, I);
  return cudaGetLastError();
}

cudaError_t launch_row_values(long long n, int nq, cudaStream_t st, const int* src, const double* inv_q64, double* q64,
                              float* q32) {
  if (n > 0)
    row_values_kernel<<<(unsigned)((n * 4 * nq + 255) / 256), 256, 0, st>>>(n, nq, src, inv_q64, q64, q32);
  return cudaGetLastError();
}

cudaError_t launch_list(cudaStream_t st, const BatchDev* b) {
  list_kernel<<<1, kSchedThreads, 0, st>>>(b);
  return cudaGetLastError();
}

cudaError_t launch_emit(int nslots, cudaStream_t st, const JuncDev* jt, const BatchDev* b) {
  emit_kernel<<<nslots, 256, 0, st>>>(jt, b);
  return cudaGetLastError();
}

cudaError_t launch_t_final(int n_e, int n_cols, cudaStream_t st, const double* t_all, const double* gr_cols,
                           double* T_out) {
  const int warps = 8;
  t_final_kernel<<<(n_e + warps - 1) / warps, 32 * warps, 0, st>>>(n_e, n_cols, t_all, gr_cols, T_out);
  return cudaGetLastError();
}

cudaError_t launch_grad_sys(int nsys, long long N, cudaStream_t st, const double2* lam, const double2* x,
                            const double* wt, double* g) {
  grad_sys_kernel<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(nsys, N, lam, x, wt, g);
  return cudaGetLastError();
}

}  // namespace rsn
