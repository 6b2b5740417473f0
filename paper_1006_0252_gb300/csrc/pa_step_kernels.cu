// pa_step_kernels.cu -- the resampling half of an annealing step and the
// per-run bookkeeping (Sec. 2 and its Algorithm), plus set-up, read-out,
// overlap (Sec. 4) and weighted-average (Sec. 3) kernels.
//
// Step pipeline for a set of runs (all state on the device):
//   k_prepare  one block per run: energy histogram -> Q' over the fixed
//              32-lane tree, ln Q and the staged -beta F~ (Eqs. (2), (4)),
//              per-bin Poisson means (Eq. (1)), Metropolis thresholds
//              (Gaussian runs: k_gprep_head, k_gweights, k_gprep_tail).
//   k_copies   one block per 256 replicas: Poisson copy counts (inverse CDF,
//              means above 32 split into pieces; long walks shared out over the
//              block), per-chunk sums.
//   k_scan     one block per run: exclusive scan of the chunk sums, R~',
//              capacity / extinction check.
//   k_scatter  one block per 256 replicas: source slot of every new slot, the
//              new slots taken in turn.
//   k_resample one block per run of at most SMALL_RUN slots (+-1 couplings): the
//              four above in one launch.
//   k_sweep*   fused copy + sweeps + measurement (pa_sweep*.cu, pa_gauss*.cu*,
//              pa_box*.cu*).
//   k_commit   one thread per run: commit the step or leave it untouched.  In a
//              schedule of small runs k_resample of the next step does this, and
//              k_commit follows the last step only.
#include <math.h>

#include "pa_dexp.cuh"
#include "pa_divk.cuh"
#include "pa_gauss.cuh"

#include <algorithm>

namespace pa {

constexpr double LN2_NEAREST = 0x1.62e42fefa39efp-1;

// ceil(C 2^53) for 0 <= C < 2^10, from the bits of C (C = M 2^(e - 1075),
// M the 53-bit significand, so C 2^53 = M 2^(e - 1022)): the smallest
// integer U with U 2^-53 >= C.
__device__ __forceinline__ uint64_t cdf_threshold(double C) {
  const uint64_t bits = (uint64_t)__double_as_longlong(C);
  const int e = (int)(bits >> 52);
  if (e == 0) return bits != 0u ? 1u : 0u;  // zero, or below 2^-1022: C 2^53 < 1
  const uint64_t M = (bits & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  const int s = e - 1022;
  if (s >= 0) return M << s;
  if (s <= -64) return 1u;
  return (M + (1ull << -s) - 1u) >> -s;
}

// ---------------------------------------------------------------------------
// Set-up
// ---------------------------------------------------------------------------

// Coupling masks of a 3D cubic lattice from int8 J[3][N] (site i = x + L(y + L z)).
__global__ void k_setup_bonds3d(const int8_t* __restrict__ J, int L, int K, int G, int W,
                                uint32_t* __restrict__ bonds) {
  const int WR = L * G;
  const int N = L * L * L;
  for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < W; w += gridDim.x * blockDim.x) {
    uint32_t m[6] = {0, 0, 0, 0, 0, 0};
    if (w < WR) {
      const int y = w / G, g = w % G;
      for (int j = 0; j < K; ++j)
        for (int x = 0; x < L; ++x) {
          const int z = g + j * G;
          const int p = j * L + x;
          const int i = x + L * (y + L * z);
          const int ixm = ((x + L - 1) % L) + L * (y + L * z);
          const int iym = x + L * (((y + L - 1) % L) + L * z);
          const int izm = x + L * (y + L * ((z + L - 1) % L));
          const int8_t jv[6] = {J[i], J[ixm], J[N + i], J[N + iym], J[2 * N + i], J[2 * N + izm]};
          for (int d = 0; d < 6; ++d)
            if (jv[d] < 0) m[d] |= 1u << p;
        }
    }
    for (int d = 0; d < 6; ++d) bonds[d * W + w] = m[d];
  }
}

// Coupling / presence masks of a chain from int8 J[N] (J[N-1] = wrap bond).
__global__ void k_setup_bonds1d(const int8_t* __restrict__ J, int N, int W,
                                uint32_t* __restrict__ bonds) {
  for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < W; w += gridDim.x * blockDim.x) {
    uint32_t jp = 0, jm = 0, pp = 0, pm = 0;
    for (int p = 0; p < 32; ++p) {
      const int i = 32 * w + p;
      if (i >= N) break;
      const int8_t a = J[i], b = J[(i + N - 1) % N];
      if (a < 0) jp |= 1u << p;
      if (b < 0) jm |= 1u << p;
      if (a != 0) pp |= 1u << p;
      if (b != 0) pm |= 1u << p;
    }
    bonds[0 * W + w] = jp;
    bonds[1 * W + w] = jm;
    bonds[2 * W + w] = pp;
    bonds[3 * W + w] = pm;
  }
}

// beta = 0 state before the init kernel fills the population (Sec. 2: ln Omega).
__global__ void k_init_state(RunDev* __restrict__ runs, const int32_t* __restrict__ ids, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  RunDev& R = runs[ids ? ids[t] : t];
  R.cur = 0;
  R.error = 0;
  R.skip = 0;
  R.step = 0;
  R.sweeps = 0;
  R.beta = 0.0;
  R.mbF = __dmul_rn((double)R.N, LN2_NEAREST);
  R.lnQ_last = 0.0;
  R.Qp_last = 0.0;
  R.sumE_next = 0ull;
  R.sumE2_next = 0ull;
  R.emin_next = 0x7FFFFFFFFFFFFFFFll;
  R.sumE2hi_next = 0ull;
  R.R_next = R.R;
}

__global__ void k_zero_hist(RunDev* __restrict__ runs, const int32_t* __restrict__ ids, int n, int which) {
  const int t = blockIdx.y;
  if (t >= n) return;
  RunDev& R = runs[ids ? ids[t] : t];
  uint32_t* h = R.hist[which];
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < R.nbins; b += gridDim.x * blockDim.x) h[b] = 0u;
}

// Energy sums of the measured population become the committed ones.  The
// Gaussian model's record keeps the bits of the physical sum of E^2 in the
// sumE2 slot (the integer sum does not fit 64 bits).
__device__ __forceinline__ void commit_energy_sums(RunDev& R) {
  R.sumE = (int64_t)R.sumE_next;
  R.sumE2 = (int64_t)R.sumE2_next;
  R.emin = R.emin_next;
  if (R.model == 1) {
    const double s = __dadd_rn(__dmul_rn((double)R.sumE2hi_next, 4294967296.0), (double)R.sumE2_next);
    R.sumE2d = __dmul_rn(s, 0x1.0p-30);
    R.sumE2 = __double_as_longlong(R.sumE2d);
  }
}

// Commit the step whose population has been measured (or, after a
// device-detected error, leave the state as it was).
__device__ __forceinline__ void commit_step(RunDev& R) {
  if (R.skip || R.error) return;
  R.cur ^= 1;
  R.R = R.R_next;
  R.beta = R.beta_next;
  R.mbF = R.mbF_staged;
  R.lnQ_last = R.lnQ_staged;
  R.Qp_last = R.Qp_staged;
  R.step += 1;
  R.sweeps += R.theta_next;
  commit_energy_sums(R);
  const int64_t k = R.step;
  if (k <= R.max_steps) {
    R.rec_beta[k] = R.beta;
    R.rec_lnQ[k] = R.lnQ_last;
    R.rec_mbF[k] = R.mbF;
    R.rec_R[k] = R.R;
    R.rec_sumE[k] = R.sumE;
    R.rec_sumE2[k] = R.sumE2;
  }
}

__global__ void k_init_finish(RunDev* __restrict__ runs, const int32_t* __restrict__ ids, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  RunDev& R = runs[ids ? ids[t] : t];
  commit_energy_sums(R);
  R.rec_beta[0] = 0.0;
  R.rec_lnQ[0] = 0.0;
  R.rec_mbF[0] = R.mbF;
  R.rec_R[0] = R.R;
  R.rec_sumE[0] = R.sumE;
  R.rec_sumE2[0] = R.sumE2;
}

// ---------------------------------------------------------------------------
// Step: Q, ln Q, -beta F~, Poisson tables, thresholds (one block per run)
// ---------------------------------------------------------------------------
constexpr int PREP_THREADS = 256;
constexpr int PREP_WIN = 2048;  // bins of one shared-memory window of the Q' sum

// Every FP64 instruction holds an SM sub-partition for about 64 cycles on
// this GPU, so the block keeps the FP64 chains short and side by side: the
// per-bin work is spread over the block, the Q' tree reads its terms from
// shared memory and visits only the occupied range of bins, and ln Q and the
// thresholds are computed by threads without bins while the others build the
// Poisson tables.  Returns false (in all threads) where the run has no step to
// take.
template <int NT>
__device__ __forceinline__ bool prepare_block(RunDev& R, int use_override, double beta_o, int theta_o, int64_t Rt_o) {
  __shared__ int s_ok, s_bmin, s_bmax, s_theta, s_nocc;
  __shared__ double s_bn, s_Qp;
  __shared__ long long s_Rt;
  __shared__ double s_term[PREP_WIN];
  const int tid = threadIdx.x;
  if (tid == 0) {
    int ok = 1;
    double bn = 0.0;
    int th = 0;
    int64_t Rt = 0;
    if (R.error) {
      ok = 0;
    } else if (use_override) {
      bn = beta_o < 0.0 ? R.beta : beta_o;
      th = theta_o;
      Rt = Rt_o < 0 ? R.R : Rt_o;
    } else if (R.step >= R.n_sched || R.step >= R.max_steps) {
      ok = 0;  // schedule exhausted: the run is finished, nothing to do
    } else {
      bn = R.sched_beta[R.step];
      th = R.sched_theta[R.step];
      Rt = R.sched_R[R.step];
    }
    if (ok && (!(bn >= R.beta) || th < 0 || Rt < 1)) {
      R.error = ERR_INVALID;
      ok = 0;
    }
    if (!ok) R.skip = 1;
    s_ok = ok;
    s_bn = bn;
    s_theta = th;
    s_Rt = Rt;
    s_bmin = 0x7FFFFFFF;
    s_bmax = -1;
    s_nocc = 0;
  }
  __syncthreads();
  if (!s_ok) return false;
  const double bn = s_bn;
  const int64_t Rt = s_Rt;
  const double dbeta = __dsub_rn(bn, R.beta);
  const uint32_t* __restrict__ h = R.hist[R.cur];
  const int nbins = R.nbins;
  double* __restrict__ w = R.bin_w;

  // occupied bins, compacted so the FP64 work below spreads evenly over the
  // block; the first and last occupied bins
  int32_t* __restrict__ occ = R.occ;
  for (int b = tid; b < nbins; b += NT)
    if (h[b] != 0u) {
      atomicMin(&s_bmin, b);
      atomicMax(&s_bmax, b);
      occ[atomicAdd(&s_nocc, 1)] = b;
    }
  __syncthreads();
  const int bmin = s_bmin, bmax = s_bmax;
  const int nocc = s_nocc;
  // reweighting factors of the occupied bins, w_b = exp(-dbeta (E_b - E_min))
  for (int i = tid; i < nocc; i += NT) {
    const int b = occ[i];
    w[b] = dexp_np(-__dmul_rn(dbeta, (double)(2 * (b - bmin))));
  }
  __syncthreads();
  // Q' = sum_b n_b w_b over the fixed tree: lane l sums the terms of bins
  // l, l+32, ... in increasing order, then butterfly levels 16, 8, 4, 2, 1.
  // An empty bin adds +0.0, which leaves the sum unchanged, so the lanes may
  // run over whole windows of the occupied range [bmin, bmax].
  double acc = 0.0;
  for (int lo = bmin & ~31; lo <= bmax; lo += PREP_WIN) {
    const int span = min(PREP_WIN, bmax + 1 - lo);
    for (int t = tid; t < span; t += NT) s_term[t] = 0.0;
    __syncthreads();
    for (int i = tid; i < nocc; i += NT) {
      const int b = occ[i];
      if (b >= lo && b < lo + span) s_term[b - lo] = __dmul_rn((double)h[b], w[b]);
    }
    __syncthreads();
    if (tid < 32)
      for (int t = tid; t < span; t += 32) acc = __dadd_rn(acc, s_term[t]);
    __syncthreads();
  }
  if (tid < 32) {
#pragma unroll
    for (int sh = 16; sh >= 1; sh >>= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, sh));
    if (tid == 0) s_Qp = acc;
  }
  __syncthreads();
  const double Qp = s_Qp;
  // ln Q, the staged -beta F~ and the thresholds by the last threads, which
  // have no bin while nocc < NT - 8
  if (tid == NT - 1) {
    const int64_t Emin = 2 * (int64_t)bmin - R.Nb;
    const double lnQ = __dsub_rn(__dsub_rn(log(Qp), log((double)R.R)), __dmul_rn(dbeta, (double)Emin));
    R.lnQ_staged = lnQ;
    R.Qp_staged = Qp;
    R.mbF_staged = __dadd_rn(R.mbF, lnQ);
    R.beta_next = bn;
    R.theta_next = s_theta;
    R.Rt_next = Rt;
    R.bmin = bmin;
    R.sumE_next = 0ull;
    R.sumE2_next = 0ull;
    R.skip = 0;
  }
  if (tid >= NT - 9 && tid < NT - 1) {
    const int d = tid - (NT - 9);
    R.thr[d] = (d == 0 || d == 7) ? 0u : metropolis_threshold(bn, 2 * d);
  }
  // Poisson means a_b = R_target w_b / Q' = (R/R~) tau_j (Eq. (1)), split in
  // m = ceil(a/32) pieces when a > 32 (a / 32 and a / 1 are exact, so they
  // are taken as a product and as a itself).
  const double Rtd = (double)Rt;
  for (int i = tid; i < nocc; i += NT) {
    const int b = occ[i];
    const double a = __ddiv_rn(__dmul_rn(Rtd, w[b]), Qp);
    int64_t m = 1;
    double am = a;
    if (a > 32.0) {
      m = (int64_t)ceil(__dmul_rn(a, 0.03125));
      am = __ddiv_rn(a, (double)m);
    }
    const double p0 = dexp_np(-am);
    R.bin_am[b] = am;
    R.bin_p0[b] = p0;
    R.bin_m[b] = m;
    // the first POISSON_TAB partial sums C_k of the walk as 53-bit integer
    // thresholds (u >= C_k iff U >= ceil(C_k 2^53), u = U 2^-53), built with
    // the walk's own recurrence, and the state after the last of them
    uint64_t* tb = R.bin_thr + (size_t)b * POISSON_TAB;
    double P = p0, C = p0;
    tb[0] = cdf_threshold(C);
#pragma unroll 1
    for (int k = 1; k < POISSON_TAB; ++k) {
      P = div_small_rn(__dmul_rn(P, am), (uint32_t)k);
      C = __dadd_rn(C, P);
      tb[k] = cdf_threshold(C);
    }
    R.bin_end[2 * b] = P;
    R.bin_end[2 * b + 1] = C;
  }
  uint32_t* hn = R.hist[R.cur ^ 1];
  for (int b = tid; b < nbins; b += NT) hn[b] = 0u;
  return true;
}

__global__ void __launch_bounds__(PREP_THREADS) k_prepare(RunDev* __restrict__ runs,
                                                          const int32_t* __restrict__ ids, int use_override,
                                                          double beta_o, int theta_o, int64_t Rt_o) {
  prepare_block<PREP_THREADS>(runs[ids ? ids[blockIdx.x] : blockIdx.x], use_override, beta_o, theta_o, Rt_o);
}

// ---------------------------------------------------------------------------
// Step: Poisson copy counts (Sec. 2: N[(R/R~) tau_j] copies of replica j)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t block_sum_i64(int64_t v, int64_t* s_warp) {
#pragma unroll
  for (int sh = 16; sh >= 1; sh >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, sh);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) s_warp[wid] = v;
  __syncthreads();
  int64_t t = 0;
  if (threadIdx.x < 32) {
    t = (lane < (int)(blockDim.x >> 5)) ? s_warp[lane] : 0;
#pragma unroll
    for (int sh = 16; sh >= 1; sh >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, sh);
  }
  return t;  // valid in thread 0
}

// Exclusive block scan (int64); returns the exclusive prefix, *total in all threads.
__device__ __forceinline__ int64_t block_exscan_i64(int64_t v, int64_t* s_warp, int64_t* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int64_t x = v;
#pragma unroll
  for (int sh = 1; sh < 32; sh <<= 1) {
    const int64_t y = __shfl_up_sync(0xFFFFFFFFu, x, sh);
    if (lane >= sh) x += y;
  }
  if (lane == 31) s_warp[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int64_t s = (lane < nw) ? s_warp[lane] : 0;
#pragma unroll
    for (int sh = 1; sh < 32; sh <<= 1) {
      const int64_t y = __shfl_up_sync(0xFFFFFFFFu, s, sh);
      if (lane >= sh) s += y;
    }
    if (lane < nw) s_warp[lane] = s;  // inclusive warp totals
  }
  __syncthreads();
  const int64_t before = (wid > 0) ? s_warp[wid - 1] : 0;
  *total = s_warp[nw - 1];
  __syncthreads();
  return before + x - v;
}

// Inverse-CDF walk of one Poisson piece (mean am, P(0) = p0) for uniform u:
// P_k = (P_{k-1} am) / k, C_k = C_{k-1} + P_k, stop at the first k with
// u < C_k (or at POISSON_KMAX).  The division by k is the exact integer one
// of div_small_rn, the same double as a correctly rounded division; u and C are
// not negative, so they compare as their bits do (at_least).
__device__ __forceinline__ bool at_least(double u, double C) {
  return __double_as_longlong(u) >= __double_as_longlong(C);
}
__device__ __forceinline__ int poisson_piece(double u, double am, double p0) {
  int k = 0;
  double P = p0, C = p0;
  while (at_least(u, C) && k < POISSON_KMAX) {
    k = k + 1;
    P = div_small_rn(__dmul_rn(P, am), (uint32_t)k);
    C = __dadd_rn(C, P);
  }
  return k;
}

// Copies of one piece of replica j from its own mean.
__device__ __forceinline__ int piece_copies(const RunDev& R, int64_t j, int64_t piece, double am, double p0) {
  const u32x4 r = philox_seeded(R.seed, (uint32_t)piece, (uint32_t)j, (uint32_t)R.step, TAG_RESAMPLE);
  return poisson_piece(u53(r.a, r.b), am, p0);
}

// The same walk from a bin's table: with U the 53-bit integer of the
// uniform, the walk stops at the first k with U < thr[k]; the thresholds do
// not decrease, so that k is the number of thresholds U reaches.  Past the
// table the walk goes on from the stored state, step by step as above.
__device__ __forceinline__ int poisson_piece_tab(uint64_t U, const uint64_t* thr, double P, double C, double am) {
  const ulonglong2* t2 = reinterpret_cast<const ulonglong2*>(thr);
  int k = 0;
#pragma unroll
  for (int q = 0; q < POISSON_TAB / 2; ++q) {
    const ulonglong2 v = t2[q];
    k += (U >= v.x) + (U >= v.y);
  }
  if (k < POISSON_TAB) return k;
  const double u = __dmul_rn((double)U, 0x1.0p-53);
  k = POISSON_TAB - 1;
  while (at_least(u, C) && k < POISSON_KMAX) {
    k = k + 1;
    P = div_small_rn(__dmul_rn(P, am), (uint32_t)k);
    C = __dadd_rn(C, P);
  }
  return k;
}

// Copies of one piece of replica j from the tables of its bin b.
__device__ __forceinline__ int piece_copies_tab(const RunDev& R, int64_t j, int64_t piece, int b) {
  const u32x4 r = philox_seeded(R.seed, (uint32_t)piece, (uint32_t)j, (uint32_t)R.step, TAG_RESAMPLE);
  const uint64_t U = ((((uint64_t)r.a) << 32) | (uint64_t)r.b) >> 11;
  return poisson_piece_tab(U, R.bin_thr + (size_t)b * POISSON_TAB, R.bin_end[2 * b], R.bin_end[2 * b + 1],
                           R.bin_am[b]);
}

// Poisson pieces of replica j of a Gaussian run from its own weight (the
// arithmetic of the per-bin tables of k_prepare).
__device__ __forceinline__ void replica_poisson(RunDev& R, int64_t j, int64_t* m, double* am, double* p0) {
  double a = __ddiv_rn(__dmul_rn((double)R.Rt_next, R.w_rep[j]), R.Qp_staged);
  // w_j <= Q' makes a <= R_target (up to rounding); anything else (a stale or
  // unset weight) draws nothing and flags the run instead of sampling an
  // unbounded mean
  if (!(a <= 2.0 * (double)R.Rt_next + 1.0)) {
    R.error = ERR_INVALID;
    a = 0.0;
  }
  int64_t mm = 1;
  double a1 = a;  // a / 1 and a / 32 are exact: taken as a itself and as a product
  if (a > 32.0) {
    mm = (int64_t)ceil(__dmul_rn(a, 0.03125));
    a1 = __ddiv_rn(a, (double)mm);
  }
  *m = mm;
  *am = a1;
  *p0 = dexp_np(-a1);
}

// A replica whose mean is above this, or that needs several pieces, is left to
// the second pass of k_copies.
constexpr double LONG_MEAN = 4.0;

// Last i in [0, N) with off[i] <= t (off does not decrease): of entries of
// which some are empty, the one that holds t.
template <int N>
__device__ __forceinline__ int holder(const int64_t* off, int64_t t) {
  int i = 0;
#pragma unroll
  for (int step = N / 2; step >= 1; step >>= 1)
    if (off[i + step] <= t) i += step;
  return i;
}

// Copy counts of a chunk of replicas.  A draw is a walk of about as many
// dependent FP64 steps as copies (each instruction holds a sub-partition for 64
// cycles), so after a large temperature step a warp waits for its heaviest
// replica, and families of heavy replicas lie side by side.  So the first pass
// draws only the short walks; the pieces of all other replicas of the chunk are
// laid out one after the other and drawn by the block's threads in turn.
// L = 10, 20000 Gaussian replicas, the first 13 of 40 steps to beta = 4: 59 us a
// launch with the heavy replicas one by one and the middling ones in their own
// threads, 27 so; 1.2e6 +-1 replicas at steps of 0.2 in beta 124 -> 85.  (The
// bound of the first pass hardly matters: 2, 4 and 7 are alike within 1 %.)
__global__ void __launch_bounds__(CHUNK) k_copies(RunDev* __restrict__ runs, const Work* __restrict__ table) {
  __shared__ int64_t s_warp[CHUNK / 32];
  __shared__ int64_t s_off[CHUNK];           // first piece of each replica in the second pass
  __shared__ unsigned long long s_cnt[CHUNK];
  __shared__ double s_am[CHUNK], s_p0[CHUNK];  // Gaussian runs
  __shared__ int32_t s_bin[CHUNK];             // +-1 runs
  const Work wk = table[blockIdx.x];
  RunDev& R = runs[wk.run];
  if (R.skip) return;
  const int tid = threadIdx.x;
  const int64_t j = (int64_t)wk.first + tid;
  const int64_t Rold = R.R;
  if ((int64_t)wk.first >= Rold) {
    if (tid == 0) R.chunk_sum[wk.first / CHUNK] = 0;
    return;
  }
  int64_t c = 0, later = 0;  // copies; pieces of the second pass
  if (j < Rold) {
    if (R.model == 0) {
      const int b = (R.E[R.cur][j] + R.Nb) >> 1;
      const int64_t m = R.bin_m[b];
      s_bin[tid] = b;
      if (m > 1 || R.bin_am[b] > LONG_MEAN) later = m;
      else c = piece_copies_tab(R, j, 0, b);
    } else {
      int64_t m;
      double am, p0;
      replica_poisson(R, j, &m, &am, &p0);
      s_am[tid] = am;
      s_p0[tid] = p0;
      if (m > 1 || am > LONG_MEAN) later = m;
      else c = piece_copies(R, j, 0, am, p0);
    }
  }
  if (__syncthreads_or(later > 0)) {
    int64_t pieces;
    s_cnt[tid] = 0ull;
    s_off[tid] = block_exscan_i64(later, s_warp, &pieces);
    __syncthreads();
    for (int64_t t = tid; t < pieces; t += CHUNK) {
      const int h = holder<CHUNK>(s_off, t);
      const int64_t piece = t - s_off[h], jh = (int64_t)wk.first + h;
      const int k = R.model == 0 ? piece_copies_tab(R, jh, piece, s_bin[h]) : piece_copies(R, jh, piece, s_am[h], s_p0[h]);
      atomicAdd(&s_cnt[h], (unsigned long long)k);
    }
    __syncthreads();
    if (later > 0) c = (int64_t)s_cnt[tid];
  }
  if (j < Rold) R.copies[j] = (int32_t)(c > 0x7FFFFFFF ? 0x7FFFFFFF : c);
  const int64_t tot = block_sum_i64(c, s_warp);
  if (tid == 0) R.chunk_sum[wk.first / CHUNK] = tot;
}

// The population after resampling; a run that dies out or outgrows its buffers
// stays as it is.
__device__ __forceinline__ void set_population(RunDev& R, int64_t total) {
  R.R_next = total;
  if (total == 0) {
    R.error = ERR_EXTINCT;
    R.skip = 1;
  } else if (total > R.R_cap) {
    R.error = ERR_CAPACITY;
    R.skip = 1;
  }
}

__global__ void __launch_bounds__(CHUNK) k_scan(RunDev* __restrict__ runs, const int32_t* __restrict__ ids) {
  __shared__ int64_t s_warp[CHUNK / 32];
  RunDev& R = runs[ids ? ids[blockIdx.x] : blockIdx.x];
  if (R.skip) return;
  const int nch = (int)((R.R + CHUNK - 1) / CHUNK);
  int64_t running = 0;
  for (int base = 0; base < nch; base += CHUNK) {
    const int i = base + threadIdx.x;
    const int64_t v = (i < nch) ? R.chunk_sum[i] : 0;
    int64_t tot;
    const int64_t ex = block_exscan_i64(v, s_warp, &tot);
    if (i < nch) R.chunk_off[i] = running + ex;
    running += tot;
  }
  if (threadIdx.x == 0) set_population(R, running);
}

// Source of every new slot.  The block's threads take the new slots of the
// chunk in turn and look their replica up in the offsets: with a thread writing
// the copies of its own replica a chunk took as long as its heaviest one (279
// us at worst in a batch of 1.2e6 replicas at steps of 0.2 in beta, 60 so).
__global__ void __launch_bounds__(CHUNK) k_scatter(RunDev* __restrict__ runs, const Work* __restrict__ table) {
  __shared__ int64_t s_warp[CHUNK / 32];
  __shared__ int64_t s_off[CHUNK];
  const Work wk = table[blockIdx.x];
  RunDev& R = runs[wk.run];
  if (R.skip) return;
  const int64_t Rold = R.R;
  if ((int64_t)wk.first >= Rold) return;
  const int64_t j = (int64_t)wk.first + threadIdx.x;
  const int64_t c = (j < Rold) ? R.copies[j] : 0;
  int64_t tot;
  s_off[threadIdx.x] = block_exscan_i64(c, s_warp, &tot);
  __syncthreads();
  int32_t* __restrict__ src = R.src + R.chunk_off[wk.first / CHUNK];
  for (int64_t q = threadIdx.x; q < tot; q += CHUNK) src[q] = wk.first + holder<CHUNK>(s_off, q);
}

// The whole resampling of a +-1 run of at most SMALL_RUN replicas by one block:
// k_prepare, k_copies and k_scatter without the launches in between.  A run of
// 1000 replicas at L = 4 took 30.7 us a step with six launches (of which 12.5
// the sweep) in a graph, 24.5 with this one and the sweep.
//
// Blocks of 256 threads for populations of up to 512 slots, which leave most of a
// larger block idle, and for more runs than SMs, where several blocks of an SM hide
// one another's waits; else of 1024, which take fewer passes.  Batches of L = 4, 40
// steps, ms with the launches apart / blocks of 1024 / of 256: 1 run of 1000 replicas
// 1.24 / 0.93 / 1.03; 100 of 1000 4.47 / 3.36 / 3.50; 300 of 1000 11.0 / 8.70 / 8.35; 1000 of
// 100 9.84 / 10.7 / 8.90; 3000 of 30 21.0 / 26.7 / 21.0.
template <int NT>
__global__ void __launch_bounds__(NT) k_resample(RunDev* __restrict__ runs, const int32_t* __restrict__ ids,
                                                 int commit_first, int use_override, double beta_o, int theta_o,
                                                 int64_t Rt_o) {
  __shared__ int64_t s_warp[NT / 32];
  __shared__ int64_t s_off[NT];
  __shared__ unsigned long long s_cnt[NT];
  __shared__ int32_t s_bin[NT];
  RunDev& R = runs[ids ? ids[blockIdx.x] : blockIdx.x];
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  if (commit_first) {
    if (threadIdx.x == 0) commit_step(R);
    __syncthreads();
  }
  if (!prepare_block<NT>(R, use_override, beta_o, theta_o, Rt_o)) return;
  __syncthreads();  // the bins' tables in place
  const int tid = threadIdx.x;
  const int64_t Rold = R.R, cap = R.R_cap;
  const int32_t* E = R.E[R.cur];
  int64_t running = 0;
  for (int64_t base = 0; base < Rold; base += NT) {
    const int64_t j = base + tid;
    int64_t c = 0, later = 0;
    if (j < Rold) {
      const int b = (E[j] + R.Nb) >> 1;
      const int64_t m = R.bin_m[b];
      s_bin[tid] = b;
      if (m > 1 || R.bin_am[b] > LONG_MEAN) later = m;
      else c = piece_copies_tab(R, j, 0, b);
    }
    if (__syncthreads_or(later > 0)) {
      int64_t pieces;
      s_cnt[tid] = 0ull;
      s_off[tid] = block_exscan_i64(later, s_warp, &pieces);
      __syncthreads();
      for (int64_t t = tid; t < pieces; t += NT) {
        const int h = holder<NT>(s_off, t);
        atomicAdd(&s_cnt[h], (unsigned long long)piece_copies_tab(R, base + h, t - s_off[h], s_bin[h]));
      }
      __syncthreads();
      if (later > 0) c = (int64_t)s_cnt[tid];
    }
    const int32_t kept = (int32_t)(c > 0x7FFFFFFF ? 0x7FFFFFFF : c);
    if (j < Rold) R.copies[j] = kept;
    int64_t tot;
    const int64_t ex = block_exscan_i64(c, s_warp, &tot);
    s_off[tid] = ex;
    __syncthreads();
    // a run past its capacity is not swept: the slots it has room for are enough
    const int64_t room = cap - running;
    for (int64_t q = tid; q < tot && q < room; q += NT) R.src[running + q] = (int32_t)(base + holder<NT>(s_off, q));
    running += tot;
    __syncthreads();  // the offsets are no longer read
  }
  if (tid == 0) set_population(R, running);
}

__global__ void k_commit(RunDev* __restrict__ runs, const int32_t* __restrict__ ids, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) commit_step(runs[ids ? ids[t] : t]);
}

// ---------------------------------------------------------------------------
// Read-out
// ---------------------------------------------------------------------------
__device__ __forceinline__ void site_word_bit(const RunDev& R, int64_t i, int* w, int* p) {
  if (R.dim == 1) {
    *w = (int)(i >> 5);
    *p = (int)(i & 31);
    return;
  }
  const int Lx = R.bx > 0 ? R.bx : R.L, Ly = R.bx > 0 ? R.by : R.L, Lz = R.bx > 0 ? R.bz : R.L;
  const int K = R.bx > 0 ? R.bk : lanes_for(R.L), G = Lz / K;
  const int x = (int)(i % Lx), y = (int)((i / Lx) % Ly), z = (int)(i / ((int64_t)Lx * Ly));
  *w = y * G + z % G;
  *p = (z / G) * Lx + x;
}

// Spins of slots [0, n) as int8 +-1 in natural site order.
__global__ void k_unpack(const RunDev* __restrict__ runs, int r, int64_t n, int8_t* __restrict__ out) {
  const RunDev& R = runs[r];
  const int64_t total = n * (int64_t)R.N;
  const uint32_t* sp = R.spins[R.cur];
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = t / R.N, i = t % R.N;
    int w, p;
    site_word_bit(R, i, &w, &p);
    const uint32_t bit = (sp[s * R.W + w] >> p) & 1u;
    out[t] = bit ? (int8_t)-1 : (int8_t)1;
  }
}

// Sec. 4 overlap: replica k of run a against replica k of run b.
__global__ void k_overlap(const RunDev* __restrict__ pa_, const RunDev* __restrict__ pb_, double qcut,
                          unsigned long long* __restrict__ count, unsigned long long* __restrict__ hist) {
  const RunDev& A = *pa_;
  const RunDev& B = *pb_;
  const int64_t n = A.R < B.R ? A.R : B.R;
  const int W = A.W;
  const double lim = __dmul_rn(qcut, (double)A.N);
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t* a = A.spins[A.cur] + k * W;
    const uint32_t* b = B.spins[B.cur] + k * W;
    int diff = 0;
    for (int w = 0; w < W; ++w) diff += __popc(a[w] ^ b[w]);
    const int dot = A.N - 2 * diff;
    if (fabs((double)dot) < lim) atomicAdd(count, 1ull);
    if (hist) atomicAdd(&hist[(dot + A.N) >> 1], 1ull);
  }
}

// Sec. 4 overlap for many pairs of runs of one batch at once: pair p counts
// the replicas k < min(R~_a, R~_b) with |q_k| < qcut, q_k the overlap of
// replica k of run ra[p] with replica k of run rb[p] (blockIdx.y = pair).
__global__ void k_overlap_pairs(const RunDev* __restrict__ runs, const int32_t* __restrict__ ra,
                                const int32_t* __restrict__ rb, int n_pairs, double qcut,
                                unsigned long long* __restrict__ count) {
  const int p = blockIdx.y;
  if (p >= n_pairs) return;
  const RunDev& A = runs[ra[p]];
  const RunDev& B = runs[rb[p]];
  const int64_t n = A.R < B.R ? A.R : B.R;
  const int W = A.W;
  const double lim = __dmul_rn(qcut, (double)A.N);
  unsigned long long local = 0ull;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t* a = A.spins[A.cur] + k * W;
    const uint32_t* b = B.spins[B.cur] + k * W;
    int diff = 0;
    for (int w = 0; w < W; ++w) diff += __popc(a[w] ^ b[w]);
    const int dot = A.N - 2 * diff;
    if (fabs((double)dot) < lim) ++local;
  }
#pragma unroll
  for (int sh = 16; sh >= 1; sh >>= 1) local += __shfl_xor_sync(0xFFFFFFFFu, local, sh);
  if ((threadIdx.x & 31) == 0 && local) atomicAdd(&count[p], local);
}

// Histogram of the overlap for each pair of runs (Sec. 4, P(q)): bin
// (N q + N) / 2 = N - (sites that differ) of replica k of run ra[p] against
// replica k of run rb[p], k < min(R~_a, R~_b), counted in shared memory
// (N + 1 bins) and added to hist[p][.].
__global__ void k_overlap_hist(const RunDev* __restrict__ runs, const int32_t* __restrict__ ra,
                               const int32_t* __restrict__ rb, int n_pairs, int nbins,
                               unsigned long long* __restrict__ hist) {
  extern __shared__ uint32_t s_bins[];
  const int p = blockIdx.y;
  if (p >= n_pairs) return;
  for (int i = threadIdx.x; i < nbins; i += blockDim.x) s_bins[i] = 0u;
  __syncthreads();
  const RunDev& A = runs[ra[p]];
  const RunDev& B = runs[rb[p]];
  const int64_t n = A.R < B.R ? A.R : B.R;
  const int W = A.W, N = A.N;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t* a = A.spins[A.cur] + k * W;
    const uint32_t* b = B.spins[B.cur] + k * W;
    int diff = 0;
    for (int w = 0; w < W; ++w) diff += __popc(a[w] ^ b[w]);
    const int bin = N - diff;  // unused bits of the words are zero, so 0 <= bin <= N
    if (bin >= 0) atomicAdd(&s_bins[bin], 1u);
  }
  __syncthreads();
  unsigned long long* hp = hist + (size_t)p * nbins;
  for (int i = threadIdx.x; i < nbins; i += blockDim.x)
    if (s_bins[i]) atomicAdd(&hp[i], (unsigned long long)s_bins[i]);
}

cudaError_t launch_overlap_hist(const RunDev* runs, const int32_t* ra, const int32_t* rb, int n_pairs, int nbins,
                                unsigned long long* hist, cudaStream_t st) {
  if (n_pairs <= 0) return cudaSuccess;
  dim3 grid(16, n_pairs);
  k_overlap_hist<<<grid, 256, sizeof(uint32_t) * (size_t)nbins, st>>>(runs, ra, rb, n_pairs, nbins, hist);
  return cudaGetLastError();
}

cudaError_t launch_overlap_pairs(const RunDev* runs, const int32_t* ra, const int32_t* rb, int n_pairs, double qcut,
                                 unsigned long long* count, cudaStream_t st) {
  if (n_pairs <= 0) return cudaSuccess;
  dim3 grid(16, n_pairs);
  k_overlap_pairs<<<grid, 256, 0, st>>>(runs, ra, rb, n_pairs, qcut, count);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Sec. 3 weighted averages: a warp or a block per group of M runs.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int sh = 16; sh >= 1; sh >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, sh));
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int sh = 16; sh >= 1; sh >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xFFFFFFFFu, v, sh));
  return v;
}

// Sum or maximum of v over a block of NT threads, in every thread; s_part: one
// value a warp.
template <int NT, bool MAX>
__device__ __forceinline__ double block_fold(double v, double* s_part) {
  v = MAX ? warp_max(v) : warp_sum(v);
  if constexpr (NT > 32) {
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
    __syncthreads();
    v = s_part[0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) v = MAX ? fmax(v, s_part[w]) : v + s_part[w];
    __syncthreads();  // s_part may be written again
  }
  return v;
}

// PAIRS: Sec. 4, Eq. (11) -- an observable of two independent runs
// (the overlap) is averaged over M pairs with weights e^{-beta (F~1 + F~2)}
// (R1 R2 e^{...} with the population factors of Eq. (6)), and fbar is
// ln[(1/M) sum_r e^{x1_r + x2_r}].  Otherwise x2 and Rw2 are unused.
//
// One block of NT threads per group.  A logarithm or an exponential is some 25
// dependent FP64 instructions of 64 cycles, so a lone group is bound by how
// many of them a thread does in turn: M = 200 takes 52 us (pairs) and 33 with a
// warp, 16 and 14 with 256 threads, which keep their first value instead of
// computing it again.
template <bool PAIRS, int NT>
__global__ void __launch_bounds__(NT) k_weighted(int M, const double* __restrict__ x, const double* __restrict__ x2,
                                                 const double* __restrict__ A, const double* __restrict__ Rw,
                                                 const double* __restrict__ Rw2, double* __restrict__ mean,
                                                 double* __restrict__ fbar) {
  __shared__ double s_part[NT / 32];
  const int g = blockIdx.x, t = threadIdx.x;
  const double* xg = x + (int64_t)g * M;
  const double* x2g = PAIRS ? x2 + (int64_t)g * M : nullptr;
  const double* Ag = A ? A + (int64_t)g * M : nullptr;
  const double* Rg = Rw ? Rw + (int64_t)g * M : nullptr;
  const double* R2g = (PAIRS && Rw2) ? Rw2 + (int64_t)g * M : nullptr;
  auto xr = [&](int r) { return PAIRS ? xg[r] + x2g[r] : xg[r]; };
  auto yr = [&](int r) {
    double y = xr(r);
    if (Rg) y = y + log(Rg[r]);
    if (PAIRS && R2g) y = y + log(R2g[r]);
    return y;
  };
  double mu = -INFINITY, mux = -INFINITY, y0 = 0.0;
  for (int r = t; r < M; r += NT) {
    const double y = yr(r);
    if (r == t) y0 = y;
    mu = fmax(mu, y);
    mux = fmax(mux, xr(r));
  }
  mu = block_fold<NT, true>(mu, s_part);
  mux = block_fold<NT, true>(mux, s_part);
  double S = 0.0, SA = 0.0, Sx = 0.0;
  for (int r = t; r < M; r += NT) {
    const double e = exp((r == t ? y0 : yr(r)) - mu);
    S += e;
    if (Ag) SA += e * Ag[r];
    Sx += exp(xr(r) - mux);
  }
  S = block_fold<NT, false>(S, s_part);
  SA = block_fold<NT, false>(SA, s_part);
  Sx = block_fold<NT, false>(Sx, s_part);
  if (t == 0) {
    mean[g] = Ag ? SA / S : 0.0;
    fbar[g] = mux + log(Sx) - log((double)M);
  }
}

// Weights of the runs of each group for k_bootstrap, one block per group: with y
// = x + ln R, tab[gk] = {e^{y_k - max y}, e^{y_k - max y} A_k, e^{x_k - max x}} for
// the M runs, then max x.  HAS_A, HAS_R: whether A and Rw are given.
constexpr int BOOT_WEIGHT_THREADS = 256;  // M = 200, one group: 24 us with a warp, 9 so
template <bool HAS_A, bool HAS_R>
__global__ void __launch_bounds__(BOOT_WEIGHT_THREADS) k_boot_weights(int M, const double* __restrict__ x,
                                                                      const double* __restrict__ A,
                                                                      const double* __restrict__ Rw,
                                                                      double* __restrict__ tab) {
  constexpr int NT = BOOT_WEIGHT_THREADS;
  __shared__ double s_part[NT / 32];
  const int gk = blockIdx.x, first = threadIdx.x;
  const double* xg = x + (int64_t)gk * M;
  double* t = tab + (int64_t)gk * (3 * (int64_t)M + 1);
  double mu = -INFINITY, mux = -INFINITY;
  for (int k = first; k < M; k += NT) {
    double y = xg[k];
    if constexpr (HAS_R) y += log(Rw[(int64_t)gk * M + k]);
    t[k] = y;
    mu = fmax(mu, y);
    mux = fmax(mux, xg[k]);
  }
  mu = block_fold<NT, true>(mu, s_part);
  mux = block_fold<NT, true>(mux, s_part);
  for (int k = first; k < M; k += NT) {  // the thread's own y
    const double e = exp(t[k] - mu);
    t[k] = e;
    if constexpr (HAS_A) t[(int64_t)M + k] = e * A[(int64_t)gk * M + k];
    else t[(int64_t)M + k] = 0.0;
    if constexpr (HAS_R) t[2 * (int64_t)M + k] = exp(xg[k] - mux);
    else t[2 * (int64_t)M + k] = e;  // without population factors y = x
  }
  if (first == 0) t[3 * (int64_t)M] = mux;
}

// Sec. 3 bootstrap: resample b draws index floor(word0 * M / 2^32) of
// Philox(ctr = (b, i, 0, TAG_BOOT)); LANES threads per resample take its draws
// in turn.  GK groups of M values each (x, A, Rw laid out [GK][M]) are resampled with the same draws;
// the results are laid out [GK][B].
//
// tab: the weights of k_boot_weights (nullptr: none).  With them a draw is its
// generator call, three loads and three FP64 additions; without, two
// exponentials and two logarithms, some 25 FP64 instructions of 64 cycles each
// (M = 200, B = 1000: 785 us with one thread a resample, 46 with tables, 11
// with eight threads, which spread 1000 resamples over more than 8 SMs).  A
// resample that misses the runs that carry the weight (all of its weights below
// 1e-200 of the largest) is summed by its first thread against its own largest
// value all the same.
template <int LANES>
__global__ void k_bootstrap(int M, const double* __restrict__ x, const double* __restrict__ A,
                            const double* __restrict__ Rw, const double* __restrict__ tab, int B, uint64_t seed,
                            int GK, double* __restrict__ bmean, double* __restrict__ bfbar) {
  const int64_t at = boot_resample(blockIdx.x, blockDim.x, threadIdx.x, LANES);
  const int lane = threadIdx.x % LANES, b = (int)min(at, (int64_t)B - 1);  // the threads past the last resample draw it again and write nothing
  for (int gk = blockIdx.y; gk < GK; gk += gridDim.y) {
    double S = 0.0, SA = 0.0, Sx = 0.0, mux = -INFINITY;
    bool direct = true;
    if (tab) {
      const double* t = tab + (int64_t)gk * (3 * (int64_t)M + 1);
      for (int i = lane; i < M; i += LANES) {
        const u32x4 r = philox_seeded(seed, (uint32_t)b, (uint32_t)i, 0u, TAG_BOOT);
        const int k = (int)(((uint64_t)r.a * (uint64_t)M) >> 32);
        S += t[k];
        SA += t[(int64_t)M + k];
        Sx += t[2 * (int64_t)M + k];
      }
#pragma unroll
      for (int sh = LANES / 2; sh >= 1; sh >>= 1) {
        S += __shfl_xor_sync(0xFFFFFFFFu, S, sh);
        SA += __shfl_xor_sync(0xFFFFFFFFu, SA, sh);
        Sx += __shfl_xor_sync(0xFFFFFFFFu, Sx, sh);
      }
      mux = t[3 * (int64_t)M];
      direct = S < 1e-200 || Sx < 1e-200;
    }
    if (lane != 0 || at >= B) continue;
    if (direct) {
      const double* xg = x + (int64_t)gk * M;
      const double* Ag = A ? A + (int64_t)gk * M : nullptr;
      const double* Rg = Rw ? Rw + (int64_t)gk * M : nullptr;
      double mu = -INFINITY;
      mux = -INFINITY;
      for (int i = 0; i < M; ++i) {
        const u32x4 r = philox_seeded(seed, (uint32_t)b, (uint32_t)i, 0u, TAG_BOOT);
        const int k = (int)(((uint64_t)r.a * (uint64_t)M) >> 32);
        const double y = Rg ? xg[k] + log(Rg[k]) : xg[k];
        mu = fmax(mu, y);
        mux = fmax(mux, xg[k]);
      }
      S = SA = Sx = 0.0;
      for (int i = 0; i < M; ++i) {
        const u32x4 r = philox_seeded(seed, (uint32_t)b, (uint32_t)i, 0u, TAG_BOOT);
        const int k = (int)(((uint64_t)r.a * (uint64_t)M) >> 32);
        const double y = Rg ? xg[k] + log(Rg[k]) : xg[k];
        const double e = exp(y - mu);
        S += e;
        if (Ag) SA += e * Ag[k];
        Sx += exp(xg[k] - mux);
      }
    }
    bmean[(int64_t)gk * B + b] = A ? SA / S : 0.0;
    bfbar[(int64_t)gk * B + b] = mux + log(Sx) - log((double)M);
  }
}

// Self-check of div_small_rn: n pairs (x, k) with x from 63 random bits
// (every exponent, zero, subnormals, infinities and NaNs) and k uniform in
// 1..POISSON_KMAX, each compared bit for bit with the division instruction;
// the number of differing pairs is added to *mismatches.
__global__ void k_check_division(int64_t n, uint64_t seed, unsigned long long* __restrict__ mismatches) {
  unsigned long long bad = 0ull;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const u32x4 r = philox_seeded(seed, (uint32_t)i, (uint32_t)(i >> 32), 0u, 0x44495643u);
    const uint64_t bits = ((((uint64_t)r.a) << 32) | r.b) & 0x7FFFFFFFFFFFFFFFull;
    // half of the draws keep the exponent within 2^-60..2^6, where the walk's
    // terms P_k am live
    const uint64_t xb = (r.d & 1u) ? bits : ((bits & 0x800FFFFFFFFFFFFFull) | ((uint64_t)(963 + r.d % 67u) << 52));
    const double x = __longlong_as_double((long long)xb);
    const uint32_t k = 1u + r.c % (uint32_t)POISSON_KMAX;
    const double q = div_small_rn(x, k), qd = __ddiv_rn(x, (double)k);
    if (__double_as_longlong(q) != __double_as_longlong(qd)) bad += 1ull;
  }
#pragma unroll
  for (int sh = 16; sh >= 1; sh >>= 1) bad += __shfl_xor_sync(0xFFFFFFFFu, bad, sh);
  if ((threadIdx.x & 31) == 0 && bad) atomicAdd(mismatches, bad);
}

// Self-check of the deterministic exponentials against CUDA's exp and expf:
// n seeded points, x uniform in [-745, 0] for dexp_np and in [-103, 0] for
// fexp_np; the largest distance in units in the last place of the CUDA value
// (both are finite and positive there; zero results count as 0 ulp apart
// only if both are zero).  out[0] = max ulp of dexp_np, out[1] = of fexp_np.
__device__ __forceinline__ unsigned long long ulp_distance_d(double a, double b) {
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  return (unsigned long long)(ia > ib ? ia - ib : ib - ia);  // same sign, finite
}

__global__ void k_check_exp(int64_t n, uint64_t seed, unsigned long long* __restrict__ out) {
  unsigned long long md = 0ull, mf = 0ull;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const u32x4 r = philox_seeded(seed, (uint32_t)i, (uint32_t)(i >> 32), 0u, 0x45585043u);
    const double xd = -745.0 * u53(r.a, r.b);
    const float xf = -103.0f * ((float)(r.c >> 8) * 0x1.0p-24f);
    md = max(md, ulp_distance_d(dexp_np(xd), exp(xd)));
    const int fa = __float_as_int(fexp_np(xf)), fb = __float_as_int(expf(xf));
    mf = max(mf, (unsigned long long)(fa > fb ? fa - fb : fb - fa));
  }
#pragma unroll
  for (int sh = 16; sh >= 1; sh >>= 1) {
    md = max(md, __shfl_xor_sync(0xFFFFFFFFu, md, sh));
    mf = max(mf, __shfl_xor_sync(0xFFFFFFFFu, mf, sh));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&out[0], md);
    atomicMax(&out[1], mf);
  }
}

cudaError_t launch_check_exp(int64_t n, uint64_t seed, unsigned long long* out, cudaStream_t st) {
  k_check_exp<<<152 * 4, 256, 0, st>>>(n, seed, out);
  return cudaGetLastError();
}

cudaError_t launch_check_division(int64_t n, uint64_t seed, unsigned long long* mismatches, cudaStream_t st) {
  k_check_division<<<152 * 8, 256, 0, st>>>(n, seed, mismatches);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Host-side launchers
// ---------------------------------------------------------------------------
cudaError_t set_exp_coefficients() {
  double c[DEXP_DEGREE + 1];
  c[0] = 1.0;
  for (int j = 1; j <= DEXP_DEGREE; ++j) c[j] = c[j - 1] / (double)j;
  cudaError_t e = cudaMemcpyToSymbol(c_dexp_coef, c, sizeof c);
  if (e != cudaSuccess) return e;
  // reciprocals floor(2^64 / k) of div_small_rn: (2^64 - 1) div k, plus one
  // where k divides 2^64
  uint64_t r[POISSON_KMAX + 1] = {0u, 0u};
  for (uint64_t k = 2; k <= (uint64_t)POISSON_KMAX; ++k) r[k] = ~0ull / k + ((~0ull % k) == k - 1u ? 1u : 0u);
  return cudaMemcpyToSymbol(c_recip_k, r, sizeof r);
}

cudaError_t launch_setup_bonds3d(const int8_t* J, int L, uint32_t* bonds, int W, cudaStream_t st) {
  const int K = lanes_for(L), G = L / K;
  k_setup_bonds3d<<<(W + 127) / 128, 128, 0, st>>>(J, L, K, G, W, bonds);
  return cudaGetLastError();
}
cudaError_t launch_setup_bonds1d(const int8_t* J, int N, uint32_t* bonds, int W, cudaStream_t st) {
  k_setup_bonds1d<<<(W + 127) / 128, 128, 0, st>>>(J, N, W, bonds);
  return cudaGetLastError();
}
cudaError_t launch_init_state(RunDev* runs, const int32_t* ids, int n, int max_bins, cudaStream_t st) {
  k_init_state<<<(n + 127) / 128, 128, 0, st>>>(runs, ids, n);
  dim3 g((max_bins + 255) / 256, n);
  k_zero_hist<<<g, 256, 0, st>>>(runs, ids, n, 0);
  return cudaGetLastError();
}
cudaError_t launch_init_finish(RunDev* runs, const int32_t* ids, int n, cudaStream_t st) {
  k_init_finish<<<(n + 127) / 128, 128, 0, st>>>(runs, ids, n);
  return cudaGetLastError();
}
cudaError_t launch_prepare(RunDev* runs, const int32_t* ids, int n, bool ovr, double beta, int theta,
                           int64_t Rt, cudaStream_t st) {
  k_prepare<<<n, PREP_THREADS, 0, st>>>(runs, ids, ovr ? 1 : 0, beta, theta, Rt);
  return cudaGetLastError();
}
cudaError_t launch_resample(int threads, RunDev* runs, const int32_t* ids, int n, bool commit_first, bool ovr,
                            double beta, int theta, int64_t Rt, cudaStream_t st) {
  return launch_dependent(threads == 256 ? k_resample<256> : k_resample<1024>, n, threads, (size_t)0, st, runs, ids,
                          commit_first ? 1 : 0, ovr ? 1 : 0, beta, theta, Rt);
}
cudaError_t launch_copies(RunDev* runs, const Work* table, int nwork, cudaStream_t st) {
  k_copies<<<nwork, CHUNK, 0, st>>>(runs, table);
  return cudaGetLastError();
}
cudaError_t launch_scan(RunDev* runs, const int32_t* ids, int n, cudaStream_t st) {
  k_scan<<<n, CHUNK, 0, st>>>(runs, ids);
  return cudaGetLastError();
}
cudaError_t launch_scatter(RunDev* runs, const Work* table, int nwork, cudaStream_t st) {
  k_scatter<<<nwork, CHUNK, 0, st>>>(runs, table);
  return cudaGetLastError();
}
cudaError_t launch_commit(RunDev* runs, const int32_t* ids, int n, cudaStream_t st) {
  k_commit<<<(n + 127) / 128, 128, 0, st>>>(runs, ids, n);
  return cudaGetLastError();
}
cudaError_t launch_unpack(const RunDev* runs, int r, int64_t n, int8_t* out, cudaStream_t st) {
  k_unpack<<<1216, 256, 0, st>>>(runs, r, n, out);
  return cudaGetLastError();
}
cudaError_t launch_overlap(const RunDev* a, const RunDev* b, double qcut, unsigned long long* count,
                           unsigned long long* hist, cudaStream_t st) {
  k_overlap<<<608, 256, 0, st>>>(a, b, qcut, count, hist);
  return cudaGetLastError();
}
// Per-step records of groups of M consecutive runs as [G][count][M] arrays:
// x = -beta F~, A = E_mean (physical units), Rw = the target population of
// the step that produced the record (R0 for the initial state).
__global__ void k_gather_records(const RunDev* __restrict__ runs, int M, int count, int G, double* __restrict__ x,
                                 double* __restrict__ A, double* __restrict__ Rw) {
  const int64_t total = (int64_t)G * count * M;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % M), k = (int)((t / M) % count), g = (int)(t / ((int64_t)M * count));
    const RunDev& R = runs[g * M + i];
    const double unit = R.model == 1 ? 0x1.0p-15 : 1.0;
    x[t] = R.rec_mbF[k];
    A[t] = __ddiv_rn(__dmul_rn((double)R.rec_sumE[k], unit), (double)R.rec_R[k]);
    Rw[t] = k == 0 ? (double)R.rec_R[0] : (double)R.sched_R[k - 1];
  }
}

// Var(x) over each group of M values (ddof 1), two passes (mean, then squared
// deviations), each summed lane-strided and by the butterfly; root = 1 gives
// the standard deviation instead.
__global__ void __launch_bounds__(32) k_variance(int M, const double* __restrict__ x, double* __restrict__ var,
                                                 int root) {
  const int g = blockIdx.x, lane = threadIdx.x;
  const double* xg = x + (int64_t)g * M;
  double s = 0.0;
  for (int r = lane; r < M; r += 32) s += xg[r];
  const double m = warp_sum(s) / (double)M;
  double v = 0.0;
  for (int r = lane; r < M; r += 32) v += (xg[r] - m) * (xg[r] - m);
  v = warp_sum(v);
  if (lane == 0) {
    const double w = M > 1 ? v / (double)(M - 1) : 0.0;
    var[g] = root ? sqrt(w) : w;
  }
}

cudaError_t launch_gather_records(const RunDev* runs, int M, int count, int G, double* x, double* A, double* Rw,
                                  cudaStream_t st) {
  const int64_t total = (int64_t)G * count * M;
  const int blocks = (int)std::min<int64_t>((total + 255) / 256, 4096);
  k_gather_records<<<blocks > 0 ? blocks : 1, 256, 0, st>>>(runs, M, count, G, x, A, Rw);
  return cudaGetLastError();
}
cudaError_t launch_variance(int G, int M, const double* x, double* var, cudaStream_t st, bool root) {
  k_variance<<<G, 32, 0, st>>>(M, x, var, root ? 1 : 0);
  return cudaGetLastError();
}

// A block of 256 threads a group or a warp.  A block shortens the chain of a
// thread but holds an SM's FP64 pipe with what its warps repeat (the folds, the
// last logarithms), so the more groups an SM has, the longer they have to be for it;
// terms: logarithms and exponentials of a group.  us, a warp / a block: 152 groups of 33
// 14.7 / 12.6, of 1000 121 / 37; 304 of 64 14.5 / 16.7, of 100 22.8 / 18.8; 400 of 200 31.8 /
// 33.0, of 400 53.5 / 49.4; 608 of 64 14.7 / 29.0, of 400 57.7 / 63.8, of 1000 135 / 129.
static bool weighted_by_block(int G, int M, bool pairs) {
  const int64_t terms = (int64_t)M * (pairs ? 2 : 1);
  return M > 32 && (G <= 152 || (G <= 304 && terms >= 100) || (G <= 456 && terms >= 400) || (G <= 608 && terms >= 800));
}
template <bool PAIRS>
static cudaError_t launch_weighted_t(int G, int M, const double* x1, const double* x2, const double* A,
                                     const double* R1, const double* R2, double* mean, double* fbar, cudaStream_t st) {
  if (weighted_by_block(G, M, PAIRS)) k_weighted<PAIRS, 256><<<G, 256, 0, st>>>(M, x1, x2, A, R1, R2, mean, fbar);
  else k_weighted<PAIRS, 32><<<G, 32, 0, st>>>(M, x1, x2, A, R1, R2, mean, fbar);
  return cudaGetLastError();
}
cudaError_t launch_weighted(int G, int M, const double* x, const double* A, const double* Rw, double* mean,
                            double* fbar, cudaStream_t st) {
  return launch_weighted_t<false>(G, M, x, nullptr, A, Rw, nullptr, mean, fbar, st);
}
cudaError_t launch_weighted_pairs(int G, int M, const double* x1, const double* x2, const double* A,
                                  const double* R1, const double* R2, double* mean, double* fbar, cudaStream_t st) {
  return launch_weighted_t<true>(G, M, x1, x2, A, R1, R2, mean, fbar, st);
}
// A thread a resample, or eight.  Eight spread a few resamples over more SMs and
// share a long one's draws, but leave lanes idle in resamples of fewer runs than
// that and repeat their folds.  Up to three runs are summed directly: the table
// saves less than its launch takes.  us of a call without population factors,
// direct / table and eight threads / now: M = 2, B = 20000 104 / 130 / 106; M = 4, B = 20000
// 108 / 128 / 105; M = 8, B = 1e5 402 / 461 / 342; a batch's 1600 groups of M = 1, B = 1000
// 640 / 2156 / 622, its 4000 of M = 8 6759 / 5360 / 1067.
template <int LANES>
static void bootstrap_lanes(int M, const double* x, const double* A, const double* Rw, const double* tab, int B,
                            uint64_t seed, int GK, double* bmean, double* bfbar, cudaStream_t st) {
  constexpr unsigned PER_BLOCK = 128 / LANES;
  const dim3 grid(((unsigned)B + PER_BLOCK - 1) / PER_BLOCK, (unsigned)std::min(GK, 65535));
  k_bootstrap<LANES><<<grid, 128, 0, st>>>(M, x, A, Rw, tab, B, seed, GK, bmean, bfbar);
}
cudaError_t launch_bootstrap(int M, const double* x, const double* A, const double* Rw, int B, uint64_t seed,
                             double* bmean, double* bfbar, double* tab, cudaStream_t st, int GK) {
  if (M <= 3) tab = nullptr;
  if (tab) {
    if (A && Rw) k_boot_weights<true, true><<<GK, BOOT_WEIGHT_THREADS, 0, st>>>(M, x, A, Rw, tab);
    else if (A) k_boot_weights<true, false><<<GK, BOOT_WEIGHT_THREADS, 0, st>>>(M, x, A, Rw, tab);
    else if (Rw) k_boot_weights<false, true><<<GK, BOOT_WEIGHT_THREADS, 0, st>>>(M, x, A, Rw, tab);
    else k_boot_weights<false, false><<<GK, BOOT_WEIGHT_THREADS, 0, st>>>(M, x, A, Rw, tab);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const bool shared = tab && (M >= 16 || (M >= 8 && (int64_t)GK * B <= 4096));
  if (shared) bootstrap_lanes<8>(M, x, A, Rw, tab, B, seed, GK, bmean, bfbar, st);
  else bootstrap_lanes<1>(M, x, A, Rw, tab, B, seed, GK, bmean, bfbar, st);
  return cudaGetLastError();
}


// ---------------------------------------------------------------------------
// Gaussian couplings: Q' over replicas (fixed two-level tree)
//   level 1: chunk c of 256 slots: lane l sums w_j, j = 256c + l + 32i,
//            i = 0..7 (j < R~), in increasing i; butterfly 16, 8, 4, 2, 1;
//   level 2: lane l sums the chunk sums c = l, l+32, ... in increasing c;
//            butterfly 16, 8, 4, 2, 1.
// w_j = exp(-dbeta * (E_j - E_min) * 2^-15) with the deterministic exp.
// ---------------------------------------------------------------------------
__global__ void k_gprep_head(RunDev* __restrict__ runs, const int32_t* __restrict__ ids, int n, int use_override,
                             double beta_o, int theta_o, int64_t Rt_o) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  RunDev& R = runs[ids ? ids[t] : t];
  int ok = 1;
  double bn = 0.0;
  int th = 0;
  int64_t Rt = 0;
  if (R.error) {
    ok = 0;
  } else if (use_override) {
    bn = beta_o < 0.0 ? R.beta : beta_o;
    th = theta_o;
    Rt = Rt_o < 0 ? R.R : Rt_o;
  } else if (R.step >= R.n_sched || R.step >= R.max_steps) {
    ok = 0;
  } else {
    bn = R.sched_beta[R.step];
    th = R.sched_theta[R.step];
    Rt = R.sched_R[R.step];
  }
  if (ok && (!(bn >= R.beta) || th < 0 || Rt < 1)) {
    R.error = ERR_INVALID;
    ok = 0;
  }
  R.skip = ok ? 0 : 1;
  if (!ok) return;
  R.beta_next = bn;
  R.theta_next = th;
  R.Rt_next = Rt;
  R.sumE_next = 0ull;
  R.sumE2_next = 0ull;
  R.sumE2hi_next = 0ull;
  R.emin_next = 0x7FFFFFFFFFFFFFFFll;
}

__global__ void __launch_bounds__(CHUNK) k_gweights(RunDev* __restrict__ runs, const Work* __restrict__ table) {
  __shared__ double s_w[CHUNK];
  const Work wk = table[blockIdx.x];
  RunDev& R = runs[wk.run];
  if (R.skip) return;
  const int64_t Rold = R.R;
  if ((int64_t)wk.first >= Rold) return;
  const int64_t j = (int64_t)wk.first + threadIdx.x;
  const double dbeta = __dsub_rn(R.beta_next, R.beta);
  double w = 0.0;
  if (j < Rold) {
    const double de = __dmul_rn((double)((long long)R.E[R.cur][j] - R.emin), GAUSS_INV_SCALE_D);
    w = dexp_np(-__dmul_rn(dbeta, de));
    R.w_rep[j] = w;
  }
  s_w[threadIdx.x] = w;
  __syncthreads();
  if (threadIdx.x < 32) {
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < CHUNK / 32; ++i)
      if (wk.first + threadIdx.x + 32 * i < Rold) acc = __dadd_rn(acc, s_w[threadIdx.x + 32 * i]);
#pragma unroll
    for (int sh = 16; sh >= 1; sh >>= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, sh));
    if (threadIdx.x == 0) R.chunk_q[wk.first / CHUNK] = acc;
  }
}

__global__ void __launch_bounds__(32) k_gprep_tail(RunDev* __restrict__ runs, const int32_t* __restrict__ ids) {
  RunDev& R = runs[ids ? ids[blockIdx.x] : blockIdx.x];
  if (R.skip) return;
  const int lane = threadIdx.x;
  const int nch = (int)((R.R + CHUNK - 1) / CHUNK);
  double acc = 0.0;
  for (int c = lane; c < nch; c += 32) acc = __dadd_rn(acc, R.chunk_q[c]);
#pragma unroll
  for (int sh = 16; sh >= 1; sh >>= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, sh));
  if (lane == 0) {
    const double Qp = acc;
    const double dbeta = __dsub_rn(R.beta_next, R.beta);
    const double emin = __dmul_rn((double)R.emin, GAUSS_INV_SCALE_D);
    const double lnQ = __dsub_rn(__dsub_rn(log(Qp), log((double)R.R)), __dmul_rn(dbeta, emin));
    R.lnQ_staged = lnQ;
    R.Qp_staged = Qp;
    R.mbF_staged = __dadd_rn(R.mbF, lnQ);
  }
}

// Gaussian coupling tables of a 3D cubic lattice from int32 J[3][N]: for
// colour c, word w and rank m of the colour-c site in the word, the couplings
// of its six bonds (x+, x-, y+, y-, z+, z-) and their sum; ranks padded with
// zeros to SP, a multiple of 4.
__global__ void k_setup_gauss3d(const int32_t* __restrict__ J, int L, int K, int G, int32_t* __restrict__ gJ,
                                int32_t* __restrict__ gS) {
  const int WR = L * G, SITES = K * L / 2, SP = (SITES + 3) & ~3, N = L * L * L;
  const int total = 2 * WR * SP;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int m = t % SP, w = (t / SP) % WR, c = t / (SP * WR);
    int32_t v[6] = {0, 0, 0, 0, 0, 0};
    if (m < SITES) {
      const int j = m / (L / 2), xh = m % (L / 2);
      const int y = w / G, g = w % G, z = g + j * G;
      const int x = 2 * xh + ((c + y + z) & 1);
      const int i = x + L * (y + L * z);
      v[0] = J[i];
      v[1] = J[((x + L - 1) % L) + L * (y + L * z)];
      v[2] = J[N + i];
      v[3] = J[N + x + L * (((y + L - 1) % L) + L * z)];
      v[4] = J[2 * N + i];
      v[5] = J[2 * N + x + L * (y + L * ((z + L - 1) % L))];
    }
    int32_t sum = 0;
    for (int d = 0; d < 6; ++d) {
      gJ[((c * 6 + d) * WR + w) * SP + m] = v[d];
      sum += v[d];
    }
    gS[(c * WR + w) * SP + m] = sum;
  }
}

cudaError_t launch_setup_gauss3d(const int32_t* J, int L, int32_t* gJ, int32_t* gS, cudaStream_t st) {
  const int K = lanes_for(L), G = L / K;
  const int total = 2 * L * G * (((K * L / 2) + 3) & ~3);
  k_setup_gauss3d<<<(total + 255) / 256, 256, 0, st>>>(J, L, K, G, gJ, gS);
  return cudaGetLastError();
}
cudaError_t launch_gprep_head(RunDev* runs, const int32_t* ids, int n, bool ovr, double beta, int theta, int64_t Rt,
                              cudaStream_t st) {
  k_gprep_head<<<(n + 127) / 128, 128, 0, st>>>(runs, ids, n, ovr ? 1 : 0, beta, theta, Rt);
  return cudaGetLastError();
}
cudaError_t launch_gweights(RunDev* runs, const Work* table, int nwork, cudaStream_t st) {
  k_gweights<<<nwork, CHUNK, 0, st>>>(runs, table);
  return cudaGetLastError();
}
cudaError_t launch_gprep_tail(RunDev* runs, const int32_t* ids, int n, cudaStream_t st) {
  k_gprep_tail<<<n, 32, 0, st>>>(runs, ids);
  return cudaGetLastError();
}

}  // namespace pa
