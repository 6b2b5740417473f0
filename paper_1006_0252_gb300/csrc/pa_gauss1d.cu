// pa_gauss1d.cu -- fused replica copy + checkerboard Metropolis sweeps +
// energy measurement for chains with Gaussian couplings (Sec. 4: the periodic
// 1D spin glass the paper compares with exact transfer matrices).
//
// Bit p of word w of a replica is site 32 w + p; colour = site parity.  The
// couplings J_q[i] (bond i -> i+1, J_q[N-1] the wrap bond, 0 = absent) are
// int32.  As in the +-1 chain kernel a block keeps its replicas split by
// colour: the 16 colour-c sites 32 w + 2 m + c of a word by rank m, of one
// replica in bits 0..15 and with RP = 2 of a second one in bits 16..31.
//
// Decision.  With J1, x1 the coupling to the neighbour at the same rank of the
// other colour's word and whether that neighbour is anti-aligned, J2, x2 the
// other neighbour's, dE = 4 (x1 J1 + x2 J2) - 2 (J1 + J2):
//   class A, x1 = x2 (the neighbours are aligned): dE = +-2 (J1 + J2),
//   class B, x1 != x2: dE = +-2 (J1 - J2),
// the sign the opposite for x1 = 0 and x1 = 1.  So a site has two thresholds
// thr(|dE|) (gauss_threshold: the Metropolis decision of pa_gauss.cuh as an
// integer, u >> 8 < thr), and whether a flip lowers the energy is a bit of a
// mask zA or zB (dE <= 0 at x1 = 0), inverted where x1 = 1.  Both classes of
// every site are compared, and the classes, the signs and the outcomes of all
// 2 x 16 sites of a word are combined by a few logic operations: no pattern is
// looked up per site.  The entry of a threshold is 2^32 - 256 thr, so that
// adding the uniform carries exactly when it rejects (thr = 2^24 never does,
// its entry is 0; thr = 0 takes 2^32 - 1, and a block with one raises its
// uniforms from 0 to 1, which no other threshold can tell apart), and the
// outcome is shifted in by an add with carry.
//
// What bounds it: instruction issue and the multiply pipe, as the +-1 chain
// (pa_sweep1d.cu), with two compares a site where that one needs one.  One
// launch, us, with packed words, one thread a replica and a threshold looked up
// per site and pattern -> now:
//   N = 256, theta = 50   2e5 replicas 1961 -> 1584   20000 413 -> 210   1000 301 -> 55
//   N = 512, theta = 10   5e4 258 -> 182
//   N = 64,  theta = 10   1e5 102 -> 61
//   N = 4096, theta = 10  5000 1050 -> 283
// (2e5, with the maxima for thresholds of 0 still in the loop: (threads a block,
// split, replicas a thread) = (128, 8, 2) 1675, (128, 4, 2) 1639, (128, 2, 2)
// 1705, (64, 1, 1) 1882; smaller populations want the finest split.)
#include "pa_gauss.cuh"
#include "pa_lattice3d.cuh"
#include "pa_patterns.cuh"

namespace pa {

__device__ __forceinline__ uint32_t gchain_valid(int w, int WR, int nl) {
  return (w + 1 < WR || nl == 32) ? 0xFFFFFFFFu : ((1u << nl) - 1u);
}

// E_q = C0 - 2 sum over anti-aligned bonds (i, i+1) of J[i], C0 = sum J
// (packed words of the initial state).
__device__ __forceinline__ int energy_gauss1d(const uint32_t* __restrict__ col, int CS,
                                              const int32_t* __restrict__ J, int WR, int nl, int32_t C0) {
  const uint32_t first = col[0];
  int32_t anti = 0;
  for (int w = 0; w < WR; ++w) {
    const uint32_t curw = col[w * CS];
    const uint32_t nbp = (w + 1 < WR) ? __funnelshift_r(curw, col[(w + 1) * CS], 1)
                                      : ((curw >> 1) | ((first & 1u) << (nl - 1)));
    uint32_t a = (curw ^ nbp) & gchain_valid(w, WR, nl);
    while (a) {
      anti += J[32 * w + __ffs(a) - 1];
      a &= a - 1u;
    }
  }
  return C0 - 2 * anti;
}

// Entry of colour c and word w, 9 uint4: {zA, zB, the word's sites, 0}, both
// halves of a mask alike, then for each four ranks the threshold entries of
// class A and of class B.
constexpr int GCHAIN_ENTRY = 9;
// uint4 of a half-sweep table per word: its four calls and one of padding, so
// that threads on neighbouring words read different banks.
constexpr int GCHAIN_CALLS = 5;

// Couplings of the colour-c site of rank m of word w: to the neighbour at the
// same rank and to the other one.
__device__ __forceinline__ void gchain_couplings(const int32_t* __restrict__ s_J, int N, int c, int w, int m,
                                                 int32_t* j1, int32_t* j2) {
  const int i = 32 * w + 2 * m + c;
  const int32_t right = s_J[i], left = s_J[i == 0 ? N - 1 : i - 1];
  *j1 = c == 0 ? right : left;
  *j2 = c == 0 ? left : right;
}

// The entries, all threads of the block (s_J in place); returns whether one
// has threshold 0.
template <int TPB>
__device__ __forceinline__ int fill_gchain(uint4* __restrict__ s_thr, const int32_t* __restrict__ s_J, int N, int WR,
                                           int nl, float beta_f) {
  uint32_t* t = reinterpret_cast<uint32_t*>(s_thr);
  int never = 0;
  for (int i = threadIdx.x; i < 2 * WR * 32; i += TPB) {
    const int m = i & 15, b = (i >> 4) & 1, cw = i >> 5;  // cw = c WR + w; b: class B
    const int c = cw >= WR, w = cw - c * WR;
    int32_t j1, j2;
    gchain_couplings(s_J, N, c, w, m, &j1, &j2);
    const uint32_t thr = gauss_threshold(abs(2 * (b ? j1 - j2 : j1 + j2)), beta_f);
    never |= thr == 0u;
    t[4 * GCHAIN_ENTRY * cw + 4 + 8 * (m >> 2) + 4 * b + (m & 3)] = thr == 0u ? 0xFFFFFFFFu : 0u - (thr << 8);
  }
  for (int cw = threadIdx.x; cw < 2 * WR; cw += TPB) {
    const int c = cw >= WR, w = cw - c * WR;
    uint32_t za = 0u, zb = 0u;
    for (int m = 0; m < 16; ++m) {
      int32_t j1, j2;
      gchain_couplings(s_J, N, c, w, m, &j1, &j2);
      za |= (j1 + j2 >= 0 ? 1u : 0u) << m;  // dE at x1 = 0: -2 (J1 + J2) and 2 (J2 - J1)
      zb |= (j1 - j2 >= 0 ? 1u : 0u) << m;
    }
    const int n = w + 1 < WR ? 16 : (nl - c + 1) >> 1;
    s_thr[GCHAIN_ENTRY * cw] =
        make_uint4(za * 0x00010001u, zb * 0x00010001u, (n >= 16 ? 0xFFFFu : (1u << n) - 1u) * 0x00010001u, 0u);
  }
  return never;
}

// Colour-C word w of a column and its neighbours in the other colour's words:
// at the same rank, and the other one (rank m - 1 for C = 0, m + 1 for C = 1,
// across the word boundary; across the ends of the chain the last site has
// rank last = (nl - 1) / 2 of the last word).
struct GchainWord {
  uint32_t s, same, other;
};
template <int C, class T>
__device__ __forceinline__ GchainWord gchain_word(const T* __restrict__ own, const T* __restrict__ oth, int CS, int w,
                                                  int WR, int last) {
  const uint32_t s = own[w * CS], nx = oth[w * CS];
  uint32_t o;
  if constexpr (C == 0) {
    const uint32_t nb = oth[(w > 0 ? w - 1 : WR - 1) * CS];
    o = ((nx << 1) & 0xFFFEFFFEu) | ((nb >> (w > 0 ? 15 : last)) & 0x00010001u);
  } else {
    const uint32_t nb = oth[(w + 1 < WR ? w + 1 : 0) * CS];
    o = ((nx >> 1) & 0x7FFF7FFFu) | ((nb & 0x00010001u) << (w + 1 < WR ? 15 : last));
  }
  return {s, nx, o};
}

// Colour-C half sweep of words w0 .. w1-1 of a column (colour-C word w at
// own[w CS], the other colour's at oth[w CS]).  The uniforms of word w are
// calls 4w .. 4w+3 of the colour; the calls are taken from the last, so that
// the outcomes are shifted in from the highest rank.
// NEVER: the table has a threshold 0 (a parameter: predicated off, the maxima
// would still take an issue slot a site).
template <int C, int RP, bool NEVER>
__device__ __forceinline__ void half_sweep_gauss1d(ColourWord<RP>* __restrict__ own,
                                                   const ColourWord<RP>* __restrict__ oth, int CS,
                                                   const uint4* __restrict__ thr, int WR, int last, int w0, int w1,
                                                   const uint4* __restrict__ half, const SweepKey (&key)[RP],
                                                   const RoundKeys& rk) {
#pragma unroll 1
  for (int w = w0; w < w1; ++w) {
    const GchainWord g = gchain_word<C>(own, oth, CS, w, WR, last);
    const uint4* e = thr + GCHAIN_ENTRY * w;
    uint32_t ga[RP] = {}, gb[RP] = {};
#pragma unroll
    for (int q = 3; q >= 0; --q) {
      const uint4 a = e[1 + 2 * q], b = e[2 + 2 * q];
#pragma unroll
      for (int k = 0; k < RP; ++k) {
        u32x4 v = philox_sweep(half[GCHAIN_CALLS * w + q], key[k], rk);
        if constexpr (NEVER) v = {max(v.a, 1u), max(v.b, 1u), max(v.c, 1u), max(v.d, 1u)};
        ga[k] = shift_in_carry(ga[k], v.d, a.w);
        gb[k] = shift_in_carry(gb[k], v.d, b.w);
        ga[k] = shift_in_carry(ga[k], v.c, a.z);
        gb[k] = shift_in_carry(gb[k], v.c, b.z);
        ga[k] = shift_in_carry(ga[k], v.b, a.y);
        gb[k] = shift_in_carry(gb[k], v.b, b.y);
        ga[k] = shift_in_carry(ga[k], v.a, a.x);
        gb[k] = shift_in_carry(gb[k], v.a, b.x);
      }
    }
    uint32_t ra = ga[0], rb = gb[0];  // rejected as class A, as class B
    if constexpr (RP == 2) {
      ra = __byte_perm(ga[0], ga[RP - 1], 0x5410u);
      rb = __byte_perm(gb[0], gb[RP - 1], 0x5410u);
    }
    const uint4 z = e[0];
    const uint32_t y = g.same ^ g.other;  // class B
    const uint32_t rise = ~(((y & z.y) | (~y & z.x)) ^ g.s ^ g.same);
    const uint32_t stay = rise & ((y & rb) | (~y & ra));
    own[w * CS] = (ColourWord<RP>)(g.s ^ (z.z & ~stay));
  }
}

// Shape of a block: NC = TPB / P columns of RP replicas, P threads a column
// (lanes l, l + 32 / P, ... of one warp) on ranges of WPP = ceil(WR / P) words;
// a column stride CS that puts the P ranges on different banks where one
// exists; NH half-sweep tables (even; the block meets once per NH half
// sweeps, the threads of a column after every one) in about 216 bytes a thread.
struct GChainShape {
  int NC, WPP, CS, NH;
  size_t words;
};
__host__ __device__ inline GChainShape gchain_shape(int TPB, int P, int RP, int WR) {
  GChainShape sh;
  sh.NC = TPB / P;
  sh.WPP = (WR + P - 1) / P;
  sh.CS = sh.NC;
  if (P > 1)
    for (int cs = sh.NC; cs < sh.NC + 8; ++cs) {
      const int m = (sh.WPP * cs) % 32;
      if (m % (32 / P) == 0 && ((m / (32 / P)) & 1)) {
        sh.CS = cs;
        break;
      }
    }
  // the threshold entries (whose memory also takes the word ranges' energies
  // at the end), the couplings padded to whole words, the colour words
  const size_t thr = 8 * (size_t)GCHAIN_ENTRY * WR;
  const size_t other = (thr > (size_t)RP * TPB ? thr : (size_t)RP * TPB) + 32 * (size_t)WR +
                       ((size_t)WR * sh.CS * RP + 3) / 4 * 4;
  const int least = P > 1 ? 2 : 6;
  const long long room = (216ll * TPB - 4ll * (long long)other) / (16ll * GCHAIN_CALLS * WR);
  sh.NH = room >= 20 ? 20 : (room < least ? least : (int)(room & ~1ll));
  sh.words = other + 4 * (size_t)sh.NH * GCHAIN_CALLS * WR;
  return sh;
}

// Sec. 2 for chains with the Gaussian couplings of Sec. 4: gather of the
// resampled population, theta checkerboard sweeps at beta', energy; block b
// takes work item b / (P / RP) (TPB slots of one run) and its share of them.
template <int TPB, int P, int RP>
__global__ void __launch_bounds__(TPB) k_sweep_gauss1d(RunDev* __restrict__ runs, const Work* __restrict__ table) {
  extern __shared__ __align__(16) uint32_t smem[];
  constexpr int NC = TPB / P, NR = NC * RP, BPI = P / RP, RW = 32 / P;
  const Work wk = table[blockIdx.x / BPI];
  RunDev& R = runs[wk.run];
  if (R.skip) return;
  const int64_t Rn = R.R_next;
  const int64_t first = (int64_t)wk.first + (int64_t)(blockIdx.x % BPI) * NR;
  if (first >= Rn) return;
  const int N = R.N, W = R.W, WR = R.Wr, nl = N - 32 * (WR - 1), last = (nl - 1) >> 1;
  const GChainShape sh = gchain_shape(TPB, P, RP, WR);
  const int CS = sh.CS;
  uint4* s_tab = reinterpret_cast<uint4*>(smem);
  uint4* s_thr = s_tab + sh.NH * GCHAIN_CALLS * WR;
  const int thr_words = 8 * GCHAIN_ENTRY * WR;
  int32_t* s_J = reinterpret_cast<int32_t*>(s_thr) + (thr_words > RP * TPB ? thr_words : RP * TPB);
  ColourWord<RP>* s_spin = reinterpret_cast<ColourWord<RP>*>(s_J + 32 * WR);  // [2 colours][WR][CS]
  const int tid = threadIdx.x, lane = tid & 31;
  for (int i = tid; i < 32 * WR; i += TPB) s_J[i] = (i < N) ? R.gJ[i] : 0;
  const RoundKeys rk = make_round_keys(R.seed);
  const int part = lane / RW, r = (tid >> 5) * RW + lane % RW;
  // replica k of column r is slot first + k NC + r
  const int64_t slot = first + r;
  const bool live = slot < Rn;
  const int cur = R.cur, nxt = cur ^ 1;
  ColourWord<RP>* col = s_spin + r;
  if (live) {
    const uint4* p4[RP];
    bool on[RP];
#pragma unroll
    for (int k = 0; k < RP; ++k) {
      on[k] = slot + k * NC < Rn;
      p4[k] = reinterpret_cast<const uint4*>(R.spins[cur] + (size_t)(on[k] ? R.src[slot + k * NC] : 0) * W);
    }
    for (int q = part; q < W / 4; q += P) {
      uint32_t v[4][RP];
#pragma unroll
      for (int k = 0; k < RP; ++k) {
        const uint4 t = on[k] ? p4[k][q] : make_uint4(0u, 0u, 0u, 0u);
        v[0][k] = t.x;
        v[1][k] = t.y;
        v[2][k] = t.z;
        v[3][k] = t.w;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int w = 4 * q + i;
        if (w < WR) {
          uint32_t a[RP], b[RP];
#pragma unroll
          for (int k = 0; k < RP; ++k) {
            a[k] = v[i][k] & 0x55555555u;
            b[k] = (v[i][k] >> 1) & 0x55555555u;
          }
          col[w * CS] = (ColourWord<RP>)gather_even<RP>(a);
          col[(WR + w) * CS] = (ColourWord<RP>)gather_even<RP>(b);
        }
      }
    }
  }
  __syncthreads();  // the couplings in place
  const int zero = fill_gchain<TPB>(s_thr, s_J, N, WR, nl, __double2float_rn(R.beta_next));
  const bool never = __syncthreads_or(zero) != 0;
  const int w0 = min(part * sh.WPP, WR), w1 = min(w0 + sh.WPP, WR);
  const int theta = R.theta_next;
  const uint32_t T0 = (uint32_t)R.sweeps;
  const int Q = 4 * WR, nhalf = 2 * theta;
  SweepKey key[RP];
#pragma unroll 1
  for (int h0 = 0; h0 < nhalf; h0 += sh.NH) {
    if (h0 > 0) __syncthreads();  // the previous chunk's tables are no longer read
    const int nh = min(sh.NH, nhalf - h0);
    for (int i = tid; i < nh * Q; i += TPB) {
      const int j = i / Q, q = i - j * Q;
      s_tab[j * GCHAIN_CALLS * WR + GCHAIN_CALLS * (q >> 2) + (q & 3)] =
          sweep_half_entry(sweep_call_entry((uint32_t)q, TAG_SWEEP + (uint32_t)(j & 1), rk),
                           PHILOX_MUL1 * (T0 + (uint32_t)((h0 + j) >> 1)));
    }
    __syncthreads();
#pragma unroll 1
    for (int j = 0; j < nh; j += 2) {  // h0 and nh are even
      const uint4* half = s_tab + j * GCHAIN_CALLS * WR;
#pragma unroll
      for (int k = 0; k < RP; ++k)
        key[k] = sweep_key((uint32_t)(slot + k * NC), T0 + (uint32_t)((h0 + j) >> 1), rk);
      const auto sweep = [&](auto nc) {
        constexpr bool NEVER = decltype(nc)::value;
        if (live)
          half_sweep_gauss1d<0, RP, NEVER>(col, col + WR * CS, CS, s_thr, WR, last, w0, w1, half, key, rk);
        __syncwarp();  // colour-1 words read what the other threads of the column wrote
        if (live)
          half_sweep_gauss1d<1, RP, NEVER>(col + WR * CS, col, CS, s_thr + GCHAIN_ENTRY * WR, WR, last, w0, w1,
                                           half + GCHAIN_CALLS * WR, key, rk);
      };
      if (never) sweep(std::true_type());
      else sweep(std::false_type());
      __syncwarp();
    }
  }
  __syncthreads();  // the thresholds are no longer read
  // Energy E = C0 - 2 sum of J over the anti-aligned bonds: those of the
  // colour-0 sites (the wrap bond of an odd chain is absent: J = 0)
  int32_t anti[RP] = {};
  if (live) {
    const uint32_t one = R.one;
    for (int w = w0; w < w1; ++w) {
      const GchainWord g = gchain_word<0>(col, col + WR * CS, CS, w, WR, last);
      const uint32_t x1 = g.s ^ g.same, x2 = g.s ^ g.other;
      const int n = w + 1 < WR ? 16 : (nl + 1) >> 1;
      for (int m = 0; m < n; ++m) {
        int32_t j1, j2;
        gchain_couplings(s_J, N, 0, w, m, &j1, &j2);
#pragma unroll
        for (int k = 0; k < RP; ++k) {
          add_if_set(anti[k], x1, 1u << (16 * k + m), j1, one);
          add_if_set(anti[k], x2, 1u << (16 * k + m), j2, one);
        }
      }
    }
    for (int q = part; q < W / 4; q += P) {
      uint32_t v[RP][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int w = 4 * q + i;
        const bool in = w < WR;
        const uint32_t a = in ? (uint32_t)col[w * CS] : 0u, b = in ? (uint32_t)col[(WR + w) * CS] : 0u;
        v[0][i] = spread_even<0>(a) | (spread_even<0>(b) << 1);
        if constexpr (RP == 2) v[RP - 1][i] = spread_even<1>(a) | (spread_even<1>(b) << 1);
      }
#pragma unroll
      for (int k = 0; k < RP; ++k)
        if (slot + k * NC < Rn)
          reinterpret_cast<uint4*>(R.spins[nxt] + (size_t)(slot + k * NC) * W)[q] =
              make_uint4(v[k][0], v[k][1], v[k][2], v[k][3]);
    }
  }
  // sum over the word ranges, then record one replica per thread
  int32_t* s_anti = reinterpret_cast<int32_t*>(s_thr);  // [P][NR]
#pragma unroll
  for (int k = 0; k < RP; ++k) s_anti[part * NR + k * NC + r] = anti[k];
  __syncthreads();
  if ((tid & ~31) >= NR) return;  // whole warps
  int E = R.gC0;
  const bool rec = tid < NR && first + tid < Rn;
  if (rec)
    for (int q = 0; q < P; ++q) E -= 2 * s_anti[q * NR + tid];
  measure_store_gauss(R, nxt, first + tid, rec, E);
}

// Sec. 2: R0 independent uniformly random microstates at beta = 0 and their
// energies, one thread per slot.
template <int TPB>
__global__ void __launch_bounds__(TPB) k_init_gauss1d(RunDev* __restrict__ runs, const Work* __restrict__ table) {
  extern __shared__ __align__(16) uint32_t smem[];
  const Work wk = table[blockIdx.x];
  RunDev& R = runs[wk.run];
  if ((int64_t)wk.first >= R.R) return;
  const int N = R.N, W = R.W, WR = R.Wr, nl = N - 32 * (WR - 1);
  const int tid = threadIdx.x;
  const int64_t slot = (int64_t)wk.first + tid;
  const bool live = slot < R.R;
  // the couplings in shared memory: a replica's energy is a chain of N / 2 loads
  // (N = 4096: 222 us a reset with them in global memory, 160 so)
  int32_t* s_J = reinterpret_cast<int32_t*>(smem);
  uint32_t* col = smem + 32 * WR + tid;
  for (int i = tid; i < N; i += TPB) s_J[i] = R.gJ[i];
  __syncthreads();
  int E = 0;
  if (live) {
    uint4* d4 = reinterpret_cast<uint4*>(R.spins[0] + (size_t)slot * W);
    for (int w4 = 0; w4 < W / 4; ++w4) {
      const u32x4 u = philox_seeded(R.seed, (uint32_t)w4, (uint32_t)slot, 0u, TAG_INIT);
      uint32_t v[4] = {u.a, u.b, u.c, u.d};
      for (int i = 0; i < 4; ++i) {
        const int w = 4 * w4 + i;
        v[i] = w < WR ? v[i] & gchain_valid(w, WR, nl) : 0u;
        if (w < WR) col[w * TPB] = v[i];
      }
      d4[w4] = make_uint4(v[0], v[1], v[2], v[3]);
    }
    E = energy_gauss1d(col, TPB, s_J, WR, nl, R.gC0);
  }
  measure_store_gauss(R, 0, slot, live, E);
}

template <int TPB, int P, int RP>
static cudaError_t launch_g1d_p(RunDev* runs, const Work* table, int nwork, int WR, cudaStream_t st, int min_smem) {
  if constexpr (P > 1 && TPB < 64) {
    return cudaErrorInvalidValue;
  } else {
    const size_t need = sizeof(uint32_t) * gchain_shape(TPB, P, RP, WR).words;
    const size_t sm = need > (size_t)min_smem ? need : (size_t)min_smem;
    if (nwork <= 0) {
      if (sm <= 48 * 1024) return cudaSuccess;
      return allow_shared(k_sweep_gauss1d<TPB, P, RP>);
    }
    k_sweep_gauss1d<TPB, P, RP><<<nwork * (P / RP), TPB, sm, st>>>(runs, table);
    return cudaGetLastError();
  }
}

template <int TPB>
static cudaError_t launch_g1d_t(int split, int rp, RunDev* runs, const Work* table, int nwork, int WR,
                                cudaStream_t st, bool init, int min_smem) {
  if (init) {
    const size_t sm = sizeof(uint32_t) * (size_t)WR * (TPB + 32);
    if (nwork <= 0) {
      if (sm <= 48 * 1024) return cudaSuccess;
      return allow_shared(k_init_gauss1d<TPB>);
    }
    k_init_gauss1d<TPB><<<nwork, TPB, sm, st>>>(runs, table);
    return cudaGetLastError();
  }
  const bool one = rp == 1;
  switch (split) {
    case 1: return launch_g1d_p<TPB, 1, 1>(runs, table, nwork, WR, st, min_smem);
    case 2:
      return one ? launch_g1d_p<TPB, 2, 1>(runs, table, nwork, WR, st, min_smem)
                 : launch_g1d_p<TPB, 2, 2>(runs, table, nwork, WR, st, min_smem);
    case 4:
      return one ? launch_g1d_p<TPB, 4, 1>(runs, table, nwork, WR, st, min_smem)
                 : launch_g1d_p<TPB, 4, 2>(runs, table, nwork, WR, st, min_smem);
    case 8:
      return one ? launch_g1d_p<TPB, 8, 1>(runs, table, nwork, WR, st, min_smem)
                 : launch_g1d_p<TPB, 8, 2>(runs, table, nwork, WR, st, min_smem);
    default: return cudaErrorInvalidValue;
  }
}

size_t gauss1d_smem_bytes(int tpb, int split, int rp, int WR) {
  return sizeof(uint32_t) * gchain_shape(tpb, split, rp, WR).words;
}

cudaError_t launch_gauss1d(int tpb, int split, int rp, RunDev* runs, const Work* table, int nwork, int WR,
                           cudaStream_t st, bool init, int min_smem) {
  switch (tpb) {
    case 32: return launch_g1d_t<32>(split, rp, runs, table, nwork, WR, st, init, min_smem);
    case 64: return launch_g1d_t<64>(split, rp, runs, table, nwork, WR, st, init, min_smem);
    case 128: return launch_g1d_t<128>(split, rp, runs, table, nwork, WR, st, init, min_smem);
    case 256: return launch_g1d_t<256>(split, rp, runs, table, nwork, WR, st, init, min_smem);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pa
