// pa_sweep1d.cu -- fused replica copy + checkerboard Metropolis sweeps +
// energy measurement for +-1 / diluted chains (Sec. 4: the 1D spin glass).
//
// Bit p of word w of a replica is site 32 w + p; colour = site parity.  A
// bond may be absent (J = 0, e.g. the wrap bond of an open chain), so the
// per-site energy change is dE = 4 n - 2 z_i with n satisfied bonds of the z_i
// present ones: n = 2 (dE = 4) and z_i = 1, n = 1 (dE = 2) are the rises that
// draw on the uniform.
//
// As in the cubic kernel a block keeps its replicas split by colour: the 16
// colour-c sites 32 w + 2 m + c of a word by rank m, of one replica in bits
// 0..15 and with RP = 2 of a second one in bits 16..31.  Of the two
// neighbours of a colour-0 site the right one has rank m of the colour-1 word
// w, the left one rank m - 1 (across the word boundary rank 15 of word
// w - 1); of a colour-1 site the left one has rank m of the colour-0 word w,
// the right one rank m + 1.  So a half sweep reads one word of the other
// colour per word and keeps the one it just read.
//
// Bound by instruction issue and the multiply pipe (see pa_sweep3d.cuh): per
// 16 sites of 32 replicas the generator takes 265 issue cycles, and half of the
// full-rate compares run on the multiply pipe, 87 % busy at beta = 1.  N =
// 4096, 2e5 replicas, theta = 5, one launch at beta = 0.1 / 1 / 4: 2604 / 2609
// / 2454 us with both colours in a word, whose compares had to be spread to
// alternate bits, 2287 / 2295 / 2202 us with this layout.
#include "pa_lattice3d.cuh"

namespace pa {

// Bond masks of one chain run: [4][W] words: JP (coupling i->i+1 is -1),
// JM (coupling i-1->i is -1), PP (bond i->i+1 present), PM (bond i-1->i present).
enum { C_JP = 0, C_JM = 1, C_PP = 2, C_PM = 3 };

__device__ __forceinline__ uint32_t chain_valid(int w, int WR, int nl) {
  return (w + 1 < WR || nl == 32) ? 0xFFFFFFFFu : ((1u << nl) - 1u);
}

// Satisfied present bonds (i, i+1) of words w0 .. w1-1 of the column.
__device__ __forceinline__ int satisfied1d(const uint32_t* __restrict__ col, int CS, const uint32_t* __restrict__ s_bond,
                                           int W, int WR, int nl, int w0, int w1) {
  const uint32_t first = col[0];
  int sat = 0;
  for (int w = w0; w < w1; ++w) {
    const uint32_t curw = col[w * CS];
    const uint32_t nbp = (w + 1 < WR) ? __funnelshift_r(curw, col[(w + 1) * CS], 1)
                                      : ((curw >> 1) | ((first & 1u) << (nl - 1)));
    sat += __popc((curw ^ nbp ^ s_bond[C_JP * W + w]) & s_bond[C_PP * W + w]);
  }
  return sat;
}

// Ranks of a chain word's sites by colour: how many there are, and the mask of
// both halves.
__device__ __forceinline__ uint32_t chain_ranks(int w, int WR, int nl, int c) {
  const int n = w + 1 < WR ? 16 : (nl - c + 1) >> 1;
  return n >= 16 ? 0xFFFFFFFFu : ((1u << n) - 1u) * 0x00010001u;
}

// Bond masks of the colour words, one entry per (c, w) and both halves alike:
// x, y the couplings of the bond to the neighbour at the same rank and to the
// other one, z, w whether they are present.  All threads of the block.
template <int TPB>
__device__ __forceinline__ void fill_bonds1d(uint4* __restrict__ s_bond, const uint32_t* __restrict__ bonds, int W,
                                             int WR) {
  for (int i = threadIdx.x; i < 2 * WR; i += TPB) {
    const int c = i >= WR, w = i - c * WR;
    uint32_t m[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const uint32_t v = (bonds[d * W + w] >> c) & 0x55555555u;
      const uint32_t x[2] = {v, v};
      m[d] = gather_even<2>(x);
    }
    s_bond[i] = c ? make_uint4(m[C_JM], m[C_JP], m[C_PM], m[C_PP]) : make_uint4(m[C_JP], m[C_JM], m[C_PP], m[C_PM]);
  }
}

// Satisfied bonds of the colour-C sites of word w: own words at own[w CS], the
// other colour's at oth[w CS], to the neighbour at the same rank and to the
// other one.  Across the ends of the chain the word before word 0 is the last
// one, whose last site has rank last = (nl - 1) / 2, and the one after the
// last word is word 0; where the wrap bond is absent its bits do not count.
struct ChainBonds {
  uint32_t s, same, other, single;  // single: sites with one bond present
};
template <int C, class T>
__device__ __forceinline__ ChainBonds chain_bonds(const T* __restrict__ own, const T* __restrict__ oth, int CS,
                                                  const uint4* __restrict__ bond, int w, int WR, int last) {
  const uint32_t s = own[w * CS], nx = oth[w * CS];
  const uint4 j = bond[w];
  uint32_t o;
  if constexpr (C == 0) {
    const uint32_t nb = oth[(w > 0 ? w - 1 : WR - 1) * CS];
    o = ((nx << 1) & 0xFFFEFFFEu) | ((nb >> (w > 0 ? 15 : last)) & 0x00010001u);
  } else {
    const uint32_t nb = oth[(w + 1 < WR ? w + 1 : 0) * CS];
    o = ((nx >> 1) & 0x7FFF7FFFu) | ((nb & 0x00010001u) << (w + 1 < WR ? 15 : last));
  }
  return {s, (s ^ nx ^ j.x) & j.z, (s ^ o ^ j.y) & j.w, j.z ^ j.w};
}

// Words w0 .. w1-1 of a column of RP replicas (colour-C word w at own[w CS],
// the other colour's at oth[w CS]).  Colour-C sites read only the other
// colour's words, which a half sweep leaves unchanged, so the word ranges of
// the P threads of a column are swept at once.  The uniforms of word w are
// calls 4w .. 4w+3 of the colour: half-sweep entries at half[4w + k].
// Compares: dE = 2 arises only at sites with one bond present (a chain's ends
// and absent bonds), so thr(dE=2) is compared only in words holding such a
// site; thr(dE=4) in every word, except that at low temperature (thr4 <
// 2^22) a word whose uniforms' minimum is not below thr4 in any lane of the
// warp skips it (then no rise is accepted).
// Every thread of a column runs WPP iterations, whatever its range holds (the
// last range may be short or empty), so that the warp votes below are taken
// by all live lanes together; an iteration past the range works on a word of
// the chain again and writes nothing.
template <int C, int RP>
__device__ __forceinline__ void half_sweep1d(ColourWord<RP>* __restrict__ own, const ColourWord<RP>* __restrict__ oth,
                                             int CS, const uint4* __restrict__ bond, int WR, int nl, int w0, int w1,
                                             int WPP, const uint4* __restrict__ half, const SweepKey (&key)[RP],
                                             const RoundKeys& rk, uint32_t T2, uint32_t T4, unsigned lanes) {
  const bool low_t = T4 < (1u << 22);
  const int last = (nl - 1) >> 1;
  const uint32_t tail = chain_ranks(WR - 1, WR, nl, C);
#pragma unroll 1
  for (int i = 0; i < WPP; ++i) {
    const int w = min(w0 + i, WR - 1);
    const ChainBonds n = chain_bonds<C>(own, oth, CS, bond, w, WR, last);
    const bool two = __any_sync(lanes, n.single != 0u);
    uint32_t e4 = 0u, e2 = 0u;
#pragma unroll
    for (int k = 0; k < RP; ++k) {
      uint32_t u[16];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const u32x4 v = philox_sweep(half[4 * w + q], key[k], rk);
        u[4 * q + 0] = v.a;
        u[4 * q + 1] = v.b;
        u[4 * q + 2] = v.c;
        u[4 * q + 3] = v.d;
      }
      if (two) e2 |= lt_mask<16, 0>(u, T2) << (16 * k);
      if (low_t && !__any_sync(lanes, min_of<16, 0>(u) < T4)) continue;
      e4 |= lt_mask<16, 0>(u, T4) << (16 * k);
    }
    const uint32_t need4 = n.same & n.other, need2 = (n.same ^ n.other) & n.single;
    const uint32_t acc = (w + 1 < WR ? 0xFFFFFFFFu : tail) & ~(need4 & ~e4) & ~(need2 & ~e2);
    if (w0 + i < w1) own[w * CS] = (ColourWord<RP>)(n.s ^ acc);
  }
}

template <int TPB>
__device__ __forceinline__ void store_column1d(uint32_t* __restrict__ dst,
                                               const uint32_t* __restrict__ col, int W, int WR) {
  uint4* d4 = reinterpret_cast<uint4*>(dst);
  for (int q = 0; q < W / 4; ++q) {
    uint4 v;
    v.x = (4 * q + 0 < WR) ? col[(4 * q + 0) * TPB] : 0u;
    v.y = (4 * q + 1 < WR) ? col[(4 * q + 1) * TPB] : 0u;
    v.z = (4 * q + 2 < WR) ? col[(4 * q + 2) * TPB] : 0u;
    v.w = (4 * q + 3 < WR) ? col[(4 * q + 3) * TPB] : 0u;
    d4[q] = v;
  }
}

// Shape of a chain sweep block: NC = TPB / P columns of RP replicas, P threads
// per column on ranges of WPP = ceil(WR / P) words (thread t takes range t /
// NC of column t mod NC); NH half-sweep tables of Q = 4 WR calls.
struct Chain1dShape {
  int NC, WPP, Q, NH;
};

__host__ __device__ inline Chain1dShape chain1d_shape(int TPB, int P, int RP, int WR) {
  Chain1dShape sh;
  sh.NC = TPB / P;
  sh.WPP = (WR + P - 1) / P;
  sh.Q = 4 * WR;
  // half-sweep tables held at once (as for the cubic kernels): with one
  // thread per column even, 2 .. 20, in about 216 bytes per thread with the
  // other arrays; with several, two, double-buffered
  const int room = 216 * TPB - (32 * WR + 4 * WR * sh.NC * RP);
  const int nh = room > 0 ? room / (16 * sh.Q) : 0;
  sh.NH = P > 1 ? 2 : (nh >= 20 ? 20 : (nh < 2 ? 2 : (nh & ~1)));
  return sh;
}

// Words: tables (which also take the word ranges' energies at the end), bond
// entries [2][WR], colour words [2][WR][NC].
__host__ __device__ inline int chain1d_tab_words(const Chain1dShape& sh, int TPB, int RP) {
  return 4 * sh.NH * sh.Q > RP * TPB ? 4 * sh.NH * sh.Q : RP * TPB;
}
__host__ __device__ inline size_t chain1d_smem_words(const Chain1dShape& sh, int TPB, int RP, int WR) {
  return (size_t)chain1d_tab_words(sh, TPB, RP) + 8 * (size_t)WR + (size_t)WR * sh.NC * RP;
}

// Sec. 2 for chains: gather of the resampled population, theta checkerboard
// sweeps at beta', energy; block b takes work item b / (P / RP) (TPB slots of
// one run) and its share of TPB / P columns.
template <int TPB, int P, int RP>
__global__ void __launch_bounds__(TPB) k_sweep1d(RunDev* __restrict__ runs, const Work* __restrict__ table) {
  extern __shared__ __align__(16) uint32_t smem[];
  constexpr int NC = TPB / P, NR = NC * RP, BPI = P / RP;
  const Work wk = table[blockIdx.x / BPI];
  RunDev& R = runs[wk.run];
  if (R.skip) return;
  const int64_t Rn = R.R_next;
  const int W = R.W, WR = R.Wr, nl = R.N - 32 * (R.Wr - 1);
  const Chain1dShape sh = chain1d_shape(TPB, P, RP, WR);
  const int64_t first = (int64_t)wk.first + (int64_t)(blockIdx.x % BPI) * NR;
  if (first >= Rn) return;
  uint4* s_tab = reinterpret_cast<uint4*>(smem);
  uint4* s_bond = reinterpret_cast<uint4*>(smem + chain1d_tab_words(sh, TPB, RP));
  ColourWord<RP>* s_spin = reinterpret_cast<ColourWord<RP>*>(s_bond + 2 * WR);
  const int tid = threadIdx.x;
  fill_bonds1d<TPB>(s_bond, R.bonds, W, WR);
  const RoundKeys rk = make_round_keys(R.seed);
  const int part = tid / NC, r = tid % NC;
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
          col[w * NC] = (ColourWord<RP>)gather_even<RP>(a);
          col[(WR + w) * NC] = (ColourWord<RP>)gather_even<RP>(b);
        }
      }
    }
  }
  const unsigned lanes = __ballot_sync(0xFFFFFFFFu, live);  // live lanes of this warp
  const uint32_t T2 = R.thr[1], T4 = R.thr[2];
  const int theta = R.theta_next;
  const uint32_t T0 = (uint32_t)R.sweeps;
  const int w0 = min(part * sh.WPP, WR), w1 = min(w0 + sh.WPP, WR);
  SweepKey key[RP];
  // half-sweep table of colour c at sweep T, all threads of the block
  const auto build = [&](uint4* tab, int c, uint32_t T) {
    const uint32_t A1 = PHILOX_MUL1 * T;
    for (int q = tid; q < sh.Q; q += TPB)
      tab[q] = sweep_half_entry(sweep_call_entry((uint32_t)q, TAG_SWEEP + (uint32_t)c, rk), A1);
  };
  const auto sweep = [&](const uint4* half, auto c) {
    constexpr int C = decltype(c)::value;
    half_sweep1d<C, RP>(col + C * WR * NC, col + (1 - C) * WR * NC, NC, s_bond + C * WR, WR, nl, w0, w1, sh.WPP, half,
                        key, rk, T2, T4, lanes);
  };
  const std::integral_constant<int, 0> c0;
  const std::integral_constant<int, 1> c1;
  if constexpr (P > 1) {
    // one table per half sweep, double-buffered, behind a block barrier that
    // also orders the word ranges' half sweeps; every thread of the block
    // passes the barriers
#pragma unroll 1
    for (int t = 0; t < theta; ++t) {
      const uint32_t T = T0 + (uint32_t)t;
#pragma unroll
      for (int k = 0; k < RP; ++k) key[k] = sweep_key((uint32_t)(slot + k * NC), T, rk);
      build(s_tab, 0, T);
      __syncthreads();
      if (live) sweep(s_tab, c0);
      build(s_tab + sh.Q, 1, T);
      __syncthreads();
      if (live) sweep(s_tab + sh.Q, c1);
    }
  } else {
    // one thread per column: half sweeps in chunks of NH tables, one block
    // barrier per chunk
    const int nhalf = 2 * theta;
#pragma unroll 1
    for (int h0 = 0; h0 < nhalf; h0 += sh.NH) {
      if (h0 > 0) __syncthreads();  // the previous chunk's tables are no longer read
      const int nh = min(sh.NH, nhalf - h0);
      // over all entries at once: table by table, a chain of one word (four
      // calls) left most threads idle for the length of the chunk
      for (int i = tid; i < nh * sh.Q; i += TPB) {
        const int j = i / sh.Q, q = i - j * sh.Q;
        s_tab[i] = sweep_half_entry(sweep_call_entry((uint32_t)q, TAG_SWEEP + (uint32_t)(j & 1), rk),
                                    PHILOX_MUL1 * (T0 + (uint32_t)((h0 + j) >> 1)));
      }
      __syncthreads();
      if (live) {
#pragma unroll 1
        for (int j = 0; j < nh; j += 2) {  // h0 and nh are even
          key[0] = sweep_key((uint32_t)slot, T0 + (uint32_t)((h0 + j) >> 1), rk);
          sweep(s_tab + j * sh.Q, c0);
          sweep(s_tab + (j + 1) * sh.Q, c1);
        }
      }
    }
  }
  __syncthreads();  // every word range swept before the energy reads its neighbour words
  // a bond joins a colour-0 and a colour-1 site: the satisfied bonds are
  // those of the colour-0 sites, or of an open chain's sites to their right
  int sat[RP] = {};
  if (live) {
    for (int w = w0; w < w1; ++w) {
      const ChainBonds n = chain_bonds<0>(col, col + WR * NC, NC, s_bond, w, WR, (nl - 1) >> 1);
#pragma unroll
      for (int k = 0; k < RP; ++k) {
        const uint32_t m = 0xFFFFu << (16 * k);
        sat[k] += __popc(n.same & m) + __popc(n.other & m);
      }
    }
    for (int q = part; q < W / 4; q += P) {
      uint32_t v[RP][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int w = 4 * q + i;
        const bool in = w < WR;
        const uint32_t a = in ? (uint32_t)col[w * NC] : 0u, b = in ? (uint32_t)col[(WR + w) * NC] : 0u;
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
  int* s_sat = reinterpret_cast<int*>(s_tab);  // [P][NR]; the tables are no longer read
#pragma unroll
  for (int k = 0; k < RP; ++k) s_sat[part * NR + k * NC + r] = sat[k];
  __syncthreads();
  if ((tid & ~31) >= NR) return;  // whole warps
  int E = R.Nb;
  const bool rec = tid < NR && first + tid < Rn;
  if (rec)
    for (int q = 0; q < P; ++q) E -= 2 * s_sat[q * NR + tid];
  measure_store(R, nxt, first + tid, rec, E);
}

template <int TPB>
__global__ void __launch_bounds__(TPB) k_init1d(RunDev* __restrict__ runs,
                                                const Work* __restrict__ table) {
  extern __shared__ uint32_t smem[];
  const Work wk = table[blockIdx.x];
  RunDev& R = runs[wk.run];
  const int64_t R0 = R.R;
  if ((int64_t)wk.first >= R0) return;
  const int W = R.W, WR = R.Wr, nl = R.N - 32 * (R.Wr - 1);
  uint32_t* s_bond = smem;
  uint32_t* s_spin = smem + 4 * W;
  const int tid = threadIdx.x;
  for (int i = tid; i < 4 * W; i += TPB) s_bond[i] = R.bonds[i];
  const int64_t slot = (int64_t)wk.first + tid;
  const bool live = slot < R0;
  uint32_t* col = s_spin + tid;
  if (live) {
    for (int w4 = 0; w4 < W / 4; ++w4) {
      const u32x4 u = philox_seeded(R.seed, (uint32_t)w4, (uint32_t)slot, 0u, TAG_INIT);
      const uint32_t v[4] = {u.a, u.b, u.c, u.d};
      for (int i = 0; i < 4; ++i) {
        const int w = 4 * w4 + i;
        if (w < WR) col[w * TPB] = v[i] & chain_valid(w, WR, nl);
      }
    }
  }
  __syncthreads();
  int E = 0;
  if (live) {
    E = R.Nb - 2 * satisfied1d(col, TPB, s_bond, W, WR, nl, 0, WR);
    store_column1d<TPB>(R.spins[0] + (size_t)slot * W, col, W, WR);
  }
  measure_store(R, 0, slot, live, E);
}

// One launch over nwork work items (with nwork <= 0 the kernel is only
// allowed its shared memory, outside any stream capture).
template <int TPB, int P, int RP>
static cudaError_t launch_sweep1d_p(RunDev* runs, const Work* table, int nwork, int WR, cudaStream_t st,
                                    int min_smem) {
  if constexpr (TPB / P < 4 || (P > 1 && TPB < 64)) {
    return cudaErrorInvalidValue;
  } else {
    const size_t need = sizeof(uint32_t) * chain1d_smem_words(chain1d_shape(TPB, P, RP, WR), TPB, RP, WR);
    const size_t sm = need > (size_t)min_smem ? need : (size_t)min_smem;
    if (nwork <= 0) {
      if (sm <= 48 * 1024) return cudaSuccess;
      return allow_shared(k_sweep1d<TPB, P, RP>);
    }
    k_sweep1d<TPB, P, RP><<<nwork * (P / RP), TPB, sm, st>>>(runs, table);
    return cudaGetLastError();
  }
}

template <int TPB>
static cudaError_t launch1d_t(RunDev* runs, const Work* table, int nwork, int W, int WR, cudaStream_t st, bool init,
                              int split, int rp, int min_smem) {
  if (!init) {
    const bool one = rp == 1;
    switch (split) {
      case 1: return launch_sweep1d_p<TPB, 1, 1>(runs, table, nwork, WR, st, min_smem);
      case 2:
        return one ? launch_sweep1d_p<TPB, 2, 1>(runs, table, nwork, WR, st, min_smem)
                   : launch_sweep1d_p<TPB, 2, 2>(runs, table, nwork, WR, st, min_smem);
      case 4:
        return one ? launch_sweep1d_p<TPB, 4, 1>(runs, table, nwork, WR, st, min_smem)
                   : launch_sweep1d_p<TPB, 4, 2>(runs, table, nwork, WR, st, min_smem);
      case 8:
        return one ? launch_sweep1d_p<TPB, 8, 1>(runs, table, nwork, WR, st, min_smem)
                   : launch_sweep1d_p<TPB, 8, 2>(runs, table, nwork, WR, st, min_smem);
      default: return cudaErrorInvalidValue;
    }
  }
  const size_t sm = sizeof(uint32_t) * (4 * (size_t)W + (size_t)WR * TPB);
  if (nwork <= 0) {
    if (sm <= 48 * 1024) return cudaSuccess;
    return allow_shared(k_init1d<TPB>);
  }
  k_init1d<TPB><<<nwork, TPB, sm, st>>>(runs, table);
  return cudaGetLastError();
}

// Threads per replica for chains: 1, 2, 4 or 8 (word ranges of ceil(WR / P)).
bool sweep1d_split_ok(int split) { return split == 1 || split == 2 || split == 4 || split == 8; }

cudaError_t launch_sweep1d(int tpb, int split, int rp, RunDev* runs, const Work* table, int nwork, int W, int WR,
                           cudaStream_t st, bool init, int min_smem) {
  switch (tpb) {
    case 32: return launch1d_t<32>(runs, table, nwork, W, WR, st, init, split, rp, min_smem);
    case 64: return launch1d_t<64>(runs, table, nwork, W, WR, st, init, split, rp, min_smem);
    case 128: return launch1d_t<128>(runs, table, nwork, W, WR, st, init, split, rp, min_smem);
    case 256: return launch1d_t<256>(runs, table, nwork, W, WR, st, init, split, rp, min_smem);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pa
