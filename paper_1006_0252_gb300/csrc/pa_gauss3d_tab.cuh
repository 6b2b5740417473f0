// pa_gauss3d_tab.cuh -- the Gaussian sweep (Sec. 4 couplings, Sec. 2 sweeps)
// with per-site acceptance thresholds, for edges L <= 10 and blocks of 512 or
// 1024 threads.
//
// A colour-c site has six neighbours; with x_d = 1 where neighbour d is
// anti-aligned with it, its energy change dE(x) = 4 sum_{d: x_d = 1} J_d - 2 S
// is one of 64 values fixed by the couplings.  The Metropolis decision of
// pa_gauss.cuh (accept iff dE <= 0 or float(u >> 8) < lim(dE)) compares an
// integer below 2^24 with a float, so it is exactly (u >> 8) < thr(dE) with
//   thr = 2^24 (dE <= 0),  thr = ceil(lim(dE)) (dE > 0),
// which is u < 256 thr.  At the start of a launch (one beta) every block
// tabulates its run's thresholds in shared memory with the decision's own
// arithmetic; a site's update is then one table load at its pattern and one
// compare.
//
// Two forms of the table:
//   full (L = 4, 6, 8: 16, 55, 128 KB): all 64 patterns; the entry is 2^32 - 256 thr,
//     so that adding the uniform carries exactly when it rejects (and never
//     for thr = 2^24, whose entry is 0).  The compare and the collection of
//     the outcome are two full-rate instructions (add with carry out, add the
//     carry in).  thr = 0 has no such entry: it takes 2^32 - 1, and a block
//     with one raises its uniforms from 0 to 1 (the same outcome for any other
//     threshold, which is a multiple of 256).
//   folded (L = 10, whose full table would take 256 KB): inverting all six
//     bits of a pattern inverts dE, so 32 patterns y_d = x_d ^ x_5 (d < 5),
//     y_5 = 0, hold thr(|dE|) and the sign z = [dE(y) <= 0]; a site flips iff
//     u >> 8 < thr or z ^ x_5.  The entry is z 2^31 - thr: of the sum with
//     u >> 8, bit 30 is the compare and bit 31 is the compare ^ z.  A table of
//     32 entries a site also never has two patterns on one bank.
//
// The spins are colour-split words (pa_colour3d.cuh) of one or two replicas:
// a 32-bit operation on neighbour words serves 2 S <= 32 sites.  The pattern
// bits of the sites are then gathered byte by byte (Patterns below), so that
// one byte permute per site yields the address of its entry.
//
// What bounds it: instruction issue and the multiply pipe, as the +-1 sweep
// (pa_sweep3d.cuh).  At L = 8 a flip takes 16.1 instructions (9.8 of them the
// generator and the walk, 3.9 the patterns and table addresses, 1.1 the loads,
// 1.3 the compare and its collection) where packed words and a compare into a
// predicate took 20.8; of a launch of 1e5 replicas the generator takes 250 us and
// the tables, the gather and the energies 44.  One launch, theta = 10, us (packed
// words, or one thread a replica and an exponential per site at L = 10 -> now):
//   L = 8   1e5 replicas 572 -> 376    2000 190 -> 29
//   L = 10  80000 2400 -> 780    20000 794 -> 213    2000 648 -> 97
//   L = 6   50000  199 -> 99      3000 168 -> 34
//   L = 4   60000   80 -> 47      2000  39 -> 17
// (populations that leave SMs idle gain most: the finest split spreads them.)
// Not kept: the seed's round keys forced into uniform registers (same
// instruction count), blocks of 512 threads (10-40 % slower; one block of 1024
// threads fills an SM's registers).
#pragma once
#include "pa_colour3d.cuh"
#include "pa_gauss3d.cuh"
#include "pa_patterns.cuh"

namespace pa {

template <int L>
constexpr bool gtab_folded() {
  return L >= 10;
}
template <int L>
constexpr int gtab_entries() {  // of one site
  return gtab_folded<L>() ? 32 : 64;
}
// Threshold table words: [2 colours][WR words][S ranks][entries].
template <int L>
constexpr int gtab_words() {
  return 2 * Geo3<L>::WR * Half<Geo3<L>>::S * gtab_entries<L>();
}

// The x neighbour of a colour-c site of rank m that sits at its own rank:
// direction 0 (+x) where q = 0, 1 (-x) where q = 1; the other x neighbour is
// at a different rank (see RowX).
template <class GEO>
__device__ __forceinline__ int same_rank_dir(int c, int w, int m) {
  const int y = w / GEO::G, z = w % GEO::G + (m / Half<GEO>::H) * GEO::G;
  return (c + y + z) & 1;
}

// sum_{d: x_d = 1} J_d of the colour-c site of rank m of word w at the four
// patterns 4 h .. 4 h + 3.  Bits 0 and 1 of the pattern are the x neighbours at
// the same and at the other rank, bits 2..5 +y, -y, +z, -z.
template <class GEO>
__device__ __forceinline__ void gtab_anti(const int32_t* __restrict__ gJ, int c, int w, int m, int h,
                                          int32_t (&a)[4]) {
  constexpr int WR = GEO::WR, SP = (Half<GEO>::S + 3) & ~3;
  const int32_t* Jw = gJ + (c * 6 * WR + w) * SP + m;
  const int d0 = same_rank_dir<GEO>(c, w, m);
  int32_t acc = 0;
#pragma unroll
  for (int d = 2; d < 6; ++d)
    if ((h >> (d - 2)) & 1) acc += __ldg(Jw + d * WR * SP);
  const int32_t j0 = __ldg(Jw + d0 * WR * SP), j1 = __ldg(Jw + (1 - d0) * WR * SP);
  a[0] = acc;
  a[1] = acc + j0;
  a[2] = acc + j1;
  a[3] = acc + j0 + j1;
}

// The threshold table, all threads of the block.  Of the two patterns p and
// 63 - p, whose energy changes are opposite, at most one takes an exponential.
// Returns whether a full entry has threshold 0.
template <int L, int TPB>
__device__ __forceinline__ int fill_thresholds(uint32_t* __restrict__ s_thr, const int32_t* __restrict__ gJ,
                                               const int32_t* __restrict__ gS, float beta_f) {
  using GEO = Geo3<L>;
  constexpr int WR = GEO::WR, S = Half<GEO>::S, SP = (S + 3) & ~3;
  uint4* s4 = reinterpret_cast<uint4*>(s_thr);
  int never = 0;
#pragma unroll 1
  for (int i = threadIdx.x; i < 2 * WR * S * 8; i += TPB) {
    const int site = i >> 3, h = i & 7;  // site = (c WR + w) S + m, patterns 4 h .. 4 h + 3
    const int m = site % S, cw = site / S, c = cw / WR, w = cw % WR;
    int32_t a[4];
    gtab_anti<GEO>(gJ, c, w, m, h, a);
    const int32_t two_s = 2 * __ldg(gS + cw * SP + m);
    uint32_t e[4], f[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int32_t dE = 4 * a[j] - two_s;
      const uint32_t thr = gauss_threshold(abs(dE), beta_f);
      if constexpr (gtab_folded<L>()) {
        e[j] = (dE <= 0 ? 0x80000000u : 0u) - thr;
      } else {
        const uint32_t up = thr == 0u ? 0xFFFFFFFFu : 0u - (thr << 8);  // the rise; the fall always goes: entry 0
        e[j] = dE > 0 ? up : 0u;
        f[3 - j] = dE < 0 ? up : 0u;
        never |= thr == 0u;
      }
    }
    if constexpr (gtab_folded<L>()) {
      s4[i] = make_uint4(e[0], e[1], e[2], e[3]);
    } else {
      s4[site * 16 + h] = make_uint4(e[0], e[1], e[2], e[3]);
      s4[site * 16 + 15 - h] = make_uint4(f[0], f[1], f[2], f[3]);
    }
  }
  return never;
}

// The word updates of one half sweep, as walk_rows calls them.  NEVER: the table
// has a threshold 0 (a parameter, not a branch: predicated off, the maxima still
// take an issue slot a site).
template <int L, int RP, bool NEVER>
struct TabUpdate {
  using GEO = Geo3<L>;
  using HF = Half<GEO>;
  uint32_t thr;       // shared address of the table of the word the walk stands at (256-byte aligned)
  const uint4* half;  // its first call's entry
  const SweepKey (&key)[RP];
  const RoundKeys& rk;
  uint32_t carry[RP][4];

  template <int K, int A, int GP>
  __device__ __forceinline__ void word(ColourWord<RP>* own, const Around& nb, const RowX<GEO>& rx) {
    constexpr int S = HF::S, EB = 4 * gtab_entries<L>();
    constexpr bool FOLD = gtab_folded<L>();
    static_assert((S * EB) % 256 == 0, "the tables of a word start on a 256-byte boundary");
    const uint32_t s = *own;
    const uint32_t ref = FOLD ? nb.zm : s;
    const uint32_t x[6] = {ref ^ nb.nx, ref ^ rx.template other<GP>(nb.nx), ref ^ nb.yp, ref ^ nb.ym, ref ^ nb.zp,
                           FOLD ? 0u : ref ^ nb.zm};
    const Patterns pat(x);
    const uint32_t base = thr + (uint32_t)(K * S * EB);
    uint32_t held[RP][4];  // the call shared with the previous word
#pragma unroll
    for (int k = 0; k < RP; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i) held[k][i] = A != 0 ? carry[k][i] : 0u;
    uint32_t lo[RP], hi[RP];  // full: bits of the rejected sites in lo; folded: pairs of the even and odd ranks
#pragma unroll
    for (int k = 0; k < RP; ++k) {
      lo[k] = hi[k] = 0u;
      // call by call from the last (see word_uniforms): the outcomes are
      // shifted in from the highest rank, and few uniforms are held at once
      static_for<0, word_calls<S, A>()>([&](auto ic) {
        constexpr int NQ = word_calls<S, A>(), q = NQ - 1 - decltype(ic)::value;
        uint32_t u[4];
        if constexpr (q == 0 && A != 0) {
#pragma unroll
          for (int i = 0; i < 4; ++i) u[i] = held[k][i];
        } else {
          const u32x4 v = philox_sweep(half[K * S / 4 + q], key[k], rk);
          u[0] = v.a;
          u[1] = v.b;
          u[2] = v.c;
          u[3] = v.d;
          if constexpr (q == NQ - 1 && (A + S) % 4 != 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) carry[k][i] = u[i];
          }
        }
        if constexpr (NEVER) {
#pragma unroll
          for (int i = 0; i < 4; ++i) u[i] = max(u[i], 1u);
        }
        static_for<0, 4>([&](auto jc) {
          constexpr int i = 3 - decltype(jc)::value, m = 4 * q + i - A;
          if constexpr (m >= 0 && m < S) {
            const int b = 16 * k + m;
            const uint32_t addr = __byte_perm(pat.f[b & 7], base, (uint32_t)(b >> 3) | 0x7650u);
            const uint32_t t = load_shared<m * EB>(addr);
            if constexpr (!FOLD) {
              lo[k] = shift_in_carry(lo[k], u[i], t);
            } else {
              const uint32_t v = (u[i] >> 8) + t;
              uint32_t& acc = (m & 1) ? hi[k] : lo[k];
              acc = __funnelshift_l(v, acc, 2);
            }
          }
        });
      });
    }
    uint32_t a = lo[0], b = hi[0];
    if constexpr (RP == 2) {
      a = __byte_perm(lo[0], lo[RP - 1], 0x5410u);
      b = __byte_perm(hi[0], hi[RP - 1], 0x5410u);
    }
    uint32_t flip;
    if constexpr (!FOLD) {
      flip = ~a;
    } else {
      const uint32_t lt = (a & 0x55555555u) | ((b << 1) & 0xAAAAAAAAu);    // compares
      const uint32_t ltz = ((a >> 1) & 0x55555555u) | (b & 0xAAAAAAAAu);  // compares ^ z
      flip = lt | (ltz ^ s ^ nb.zm);  // where not lt, ltz is z
    }
    *own = (ColourWord<RP>)(s ^ (HF::BOTH & flip));
  }
  template <int N>
  __device__ __forceinline__ void advance() {
    thr += (uint32_t)(N * HF::S * 4 * gtab_entries<L>());
    half += N * HF::S / 4;
  }
};

// P threads share a column of RP replicas (ranges of L / P rows).  Where P is
// a power of two they are lanes of one warp, and between the half sweeps only
// the warp waits (the block meets once per chunk of NH uniform tables).  Else
// thread t takes range t / ncol of column t mod ncol, and the block meets after
// every half sweep.
constexpr bool pow2(int P) { return (P & (P - 1)) == 0; }

// Column stride of words of `per_bank` columns a bank: the P row ranges of a
// column, D words apart, start on different banks.
constexpr int column_stride(int NC, int D, int P, int per_bank) {
  const int n = 32 * per_bank;
  for (int cs = NC; cs < NC + n; ++cs) {
    const int m = (D * cs) % n;
    if (m % (n / P) == 0 && ((m / (n / P)) & 1)) return cs;
  }
  return NC;
}

template <int L, int TPB, int P, int RP>
struct GTabShape {
  using GEO = Geo3<L>;
  static constexpr int NC = TPB / P;  // columns
  static constexpr int NR = NC * RP;  // replicas per block
  static constexpr int RPP = L / P;
  static constexpr int CS = pow2(P) && P > 1 ? column_stride(NC, RPP * GEO::G, P, 2 / RP) : NC;
  static constexpr int TAB = gtab_words<L>();
  static constexpr int SPIN_WORDS = (GEO::WR * CS * RP + 3) / 4 * 4;  // [2 colours][WR][CS] colour words
  // uniform tables held at once: as many as fit in the SM's shared memory
  // where the threshold table leaves room for one block, else in what does
  // not lower the occupancy the registers allow
  static constexpr int ROOM = (TPB == 1024 || TAB > 16384 ? 224 * 1024 : 216 * TPB) - 256 -
                              4 * (TAB + SPIN_WORDS + sweep_table_words<GEO, P>(0));
  static constexpr int FIT = ROOM > 0 ? ROOM / (16 * half_buffer_entries<GEO, P>()) : 0;
  static constexpr int NH = FIT >= 20 ? 20 : (FIT < 2 ? 2 : (FIT & ~1));
  // + 64 words: the table starts at the first 256-byte boundary of the
  // block's shared memory
  static constexpr size_t SMEM_WORDS = 64 + (size_t)TAB + sweep_table_words<GEO, P>(NH) + SPIN_WORDS;
  static_assert(GEO::WR * Half<GEO>::S * 64 <= TAB, "the energy table takes the threshold table's memory");
  static_assert(P * NR <= TAB, "the row ranges' energies take the threshold table's memory at the end");
  static_assert(NR <= TPB, "one thread records a replica");
  static_assert(4 * SMEM_WORDS <= SMEM_LIMIT, "shared memory of a block");
};

// Sec. 2 with the Gaussian couplings of Sec. 4: gather of the resampled
// population, theta checkerboard sweeps at beta', the energy of every replica.
// A work item stands for `slots` slots of one run; the run's blocks share its
// population evenly (whole warps of columns), so that none is left with a few
// replicas that would hold an SM for the length of a sweep.  Replica k of
// column r is slot first + k ncol + r, ncol = the columns the block's slots
// fill.
template <int L, int TPB, int P, int RP>
__global__ void __launch_bounds__(TPB) k_sweep_gtab3d(RunDev* __restrict__ runs, const Work* __restrict__ table,
                                                      int slots) {
  using GEO = Geo3<L>;
  using HF = Half<GEO>;
  using SH = GTabShape<L, TPB, P, RP>;
  constexpr int WR = GEO::WR, W = GEO::W, G = GEO::G, S = HF::S;
  constexpr int RPP = SH::RPP, CS = SH::CS, E = gtab_entries<L>();
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t smem_addr = (uint32_t)__cvta_generic_to_shared(smem);
  uint32_t* s_thr = smem + ((256u - (smem_addr & 255u)) & 255u) / 4u;
  uint4* s_tab = reinterpret_cast<uint4*>(s_thr + SH::TAB);
  ColourWord<RP>* s_spin =
      reinterpret_cast<ColourWord<RP>*>(s_thr + SH::TAB + sweep_table_words<GEO, P>(SH::NH));  // [2][WR][CS]
  const Work wk = table[blockIdx.x];
  RunDev& R = runs[wk.run];
  if (R.skip) return;
  const int64_t Rn = R.R_next;
  const int blocks = (int)((Rn + slots - 1) / slots), unit = pow2(P) ? 32 / P * RP : RP;
  const int share = (int)((Rn + (int64_t)blocks * unit - 1) / ((int64_t)blocks * unit)) * unit;  // <= slots
  const int64_t first = (int64_t)(wk.first / slots) * share;
  if (first >= Rn) return;
  const int n = (int)min((int64_t)share, Rn - first);  // slots of this block
  const int ncol = (n + RP - 1) / RP;  // columns with live slots
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float beta_f = __double2float_rn(R.beta_next);
  const int zero = fill_thresholds<L, TPB>(s_thr, R.gJ, R.gS, beta_f);
  const RoundKeys rk = make_round_keys(R.seed);
  fill_call_table<GEO, TPB>(s_tab, rk);
  const bool never = __syncthreads_or(zero) != 0;
  int part, r;
  if constexpr (pow2(P)) {
    part = lane / (32 / P);
    r = warp * (32 / P) + lane % (32 / P);
  } else {
    part = tid / ncol;
    r = tid - part * ncol;
  }
  const bool live = part < P && r < ncol;
  const int cur = R.cur, nxt = cur ^ 1;
  ColourWord<RP>* col = s_spin + r;
  bool on[RP];
#pragma unroll
  for (int k = 0; k < RP; ++k) on[k] = live && k * ncol + r < n;
  if (live) {
    const uint4* p4[RP];
#pragma unroll
    for (int k = 0; k < RP; ++k)
      p4[k] = reinterpret_cast<const uint4*>(R.spins[cur] + (size_t)(on[k] ? R.src[first + k * ncol + r] : 0) * W);
#pragma unroll 1
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
          const uint32_t e = (uint32_t)(w / G + w % G) & 1u;
          col[w * CS] = (ColourWord<RP>)take_colour<GEO, RP>(v[i], e);
          col[(WR + w) * CS] = (ColourWord<RP>)take_colour<GEO, RP>(v[i], e ^ 1u);
        }
      }
    }
  }
  const int theta = R.theta_next;
  const uint32_t T0 = (uint32_t)R.sweeps;
  const int y0 = part * RPP, w0 = y0 * G;
  const uint32_t thr0 = (uint32_t)__cvta_generic_to_shared(s_thr) + (uint32_t)(w0 * S * 4 * E);
  SweepKey key[RP];
  const int nhalf = 2 * theta;
#pragma unroll 1
  for (int h0 = 0; h0 < nhalf; h0 += SH::NH) {
    if (h0 > 0) __syncthreads();  // the previous chunk's tables are no longer read
    const int nh = min(SH::NH, nhalf - h0);
    build_half_tables<GEO, TPB, P>(s_tab, h0, nh, T0);
#pragma unroll 1
    for (int j = 0; j < nh; ++j) {
      const int c = j & 1;  // h0 is even
      if (c == 0) {
#pragma unroll
        for (int k = 0; k < RP; ++k)
          key[k] = sweep_key((uint32_t)(first + k * ncol + r), T0 + (uint32_t)((h0 + j) >> 1), rk);
      }
      if (live) {
        const uint32_t thr = thr0 + (uint32_t)(c * WR * S * 4 * E);
        const uint4* half = half_table<GEO, P>(s_tab, j) + part + w0 * S / 4;
        if (!gtab_folded<L>() && never) {
          TabUpdate<L, RP, !gtab_folded<L>()> upd{thr, half, key, rk, {}};
          walk_rows<GEO, CS, RPP>(col, c, y0, upd);
        } else {
          TabUpdate<L, RP, false> upd{thr, half, key, rk, {}};
          walk_rows<GEO, CS, RPP>(col, c, y0, upd);
        }
      }
      // the next half sweep reads the words the other threads of the column wrote
      if constexpr (!pow2(P)) __syncthreads();
      else if constexpr (P > 1) __syncwarp();
    }
  }
  __syncthreads();  // the threshold table is no longer read
  // Energy E = C0 - 2 sum of J over the anti-aligned bonds; every bond joins a
  // colour-0 and a colour-1 site, so the sums of the colour-0 sites at their
  // patterns, tabulated where the thresholds were.
#pragma unroll 1
  for (int i = tid; i < WR * S * 16; i += TPB) {
    const int site = i >> 4, m = site % S, w = site / S;
    int32_t a[4];
    gtab_anti<GEO>(R.gJ, 0, w, m, i & 15, a);
    reinterpret_cast<uint4*>(s_thr)[i] = make_uint4((uint32_t)a[0], (uint32_t)a[1], (uint32_t)a[2], (uint32_t)a[3]);
  }
  __syncthreads();
  int32_t anti[2] = {0, 0};
  if (live) {
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(s_thr);
#pragma unroll 1
    for (int y = y0; y < y0 + RPP; ++y) {
      const int yp = row_up<GEO>(y) * CS, ym = row_down<GEO>(y) * CS;
      static_for<0, G>([&](auto gc) {
        constexpr int g = decltype(gc)::value;
        const RowX<GEO> rx((uint32_t)y & 1u);  // words of odd G take the mask pair of their own parity
        const int w = y * G + g;
        const Around nb = around<GEO, CS>(col + (WR + y * G) * CS, yp, ym, gc);
        const uint32_t s = col[w * CS];
        const uint32_t x[6] = {s ^ nb.nx, s ^ rx.template other<(g & 1)>(nb.nx), s ^ nb.yp, s ^ nb.ym, s ^ nb.zp,
                               s ^ nb.zm};
        const Patterns pat(x);
        static_for<0, RP * S>([&](auto ic) {
          constexpr int k = decltype(ic)::value / S, m = decltype(ic)::value % S, b = 16 * k + m;
          const uint32_t four_p = __byte_perm(pat.f[b & 7], 0u, (uint32_t)(b >> 3) | 0x4440u);
          anti[k] += (int32_t)load_shared<m * 256>(base + (uint32_t)(w * S * 256) + four_p);
        });
      });
    }
  }
  __syncthreads();  // the sums are no longer read
  int32_t* s_anti = reinterpret_cast<int32_t*>(s_thr);  // [P][NR]
  if (live) {
#pragma unroll
    for (int k = 0; k < RP; ++k)
      if (on[k]) s_anti[part * SH::NR + k * ncol + r] = anti[k];
    uint4* d4[RP];
#pragma unroll
    for (int k = 0; k < RP; ++k)
      d4[k] = reinterpret_cast<uint4*>(R.spins[nxt] + (size_t)(first + k * ncol + r) * W);
#pragma unroll 1
    for (int q = part; q < W / 4; q += P) {
      uint32_t v[RP][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int w = 4 * q + i;
        const bool in = w < WR;
        const uint32_t e = (uint32_t)(w / G + w % G) & 1u;
        const uint32_t a = in ? (uint32_t)col[w * CS] : 0u, b = in ? (uint32_t)col[(WR + w) * CS] : 0u;
        v[0][i] = place_colour<GEO, 0>(a, e) | place_colour<GEO, 0>(b, e ^ 1u);
        if constexpr (RP == 2) v[RP - 1][i] = place_colour<GEO, 1>(a, e) | place_colour<GEO, 1>(b, e ^ 1u);
      }
#pragma unroll
      for (int k = 0; k < RP; ++k)
        if (on[k]) d4[k][q] = make_uint4(v[k][0], v[k][1], v[k][2], v[k][3]);
    }
  }
  __syncthreads();
  if ((tid & ~31) >= n) return;  // whole warps
  int En = R.gC0;
  if (tid < n)
    for (int q = 0; q < P; ++q) En -= 2 * s_anti[q * SH::NR + tid];
  measure_store_gauss(R, nxt, first + tid, tid < n, En);
}

template <int L, int TPB, int P, int RP>
cudaError_t launch_gtab3d_p(const Sweep3dLaunch& a) {
  if constexpr (!gtab_shape_ok(L, P, RP)) {
    return cudaErrorInvalidValue;
  } else {
    using SH = GTabShape<L, TPB, P, RP>;
    if (a.slots > SH::NR) return cudaErrorInvalidValue;
    const size_t sm = sizeof(uint32_t) * SH::SMEM_WORDS;
    if (a.nwork <= 0) {
      if (sm <= 48 * 1024) return cudaSuccess;
      return allow_shared(k_sweep_gtab3d<L, TPB, P, RP>);
    }
    k_sweep_gtab3d<L, TPB, P, RP><<<a.nwork, TPB, sm, a.st>>>(a.runs, a.table, a.slots);
    return cudaGetLastError();
  }
}

template <int L, int TPB>
cudaError_t launch_gtab3d_t(const Sweep3dLaunch& a) {
  const bool one = a.rp == 1;
  switch (a.split) {
    case 1: return one ? launch_gtab3d_p<L, TPB, 1, 1>(a) : cudaErrorInvalidValue;
    case 2: return one ? cudaErrorInvalidValue : launch_gtab3d_p<L, TPB, 2, 2>(a);
    case 3: return one ? launch_gtab3d_p<L, TPB, 3, 1>(a) : launch_gtab3d_p<L, TPB, 3, 2>(a);
    case 4: return one ? launch_gtab3d_p<L, TPB, 4, 1>(a) : launch_gtab3d_p<L, TPB, 4, 2>(a);
    case 5: return one ? launch_gtab3d_p<L, TPB, 5, 1>(a) : launch_gtab3d_p<L, TPB, 5, 2>(a);
    case 8: return one ? launch_gtab3d_p<L, TPB, 8, 1>(a) : launch_gtab3d_p<L, TPB, 8, 2>(a);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pa

// Edges with threshold tables: blocks of 32 .. 256 threads take the
// estimate-and-window kernel of pa_gauss3d.cuh, 512 and 1024 the tables.
#define PA_INSTANTIATE_GAUSS3D_TAB(LL)                                                                \
  namespace pa {                                                                                      \
  cudaError_t launch_gauss3d_L##LL(const Sweep3dLaunch& a, bool init) {                               \
    if (!init && a.tpb == 512) return launch_gtab3d_t<LL, 512>(a);                                    \
    if (!init && a.tpb == 1024) return launch_gtab3d_t<LL, 1024>(a);                                  \
    return init ? launch_gauss3d_init_any<LL>(a) : launch_gauss3d_any<LL>(a);                         \
  }                                                                                                   \
  bool gauss3d_split_ok_L##LL(int split) { return split <= 4 && split_ok<Geo3<LL>>(split); }          \
  }
