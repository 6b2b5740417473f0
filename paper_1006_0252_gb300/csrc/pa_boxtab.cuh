// pa_boxtab.cuh -- sweeps of general Lx x Ly x Lz boxes (any axes open, either
// coupling model) with a threshold table per site, for boxes whose table fits
// a block's shared memory (256 bytes a site, up to about 800 sites).
//
// The pattern of a site is which of its six neighbours are anti-aligned with
// it; its energy change dE(x) = 4 sum_{d: x_d = 1} J_d - 2 S takes at most 64
// values, fixed by the couplings (an absent bond has J = 0, so its bit does not
// matter and may be junk).  Every block tabulates, once per launch, for each
// site and pattern 2^32 - t, where the site flips iff its uniform u < t (t =
// 2^32 for dE <= 0, whose entry is 0): adding the uniform carries exactly when
// it rejects, as in the Gaussian cubic kernel (pa_gauss3d_tab.cuh).  t = 0 has
// no entry; it takes that of t = 1.  So every thread keeps the minimum of its
// uniforms of a half sweep, and in a block with such an entry a minimum of 0
// sends it to decide_zeros.
//
// Words are split by colour as in pa_colour3d.cuh, with the geometry known only
// at run time: the S = k Lx / 2 colour-c sites of a word by rank m = j Lx/2 +
// h, up to RP = 4 (S <= 8) or 2 replicas side by side at multiples of T = 8 or
// 16 bits.  The neighbours of a colour-c site are at its own rank in the words
// y +- 1 and z +- 1 of the other colour (moved by a lane across the end of a
// row of words), at its own rank in the word itself, and one rotated within
// the lane.  S is a template parameter, because the uniforms of a word start
// at rank w S of the colour and a generator call serves four ranks.
//
// P threads (lanes of one warp) share a column of replicas on ranges of words.
//
// What bounds it: instruction issue at full blocks (27 instructions a flip at
// four sites a word: the generator 8.5, the walk and the patterns of a word shared
// by 16 flips), in small populations the 15-20 us of tables, gather and energies.
// One launch, theta = 10, us at beta = 0.5, site at a time (pa_box.cu, every box
// before) -> this kernel:
//   8 x 6 x 5, +-1       20000 replicas 832 -> 82      1000 775 -> 31
//   8 x 6 x 5, Gaussian  20000          903 -> 82
//   6 x 8 x 8, +-1       30000         1311 -> 130
//   8 x 8 x 8, Gaussian  10000         1765 -> 70      (open z)
//   6 x 6 x 7, Gaussian   3000          955 -> 64
// (Uniforms of 0 looked for site by site under a flag took 46 instructions and
// 109 us of the first: predicated off, they are issued all the same.)
#pragma once
#include "pa_gauss.cuh"
#include "pa_lattice3d.cuh"
#include "pa_patterns.cuh"

namespace pa {

// Run-time geometry of a box in rank space (RP copies of every mask).
template <int S>
struct BoxWords {
  static constexpr int T = S <= 8 ? 8 : 16;
  static constexpr int RP = 32 / T;
  static constexpr uint32_t rep(uint32_t m) {
    uint32_t r = 0;
    for (int k = 0; k < RP; ++k) r |= m << (T * k);
    return r;
  }
  static constexpr uint32_t ALL = rep((1u << S) - 1u);
  int H, G, Ly, WR;         // sites of a lane, words of a row, rows, words
  uint32_t f0, fh, low, up;  // h = 0, h = H - 1; ranks below S - H, from H on
  uint32_t odd;              // lanes of odd j where G is odd, else none
  __device__ __forceinline__ BoxWords(const BoxShape& b, int wr) : H(b.Lx / 2), G(b.G), Ly(b.Ly), WR(wr) {
    uint32_t first = 0u, o = 0u;
    for (int j = 0; j * H < S; ++j) {
      first |= 1u << (j * H);
      if (j & 1) o |= ((1u << H) - 1u) << (j * H);
    }
    f0 = rep(1u) * first;
    fh = f0 << (H - 1);
    low = rep(1u) * ((1u << (S - H)) - 1u);
    up = (low << H) & ALL;
    odd = (G & 1) ? rep(1u) * o : 0u;
  }
  // Ranks of word (y, g) whose colour-c sites have odd x.
  __device__ __forceinline__ uint32_t odd_x(int c, int y, int g) const { return ((c + y + g) & 1) ? ~odd : odd; }
  __device__ __forceinline__ uint32_t lane_next(uint32_t x) const {
    return ((x >> H) & low) | ((x << (S - H)) & (ALL & ~low));
  }
  __device__ __forceinline__ uint32_t lane_prev(uint32_t x) const {
    return ((x << H) & up) | ((x >> (S - H)) & (ALL & ~up));
  }
  // The x neighbour at another rank: h + 1 where x is odd, h - 1 where even.
  __device__ __forceinline__ uint32_t other(uint32_t b, uint32_t m) const {
    const uint32_t down = ((b << 1) & ~f0) | ((b >> (H - 1)) & f0);
    const uint32_t more = ((b >> 1) & ~fh) | ((b << (H - 1)) & fh);
    return (more & m) | (down & ~m);
  }
  // Anti-alignment words of the colour-c sites s of word (y, g): bits x at the
  // same and at the other rank, +y, -y, +z, -z; oth: the other colour's words.
  __device__ __forceinline__ void around(const uint32_t* __restrict__ oth, int CS, int c, int y, int g, uint32_t s,
                                         uint32_t (&x)[6]) const {
    const int w = y * G + g;
    const uint32_t nx = oth[w * CS];
    x[0] = s ^ nx;
    x[1] = s ^ other(nx, odd_x(c, y, g));
    x[2] = s ^ oth[(y + 1 < Ly ? w + G : g) * CS];
    x[3] = s ^ oth[(y > 0 ? w - G : w + (Ly - 1) * G) * CS];
    const uint32_t zp = oth[(g + 1 < G ? w + 1 : w + 1 - G) * CS], zm = oth[(g > 0 ? w - 1 : w + G - 1) * CS];
    x[4] = s ^ (g + 1 < G ? zp : lane_next(zp));
    x[5] = s ^ (g > 0 ? zm : lane_prev(zm));
  }
};

// sum_{d: x_d = 1} J_d at the patterns 4 h .. 4 h + 3 of a site.  gJ: of the
// site, direction d at d * plane (+x, -x, +y, -y, +z, -z); the x neighbour at
// its own rank is +x where x is even.
__device__ __forceinline__ void box_anti(const int32_t* __restrict__ gJ, int plane, int odd, int h, int32_t (&a)[4]) {
  int32_t acc = 0;
#pragma unroll
  for (int d = 2; d < 6; ++d)
    if ((h >> (d - 2)) & 1) acc += __ldg(gJ + d * plane);
  const int32_t j0 = __ldg(gJ + odd * plane), j1 = __ldg(gJ + (1 - odd) * plane);
  a[0] = acc;
  a[1] = acc + j0;
  a[2] = acc + j1;
  a[3] = acc + j0 + j1;
}

// Words w0 .. w1-1 of a column after a colour-c half sweep at sweep T: sites whose
// uniform was 0 were flipped (no entry makes 0 carry), and those that rise with
// threshold 0 go back.  Their neighbours have the other colour and are as they
// were.  Slow: a uniform is 0 once in 2^32 draws.  (Inline: a call here would
// cost registers in the sweep, 5 us of 34 in a launch of 1000 replicas.)
__device__ __forceinline__ void decide_zeros(const RunDev& R, uint32_t* own, const uint32_t* oth, int CS, int S,
                                             int field, int c, int w0, int w1, int reps, int64_t slot, int ncol,
                                             uint32_t T, float beta_f) {
  const int plane = R.Wr * S, H = R.bx / 2;
#pragma unroll 1
  for (int w = w0; w < w1; ++w)
#pragma unroll 1
    for (int m = 0; m < S; ++m)
#pragma unroll 1
      for (int k = 0; k < reps; ++k) {
        const int at = w * S + m;
        const uint32_t call = (uint32_t)at >> 2, s_k = (uint32_t)(slot + (int64_t)k * ncol);
        if (pick(philox_seeded(R.seed, call, s_k, T, TAG_SWEEP + (uint32_t)c), at & 3) != 0u) continue;
        const uint32_t bit = 1u << (field * k + m);
        const uint32_t s = (own[w * CS] & bit) ? 0u : 1u;  // before the flip
        int32_t acc = 0;
        for (int d = 0; d < 6; ++d) {
          const int32_t J = R.gJ[(c * 6 + d) * plane + at];
          if (J == 0) continue;
          const int code = R.box_code[(c * 7 + 1 + d) * plane + at], p = code & 31;  // the neighbour's packed place
          const int rank = p / R.bx * H + p % R.bx / 2;
          if (((oth[(code >> 5) * CS] >> (field * k + rank)) & 1u) != s) acc += J;
        }
        const int32_t dE = 4 * acc - 2 * R.gS[c * plane + at];
        if (dE > 0 && (R.model == 1 ? gauss_threshold(dE, beta_f) : R.thr[dE >> 1]) == 0u) own[w * CS] ^= bit;
      }
}

// Sec. 2: gather of the resampled population, theta checkerboard sweeps at
// beta', the energy of every replica.  A work item stands for a.slots slots of
// one run; the run's blocks share its population evenly.  Replica k of column
// r is slot first + k ncol + r, k < a.rp.
template <int S>
__global__ void __launch_bounds__(BOX_TPB) k_sweep_boxtab(RunDev* __restrict__ runs, const Work* __restrict__ table,
                                                          BoxShape box) {
  using B = BoxWords<S>;
  constexpr int T = B::T, RP = B::RP, U = S % 4 == 0 ? 1 : (S % 2 == 0 ? 2 : 4);
  extern __shared__ __align__(16) uint32_t smem[];
  const Work wk = table[blockIdx.x];
  RunDev& R = runs[wk.run];
  if (R.skip) return;
  const int P = box.P, RW = 32 / P, reps = box.reps;
  const int64_t Rn = R.R_next;
  const int blocks = (int)((Rn + box.slots - 1) / box.slots), unit = RW * reps;
  const int share = (int)((Rn + (int64_t)blocks * unit - 1) / ((int64_t)blocks * unit)) * unit;  // <= slots
  const int64_t first = (int64_t)(wk.first / box.slots) * share;
  if (first >= Rn) return;
  const int n = (int)min((int64_t)share, Rn - first);  // slots of this block
  const int ncol = (n + reps - 1) / reps;
  const int W = R.W, WR = R.Wr, plane = WR * S;
  const BoxTabShape sh = boxtab_shape(WR, S, box);
  const int CS = sh.CS;
  const uint32_t smem_addr = (uint32_t)__cvta_generic_to_shared(smem);
  uint32_t* s_thr = smem + ((256u - (smem_addr & 255u)) & 255u) / 4u;
  uint4* s_tab = reinterpret_cast<uint4*>(s_thr + sh.thr_words);
  uint32_t* s_spin = reinterpret_cast<uint32_t*>(s_tab + sh.NH * sh.Q);  // [2 colours][WR][CS]
  const B bw(box, WR);
  const int tid = threadIdx.x, lane = tid & 31;
  const float beta_f = __double2float_rn(R.beta_next);
  const int model = R.model;
  // thresholds: of the patterns p and 63 - p, whose energy changes are
  // opposite, at most one rises
  int zero = 0;
  uint4* s4 = reinterpret_cast<uint4*>(s_thr);
#pragma unroll 1
  for (int i = tid; i < 2 * plane * 8; i += BOX_TPB) {
    const int site = i >> 3, h = i & 7, c = site >= plane, at = site - c * plane, w = at / S, m = at - w * S;
    const int y = w / bw.G, z = w - y * bw.G + (m / bw.H) * bw.G;
    int32_t a[4];
    box_anti(R.gJ + (size_t)c * 6 * plane + at, plane, (c + y + z) & 1, h, a);
    const int32_t two_s = 2 * __ldg(R.gS + site);
    uint32_t e[4], f[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int32_t dE = 4 * a[j] - two_s;
      uint32_t t = 0u;  // the entry of the rise
      if (dE != 0) {
        t = model == 1 ? gauss_threshold(abs(dE), beta_f) : R.thr[abs(dE) >> 1];
        if (t == 0u) {
          zero = 1;
          t = 0xFFFFFFFFu;
        } else {
          t = model == 1 ? 0u - (t << 8) : 0u - t;
        }
      }
      e[j] = dE > 0 ? t : 0u;
      f[3 - j] = dE < 0 ? t : 0u;
    }
    s4[site * 16 + h] = make_uint4(e[0], e[1], e[2], e[3]);
    s4[site * 16 + 15 - h] = make_uint4(f[0], f[1], f[2], f[3]);
  }
  const bool never = __syncthreads_or(zero) != 0;
  const RoundKeys rk = make_round_keys(R.seed);
  const int part = lane / RW, r = (tid >> 5) * RW + lane % RW;
  const bool live = r < ncol;
  const int cur = R.cur, nxt = cur ^ 1;
  uint32_t* col = s_spin + r;
  const auto on = [&](int k) { return live && k < reps && k * ncol + r < n; };
  if (live) {
    int64_t src[RP];
#pragma unroll
    for (int k = 0; k < RP; ++k) src[k] = on(k) ? R.src[first + k * ncol + r] : 0;
    for (int w = part; w < WR; w += P) {
      const int y = w / bw.G, g = w - y * bw.G;
      const uint32_t m0 = spread_even<0>(bw.odd_x(0, y, g) & 0xFFFFu);  // even places of lanes whose colour-0 x is odd
      uint32_t a = 0u, b = 0u;
#pragma unroll
      for (int k = 0; k < RP; ++k) {
        const uint32_t v = on(k) ? R.spins[cur][(size_t)src[k] * W + w] : 0u;
        const uint32_t x0[1] = {((v & ~m0) | ((v >> 1) & m0)) & 0x55555555u};
        const uint32_t x1[1] = {(((v >> 1) & ~m0) | (v & m0)) & 0x55555555u};
        a |= (gather_even<1>(x0) & ((1u << S) - 1u)) << (T * k);
        b |= (gather_even<1>(x1) & ((1u << S) - 1u)) << (T * k);
      }
      col[w * CS] = a;
      col[(WR + w) * CS] = b;
    }
  }
  const uint32_t thr = (uint32_t)__cvta_generic_to_shared(s_thr);
  const int theta = R.theta_next, nhalf = 2 * theta;
  const uint32_t T0 = (uint32_t)R.sweeps;
  const int groups = (WR + U - 1) / U, gpp = (groups + P - 1) / P;
  const int w0 = min(part * gpp, groups) * U, w1 = min(w0 + gpp * U, WR);
  SweepKey key[RP];
#pragma unroll 1
  for (int h0 = 0; h0 < nhalf; h0 += sh.NH) {
    if (h0 > 0) __syncthreads();  // the previous chunk's tables are no longer read
    const int nh = min(sh.NH, nhalf - h0);
    for (int i = tid; i < nh * sh.Q; i += BOX_TPB) {
      const int j = i / sh.Q, q = i - j * sh.Q;
      s_tab[i] = sweep_half_entry(sweep_call_entry((uint32_t)q, TAG_SWEEP + (uint32_t)(j & 1), rk),
                                  PHILOX_MUL1 * (T0 + (uint32_t)((h0 + j) >> 1)));
    }
    __syncthreads();
#pragma unroll 1
    for (int j = 0; j < nh; ++j) {
      const int c = j & 1;  // h0 is even
      if (c == 0) {
#pragma unroll
        for (int k = 0; k < RP; ++k)
          key[k] = sweep_key((uint32_t)(first + k * ncol + r), T0 + (uint32_t)((h0 + j) >> 1), rk);
      }
      uint32_t* own = col + c * WR * CS;
      const uint32_t* oth = col + (1 - c) * WR * CS;
      uint32_t low = ~0u;  // the minimum of the half sweep's uniforms
      uint32_t carry[RP][4];
#pragma unroll
      for (int k = 0; k < RP; ++k) carry[k][0] = carry[k][1] = carry[k][2] = carry[k][3] = 0u;
      int y = w0 / bw.G, g = w0 - y * bw.G;
#pragma unroll 1
      for (int wg = live ? w0 : w1; wg < w1; wg += U) {
        const uint4* half = s_tab + j * sh.Q + wg * S / 4;
        static_for<0, U>([&](auto uc) {
          constexpr int K = decltype(uc)::value, A = (K * S) % 4, NQ = word_calls<S, A>();
          const int w = wg + K;
          if (w < w1) {
            const uint32_t s = own[w * CS];
            uint32_t x[6];
            bw.around(oth, CS, c, y, g, s, x);
            const Patterns pat(x);
            const uint32_t base = thr + (uint32_t)(c * plane + w * S) * 256u;
            uint32_t stay = ~0u;
#pragma unroll
            for (int k = 0; k < RP; ++k) {
              if (k >= reps) break;
              uint32_t ge = 0u;
              uint32_t held[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) held[i] = carry[k][i];
              // call by call from the last, so that the outcomes are shifted in
              // from the highest rank
              static_for<0, NQ>([&](auto ic) {
                constexpr int q = NQ - 1 - decltype(ic)::value;
                uint32_t u[4];
                if constexpr (q == 0 && A != 0) {
#pragma unroll
                  for (int i = 0; i < 4; ++i) u[i] = held[i];
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
                low = __vimin3_u32(__vimin3_u32(low, u[0], u[1]), u[2], u[3]);
                static_for<0, 4>([&](auto jc) {
                  constexpr int i = 3 - decltype(jc)::value, m = 4 * q + i - A;
                  if constexpr (m >= 0 && m < S) {
                    const int b = T * k + m;
                    const uint32_t addr = __byte_perm(pat.f[b & 7], base, (uint32_t)(b >> 3) | 0x7650u);
                    ge = shift_in_carry(ge, u[i], load_shared<m * 256>(addr));
                  }
                });
              });
              stay &= ~(((~ge) & ((1u << S) - 1u)) << (T * k));
            }
            own[w * CS] = s ^ (B::ALL & ~stay);
          }
          if (++g == bw.G) {
            g = 0;
            ++y;
          }
        });
      }
      if (never && low == 0u)
        decide_zeros(R, own, oth, CS, S, T, c, w0, w1, reps, first + r, ncol, T0 + (uint32_t)((h0 + j) >> 1), beta_f);
      __syncwarp();  // the next half sweep reads what the other threads of the column wrote
    }
  }
  __syncthreads();  // the thresholds are no longer read
  // Energy E = C0 - 2 sum of J over the anti-aligned bonds; every bond joins a
  // colour-0 and a colour-1 site: the sums of the colour-0 sites at their
  // patterns, tabulated where the thresholds were.
#pragma unroll 1
  for (int i = tid; i < plane * 16; i += BOX_TPB) {
    const int at = i >> 4, w = at / S, m = at - w * S, y = w / bw.G, z = w - y * bw.G + (m / bw.H) * bw.G;
    int32_t a[4];
    box_anti(R.gJ + at, plane, (y + z) & 1, i & 15, a);
    s4[i] = make_uint4((uint32_t)a[0], (uint32_t)a[1], (uint32_t)a[2], (uint32_t)a[3]);
  }
  __syncthreads();
  int32_t anti[RP] = {};
  if (live) {
    for (int w = w0; w < w1; ++w) {
      const int y = w / bw.G, g = w - y * bw.G;
      const uint32_t s = col[w * CS];
      uint32_t x[6];
      bw.around(col + WR * CS, CS, 0, y, g, s, x);
      const Patterns pat(x);
      const uint32_t base = thr + (uint32_t)(w * S) * 256u;
      static_for<0, RP * S>([&](auto ic) {
        constexpr int k = decltype(ic)::value / S, m = decltype(ic)::value % S, b = T * k + m;
        const uint32_t addr = __byte_perm(pat.f[b & 7], base, (uint32_t)(b >> 3) | 0x7650u);
        anti[k] += (int32_t)load_shared<m * 256>(addr);
      });
    }
    for (int w = part; w < W; w += P) {
      const bool in = w < WR;
      const int y = in ? w / bw.G : 0, g = in ? w - y * bw.G : 0;
      const uint32_t m0 = spread_even<0>(bw.odd_x(0, y, g) & 0xFFFFu);
      const uint32_t a = in ? col[w * CS] : 0u, b = in ? col[(WR + w) * CS] : 0u;
#pragma unroll
      for (int k = 0; k < RP; ++k) {
        const uint32_t ea = spread_even<0>((a >> (T * k)) & ((1u << S) - 1u));
        const uint32_t eb = spread_even<0>((b >> (T * k)) & ((1u << S) - 1u));
        if (on(k))
          R.spins[nxt][(size_t)(first + k * ncol + r) * W + w] =
              (ea & ~m0) | ((ea & m0) << 1) | (eb & m0) | ((eb & ~m0) << 1);
      }
    }
  }
  __syncthreads();  // the sums are no longer read
  int32_t* s_anti = reinterpret_cast<int32_t*>(s_thr);  // [P][slots]
#pragma unroll
  for (int k = 0; k < RP; ++k)
    if (on(k)) s_anti[part * box.slots + k * ncol + r] = anti[k];
  __syncthreads();
  for (int i0 = 0; i0 < n; i0 += BOX_TPB) {
    const int i = i0 + tid;
    if ((i & ~31) >= n) return;  // whole warps
    int En = R.gC0;
    if (i < n)
      for (int q = 0; q < P; ++q) En -= 2 * s_anti[q * box.slots + i];
    if (model == 1) measure_store_gauss(R, nxt, first + i, i < n, En);
    else measure_store(R, nxt, first + i, i < n, En);
  }
}

template <int S>
cudaError_t launch_boxtab_s(const BoxShape& box, RunDev* runs, const Work* table, int nwork, int WR,
                            cudaStream_t st) {
  const size_t sm = sizeof(uint32_t) * boxtab_shape(WR, S, box).words;
  if (nwork <= 0) {
    if (sm <= 48 * 1024) return cudaSuccess;
    return allow_shared(k_sweep_boxtab<S>);
  }
  k_sweep_boxtab<S><<<nwork, BOX_TPB, sm, st>>>(runs, table, box);
  return cudaGetLastError();
}

}  // namespace pa
