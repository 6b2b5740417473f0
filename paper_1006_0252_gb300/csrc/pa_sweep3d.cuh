// pa_sweep3d.cuh -- fused replica copy + checkerboard Metropolis sweeps +
// energy measurement for 3D periodic cubic +-1 spin glasses (Sec. 2: "all
// replicas are now subject to an equilibrating MCMC process at the new
// temperature"; Algorithm: "Equilibrate replica j for theta sweeps", then
// "Compute observables").
//
// A block keeps its replicas in shared memory split by colour: for colour c
// and word w = y G + g of the packed lattice, one 32-bit word holds the word's
// S = K L / 2 colour-c sites by rank m = j L/2 + h (lane j, site x = 2h + q,
// q = (c + y + z) mod 2) of one replica in bits 0..15 and, with RP = 2, of a
// second replica in bits 16..31.  A colour-c site's neighbours all have the
// other colour, and they sit at these ranks of the other colour's words:
//   y +- 1   rank m of the words w +- G (x and the lane stay),
//   z +- 1   rank m of the words w +- 1; across the end of a row of words
//            (g = G-1 -> 0, g = 0 -> G-1) the lane moves by one: m +- L/2,
//   x +- 1   one of the two at rank m of the word w itself; the other at
//            h - 1 (q = 0) or h + 1 (q = 1), a rotation of every lane's field.
// So one 32-bit operation serves 2 S <= 32 sites of one colour (a layout with
// both colours in a word serves at most 16), the threshold compares need no
// spreading to alternate bits, and words are written in place: a half sweep
// writes colour-c words and reads colour-(1-c) words only.
//
// For every direction d the bond bit b_d = s ^ s_nb ^ j_d is 1 where the bond
// is satisfied (J s s' = -1), a carry-save adder counts the n satisfied bonds
// per site (dE = 4n - 12), and a site flips iff n <= 3 or its uniform
// u < threshold[dE/2] (only energy rises draw on the uniform).
//
// P threads share the replicas of a column (ranges of L / P rows).
//
// What bounds it.  A scheduler issues one full-rate integer instruction (two
// register operands: add, two-input logic) a cycle and a half-rate one (three
// operands, shifts, permutes, minima, multiplies) every two cycles, whatever
// pipe takes it; a wide multiply also holds the multiply pipe four cycles.  A
// generator round of a warp is 2 wide multiplies and 2 three-input XORs: 8.2
// cycles on the multiply pipe and 8 of issue (8.66 measured alone), so every
// other instruction of the sweep adds to the generator's time.  Per 16 sites
// of 32 replicas at L = 8 the generator takes 265 cycles and the launch 349
// (beta = 4) to 442 (beta = 0.1): it is issue bound, and only fewer or
// cheaper instructions help.  This layout needs 180 instructions there at
// beta = 4 where a word of both colours needed 202.  One launch, theta = 10,
// us at beta = 0.1 / 1.0 / 4.0 (both colours in a word -> this layout):
//   L = 8,  1e5 replicas    404 / 371 / 304 -> 360 / 333 / 281
//   L = 12, 30011 replicas  511 / 464 / 382 -> 420 / 389 / 330
//   L = 10, 30000 replicas  427 / 407 / 284 -> 252 / 238 / 205
//   L = 6,  40000 replicas  131 / 119 / 96  ->  97 /  91 /  79
//   L = 16, 20000 replicas  864 / 804 / 617 -> 681 / 632 / 544
//   L = 14, 20000 replicas 1083 / 995 / 687 -> 469 / 435 / 371
// (L = 6, 10 and 14 had one thread per replica before; they split in pairs of
// rows now.)
#pragma once
#include "pa_colour3d.cuh"

namespace pa {

// Bond masks of one run: [6][W] words; direction order x+, x-, y+, y-, z+, z-;
// bit (w, p) set iff the coupling of that bond of site (w, p) is -1.
enum { DXP = 0, DXM = 1, DYP = 2, DYM = 3, DZP = 4, DZM = 5 };

// Satisfied-bond counts of the "+" bonds of one word (energy measurement).
template <class GEO>
__device__ __forceinline__ int plus_bonds_satisfied(uint32_t s, uint32_t yp, uint32_t zp, uint32_t jxp, uint32_t jyp,
                                                    uint32_t jzp) {
  const uint32_t bx = s ^ rot_xp<GEO>(s) ^ jxp;
  const uint32_t by = s ^ yp ^ jyp;
  const uint32_t bz = s ^ zp ^ jzp;
  return __popc(bx & GEO::VALID) + __popc(by & GEO::VALID) + __popc(bz & GEO::VALID);
}

// Satisfied "+" bonds of rows y0 .. y1-1 of the replica in a shared-memory
// column (word w at col[w * CS]).
template <class GEO, int CS>
__device__ __forceinline__ int satisfied_rows(const uint32_t* __restrict__ col, const uint32_t* __restrict__ s_bond,
                                              int y0, int y1) {
  constexpr int G = GEO::G, L = GEO::L, W = GEO::W;
  int sat = 0;
  for (int y = y0; y < y1; ++y) {
    const int yn = (y + 1 == L) ? 0 : y + 1;
    uint32_t row[G], rowp[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      row[g] = col[(y * G + g) * CS];
      rowp[g] = col[(yn * G + g) * CS];
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int w = y * G + g;
      const uint32_t zp = (g + 1 < G) ? row[(g + 1) % G] : lanes_down<GEO>(row[0]);
      sat += plus_bonds_satisfied<GEO>(row[g], rowp[g], zp, s_bond[DXP * W + w], s_bond[DYP * W + w],
                                       s_bond[DZP * W + w]);
    }
  }
  return sat;
}

// Bond masks of the colour words, one 32-byte entry for (c, w): the x bond to
// the same rank, the x bond to the other rank, y+, y-, z+, z- (both halves
// alike).  All threads of the block; a barrier must follow.
template <class GEO, int TPB>
__device__ __forceinline__ void fill_bonds(uint4* __restrict__ s_bond, const uint32_t* __restrict__ bonds) {
  constexpr int WR = GEO::WR, W = GEO::W, G = GEO::G;
  for (int i = threadIdx.x; i < 2 * WR; i += TPB) {
    const int c = i / WR, w = i - c * WR;
    const uint32_t e = (uint32_t)(c + w / G + w % G) & 1u;
    uint32_t m[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      const uint32_t v[2] = {bonds[d * W + w], bonds[d * W + w]};
      m[d] = take_colour<GEO, 2>(v, e);
    }
    const uint32_t q = (GEO::G & 1) == 0 ? (e ? 0xFFFFFFFFu : 0u) : (e ? ~Half<GEO>::ODD : Half<GEO>::ODD);
    s_bond[2 * i] = make_uint4((m[DXM] & q) | (m[DXP] & ~q), (m[DXP] & q) | (m[DXM] & ~q), m[DYP], m[DYM]);
    s_bond[2 * i + 1] = make_uint4(m[DZP], m[DZM], 0u, 0u);
  }
}

// Satisfied-bond counts n = 4 n2 + 2 n1 + n0 of the colour-c sites s of a
// word; GP = g mod 2.
struct Count3 {
  uint32_t n0, n1, n2;
};
template <class GEO, int GP>
__device__ __forceinline__ Count3 count_satisfied(uint32_t s, const Around& n, const uint4* __restrict__ bond,
                                                  const RowX<GEO>& rx) {
  const uint4 j0 = bond[0];
  const uint2 j1 = *reinterpret_cast<const uint2*>(bond + 1);
  const uint32_t b0 = s ^ n.nx ^ j0.x;
  const uint32_t b1 = s ^ rx.template other<GP>(n.nx) ^ j0.y;
  const uint32_t b2 = s ^ n.yp ^ j0.z;
  const uint32_t b3 = s ^ n.ym ^ j0.w;
  const uint32_t b4 = s ^ n.zp ^ j1.x;
  const uint32_t b5 = s ^ n.zm ^ j1.y;
  const uint32_t sa = b0 ^ b1 ^ b2, ca = (b0 & b1) | (b2 & (b0 ^ b1));
  const uint32_t sb = b3 ^ b4 ^ b5, cb = (b3 & b4) | (b5 & (b3 ^ b4));
  const uint32_t n0 = sa ^ sb, c0 = sa & sb;
  return {n0, ca ^ cb ^ c0, (ca & cb) | (c0 & (ca ^ cb))};
}

// Everything a word's update needs beyond the lattice: the slots' keys and the
// thresholds of dE = 4, 8, 12.
template <int RP>
struct HalfSweep {
  SweepKey key[RP];
  uint32_t T4, T8, T12;
  bool low_t;      // T4 < 2^22: most words draw no uniform below T4
  bool high_t;     // T4 >= 2^24: almost every word needs the compares with T4 and T8
  unsigned lanes;  // live lanes of the warp
};

// Word g of a row of a half sweep: satisfied-bond count of all its replicas'
// sites at once, then per replica the word's uniforms and the compares, then
// the flips.  T4 >= T8 >= T12, a site with n = 4, 5, 6 takes the compare with
// T4, T8, T12, so T8 is compared only where a lane of the warp has a site of
// n >= 5 with u < T4, T12 where one of n = 6 has u < T8.  At low temperature
// the word's uniforms are first reduced to their minimum and all compares
// skipped when no lane's minimum is below T4.  half: the word's first call; A
// the alignment of its first uniform (see word_uniforms); GP = g mod 2.
template <class GEO, int RP, int A, int GP>
__device__ __forceinline__ void word3d(ColourWord<RP>* __restrict__ own, const Around& nb,
                                       const uint4* __restrict__ bond, const RowX<GEO>& rx,
                                       const uint4* __restrict__ half, const HalfSweep<RP>& hs, const RoundKeys& rk,
                                       uint32_t (&carry)[RP][4]) {
  constexpr int S = Half<GEO>::S;
  const uint32_t s = *own;
  const Count3 n = count_satisfied<GEO, GP>(s, nb, bond, rx);
  uint32_t e4 = 0u, e8 = 0u, e12 = 0u;
#pragma unroll
  for (int k = 0; k < RP; ++k) {
    uint32_t u[4 * word_calls<S, A>()];
    word_uniforms<S, A>(0u, half, hs.key[k], rk, carry[k], u);
    if (hs.low_t && !__any_sync(hs.lanes, min_of<S, A>(u) < hs.T4)) continue;
    const uint32_t m4 = lt_mask<S, A>(u, hs.T4);
    e4 |= m4 << (16 * k);
    const uint32_t n5 = (n.n2 & (n.n1 | n.n0)) >> (16 * k), n6 = (n.n2 & n.n1) >> (16 * k);
    if (!hs.high_t && !__any_sync(hs.lanes, (m4 & n5) != 0u)) continue;
    const uint32_t m8 = lt_mask<S, A>(u, hs.T8);
    e8 |= m8 << (16 * k);
    if (__any_sync(hs.lanes, (m8 & n6) != 0u)) e12 |= lt_mask<S, A>(u, hs.T12) << (16 * k);
  }
  const uint32_t sel = (n.n1 & e12) | (~n.n1 & ((n.n0 & e8) | (~n.n0 & e4)));
  *own = (ColourWord<RP>)(s ^ (Half<GEO>::BOTH & (~n.n2 | sel)));
}

// The word updates of one half sweep, as walk_rows calls them.
template <class GEO, int RP>
struct PmUpdate {
  const uint4* bond;  // of the word the walk stands at
  const uint4* half;  // its first call's entry
  const HalfSweep<RP>& hs;
  const RoundKeys& rk;
  uint32_t carry[RP][4];
  template <int K, int A, int GP>
  __device__ __forceinline__ void word(ColourWord<RP>* own, const Around& nb, const RowX<GEO>& rx) {
    word3d<GEO, RP, A, GP>(own, nb, bond + 2 * K, rx, half + K * Half<GEO>::S / 4, hs, rk, carry);
  }
  template <int N>
  __device__ __forceinline__ void advance() {
    bond += 2 * N;
    half += N * Half<GEO>::S / 4;
  }
};

// One Metropolis half sweep over the colour-c sites of the RPP rows from y0
// of the replicas of one column.  half: the column's uniform table of this
// half sweep.
template <class GEO, int CS, int RP, int RPP, class COLOUR>
__device__ __forceinline__ void half_sweep3d(ColourWord<RP>* __restrict__ col, const uint4* __restrict__ s_bond,
                                             const uint4* __restrict__ half, COLOUR c, const HalfSweep<RP>& hs,
                                             const RoundKeys& rk, int y0) {
  const int w0 = y0 * GEO::G;
  PmUpdate<GEO, RP> upd{s_bond + 2 * (c * GEO::WR + w0), half + w0 * Half<GEO>::S / 4, hs, rk, {}};
  walk_rows<GEO, CS, RPP>(col, c, y0, upd);
}

// Block of TPB threads: P threads per column of RP replicas, thread t takes
// row range t / NC of column t mod NC (NC = TPB / P columns; the last TPB - P
// NC threads of an odd P only help with the tables).  A block is a multiple of
// four warps wherever it can be: its warps go to the SM's four schedulers in
// turn, so blocks of 5 warps (one per row range, L = 10) gave one scheduler
// twice the work of the others.  Block b takes work item b / BPI of the class
// table (SLOTS consecutive slots of one run) and its (b mod BPI)-th share.
template <int L, int TPB, int P, int RP>
struct SweepShape {
  using GEO = Geo3<L>;
  static constexpr int NC = TPB / P;              // columns
  static constexpr int NR = NC * RP;              // replicas per block
  static constexpr int RPP = L / P;               // rows per thread
  static constexpr int WPP = RPP * GEO::G;        // words per thread
  static constexpr int SLOTS = (P & (P - 1)) == 0 ? TPB : NR;  // slots of a work item (LatticeClass::slots)
  static constexpr int BPI = SLOTS / NR;
  static constexpr int CS = NC;
  static constexpr int BOND_WORDS = 16 * GEO::WR;
  static constexpr int SPIN_WORDS = (GEO::WR * CS * RP + 3) / 4 * 4;  // [2 colours][WR][CS] colour words
  static constexpr int Q = calls_per_colour<GEO>();
  // half-sweep tables held at once: with one thread per column as many as
  // fit, else two, double-buffered behind one block barrier per half sweep
  static constexpr int room() {
    const int n = (216 * TPB - 4 * (BOND_WORDS + SPIN_WORDS)) / (16 * Q);
    return n >= 20 ? 20 : (n < 2 ? 2 : (n & ~1));
  }
  static constexpr int NH = P > 1 ? 2 : room();
  // the tables' memory also takes the row ranges' energies at the end
  static constexpr int TAB_WORDS = 4 * NH * Q > RP * TPB ? 4 * NH * Q : RP * TPB;
  static constexpr size_t SMEM_WORDS = (size_t)TAB_WORDS + BOND_WORDS + SPIN_WORDS;
  static constexpr bool OK = SLOTS % NR == 0 && NR <= TPB && NC >= 4 && (P == 1 || TPB >= 64);
};

// Half-sweep tables h0 .. h0 + nh - 1 (half sweep h = 2t + c is colour c of
// sweep T0 + t) at tab[(buf + j) Q + q], all threads of the block.
template <class SH, int TPB>
__device__ __forceinline__ void build_tables3d(uint4* __restrict__ tab, int buf, int h0, int nh, uint32_t T0,
                                               const RoundKeys& rk) {
  for (int i = threadIdx.x; i < nh * SH::Q; i += TPB) {
    const int j = i / SH::Q, q = i - j * SH::Q;
    const int h = h0 + j;
    const uint32_t A1 = PHILOX_MUL1 * (T0 + (uint32_t)(h >> 1));
    tab[(buf + j) * SH::Q + q] =
        sweep_half_entry(sweep_call_entry((uint32_t)q, TAG_SWEEP + (uint32_t)(h & 1), rk), A1);
  }
}

// Sec. 2: the gather of the resampled population (slot s <- old slot src(s)),
// theta checkerboard sweeps at beta', and the energy of every replica.
template <int L, int TPB, int P, int RP>
__global__ void __launch_bounds__(TPB) k_sweep3d(RunDev* __restrict__ runs, const Work* __restrict__ table) {
  using GEO = Geo3<L>;
  using SH = SweepShape<L, TPB, P, RP>;
  using HF = Half<GEO>;
  constexpr int WR = GEO::WR, W = GEO::W, G = GEO::G, CS = SH::CS, RPP = SH::RPP;
  extern __shared__ __align__(16) uint32_t smem[];
  uint4* s_tab = reinterpret_cast<uint4*>(smem);
  uint4* s_bond = reinterpret_cast<uint4*>(smem + SH::TAB_WORDS);
  ColourWord<RP>* s_spin = reinterpret_cast<ColourWord<RP>*>(smem + SH::TAB_WORDS + SH::BOND_WORDS);  // [2][WR][CS]
  const Work wk = table[blockIdx.x / SH::BPI];
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  RunDev& R = runs[wk.run];
  if (R.skip) return;
  const int64_t Rn = R.R_next;
  const int64_t first = (int64_t)wk.first + (int64_t)(blockIdx.x % SH::BPI) * SH::NR;
  if (first >= Rn) return;
  const int tid = threadIdx.x;
  fill_bonds<GEO, TPB>(s_bond, R.bonds);
  const RoundKeys rk = make_round_keys(R.seed);
  const int part = tid / SH::NC, r = tid - part * SH::NC;  // row range and column of this thread
  // replica k of column r is slot first + k NC + r
  const int64_t slot = first + r;
  const bool live = part < P && slot < Rn;
  const int cur = R.cur, nxt = cur ^ 1;
  ColourWord<RP>* col = s_spin + r;
  if (live) {
    const uint4* p4[RP];
    bool on[RP];
#pragma unroll
    for (int k = 0; k < RP; ++k) {
      on[k] = slot + k * SH::NC < Rn;
      p4[k] = reinterpret_cast<const uint4*>(R.spins[cur] + (size_t)(on[k] ? R.src[slot + k * SH::NC] : 0) * W);
    }
#pragma unroll 2
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
  HalfSweep<RP> hs;
  hs.T4 = R.thr[2];
  hs.T8 = R.thr[4];
  hs.T12 = R.thr[6];
  hs.low_t = hs.T4 < (1u << 22);
  hs.high_t = hs.T4 >= (1u << 24);
  hs.lanes = __ballot_sync(0xFFFFFFFFu, live);
  const int theta = R.theta_next;
  const uint32_t T0 = (uint32_t)R.sweeps;
  const int y0 = part * RPP;
  if constexpr (P > 1) {
    // one table per half sweep, double-buffered: the block barrier after the
    // build orders the word ranges too (a colour-c half sweep reads the
    // colour-(1-c) words the other threads just wrote) and keeps a table
    // until every thread has left the half sweep that reads it; every thread
    // of the block passes the barriers
    const auto half_sweep = [&](int t, auto c) {
      build_tables3d<SH, TPB>(s_tab, c, 2 * t + c, 1, T0, rk);
      __syncthreads();
      if (live) half_sweep3d<GEO, CS, RP, RPP>(col, s_bond, s_tab + c * SH::Q, c, hs, rk, y0);
    };
#pragma unroll 1
    for (int t = 0; t < theta; ++t) {
#pragma unroll
      for (int k = 0; k < RP; ++k) hs.key[k] = sweep_key((uint32_t)(slot + k * SH::NC), T0 + (uint32_t)t, rk);
      if constexpr (G != 2 || HF::S % 4 == 0) {
        // the colour known at compile time: the addresses of a row's words
        // and tables are then offsets of values kept over the whole launch
        half_sweep(t, std::integral_constant<int, 0>{});
        half_sweep(t, std::integral_constant<int, 1>{});
      } else {
#pragma unroll 1
        for (int c = 0; c < 2; ++c) half_sweep(t, c);
      }
    }
  } else {
    // one thread per column: the half sweeps in chunks of NH tables, one
    // block barrier per chunk
    const int nhalf = 2 * theta;
#pragma unroll 1
    for (int h0 = 0; h0 < nhalf; h0 += SH::NH) {
      if (h0 > 0) __syncthreads();  // the previous chunk's tables are no longer read
      const int nh = min(SH::NH, nhalf - h0);
      build_tables3d<SH, TPB>(s_tab, 0, h0, nh, T0, rk);
      __syncthreads();
      if (live) {
#pragma unroll 1
        for (int j = 0; j < nh; ++j) {
          const int c = j & 1;  // h0 is even
          if (c == 0) {
#pragma unroll
            for (int k = 0; k < RP; ++k)
              hs.key[k] = sweep_key((uint32_t)(slot + k * SH::NC), T0 + (uint32_t)((h0 + j) >> 1), rk);
          }
          half_sweep3d<GEO, CS, RP, RPP>(col, s_bond, s_tab + j * SH::Q, c, hs, rk, y0);
        }
      }
    }
  }
  __syncthreads();  // every word range swept before the energy reads its neighbours
  // every bond joins a colour-0 and a colour-1 site: the satisfied bonds are
  // the counts n of the colour-0 sites
  int sat[2] = {0, 0};
  if (live) {
#pragma unroll 1
    for (int y = y0; y < y0 + RPP; ++y) {
      const int yp = row_up<GEO>(y) * CS, ym = row_down<GEO>(y) * CS;
      static_for<0, G>([&](auto gc) {
        constexpr int g = decltype(gc)::value, w = g;
        // words of odd G take the mask pair of their own parity
        const RowX<GEO> rx((uint32_t)y & 1u);
        const Around nb = around<GEO, CS>(col + (WR + y * G) * CS, yp, ym, gc);
        const Count3 n = count_satisfied<GEO, (g & 1)>(col[(y * G + w) * CS], nb, s_bond + 2 * (y * G + w), rx);
#pragma unroll
        for (int k = 0; k < RP; ++k) {
          const uint32_t m = HF::ONE << (16 * k);
          sat[k] += __popc(n.n0 & m) + 2 * __popc(n.n1 & m) + 4 * __popc(n.n2 & m);
        }
      });
    }
    uint4* d4[RP];
#pragma unroll
    for (int k = 0; k < RP; ++k) d4[k] = reinterpret_cast<uint4*>(R.spins[nxt] + (size_t)(slot + k * SH::NC) * W);
#pragma unroll 2
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
        if (slot + k * SH::NC < Rn) d4[k][q] = make_uint4(v[k][0], v[k][1], v[k][2], v[k][3]);
    }
  }
  // sum over the row ranges, then record one replica per thread
  int* s_sat = reinterpret_cast<int*>(s_tab);  // [P][NR]; the tables are no longer read
  if (part < P) {
#pragma unroll
    for (int k = 0; k < RP; ++k) s_sat[part * SH::NR + k * SH::NC + r] = sat[k];
  }
  __syncthreads();
  if ((tid & ~31) >= SH::NR) return;  // whole warps
  int E = GEO::NB;
  const bool rec = tid < SH::NR && first + tid < Rn;
  if (rec)
    for (int q = 0; q < P; ++q) E -= 2 * s_sat[q * SH::NR + tid];
  measure_store(R, nxt, first + tid, rec, E);
}

// Sec. 2: R0 independent uniformly random microstates at beta = 0.  Word w of
// slot s is word (w mod 4) of Philox(ctr = (w div 4, s, 0, TAG_INIT)),
// restricted to the valid lanes.  One thread per slot of a work item.
template <int L, int TPB>
__global__ void __launch_bounds__(TPB) k_init3d(RunDev* __restrict__ runs, const Work* __restrict__ table,
                                                int slots) {
  using GEO = Geo3<L>;
  constexpr int WR = GEO::WR, W = GEO::W;
  extern __shared__ uint32_t smem[];
  uint32_t* s_bond = smem;
  uint32_t* s_spin = smem + 6 * W;
  const Work wk = table[blockIdx.x];
  RunDev& R = runs[wk.run];
  const int64_t R0 = R.R;
  if ((int64_t)wk.first >= R0) return;
  const int tid = threadIdx.x;
  for (int i = tid; i < 6 * W; i += TPB) s_bond[i] = R.bonds[i];
  const int64_t slot = (int64_t)wk.first + tid;
  const bool live = tid < slots && slot < R0;
  uint32_t* col = s_spin + tid;
  if (live) {
    for (int w4 = 0; w4 < W / 4; ++w4) {
      const u32x4 u = philox_seeded(R.seed, (uint32_t)w4, (uint32_t)slot, 0u, TAG_INIT);
      if (4 * w4 + 0 < WR) col[(4 * w4 + 0) * TPB] = u.a & GEO::VALID;
      if (4 * w4 + 1 < WR) col[(4 * w4 + 1) * TPB] = u.b & GEO::VALID;
      if (4 * w4 + 2 < WR) col[(4 * w4 + 2) * TPB] = u.c & GEO::VALID;
      if (4 * w4 + 3 < WR) col[(4 * w4 + 3) * TPB] = u.d & GEO::VALID;
    }
  }
  __syncthreads();
  int E = 0;
  if (live) {
    E = GEO::NB - 2 * satisfied_rows<GEO, TPB>(col, s_bond, 0, L);
    store_column<GEO, TPB>(R.spins[0] + (size_t)slot * W, col);
  }
  measure_store(R, 0, slot, live, E);
}

template <int L, int TPB>
inline size_t init3d_smem() {
  using GEO = Geo3<L>;
  return sizeof(uint32_t) * (6 * GEO::W + GEO::WR * TPB);
}

// One launch over nwork work items (with nwork <= 0 the kernel is only
// allowed its shared memory, outside any stream capture).
template <int L, int TPB, int P, int RP>
cudaError_t sweep3d_p(const Sweep3dLaunch& a) {
  if constexpr (!rows_split<Geo3<L>>(P)) {
    return cudaErrorInvalidValue;
  } else if constexpr (!SweepShape<L, TPB, P, RP>::OK) {
    return cudaErrorInvalidValue;
  } else {
    using SH = SweepShape<L, TPB, P, RP>;
    const int need = (int)(sizeof(uint32_t) * SH::SMEM_WORDS), sm = need > a.min_smem ? need : a.min_smem;
    if (a.nwork <= 0) {
      if (sm <= 48 * 1024) return cudaSuccess;
      return allow_shared(k_sweep3d<L, TPB, P, RP>);
    }
    return launch_dependent(k_sweep3d<L, TPB, P, RP>, a.nwork * SH::BPI, TPB, (size_t)sm, a.st, a.runs, a.table);
  }
}

template <int L, int TPB>
cudaError_t launch_init3d_t(int slots, RunDev* runs, const Work* table, int nwork, cudaStream_t st) {
  const size_t sm = init3d_smem<L, TPB>();
  if (sm > 48 * 1024) {
    const cudaError_t e = allow_shared(k_init3d<L, TPB>);
    if (e != cudaSuccess) return e;
  }
  if (nwork <= 0) return cudaSuccess;
  k_init3d<L, TPB><<<nwork, TPB, sm, st>>>(runs, table, slots);
  return cudaGetLastError();
}

template <int L, int TPB>
cudaError_t sweep3d_t(const Sweep3dLaunch& a) {
  const bool one = a.rp == 1;
  switch (a.split) {
    case 1: return one ? sweep3d_p<L, TPB, 1, 1>(a) : cudaErrorInvalidValue;
    case 2: return one ? sweep3d_p<L, TPB, 2, 1>(a) : sweep3d_p<L, TPB, 2, 2>(a);
    case 4: return one ? sweep3d_p<L, TPB, 4, 1>(a) : sweep3d_p<L, TPB, 4, 2>(a);
    case 8: return one ? sweep3d_p<L, TPB, 8, 1>(a) : sweep3d_p<L, TPB, 8, 2>(a);
    default: return cudaErrorInvalidValue;
  }
}

// Further splits, not powers of two: whole pairs of rows where a row's
// uniforms end within a call (L = 6, 10, 14), one or two rows at L = 12.
template <int L>
constexpr bool extra_split(int P) {
  return (L == 6 && P == 3) || (L == 10 && P == 5) || (L == 14 && P == 7) || (L == 12 && (P == 6 || P == 12));
}

template <int L, int P>
cudaError_t sweep3d_extra(const Sweep3dLaunch& a) {
  if constexpr (extra_split<L>(P)) {
    const bool one = a.rp == 1;
    switch (a.tpb) {
      case 64: return one ? sweep3d_p<L, 64, P, 1>(a) : sweep3d_p<L, 64, P, 2>(a);
      case 128: return one ? sweep3d_p<L, 128, P, 1>(a) : sweep3d_p<L, 128, P, 2>(a);
      case 256: return one ? sweep3d_p<L, 256, P, 1>(a) : sweep3d_p<L, 256, P, 2>(a);
    }
  }
  return cudaErrorInvalidValue;
}

template <int L>
cudaError_t sweep3d_any(const Sweep3dLaunch& a) {
  switch (a.split) {
    case 3: return sweep3d_extra<L, 3>(a);
    case 5: return sweep3d_extra<L, 5>(a);
    case 6: return sweep3d_extra<L, 6>(a);
    case 7: return sweep3d_extra<L, 7>(a);
    case 12: return sweep3d_extra<L, 12>(a);
  }
  switch (a.tpb) {
    case 32: return sweep3d_t<L, 32>(a);
    case 64: return sweep3d_t<L, 64>(a);
    case 128: return sweep3d_t<L, 128>(a);
    case 256: return sweep3d_t<L, 256>(a);
    default: return cudaErrorInvalidValue;
  }
}

template <int L>
cudaError_t launch_init3d(int slots, RunDev* runs, const Work* table, int nwork, cudaStream_t st) {
  if (slots <= 32) return launch_init3d_t<L, 32>(slots, runs, table, nwork, st);
  if (slots <= 64) return launch_init3d_t<L, 64>(slots, runs, table, nwork, st);
  if (slots <= 128) return launch_init3d_t<L, 128>(slots, runs, table, nwork, st);
  return slots <= 256 ? launch_init3d_t<L, 256>(slots, runs, table, nwork, st) : cudaErrorInvalidValue;
}

}  // namespace pa

#define PA_INSTANTIATE_SWEEP3D(LL)                                                                        \
  namespace pa {                                                                                          \
  cudaError_t sweep3d_L##LL(const Sweep3dLaunch& a) { return sweep3d_any<LL>(a); }                        \
  cudaError_t launch_init3d_L##LL(int slots, RunDev* runs, const Work* table, int nwork,                  \
                                  cudaStream_t st) {                                                      \
    return launch_init3d<LL>(slots, runs, table, nwork, st);                                              \
  }                                                                                                       \
  bool sweep3d_split_ok_L##LL(int split) { return split_ok<Geo3<LL>>(split) || extra_split<LL>(split); } \
  }
