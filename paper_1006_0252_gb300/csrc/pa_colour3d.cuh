// pa_colour3d.cuh -- colour-split words of the cubic lattices (+-1 and
// Gaussian couplings): neighbour words, conversion from and to the packed
// words, and the walk over a column's words in a half sweep.
//
// For colour c and word w = y G + g of the packed lattice, one word holds the
// word's S = K L / 2 colour-c sites by rank m = j L/2 + h (lane j, site x = 2h
// + q, q = (c + y + z) mod 2) of one replica in bits 0..15 and, with RP = 2, of
// a second replica in bits 16..31.
#pragma once
#include "pa_lattice3d.cuh"

namespace pa {

// ---------------------------------------------------------------------------
// Colour-split words.
// ---------------------------------------------------------------------------
template <class GEO>
struct Half {
  static constexpr int H = GEO::L / 2;       // colour-c sites of a lane
  static constexpr int S = GEO::K * H;       // colour-c sites of a word, <= 16
  static constexpr uint32_t ONE = (1u << S) - 1u;  // bits of one replica (S <= 16)
  static constexpr uint32_t BOTH = ONE | (ONE << 16);
  static constexpr uint32_t fields(uint32_t f) {  // f in every lane's field, both replicas
    uint32_t m = 0;
    for (int j = 0; j < GEO::K; ++j) m |= f << (j * H);
    return m | (m << 16);
  }
  static constexpr uint32_t F0 = fields(1u);             // h = 0
  static constexpr uint32_t FH = fields(1u << (H - 1));  // h = H - 1
  static constexpr uint32_t odd_lanes() {                // lanes with odd j
    uint32_t m = 0;
    for (int j = 1; j < GEO::K; j += 2) m |= ((1u << H) - 1u) << (j * H);
    return m | (m << 16);
  }
  static constexpr uint32_t ODD = odd_lanes();
  // lane moves: bits that stay inside the word when m shifts by H
  static constexpr uint32_t LOW = ((1u << (S - H)) - 1u) | (((1u << (S - H)) - 1u) << 16);
};

// Neighbour one lane up (z + 1 across the end of a row of words) and down.
template <class GEO>
__device__ __forceinline__ uint32_t lane_next(uint32_t x) {
  using HF = Half<GEO>;
  if constexpr (GEO::K == 1) return x;
  return ((x >> HF::H) & HF::LOW) | ((x << (HF::S - HF::H)) & (HF::BOTH & ~HF::LOW));
}
template <class GEO>
__device__ __forceinline__ uint32_t lane_prev(uint32_t x) {
  using HF = Half<GEO>;
  constexpr uint32_t UP = (HF::LOW << HF::H) & HF::BOTH;  // bits H .. S-1 of both replicas
  if constexpr (GEO::K == 1) return x;
  return ((x << HF::H) & UP) | ((x >> (HF::S - HF::H)) & (HF::BOTH & ~UP));
}

// The x neighbour that is not at the same rank: h - 1 where q = 0, h + 1
// where q = 1.  With e = (c + y) mod 2 of a row, q = e ^ (g mod 2) in every
// lane of word g when G is even: one rotation of the fields, whose shifts and
// masks are set once per row; when G is odd q also alternates with the lane,
// and both rotations are taken.  Bits past S are junk (the flips are masked).
template <class GEO>
struct RowX {
  uint32_t l, r;    // G even: shifts of the words with g even (exchanged for g odd)
  uint32_t m0, m1;  // G even: bits taken from the left shift, g even / odd; G odd: lanes with q = 1
  __device__ __forceinline__ explicit RowX(uint32_t e) {
    using HF = Half<GEO>;
    constexpr uint32_t D = HF::BOTH & ~HF::F0;
    if constexpr ((GEO::G & 1) == 0) {
      l = e ? (uint32_t)(HF::H - 1) : 1u;
      r = e ? 1u : (uint32_t)(HF::H - 1);
      m0 = e ? HF::FH : D;
      m1 = e ? D : HF::FH;
    } else {
      l = r = 0u;
      m0 = e ? ~HF::ODD : HF::ODD;
      m1 = ~m0;
    }
  }
  template <int GP>  // g mod 2
  __device__ __forceinline__ uint32_t other(uint32_t b) const {
    using HF = Half<GEO>;
    constexpr uint32_t D = HF::BOTH & ~HF::F0, U = HF::BOTH & ~HF::FH;
    const uint32_t m = GP == 0 ? m0 : m1;
    if constexpr ((GEO::G & 1) == 0) {
      return GP == 0 ? (((b << l) & m) | ((b >> r) & ~m)) : (((b << r) & m) | ((b >> l) & ~m));
    } else {
      const uint32_t down = ((b << 1) & D) | ((b >> (HF::H - 1)) & HF::F0);
      const uint32_t up = ((b >> 1) & U) | ((b << (HF::H - 1)) & HF::FH);
      return (up & m) | (down & ~m);
    }
  }
};

// Two replicas' packed words as the colour-c word (e = (c + y + g) mod 2),
// and the packed words of the replicas back from a colour word.
template <class GEO, int RP>
__device__ __forceinline__ uint32_t take_colour(const uint32_t (&v)[RP], uint32_t e) {
  uint32_t x[RP];
#pragma unroll
  for (int k = 0; k < RP; ++k) x[k] = from_colour_positions<GEO>(v[k], e);  // sites at even positions 2m
  return gather_even<RP>(x);
}
template <class GEO, int K_>
__device__ __forceinline__ uint32_t place_colour(uint32_t a, uint32_t e) {  // replica K_ (0 or 1)
  return to_colour_positions<GEO>(spread_even<K_>(a), e);
}

// The other colour's words around word g of a row: the word at the same (y,
// g), those of the rows y + 1 and y - 1, and the next and previous word of the
// row (z +- 1), moved by a lane across the row's ends.  same: word 0 of the
// row; yp, ym: distance of its neighbour rows.
struct Around {
  uint32_t nx, yp, ym, zp, zm;
};
template <class GEO, int CS, class T, class INT>
__device__ __forceinline__ Around around(const T* __restrict__ same, int yp, int ym, INT g) {
  constexpr int G = GEO::G;
  Around n;
  const T* o = same + g * CS;
  n.nx = o[0];
  n.yp = o[yp];
  n.ym = o[ym];
  n.zp = o[(g + 1 < G ? 1 : 1 - G) * CS];
  n.zm = o[(g > 0 ? -1 : G - 1) * CS];
  if (g + 1 == G) n.zp = lane_next<GEO>(n.zp);
  if (g == 0) n.zm = lane_prev<GEO>(n.zm);
  return n;
}
// Distances of the neighbour rows of row y (in words of a column).
template <class GEO>
__device__ __forceinline__ int row_up(int y) {
  return y + 1 == GEO::L ? -(GEO::L - 1) * GEO::G : GEO::G;
}
template <class GEO>
__device__ __forceinline__ int row_down(int y) {
  return y == 0 ? (GEO::L - 1) * GEO::G : -GEO::G;
}

// Walk over the words of the RPP rows from y0 of a column in a half sweep of
// colour c (whole pairs of rows where the colour-c sites of a row are not a
// multiple of 4, since a Philox call serves four consecutive ranks).  The
// update is `upd`: word<K, A, GP>(own, around, rx) for the word K past the one
// its pointers stand at (A: alignment of its first uniform, see word_uniforms;
// GP = g mod 2), advance<N>() past N words.  The loop body stays short (a few
// words), so that the half sweeps of both colours fit the instruction cache:
// whole rows unrolled stalled 15-30 % of the cycles on instruction fetch at
// L = 10 and 16.
template <class GEO, int CS, int RPP, class T, class COLOUR, class UPDATE>
__device__ __forceinline__ void walk_rows(T* __restrict__ col, COLOUR c, int y0, UPDATE& upd) {
  constexpr int G = GEO::G, WR = GEO::WR, S = Half<GEO>::S;
  T* own = col + (c * WR + y0 * G) * CS;
  const T* oth = col + ((1 - c) * WR + y0 * G) * CS;
  if constexpr (G <= 2) {
    // whole rows, pairs of them where a row's uniforms end within a call
    constexpr int YU = (G * S) % 4 == 0 ? 1 : 2;
#pragma unroll 1
    for (int i = 0; i < RPP; i += YU) {
      static_for<0, YU>([&](auto yc) {
        constexpr int yi = decltype(yc)::value;
        const int y = y0 + i + yi, yp = row_up<GEO>(y) * CS, ym = row_down<GEO>(y) * CS;
        const RowX<GEO> rx((uint32_t)(c + y) & 1u);
        static_for<0, G>([&](auto gc) {
          constexpr int g = decltype(gc)::value, w = yi * G + g;
          const Around nb = around<GEO, CS>(oth + yi * G * CS, yp, ym, gc);
          upd.template word<w, (w * S) % 4, (g & 1)>(own + w * CS, nb, rx);
        });
      });
      own += YU * G * CS;
      oth += YU * G * CS;
      upd.template advance<YU * G>();
    }
  } else if constexpr (G % 2 == 0) {
    // pairs of words of a row
    static_assert(S % 4 == 0, "a word's uniforms are whole calls");
#pragma unroll 1
    for (int y = y0; y < y0 + RPP; ++y) {
      const int yp = row_up<GEO>(y) * CS, ym = row_down<GEO>(y) * CS;
      const RowX<GEO> rx((uint32_t)(c + y) & 1u);
#pragma unroll 1
      for (int g = 0; g < G; g += 2) {
        static_for<0, 2>([&](auto kc) {
          constexpr int k = decltype(kc)::value;
          const Around nb = around<GEO, CS>(oth - g * CS, yp, ym, g + k);
          upd.template word<k, 0, k>(own + k * CS, nb, rx);
        });
        own += 2 * CS;
        oth += 2 * CS;
        upd.template advance<2>();
      }
    }
  } else {
    // pairs of words across the rows of a pair (y0 even, so the word number's
    // parity is that of y + g)
    static_assert(S % 2 == 0 && RPP % 2 == 0 || RPP == GEO::L, "whole pairs of rows");
    const RowX<GEO> rx((uint32_t)c & 1u);
    int y = y0, g = 0, yp = row_up<GEO>(y) * CS, ym = row_down<GEO>(y) * CS;
#pragma unroll 1
    for (int i = 0; i < RPP * G; i += 2) {
      static_for<0, 2>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        const Around nb = around<GEO, CS>(oth + (k - g) * CS, yp, ym, g);
        upd.template word<k, (k * S) % 4, k>(own + k * CS, nb, rx);
        if (++g == G) {
          g = 0;
          ++y;
          yp = row_up<GEO>(y) * CS;
          ym = row_down<GEO>(y) * CS;
        }
      });
      own += 2 * CS;
      oth += 2 * CS;
      upd.template advance<2>();
    }
  }
}

}  // namespace pa
