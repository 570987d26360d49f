// The independent sums behind the nine components of the 4PCF multipoles.
//
// Every component is a sum over centres of a centre factor times three neighbour multipoles,
// one per radial bin, and a permutation of the bins turns one component into another (the
// symmetries of Table tab:4PCFSymm).  With the multipoles ordered by their own indices instead
// of by (n2, n3), five families of sums hold everything:
//   F0[sg, a](b1; b2, b3) = sum_i x   G_{-sg-8}(b1)  G_a(b2) G_{sg-a}(b3)
//   F1                    = sum_i x^* G_{-sg-4}(b1)  G_a(b2) G_{sg-a}(b3)
//   F2                    = sum_i x   G_{sg+4}^*(b1) G_a(b2) G_{sg-a}(b3)
//   F3                    = sum_i x^* G_sg^*(b1)     G_a(b2) G_{sg-a}(b3)
//   FW                    = sum_i w   W_{-sg}(b1)    W_a(b2) W_{sg-a}(b3)
// With s = n2 + n3 the components are (third column: which bins take the places b1; b2, b3)
//   Upsilon_0  F0[-s-5, -n2-2]   (1; 2, 3)     Upsilon_1  F1[-s-3, -n2-2]   (1; 2, 3)
//   Upsilon_2  F2[-s-5, -n2-2]   (1; 2, 3)     Upsilon_5  F3[-s-3, -n2-2]   (1; 2, 3)
//   Upsilon_3  F2[n2-6, s-3]     (2; 1, 3)     Upsilon_6  F3[n2-2, s-1]     (2; 1, 3)
//   Upsilon_4  F2[n3-5, s-3]     (3; 1, 2)     Upsilon_7  F3[n3-3, s-1]     (3; 1, 2)
//   N          FW[-s, -n2]       (1; 2, 3)
// All five are unchanged when (a, b2) and (sg - a, b3) trade places, so they are kept for
// b2 <= b3 only; F0 and F1 are unchanged under any permutation of their three (index, bin)
// pairs, so only b1 <= b2 <= b3 is ever read of them; and FW[-sg, -a] = FW[sg, a]^*, so it is
// kept for sg <= 0.  F0..F3 share their row products G_a(b2) G_{sg-a}(b3): 2839 (sg, a) at
// n_max = 20 (861 more for FW) take the place of the 11767 (row type, n2, n3) that the nine
// components need when only b2 <= b3 is used component by component.
#pragma once
#include "common.cuh"

namespace ext4pcf {

constexpr int kMaxSg = 168;  // values of sg at n_max = 40 (4 n_max + 3)

// Rows (sg, a) of the reduced array.  X rows (F0..F3): sg = sg0 + k, a in [xlo[k], xlo[k] +
// xlen[k]), row xbase[k] + a - xlo[k].  W rows (FW): s = -sg = 0 .. 2N, a in [-N, N - s].
struct Basis {
  int N, nb, npairs;
  int sg0, nsg;
  int rx, rw;  // rows of both kinds
  int xbase[kMaxSg];
  short xlo[kMaxSg], xlen[kMaxSg];
  __host__ __device__ int wbase(int s) const { return s * (2 * N + 1) - s * (s - 1) / 2; }
  __host__ __device__ int wlen(int s) const { return 2 * N + 1 - s; }
  // complex elements: [rx][4 nb][npairs] then [rw][nb][npairs]
  __host__ __device__ size_t woff() const { return (size_t)rx * 4 * nb * npairs; }
  __host__ __device__ size_t elems() const { return woff() + (size_t)rw * nb * npairs; }
};

// multipole index and conjugation of the column factor of family q (0..3) at sg, and whether the
// centre factor is x^* (1) or x (0)
__host__ __device__ inline int basis_col_index(int q, int sg) {
  return q == 0 ? -sg - 8 : q == 1 ? -sg - 4 : q == 2 ? sg + 4 : sg;
}
__host__ __device__ inline bool basis_col_conj(int q) { return q >= 2; }
__host__ __device__ inline bool basis_centre_conj(int q) { return (q & 1) != 0; }
// G index within the record
__host__ __device__ inline bool basis_in_g(int N, int m) { return m >= -2 * N - 3 && m <= 2 * N - 1; }

// Where component mu (0..7, 8: N) at (n2, n3) is found among the families (the table above): the expansion,
// the rows of the reduced array and the table of ext4pcf_contraction_tables all follow from this.
// k: the multipole index of the factor of bins 1, 2, 3 (of a column of F2, F3, which is conjugated, the one
// that F0, F1 would have in its place); place: the column's factor, sg: its sums' (F0 and F1 have any
// factor in the column's place); flip: N at s < 0, the conjugate of the sum with these indices.
struct BasisTerm {
  int q, place, sg, k[3];
  bool flip;
};
__host__ __device__ inline int basis_total(int q) { return q == 4 ? 0 : basis_centre_conj(q) ? -4 : -8; }  // sum of the k
__host__ __device__ inline BasisTerm basis_term(int mu, int n2, int n3) {
  const int s = n2 + n3;
  const bool odd = mu == 1 || (mu >= 5 && mu < 8);  // x^* at the centre: F1 or F3
  BasisTerm t;
  t.q = mu == 8 ? 4 : mu < 2 ? mu : odd ? 3 : 2;
  t.place = mu == 3 || mu == 6 ? 1 : mu == 4 || mu == 7 ? 2 : 0;
  t.flip = mu == 8 && s < 0;  // FW[-sg, -a] = FW[sg, a]^*
  t.k[0] = mu == 8 ? (t.flip ? -s : s) : odd ? s - 1 : s - 3;
  t.k[1] = mu == 8 ? (t.flip ? n2 : -n2) : -n2 - 2;
  t.k[2] = mu == 8 ? (t.flip ? n3 : -n3) : odd ? -n3 - 1 : -n3 - 3;
  t.sg = basis_total(t.q) - (t.place == 0 ? t.k[0] : t.place == 1 ? t.k[1] : t.k[2]);
  return t;
}

bool basis_make(const Layout& L, Basis& B);

// bin pair p -> (b2, b3), b2 <= b3, pairs in row-major order of (b2, b3)
__device__ __forceinline__ void basis_pair(int p, int nb, int& b2, int& b3) {
  int b = 0, first = 0;
  while (p >= first + (nb - b)) {
    first += nb - b;
    ++b;
  }
  b2 = b;
  b3 = b + (p - first);
}

// Sums of the multiple-counting terms (two or three of a quadruplet's neighbours the same galaxy; App.
// A.1, Table tab:4PCFMCCorr).  Merging two factors of a family leaves the bin sum of their
// per-galaxy product (XX, XA or WW of the record) times the third factor, so the terms of every
// component come from seven arrays (bm: the merged pair's bin, bo: the third factor's):
//   0: sum x   XX_sg(bm) G_{-sg-8}(bo)     F0, any two      1: sum x^* XX_sg(bm) G_{-sg-4}(bo)  F1, any two
//   2: sum x   XX_sg(bm) G_{sg+4}^*(bo)    F2, rows merged  3: sum x   XA_{sg+4}(bm) G_{-sg-8}(bo)  F2, column merged
//   4: sum x^* XX_sg(bm) G_sg^*(bo)        F3, rows merged  5: sum x^* XA_{sg+4}(bm) G_{-sg-4}(bo)  F3, column merged
//   6: sum w   WW_c^*(bm) W_c(bo), c >= 0  FW, any two
// and five triple sums.  Layout of a copy, complex: [6][nsig][nb][nb] (sg = -2N-6 + i), [2N+1][nb][nb],
// triple [5][nb], xi accumulators [3][nb].
struct CorrLayout {
  int N, nb, nsig;
  size_t ow, ot, ox, elems;
  __host__ __device__ static CorrLayout make(int N, int nb) {
    CorrLayout c;
    c.N = N;
    c.nb = nb;
    c.nsig = 4 * N + 5;
    c.ow = (size_t)6 * c.nsig * nb * nb;
    c.ot = c.ow + (size_t)(2 * N + 1) * nb * nb;
    c.ox = c.ot + (size_t)5 * nb;
    c.elems = c.ox + (size_t)3 * nb;
    return c;
  }
};

// every ordered triple of bins at |n| <= N from the reduced array (the sum of `slices` arrays, one
// after the other; none if red is null) less the multiple-counting terms of the slot's first copy of
// correction sums, added into ups
cudaError_t basis_expand(const Basis& B, const double* red, int slices, const double* corr, double* ups,
                         cudaStream_t s);

// contract.cu: reduced arrays (slices of a wave's centres) of the CUDA-core contraction
int contract_slices(const Basis& B);

}  // namespace ext4pcf
