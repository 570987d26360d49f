// Host tables of the independent sums (basis.cuh) and the expansion into all nine components.
#include <algorithm>
#include <vector>

#include "basis.cuh"

namespace ext4pcf {

// The (sg, a) that some component at |n2|, |n3| <= N reads, as one range of a per sg.
bool basis_make(const Layout& L, Basis& B) {
  const int N = L.N;
  B.N = N;
  B.nb = L.nb;
  B.npairs = L.nb * (L.nb + 1) / 2;
  B.sg0 = std::min(-2 * N - 5, -N - 6);
  const int hi = std::max(2 * N - 3, N - 2);
  B.nsg = hi - B.sg0 + 1;
  if (B.nsg > kMaxSg) return false;
  std::vector<int> lo(B.nsg, 1 << 20), up(B.nsg, -(1 << 20));
  for (int n2 = -N; n2 <= N; ++n2)
    for (int n3 = -N; n3 <= N; ++n3)
      for (int mu = 0; mu < 8; ++mu) {
        const BasisTerm t = basis_term(mu, n2, n3);
        for (int i = 0; i < 3; ++i) {
          if (t.q >= 2 && i != t.place) continue;  // (F0, F1: any factor can stand in the column's place)
          const int q = basis_total(t.q) - t.k[i] - B.sg0;
          if (q < 0 || q >= B.nsg) return false;
          for (int j = 0; j < 3; ++j) {
            if (i == j) continue;
            lo[q] = std::min(lo[q], t.k[j]);
            up[q] = std::max(up[q], t.k[j]);
          }
        }
      }
  B.rx = 0;
  for (int q = 0; q < B.nsg; ++q) {
    B.xbase[q] = B.rx;
    B.xlo[q] = 0;
    B.xlen[q] = 0;
    if (lo[q] > up[q]) continue;  // (n_max = 0 leaves one sg out)
    if (!basis_in_g(N, lo[q]) || !basis_in_g(N, up[q])) return false;
    B.xlo[q] = (short)lo[q];
    B.xlen[q] = (short)(up[q] - lo[q] + 1);
    B.rx += B.xlen[q];
  }
  B.rw = B.wbase(2 * N + 1);
  return true;
}

namespace {

// exchange two (index, bin) pairs so that their bins do not decrease
__device__ __forceinline__ void order2(int& k0, int& b0, int& k1, int& b1) {
  if (b0 > b1) {
    int t = k0; k0 = k1; k1 = t;
    t = b0; b0 = b1; b1 = t;
  }
}

// Block = (component, n2, n3): its nb^3 values come from one or a few rows (sg, a) of the
// reduced array (nb npairs complex each), which stay in the cache, and are added into one
// contiguous stretch of the output, less the multiple-counting terms where two bins are the same:
// one nb x nb matrix for each pair of factors that can merge, staged in shared memory.  The output's
// read and write bound it, and the FP64 additions next (16 clocks a warp instruction and SM).
// n_max = 20, 10 bins (242 MB of output): 199 us, expansion and corrections as two kernels 491 us.
constexpr int kExpandThreads = 256, kExpandValues = 4;
template <bool SLICES>
__global__ void __launch_bounds__(kExpandThreads) expand_kernel(const __grid_constant__ Basis B,
                                                                const double2* __restrict__ red, int slices,
                                                                const double2* __restrict__ corr, int inv,
                                                                double2* __restrict__ ups) {
  extern __shared__ double2 merged[];  // [3][nb][nb]: factors (1, 2), (1, 3), (2, 3); triple [nb]
  const int N = B.N, nb = B.nb, np = B.npairs, nn = 2 * N + 1, nb2 = nb * nb, nb3 = nb2 * nb;
  const int mu = blockIdx.x / (nn * nn), n2 = (blockIdx.x / nn) % nn - N, n3 = blockIdx.x % nn - N;
  const size_t stride = B.elems();
  const BasisTerm term = basis_term(mu, n2, n3);
  const int q = term.q, place = term.place, sgc = term.sg, total = basis_total(q);
  const int(&k)[3] = term.k;
  const bool flip = term.flip;
  const CorrLayout C = CorrLayout::make(N, nb);
  for (int i = threadIdx.x; i < 3 * nb2 + nb; i += kExpandThreads) {
    double2 v;
    if (i >= 3 * nb2) {
      v = corr[C.ot + (size_t)q * nb + (i - 3 * nb2)];
    } else {
      const int m = i / nb2, third = 2 - m;  // pairs (0, 1), (0, 2), (1, 2) leave factor 2, 1, 0
      const int c = third == 2 ? k[2] : third == 1 ? k[1] : k[0];
      size_t at;
      if (q == 4) {
        at = C.ow + (size_t)(c < 0 ? -c : c) * nb2;
      } else if (q >= 2 && third == place) {  // both row factors merged: the third is the column
        at = (size_t)(q == 2 ? 2 : 4) * C.nsig * nb2 + (size_t)(sgc + 2 * N + 6) * nb2;
      } else {
        at = (size_t)(q < 2 ? q : q == 2 ? 3 : 5) * C.nsig * nb2 + (size_t)(2 * N + 6 + total - c) * nb2;
      }
      v = corr[at + (i - m * nb2)];
      if (q == 4 && c < 0) v.y = -v.y;
    }
    merged[i] = v;
  }
  __syncthreads();
  // (all three bins the same: the three terms less twice the triple one, at the first matrix' diagonal)
  if ((int)threadIdx.x < nb) {
    const int i = threadIdx.x * (nb + 1);
    const double2 t = merged[3 * nb2 + threadIdx.x], m1 = merged[nb2 + i], m2 = merged[2 * nb2 + i];
    merged[i].x += m1.x + m2.x - 2.0 * t.x;
    merged[i].y += m1.y + m2.y - 2.0 * t.y;
  }
  __syncthreads();
  double2* out = ups + (size_t)blockIdx.x * nb3;
  // the reduced array's value of the triple (b0, b1, b2)
  auto value = [&](int b0, int b1, int b2) -> double2 {
    if (!red) return make_double2(0.0, 0.0);
    int k0 = k[0], k1 = k[1], k2 = k[2], c0 = b0, c1 = b1, c2 = b2, sg = sgc;
    if (q < 2) {  // any order of the three
      order2(k0, c0, k1, c1);
      order2(k1, c1, k2, c2);
      order2(k0, c0, k1, c1);
      sg = total - k0;
    } else if (q == 4) {
      order2(k1, c1, k2, c2);
    } else {
      if (place == 1) { k1 = k0; c1 = c0; c0 = b1; }
      else if (place == 2) { k2 = k0; c2 = c0; c0 = b2; }
      order2(k1, c1, k2, c2);
    }
    size_t at;
    if (q == 4) at = B.woff() + ((size_t)(B.wbase(k0) + k1 + N) * nb + c0) * np;
    else at = ((size_t)(B.xbase[sg - B.sg0] + k1 - B.xlo[sg - B.sg0]) * 4 * nb + q * nb + c0) * np;
    at += c1 * nb - c1 * (c1 - 1) / 2 + (c2 - c1);
    double2 v = red[at];
    for (int z = 1; SLICES && z < slices; ++z) {
      const double2 a = red[at + z * stride];
      v.x += a.x;
      v.y += a.y;
    }
    return v;
  };
  auto flipped = [&](double y) { return flip ? -y : y; };
  // three different bins: nothing to take off
  for (int e0 = threadIdx.x; e0 < nb3 && red; e0 += kExpandThreads * kExpandValues) {
    double2 v[kExpandValues], u[kExpandValues];
    bool use[kExpandValues];
#pragma unroll
    for (int i = 0; i < kExpandValues; ++i) {
      const int e = e0 + i * kExpandThreads;
      const int d = (e * inv) >> 20, b2 = e - d * nb, b0 = (d * inv) >> 20, b1 = d - b0 * nb;
      use[i] = e < nb3 && b0 != b1 && b0 != b2 && b1 != b2;
      if (use[i]) {
        u[i] = out[e];
        v[i] = value(b0, b1, b2);
      }
    }
#pragma unroll
    for (int i = 0; i < kExpandValues; ++i)
      if (use[i]) out[e0 + i * kExpandThreads] = make_double2(u[i].x + v[i].x, u[i].y + flipped(v[i].y));
  }
  // two or three the same: the nb (3 nb - 2) others, each with the term of its equal pair (they get
  // lanes of their own: a predicated FP64 instruction takes its turn in the pipe whether it runs or not)
  for (int i = threadIdx.x; i < nb * (3 * nb - 2); i += kExpandThreads) {
    int m = 0, bm, bo;
    if (i < nb2) {
      bm = i / nb;
      bo = i - bm * nb;
    } else {
      const int j = i - nb2, w = nb * (nb - 1), r = j % (nb - 1);
      m = 1 + j / w;
      bm = (j % w) / (nb - 1);
      bo = r + (r >= bm);
    }
    const int b0 = m == 2 ? bo : bm, b1 = m == 1 ? bo : bm, b2 = m == 0 ? bo : bm;
    const size_t e = ((size_t)b0 * nb + b1) * nb + b2;
    const double2 u = out[e], v = value(b0, b1, b2), t = merged[m * nb2 + bm * nb + bo];
    out[e] = make_double2(u.x + (v.x - t.x), u.y + flipped(v.y - t.y));
  }
}

}  // namespace

// The factors of every component from basis_term and the families' columns, in the layout of
// ext4pcf_nth_order_factors at order 4: sign, centre code, then per bin (array, conj, coefficient of n2,
// coefficient of n3, constant).  Indices are linear in (n2, n3) (for N at s >= 0, and past it by flip).
int contraction_table_cc(int* out) {
  for (int mu = 0; mu < 9; ++mu) {
    int* t = out + mu * 17;
    int idx[3][3];  // factor, at (0, 0), (1, 0), (0, 1)
    for (int e = 0; e < 3; ++e) {
      const BasisTerm b = basis_term(mu, e == 1, e == 2);
      t[0] = 1;
      t[1] = b.q == 4 ? 2 : basis_centre_conj(b.q);
      for (int l = 0; l < 3; ++l) {
        const bool column = b.q < 4 && l == b.place;
        idx[l][e] = column ? basis_col_index(b.q, b.sg) : b.k[l];
        t[2 + 5 * l] = b.q == 4;
        t[3 + 5 * l] = column && basis_col_conj(b.q);
      }
    }
    for (int l = 0; l < 3; ++l) {
      t[4 + 5 * l] = idx[l][1] - idx[l][0];
      t[5 + 5 * l] = idx[l][2] - idx[l][0];
      t[6 + 5 * l] = idx[l][0];
    }
  }
  return 9 * 17;
}

cudaError_t basis_expand(const Basis& B, const double* red, int slices, const double* corr, double* ups,
                         cudaStream_t s) {
  const int nn = 2 * B.N + 1, blocks = 9 * nn * nn;
  const int inv = ((1 << 20) + B.nb - 1) / B.nb;  // e / nb = (e inv) >> 20 for e < 32768, nb <= 32
  const double2* r = reinterpret_cast<const double2*>(red);
  const double2* c = reinterpret_cast<const double2*>(corr);
  double2* u = reinterpret_cast<double2*>(ups);
  const size_t smem = (size_t)(3 * B.nb * B.nb + B.nb) * sizeof(double2);
  auto kernel = slices > 1 ? expand_kernel<true> : expand_kernel<false>;
  cudaError_t e = allow_smem(kernel);
  if (e != cudaSuccess) return e;
  kernel<<<blocks, kExpandThreads, smem, s>>>(B, r, slices, c, inv, u);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace ext4pcf
