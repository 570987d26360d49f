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
      for (int f = 0; f < 2; ++f) {  // the three multipole indices of F0 / F2 and of F1 / F3
        const int s = n2 + n3;
        const int k[3] = {f ? s - 1 : s - 3, -n2 - 2, f ? -n3 - 1 : -n3 - 3};
        const int total = f ? -4 : -8;
        for (int i = 0; i < 3; ++i)  // any of them can stand in the column's place
          for (int j = 0; j < 3; ++j) {
            if (i == j) continue;
            const int q = total - k[i] - B.sg0;
            if (q < 0 || q >= B.nsg) return false;
            lo[q] = std::min(lo[q], k[j]);
            up[q] = std::max(up[q], k[j]);
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
// contiguous stretch of the output.
template <bool SLICES>
__global__ void __launch_bounds__(256) expand_kernel(const __grid_constant__ Basis B, const double2* __restrict__ red,
                                                     int slices, double2* __restrict__ ups) {
  const int N = B.N, nb = B.nb, nn = 2 * N + 1, np = B.npairs;
  const int mu = blockIdx.x / (nn * nn), n2 = (blockIdx.x / nn) % nn - N, n3 = blockIdx.x % nn - N, s = n2 + n3;
  const bool odd = mu == 1 || mu >= 5;  // x^* at the centre: F1 or F3
  const size_t stride = B.elems();
  double2* out = ups + (size_t)blockIdx.x * nb * nb * nb;
  for (int e = threadIdx.x; e < nb * nb * nb; e += blockDim.x) {
    const int b[3] = {e / (nb * nb), (e / nb) % nb, e % nb};
    size_t at;
    double sign = 1.0;
    if (mu == 8) {
      const bool flip = s < 0;  // FW[-sg, -a] = FW[sg, a]^*
      int k2 = flip ? n2 : -n2, k3 = flip ? n3 : -n3, c2 = b[1], c3 = b[2];
      order2(k2, c2, k3, c3);
      const int as = flip ? -s : s;
      const size_t row = (size_t)(B.wbase(as) + k2 + N);
      at = B.woff() + (row * nb + b[0]) * np + c2 * nb - c2 * (c2 - 1) / 2 + (c3 - c2);
      if (flip) sign = -1.0;
    } else {
      // the three (index, bin) pairs: the column's, then the row's two
      int k0 = odd ? s - 1 : s - 3, k1 = -n2 - 2, k2 = odd ? -n3 - 1 : -n3 - 3;
      int c0 = b[0], c1 = b[1], c2 = b[2], sg, q;
      if (mu < 2) {
        order2(k0, c0, k1, c1);
        order2(k1, c1, k2, c2);
        order2(k0, c0, k1, c1);
        sg = (mu ? -4 : -8) - k0;
        q = mu;
      } else {
        // the conjugated factor is the column's: its place is bin 1, 2 or 3
        const int place = (mu == 2 || mu == 5) ? 0 : (mu == 3 || mu == 6) ? 1 : 2;
        if (place == 0) sg = odd ? -s - 3 : -s - 5;
        else if (place == 1) { sg = odd ? n2 - 2 : n2 - 6; k1 = k0; c1 = c0; c0 = b[1]; }
        else { sg = odd ? n3 - 3 : n3 - 5; k2 = k0; c2 = c0; c0 = b[2]; }
        order2(k1, c1, k2, c2);
        q = odd ? 3 : 2;
      }
      const int si = sg - B.sg0;
      const size_t row = (size_t)(B.xbase[si] + k1 - B.xlo[si]);
      at = (row * 4 * nb + q * nb + c0) * np + c1 * nb - c1 * (c1 - 1) / 2 + (c2 - c1);
    }
    double2 v = red[at];
    for (int z = 1; SLICES && z < slices; ++z) {
      const double2 t = red[at + z * stride];
      v.x += t.x;
      v.y += t.y;
    }
    double2 u = out[e];
    u.x += v.x;
    u.y += sign * v.y;
    out[e] = u;
  }
}

}  // namespace

cudaError_t basis_expand(const Basis& B, const double* red, int slices, double* ups, cudaStream_t s) {
  const int nn = 2 * B.N + 1;
  const double2* r = reinterpret_cast<const double2*>(red);
  double2* u = reinterpret_cast<double2*>(ups);
  if (slices > 1) expand_kernel<true><<<9 * nn * nn, 256, 0, s>>>(B, r, slices, u);
  else expand_kernel<false><<<9 * nn * nn, 256, 0, s>>>(B, r, 1, u);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace ext4pcf
