// Contraction of a wave of per-centre multipole records into the 4PCF multipoles
//   Upsilon_{mu,n}(Theta1,Theta2,Theta3) += sum_i xt_i A_i(Theta1) B_i(Theta2) C_i(Theta3)
// (paper Eq. 4PCFUpsilon0 and the seven equations after it; Eq. Nnmultipoles).  CUDA-core version, templated
// on the arithmetic type: FP64 throughout, or FP32 within a wave with the wave totals added
// into the FP64 reduced array of the independent sums (basis.cuh).
#include <algorithm>

#include "basis.cuh"

namespace ext4pcf {

namespace {

constexpr int kChunk = 32;  // centres staged per pass of the contraction kernel

// One thread per row (sg, a, b2 <= b3) of the reduced array: it forms the row product
// G_a(b2) G_{sg-a}(b3) of a centre once and folds it into the NC NBT sums of its families and
// Theta1 bins, held in registers; the column factors (x G_m of the wave's centres) are formed
// once per block and read back as broadcasts.
// FP64 (2 fused multiply-adds per clock and SM) is bound by that pipe, so the rows run pair by
// pair (all a of one bin pair side by side): a warp then mostly holds one b2 and leaves out the
// Theta1 > b2 columns of F0 and F1, which the expansion never reads.  FP32 has no pipe to save
// and runs the rows a by a, so that neighbouring lanes read neighbouring bins of the records.
// Measured against one block per (component, n2, n3) with a thread per (Theta2, Theta3): FP64,
// 1000 centres at n_max = 20, 10 bins 188.6 -> 45.0 ms (its 8.06e8 FP64 warp instructions take
// 42 ms at 16 clocks each: pipe 96% busy), 2000 centres at n_max = 10, 8 bins 36 -> 13.9 ms; FP32,
// 1500 centres at n_max = 16, 9 bins 6.71 -> 1.94 ms.
template <typename R> constexpr int kRowThreadsOf = sizeof(R) == 8 ? 32 : 64;

// NC families per block of NBT >= nb columns.  Grid: x the tile of kRowThreads rows within sg,
// y the sg of the X rows (times the groups of families), then s = -sg of the W rows, z the slice
// of the wave's centres (each with its own reduced array).
template <typename R, int NBT, int NC>
__global__ void __launch_bounds__(kRowThreadsOf<R>)
contract_rows(const Layout L, const __grid_constant__ Basis B, const cplx_t<R>* __restrict__ rec,
              const cplx_t<R>* __restrict__ xw, int T, const int* __restrict__ n_live, int w0,
              double2* __restrict__ red) {
  using Cx = cplx_t<R>;
  constexpr bool kPairMajor = sizeof(R) == 8;
  constexpr int kRowThreads = kRowThreadsOf<R>;
  static_assert(NC == 1 || NC == 2, "families per block");
  T = wave_centres(T, n_live, w0);
  // this block's slice of the wave's centres
  const int t0 = (int)((long long)T * blockIdx.z / gridDim.z), t1 = (int)((long long)T * (blockIdx.z + 1) / gridDim.z);
  if (t0 == t1) return;
  red += blockIdx.z * B.elems();
  __shared__ __align__(16) Cx sA[kChunk][NC * NBT];
  const int N = L.N, nb = L.nb, np = B.npairs;
  constexpr int kGroups = 4 / NC;
  const bool wk = (int)blockIdx.y >= B.nsg * kGroups;
  const int grp = wk ? 0 : blockIdx.y / B.nsg, q0 = blockIdx.y % B.nsg;
  const int sg = wk ? -((int)blockIdx.y - B.nsg * kGroups) : B.sg0 + q0;
  const int alo = wk ? -N : B.xlo[q0], len = wk ? B.wlen(-sg) : B.xlen[q0];
  const int row0 = wk ? B.wbase(-sg) : B.xbase[q0];
  const int tid = threadIdx.x, first = blockIdx.x * kRowThreads;
  if (first >= len * np) return;
  const bool active = first + tid < len * np;
  const int r = active ? first + tid : first;
  const int a = alo + (kPairMajor ? r % len : r / np), pair = kPairMajor ? r / len : r % np;
  int b2, b3;
  basis_pair(pair, nb, b2, b3);
  // where this row's two factors sit in a record, and the sign of their imaginary parts
  const int m3 = sg - a;
  const int i2 = wk ? L.W(a >= 0 ? a : -a, b2) : L.G(a, b2);
  const int i3 = wk ? L.W(m3 >= 0 ? m3 : -m3, b3) : L.G(m3, b3);
  const R g2s = wk && a < 0 ? R(-1) : R(1), g3s = wk && m3 < 0 ? R(-1) : R(1);
  // columns: family of slot j.  Two families a block: group 0 holds F2 and F3 (every Theta1),
  // group 1 F0 and F1; one family a block: group g holds family g.
  int fam[NC];
  bool use[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    fam[j] = wk ? 4 : NC == 2 ? (grp == 0 ? 2 + j : j) : grp;
    use[j] = wk ? j == 0 : basis_in_g(N, basis_col_index(fam[j], sg));
  }
  int kmax = nb - 1;
  if (kPairMajor && !wk && fam[0] < 2) {  // Theta1 <= b2, over the warp's rows
    kmax = b2;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kmax = max(kmax, __shfl_xor_sync(0xFFFFFFFFu, kmax, o));
  }
  Cx acc[NC * NBT];
#pragma unroll
  for (int k = 0; k < NC * NBT; ++k) acc[k] = cmk<Cx>(R(0), R(0));
  Cx n2v = rec[(size_t)t0 * L.rec + i2], n3v = rec[(size_t)t0 * L.rec + i3];
  for (int c0 = t0; c0 < t1; c0 += kChunk) {
    const int nc = min(kChunk, t1 - c0);
    __syncthreads();
    for (int k = tid; k < nc * NC * NBT; k += kRowThreads) {
      const int cc = k / (NC * NBT), j = (k / NBT) % NC, b = k % NBT;
      const Cx* rc = rec + (size_t)(c0 + cc) * L.rec;
      const int q = wk ? 4 : NC == 2 ? (grp == 0 ? 2 + j : j) : grp;
      Cx v = cmk<Cx>(R(0), R(0));
      if (b < nb && (wk ? j == 0 : basis_in_g(N, basis_col_index(q, sg)))) {
        Cx t, f;
        if (q == 4) {
          t = xw[2 * (size_t)(c0 + cc) + 1];
          f = rc[L.W(-sg, b)];
        } else {
          t = xw[2 * (size_t)(c0 + cc)];
          if (basis_centre_conj(q)) t = cconj(t);
          f = rc[L.G(basis_col_index(q, sg), b)];
          if (basis_col_conj(q)) f = cconj(f);
        }
        v = cmul(t, f);
      }
      sA[cc][j * NBT + b] = v;
    }
    __syncthreads();
    for (int cc = 0; cc < nc; ++cc) {
      const Cx g2 = cmk<Cx>(n2v.x, g2s * n2v.y), g3 = cmk<Cx>(n3v.x, g3s * n3v.y);
      if (c0 + cc + 1 < t1) {  // the next centre's factors, used one round later
        const Cx* rc = rec + (size_t)(c0 + cc + 1) * L.rec;
        n2v = rc[i2];
        n3v = rc[i3];
      }
      const Cx kr = cmul(g2, g3);
      // two columns at a time, left by a branch after the last one in use (a predicate on every
      // multiply-add would still take its turn in the FP64 pipe); unused slots hold zeros
#pragma unroll
      for (int k = 0; k < NBT; k += 2) {
        if (sizeof(R) == 8 && k > kmax) break;
#pragma unroll
        for (int j = 0; j < NC; ++j)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const Cx v = sA[cc][j * NBT + k + i];
            Cx& s = acc[j * NBT + k + i];
            s.x += v.x * kr.x;  // separate multiply-adds: a sum of products would
            s.x -= v.y * kr.y;  // cost an extra multiply and add
            s.y += v.x * kr.y;
            s.y += v.y * kr.x;
          }
      }
    }
  }
  if (active) {
    const size_t row = (size_t)row0 + (a - alo);
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      if (!use[j]) continue;
      double2* o = wk ? red + B.woff() + row * nb * np + pair : red + (row * 4 + fam[j]) * nb * np + pair;
#pragma unroll
      for (int k = 0; k < NBT; ++k)
        if (k <= kmax) {
          double2 v = o[(size_t)k * np];
          v.x += (double)acc[j * NBT + k].x;
          v.y += (double)acc[j * NBT + k].y;
          o[(size_t)k * np] = v;
        }
    }
  }
}

template <typename R, int NBT, int NC>
cudaError_t launch_rows(const Layout& L, const Basis& B, const cplx_t<R>* rec, const cplx_t<R>* xw, int T,
                        const int* n_live, int w0, double* red, cudaStream_t s) {
  constexpr int kRowThreads = kRowThreadsOf<R>;
  int len = 2 * L.N + 1;  // the most rows (sg, a) of one sg
  for (int q = 0; q < B.nsg; ++q) len = std::max(len, (int)B.xlen[q]);
  const dim3 grid((len * B.npairs + kRowThreads - 1) / kRowThreads, B.nsg * (4 / NC) + 2 * L.N + 1,
                  contract_slices(B));
  // FP64: about nine blocks (warps) per SM keep its pipe full; more would only lengthen every
  // block, and with it the last round (shared memory that is not used holds the others back)
  const size_t held = sizeof(R) == 8 ? 24 * 1024 - sizeof(cplx_t<R>) * kChunk * NC * NBT : 0;
  contract_rows<R, NBT, NC><<<grid, kRowThreads, held, s>>>(L, B, rec, xw, T, n_live, w0,
                                                            reinterpret_cast<double2*>(red));
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace

// Slices of a wave's centres, each summed by blocks of its own into a reduced array of its own
// (the expansion adds them in order).  Few rows (n_max = 10, 8 bins: 2100 FP64 blocks of one
// warp, all resident at once and unevenly spread over the SMs) leave FP64 pipes idle at the end:
// enough slices for about ten rounds of blocks.
int contract_slices(const Basis& B) {
  const int warps = (B.rx * 2 + B.rw) * B.npairs / 32 + 1;
  return std::min(16, std::max(1, (16384 + warps / 2) / warps));
}

// two families a block up to 16 bins (at most 32 complex sums a thread), one beyond
template <typename R>
cudaError_t contract_wave(const Layout& L, const Basis& B, const cplx_t<R>* rec, const cplx_t<R>* xw, int T,
                          const int* n_live, int w0, double* red, cudaStream_t s) {
  if (T <= 0) return cudaSuccess;
  const int nb = L.nb;
#define EXT4PCF_ROWS(NBT, NC) \
  if (nb <= NBT) return launch_rows<R, NBT, NC>(L, B, rec, xw, T, n_live, w0, red, s)
  EXT4PCF_ROWS(4, 2);
  EXT4PCF_ROWS(6, 2);
  EXT4PCF_ROWS(8, 2);
  EXT4PCF_ROWS(10, 2);
  EXT4PCF_ROWS(12, 2);
  EXT4PCF_ROWS(16, 2);
  EXT4PCF_ROWS(24, 1);
  EXT4PCF_ROWS(32, 1);
#undef EXT4PCF_ROWS
  return cudaErrorInvalidValue;
}

template cudaError_t contract_wave<float>(const Layout&, const Basis&, const float2*, const float2*, int, const int*,
                                          int, double*, cudaStream_t);
template cudaError_t contract_wave<double>(const Layout&, const Basis&, const double2*, const double2*, int,
                                           const int*, int, double*, cudaStream_t);

}  // namespace ext4pcf

