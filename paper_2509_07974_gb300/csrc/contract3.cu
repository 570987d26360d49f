// Third-order multipoles (the shear 3PCF, N = 3 of paper App. F) from the per-centre records
// of the neighbour gather, with the factor tables generated for order 3
// (ext4pcf_nth_order_factors) rather than written by hand:
//   Upsilon_{mu,n}(Theta1, Theta2) = sign sum_i t_i [F1(Theta1) F2(Theta2) - delta_{Theta1 Theta2} D],
// F_l = G_m, conj(G_m) or W_m with m = a n + b, and D the product of the two factors' terms of
// one and the same neighbour (their sum over the bin is XX, XA or WW of the record), which
// removes the triplets whose two neighbours coincide.  Records in FP64 or FP32, products and
// sums in FP64, each slice's centres summed in order; the slices' partial sums are then added in
// slice order.
#include <algorithm>
#include <cstdlib>

#include "common.cuh"

extern "C" int ext4pcf_nth_order_factors(int order, int mu, int* table, int cap);

namespace ext4pcf {
namespace {

struct F3 {
  int arr, conj, a, b;  // arr 0: G, 1: W; index m = a n + b
};
struct D3 {
  int arr, idx, conj;  // arr 0: XX, 1: XA, 2: WW
};
struct C3 {
  int sign, centre;  // centre 0: x_i, 1: x_i^*, 2: w_i
  F3 f[2];
  D3 d;
};
// Component mu at n with (Theta1, Theta2) is component mir at -n with (Theta2, Theta1) where their
// factors are each other's, swapped (mu 0, 1 and the normalisation with themselves, 2 with 3): of
// such a pair only n >= 0, or only one component, is summed.  D does not depend on n.
struct Table3 {
  C3 c[5];      // mu = 0..3, 4: normalisation
  int mir[5];   // -1: none
  int nitem;    // what is summed at |n|: component, sign of n (0 at n = 0 only once)
  signed char mu[10], sg[10];
};

__device__ __forceinline__ double2 cj(double2 v) { return make_double2(v.x, -v.y); }
__device__ __forceinline__ double2 d2(float2 v) { return make_double2((double)v.x, (double)v.y); }
__device__ __forceinline__ double2 d2(double2 v) { return v; }

template <typename Cx>
__device__ __forceinline__ double2 factor(const Cx* __restrict__ r, const Layout& L, const F3& f, int n, int b) {
  const int m = f.a * n + f.b;
  double2 v;
  if (f.arr == 0) v = d2(r[L.G(m, b)]);
  else v = m >= 0 ? d2(r[L.W(m, b)]) : cj(d2(r[L.W(-m, b)]));  // W_{-m} = W_m^*
  return f.conj ? cj(v) : v;
}

template <typename Cx>
__device__ __forceinline__ double2 same_galaxy(const Cx* __restrict__ r, const Layout& L, const D3& d, int b) {
  double2 v;
  if (d.arr == 0) v = d2(r[L.XX(d.idx, b)]);
  else if (d.arr == 1) v = d.idx >= 0 ? d2(r[L.XA(d.idx, b)]) : cj(d2(r[L.XA(-d.idx, b)]));
  else v = d.idx >= 0 ? d2(r[L.WW(d.idx, b)]) : cj(d2(r[L.WW(-d.idx, b)]));
  return d.conj ? cj(v) : v;
}

// Block = (n >= 0, slice of the centres, 512 of the sums at +-n): the products of a sum are those of
// two rows of nb factors, so kC3Centres centres at a time have their rows t F1 and F2 put into shared
// memory as doubles and every sum takes one product from them.  The FP64 pipe bounds it (2
// multiply-adds per clock and SM): four per sum and centre, where forming F1 F2, t and the same
// neighbour's term for each sum took twelve, and all sums of |n| in one block leave few lanes idle.
// 50000 centres, n_max = 20, 10 bins, FP32 records: 62 -> 7.3 ms.
constexpr int kC3Threads = 256, kC3Out = 2, kC3Centres = 8;
template <typename Cx>
__global__ void __launch_bounds__(kC3Threads) contract3_kernel(const Layout L, const Table3 tab,
                                                               const Cx* __restrict__ rec,
                                                               const Cx* __restrict__ xw, int T, int S, int chunks,
                                                               double2* __restrict__ part) {
  extern __shared__ double2 rows[];  // [kC3Centres][items of the block][2][nb]
  const int nn = 2 * L.N + 1, nb = L.nb, nb2 = nb * nb, tid = threadIdx.x;
  const int n = blockIdx.x / (S * chunks), sl = blockIdx.x / chunks % S, ch = blockIdx.x % chunks;
  const int i0 = (int)((long long)T * sl / S), i1 = (int)((long long)T * (sl + 1) / S);
  const int o0 = ch * kC3Threads * kC3Out, o1 = min(o0 + kC3Threads * kC3Out, tab.nitem * nb2);
  const int it0 = o0 / nb2, nit = (o1 - 1) / nb2 + 1 - it0, per = nit * 2 * nb;
  int ra[kC3Out], rb[kC3Out];
  double2 acc[kC3Out];
#pragma unroll
  for (int r = 0; r < kC3Out; ++r) {
    const int o = o0 + r * kC3Threads + tid, it = o / nb2 - it0, b = o % nb2;
    ra[r] = o < o1 ? it * 2 * nb + b / nb : -1;
    rb[r] = it * 2 * nb + nb + b % nb;
    acc[r] = make_double2(0.0, 0.0);
  }
  for (int i = i0; i < i1; i += kC3Centres) {
    const int nc = min(kC3Centres, i1 - i);
    __syncthreads();  // the rows before have been used
    for (int k = tid; k < nc * per; k += kC3Threads) {
      const int ci = i + k / per, e = k % per, it = it0 + e / (2 * nb), side = e / nb % 2, b = e % nb;
      const C3& c = tab.c[tab.mu[it]];
      double2 v = factor(rec + (size_t)ci * L.rec, L, c.f[side], tab.sg[it] * n, b);
      if (side == 0) {
        const double2 x = d2(xw[2 * (size_t)ci + (c.centre == 2)]);
        v = cmul(c.centre == 1 ? cj(x) : x, v);
      }
      rows[k] = v;
    }
    __syncthreads();
    for (int k = 0; k < nc; ++k) {
      const double2* rw = rows + k * per;
#pragma unroll
      for (int r = 0; r < kC3Out; ++r) {
        if (ra[r] < 0) break;
        const double2 u = rw[ra[r]], v = rw[rb[r]];
        acc[r].x += u.x * v.x;
        acc[r].y += u.x * v.y;
        acc[r].x -= u.y * v.y;
        acc[r].y += u.y * v.x;
      }
    }
  }
  double2* out = part + (size_t)sl * (5 * nn * nb2 + 5 * nb);
#pragma unroll
  for (int r = 0; r < kC3Out; ++r) {
    if (ra[r] < 0) break;
    const int o = o0 + r * kC3Threads + tid, it = o / nb2;
    if (n == 0 && tab.sg[it] < 0) continue;  // the same sum as at + n
    out[(size_t)(tab.mu[it] * nn + tab.sg[it] * n + L.N) * nb2 + o % nb2] = acc[r];
  }
  // the same neighbour's terms t D of the slice
  if (n == 0 && ch == 0) {
    for (int k = tid; k < 5 * nb; k += kC3Threads) {
      const C3& c = tab.c[k / nb];
      double2 sum = make_double2(0.0, 0.0);
#pragma unroll 4
      for (int i = i0; i < i1; ++i) {
        const double2 x = d2(xw[2 * (size_t)i + (c.centre == 2)]);
        sum = cadd(sum, cmul(c.centre == 1 ? cj(x) : x, same_galaxy(rec + (size_t)i * L.rec, L, c.d, k % nb)));
      }
      out[(size_t)5 * nn * nb2 + k] = sum;
    }
  }
}

// thread = output entry: the slices' partial sums in slice order, with the component's sign
__global__ void contract3_sum(const Layout L, const Table3 tab, int S, const double2* __restrict__ part,
                              double* __restrict__ ups3) {
  const int nn = 2 * L.N + 1, nb = L.nb, nb2 = nb * nb;
  const size_t total = (size_t)5 * nn * nb2, stride = total + 5 * nb;
  for (size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o < total; o += (size_t)gridDim.x * blockDim.x) {
    const int mu = (int)(o / ((size_t)nn * nb2)), n = (int)(o / nb2 % nn) - L.N;
    const int b1 = (int)(o % nb2) / nb, b2 = (int)(o % nb2) % nb;
    const int m = tab.mir[mu];
    const bool mirrored = m >= 0 && (m == mu ? n < 0 : m > mu);
    const size_t src = mirrored ? (size_t)(m * nn - n + L.N) * nb2 + b2 * nb + b1 : o;
    double re = 0.0, im = 0.0;
    for (int sl = 0; sl < S; ++sl) {
      const double2 v = part[(size_t)sl * stride + src];
      re += v.x;
      im += v.y;
      if (b1 == b2) {
        const double2 d = part[(size_t)sl * stride + total + mu * nb + b1];
        re -= d.x;
        im -= d.y;
      }
    }
    ups3[2 * o] += tab.c[mu].sign * re;
    ups3[2 * o + 1] += tab.c[mu].sign * im;
  }
}

// m = a n + b over |n| <= N stays inside [lo, hi]
bool in_range(const F3& f, int N, int lo, int hi) {
  const int m1 = f.a * N + f.b, m2 = -f.a * N + f.b;
  return std::min(m1, m2) >= lo && std::max(m1, m2) <= hi;
}

// Order-3 tables from the generator, with the same-neighbour term of each component; false
// if a needed index lies outside the gather's record (Layout) for this N.
bool build_table3(int N, Table3& t) {
  for (int k = 0; k < 5; ++k) {
    const int mu = k < 4 ? k : -1;
    int raw[10];
    if (ext4pcf_nth_order_factors(3, mu, raw, 10) != 10) return false;
    C3& c = t.c[k];
    c.sign = raw[0];
    c.centre = raw[1];
    for (int l = 0; l < 2; ++l) c.f[l] = F3{raw[2 + 4 * l], raw[3 + 4 * l], raw[4 + 4 * l], raw[5 + 4 * l]};
    const F3 &f0 = c.f[0], &f1 = c.f[1];
    if (f0.arr != f1.arr) return false;
    if (f0.arr == 1) {  // w_j e^{i m0 phi} w_j e^{i m1 phi}
      // the same-galaxy term below is W W at the summed index, valid only when neither W
      // factor is conjugated; a table with a conjugated W factor is refused
      if (f0.conj || f1.conj) return false;
      if (f0.a + f1.a != 0) return false;
      c.d = D3{2, f0.b + f1.b, 0};
      if (!in_range(f0, N, -2 * N, 2 * N) || !in_range(f1, N, -2 * N, 2 * N) || std::abs(c.d.idx) > 2 * N)
        return false;
      continue;
    }
    if (f0.conj == f1.conj) {  // x_j^2 e^{i (m0 + m1) phi}, conjugated if both factors are
      if (f0.a + f1.a != 0) return false;
      c.d = D3{0, f0.b + f1.b, f0.conj};
      if (c.d.idx < -2 * N - 6 || c.d.idx > 2 * N - 2) return false;
    } else {  // |x_j|^2 e^{i (m_plain - m_conj) phi}
      const F3& pl = f0.conj ? f1 : f0;
      const F3& cn = f0.conj ? f0 : f1;
      if (pl.a - cn.a != 0) return false;
      c.d = D3{1, pl.b - cn.b, 0};
      if (std::abs(c.d.idx) > 2 * N + 2) return false;
    }
    if (!in_range(f0, N, -2 * N - 3, 2 * N - 1) || !in_range(f1, N, -2 * N - 3, 2 * N - 1)) return false;
  }
  auto same = [](const F3& f, const F3& g) { return f.arr == g.arr && f.conj == g.conj && f.a == -g.a && f.b == g.b; };
  t.nitem = 0;
  for (int k = 0; k < 5; ++k) {
    t.mir[k] = -1;
    for (int m = 0; m < 5 && t.mir[k] < 0; ++m)
      if (t.c[m].centre == t.c[k].centre && same(t.c[m].f[0], t.c[k].f[1]) && same(t.c[m].f[1], t.c[k].f[0]))
        t.mir[k] = m;
    if (t.mir[k] > k) continue;  // taken from that component
    for (int sg = 1; sg >= -1; sg -= 2)
      if (sg > 0 || t.mir[k] != k) {
        t.mu[t.nitem] = (signed char)k;
        t.sg[t.nitem++] = (signed char)sg;
      }
  }
  return true;
}

}  // namespace

bool contract3_supported(int N) {
  Table3 t;
  return build_table3(N, t);
}

// at least 32 centres to a slice
int contract3_slices(int T) { return std::max(1, std::min(32, T / 32)); }
size_t contract3_scratch_bytes(const Layout& L, int T) {
  return (size_t)contract3_slices(T) * 5 * ((2 * L.N + 1) * L.nb * L.nb + L.nb) * sizeof(double2);
}

template <typename Cx>
cudaError_t contract3_wave(const Layout& L, const Cx* rec, const Cx* xw, int T, double* ups3, double2* scratch,
                           cudaStream_t s) {
  Table3 t;
  if (!build_table3(L.N, t)) return cudaErrorInvalidValue;
  if (T <= 0) return cudaSuccess;
  const int S = contract3_slices(T);
  const int nb2 = L.nb * L.nb, outs = kC3Threads * kC3Out, chunks = (t.nitem * nb2 + outs - 1) / outs;
  // components that 512 consecutive sums touch, at most
  const int items = std::min(t.nitem, (outs + nb2 - 2) / nb2 + 1);
  const size_t smem = (size_t)kC3Centres * items * 2 * L.nb * sizeof(double2);
  cudaError_t e = allow_smem(contract3_kernel<Cx>);
  if (e != cudaSuccess) return e;
  contract3_kernel<Cx><<<(L.N + 1) * S * chunks, kC3Threads, smem, s>>>(L, t, rec, xw, T, S, chunks, scratch);
  const int total = 5 * (2 * L.N + 1) * nb2;
  contract3_sum<<<std::min(4 * device_sms(), (total + 127) / 128), 128, 0, s>>>(L, t, S, scratch, ups3);
  g_launches += 2;
  return cudaGetLastError();
}
template cudaError_t contract3_wave<float2>(const Layout&, const float2*, const float2*, int, double*, double2*,
                                            cudaStream_t);
template cudaError_t contract3_wave<double2>(const Layout&, const double2*, const double2*, int, double*,
                                             double2*, cudaStream_t);

}  // namespace ext4pcf
