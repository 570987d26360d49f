// Sums over a wave's centres of the multiple-counting terms (paper App. A.1, Table tab:4PCFMCCorr) and
// the xi accumulators, for the layout of basis.cuh.
//
// One block takes one sg and one slice of the wave's centres.  It stages the two merged factors XX_sg
// and XA_{sg+4} and the four columns x G_{-sg-8}, x^* G_{-sg-4}, x G_{sg+4}^*, x^* G_sg^* of 32 centres
// (corr_chunk; each loaded once for the six arrays they serve), and a thread holds a 2 x 2 tile of bins of one
// array, or with few bins its part of the centres.  Products and sums over corr_run centres are in R,
// the rest in FP64; every slice adds into a copy of its own (one writer, no atomics), and the copies
// are added in order at the end of the call.
// One block per (component, kind, index), 27 arrays of terms where seven hold them all, took 1.56 ms
// a wave of 8192 centres at n_max = 20, 10 bins (and the xi sums 76 us); this takes 0.52 ms, a
// quarter of it FP64 additions (16 clocks a warp instruction and SM).
#include <algorithm>

#include "basis.cuh"

namespace ext4pcf {

namespace {

// Few bins have few tiles: up to kCorrParts threads share one, each with every parts-th centre.
constexpr int kCorrParts = 8;
// Centres that a thread sums in FP32 before it adds them in FP64.  Few bins are the cheaper ones and keep
// more of their sums in FP64: the 1, 3, 7, 11 centres that 192 threads sharing the tiles of 2, 4, 6, 8
// bins have of 128 each (at 10 bins and more it would be 19 and up).  16 for every number of bins lost what lies 2^-24
// below the largest of 16 terms.  Whole split-FP16 calls on 3000 galaxies with 16 everywhere, with runs of 1, 2, 4,
// 8 and one thread to a tile, and as it is: 0.72, 1.07, 0.77 ms (2 bins, n_max = 20); 0.57, 0.67, 0.59 ms
// (4, 10); 1.03, 1.13, 1.06 ms (5, 20).
__host__ __device__ constexpr int corr_run(int nb) { return nb <= 2 ? 1 : nb <= 4 ? 3 : nb <= 6 ? 7 : nb <= 8 ? 11 : 16; }
// Centres staged at once: two full runs of every thread that shares a tile (8, 3, 2 of them for 4, 6, 8 bins)
__host__ __device__ constexpr int corr_chunk(int nb) { return nb <= 2 ? 32 : nb <= 4 ? 48 : nb <= 6 ? 42 : nb <= 8 ? 44 : 32; }

template <typename Cx> struct __align__(16) Pair2 { Cx a, b; };

// The arrays of an X block: which merged factor (0: XX, 1: XA) and which column
__constant__ signed char kArrP[6] = {0, 0, 0, 1, 0, 1};
__constant__ signed char kArrO[6] = {0, 1, 2, 0, 3, 1};

// whether array k of sg is made of entries that the record holds
__device__ __forceinline__ bool corr_valid(const Layout& L, int k, int sg) {
  const int N = L.N, q = kArrO[k];
  const bool p = kArrP[k] ? (sg + 4 <= 2 * N + 2 && sg + 4 >= -2 * N - 2) : (sg >= -2 * N - 6 && sg <= 2 * N - 2);
  return p && basis_in_g(N, basis_col_index(q, sg));
}

// SHARED: tiles that several threads share (up to eight bins)
template <typename R, bool SHARED>
__global__ void __launch_bounds__(384) corrections_kernel(const Layout L, const CorrLayout C,
                                                          const cplx_t<R>* __restrict__ rec,
                                                          const cplx_t<R>* __restrict__ xw,
                                                          const __grid_constant__ WavePlan plan,
                                                          double2* __restrict__ corr, size_t slot_stride, bool xi) {
  using Cx = cplx_t<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nb = L.nb, N = L.N, tid = threadIdx.x, job = blockIdx.x, slice = blockIdx.y, ns = gridDim.y;
  const int nt = (nb + 1) / 2, nbp = 2 * nt;
  const size_t nb2 = (size_t)nb * nb;
  double2* copy = corr + (size_t)slice * C.elems;
  if (job == C.nsig + 2 * N + 1) {
    // ---- triple sums and xi accumulators: thread (part of the slice's centres, item), items
    // [5][nb] triple then [3][nb] xi; FP64 sums of products in R (xi: in FP64), parts in order
    double2* red = reinterpret_cast<double2*>(smem_raw);
    const int items = (xi ? 8 : 5) * nb, parts = max(1, (int)blockDim.x / items);
    for (int si = 0; si < plan.nseg; ++si) {
      const WaveSeg& g = plan.seg[si];
      const int live = seg_live(g);
      const int t0 = (int)((long long)live * slice / ns), t1 = (int)((long long)live * (slice + 1) / ns);
      for (int i0 = 0; i0 < items; i0 += blockDim.x) {  // (more items than threads: one part, several passes)
        const int item = i0 + tid % min(items, (int)blockDim.x), part = parts > 1 ? tid / items : 0;
        double ar = 0.0, ai = 0.0;
        if (item < items && part < parts) {
          const int k = item / nb, b = item % nb;
          for (int c = t0 + part; c < t1; c += parts) {
            const Cx* rc = rec + (size_t)(g.off + c) * L.rec;
            const Cx x = xw[2 * (size_t)(g.off + c)], w = xw[2 * (size_t)(g.off + c) + 1];
            if (k < 5) {
              const Cx f = rc[L.TR(k, b)];
              const Cx v = cmul(k == 4 ? w : (k & 1) ? cconj(x) : x, f);
              ar += (double)v.x;
              ai += (double)v.y;
            } else {  // x^* G_0, x G_-4, w W_0
              const Cx f = k == 5 ? rc[L.G(0, b)] : k == 6 ? rc[L.G(-4, b)] : rc[L.W(0, b)];
              const double xr = k == 7 ? (double)w.x : (double)x.x, xm = k == 7 ? 0.0 : k == 5 ? -(double)x.y : (double)x.y;
              ar += xr * (double)f.x - xm * (double)f.y;
              ai += xr * (double)f.y + xm * (double)f.x;
            }
          }
        }
        __syncthreads();
        red[tid] = make_double2(ar, ai);
        __syncthreads();
        if (item < items && part == 0) {
          double2 s = red[tid];
          for (int p = 1; p < parts; ++p) {
            s.x += red[tid + p * items].x;
            s.y += red[tid + p * items].y;
          }
          double2* o = copy + (size_t)g.slot * slot_stride + C.ot + item;
          o->x += s.x;
          o->y += s.y;
        }
      }
    }
    return;
  }
  const bool wk = job >= C.nsig;
  const int sg = wk ? job - C.nsig : -2 * N - 6 + job;  // (W blocks: the index c)
  const int width = (wk ? 2 : 6) * nbp;                 // staged values per centre
  const int tiles = (wk ? 1 : 6) * nt * nt;
  const int run = SHARED && sizeof(R) == 4 ? corr_run(nb) : 16, chunk = SHARED ? corr_chunk(nb) : 32;
  Cx* st = reinterpret_cast<Cx*>(smem_raw);  // [chunk][width]
  // the value this thread stages of every (blockDim / width)-th centre: its place in a record (-1: a
  // zero), its conjugation and its centre factor (0: none, 1: x, 2: x^*, 3: w)
  const int cper = blockDim.x / width, scol = tid % width, scc = tid / width;
  int soff = -1, sfac = 0;
  R ssign = R(1);
  {
    const int b = scol % nbp, f = scol / nbp;
    if (b < nb && scc < cper) {
      if (wk) {
        soff = f == 0 ? L.WW(sg, b) : L.W(sg, b);
        if (f == 0) ssign = R(-1);
        else sfac = 3;
      } else if (f == 0) {
        soff = L.XX(sg, b);
      } else if (f == 1) {
        const int m = sg + 4;
        if (m <= 2 * N + 2 && m >= -2 * N - 2) soff = L.XA(m >= 0 ? m : -m, b);
        if (m < 0) ssign = R(-1);
      } else {
        const int q = f - 2, m = basis_col_index(q, sg);
        if (basis_in_g(N, m)) {
          soff = L.G(m, b);
          sfac = basis_centre_conj(q) ? 2 : 1;
          if (basis_col_conj(q)) ssign = R(-1);
        }
      }
    }
  }
  const int parts = SHARED ? max(1, min(kCorrParts, (int)blockDim.x / tiles)) : 1;
  for (int i0 = 0; i0 < tiles; i0 += blockDim.x) {
    const int tile = parts > 1 ? tid % tiles : i0 + tid, part = parts > 1 ? tid / tiles : 0;
    const int k = tile / (nt * nt), ta = 2 * ((tile / nt) % nt), tb = 2 * (tile % nt);
    const bool active = tile < tiles && part < parts && (wk || corr_valid(L, k, sg));
    const int po = wk ? ta : kArrP[active ? k : 0] * nbp + ta, oo = wk ? nbp + tb : (2 + kArrO[active ? k : 0]) * nbp + tb;
    for (int si = 0; si < plan.nseg; ++si) {
      const WaveSeg& g = plan.seg[si];
      const int live = seg_live(g);
      const int t0 = (int)((long long)live * slice / ns), t1 = (int)((long long)live * (slice + 1) / ns);
      if (t0 == t1) continue;
      double a64[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) a64[i][0] = a64[i][1] = 0.0;
      for (int c0 = t0; c0 < t1; c0 += chunk) {
        const int nc = min(chunk, t1 - c0);
        __syncthreads();
        if (scc < cper) {
#pragma unroll 4
          for (int cc = scc; cc < nc; cc += cper) {
            const size_t c = (size_t)(g.off + c0 + cc);
            Cx v = cmk<Cx>(R(0), R(0));
            if (soff >= 0) {
              v = rec[c * L.rec + soff];
              v.y *= ssign;
              if (sfac) {
                Cx x = xw[2 * c + (sfac == 3 ? 1 : 0)];
                if (sfac == 2) x.y = -x.y;
                v = cmul(x, v);
              }
            }
            st[cc * width + scol] = v;
          }
        }
        __syncthreads();
        if (active) {
          for (int h = part; h < nc; h += run * parts) {
            Cx acc[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = cmk<Cx>(R(0), R(0));
            const int he = min(nc, h + run * parts);
            for (int cc = h; cc < he; cc += parts) {
              const Cx* row = st + cc * width;  // (po, oo and width are even: aligned pairs)
              const Pair2<Cx> p = *reinterpret_cast<const Pair2<Cx>*>(row + po);
              const Pair2<Cx> o = *reinterpret_cast<const Pair2<Cx>*>(row + oo);
              acc[0] = cadd(acc[0], cmul(p.a, o.a));
              acc[1] = cadd(acc[1], cmul(p.a, o.b));
              acc[2] = cadd(acc[2], cmul(p.b, o.a));
              acc[3] = cadd(acc[3], cmul(p.b, o.b));
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              a64[i][0] += (double)acc[i].x;
              a64[i][1] += (double)acc[i].y;
            }
          }
        }
      }
      double2* out = copy + (size_t)g.slot * slot_stride;
      auto add = [&](int tl, int i, double2 sum) {  // value i of tile tl
        const int a = tl / (nt * nt), ba = 2 * ((tl / nt) % nt) + (i >> 1), bb = 2 * (tl % nt) + (i & 1);
        if (ba >= nb || bb >= nb || !(wk || corr_valid(L, a, sg))) return;
        double2* o = out + (wk ? C.ow + (size_t)sg * nb2 : ((size_t)a * C.nsig + job) * nb2) + ba * nb + bb;
        const double2 v = *o;
        *o = make_double2(v.x + sum.x, v.y + sum.y);
      };
      if (parts > 1) {  // the parts' sums in order (the staged values have been used)
        double2* red = reinterpret_cast<double2*>(smem_raw);  // [parts][tiles][4]
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (part < parts) red[tid * 4 + i] = make_double2(a64[i][0], a64[i][1]);
        __syncthreads();
        for (int e = tid; e < 4 * tiles; e += blockDim.x) {
          double2 sum = red[e];
          for (int p = 1; p < parts; ++p) {
            sum.x += red[e + p * 4 * tiles].x;
            sum.y += red[e + p * 4 * tiles].y;
          }
          add(e / 4, e % 4, sum);
        }
      } else if (active) {
#pragma unroll
        for (int i = 0; i < 4; ++i) add(tile, i, make_double2(a64[i][0], a64[i][1]));
      }
    }
  }
}

// the copies of every slot added into the first, in order, and its xi sums into the caller's
__global__ void corrections_sum(const CorrLayout C, int copies, size_t slot_stride, double2* __restrict__ corr,
                                double* __restrict__ xi) {
  double2* c = corr + (size_t)blockIdx.y * slot_stride;
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= C.elems) return;
  double2 v = c[e];
  for (int k = 1; k < copies; ++k) {
    const double2 t = c[e + (size_t)k * C.elems];
    v.x += t.x;
    v.y += t.y;
  }
  c[e] = v;
  if (xi && e >= C.ox) {
    const int i = (int)(e - C.ox), q = i / C.nb, b = i % C.nb;
    double* o = xi + (size_t)blockIdx.y * 6 * C.nb + 6 * b + 2 * q;
    o[0] += v.x;
    o[1] += v.y;
  }
}

}  // namespace

// Copies per slot, of n_out slots that are summed at once: slices enough to fill the SMs from one sg each while the
// slots are few (with many a wave's segments are short), and no more than two where all of them would
// take over 128 MB (16 copies of 8 slots are 56 MB at n_max = 20, 10 bins, 2.25 GB at 40, 32).
static int corrections_copies(const CorrLayout& C, int n_out) {
  const size_t fit = ((size_t)128 << 20) / (C.elems * sizeof(double2) * (size_t)n_out);
  return (int)std::min<size_t>(n_out <= 8 ? 16 : n_out < 32 ? 4 : 2, std::max<size_t>(fit, 2));
}
size_t corrections_slot_doubles(const Layout& L, int n_out) {
  const CorrLayout C = CorrLayout::make(L.N, L.nb);
  return 2 * C.elems * corrections_copies(C, n_out);
}

template <typename R>
cudaError_t corrections_wave(const Layout& L, const cplx_t<R>* rec, const cplx_t<R>* xw, const WavePlan& plan, int n_out,
                             double* corr, bool xi, cudaStream_t s) {
  if (plan.total <= 0 || plan.nseg <= 0) return cudaSuccess;
  const CorrLayout C = CorrLayout::make(L.N, L.nb);
  const int nt = (L.nb + 1) / 2;
  // up to eight bins 192 threads: 8, 8, 3 and 2 to a tile of the six X arrays
  const bool shared = nt <= 4;
  const int threads = std::min(384, std::max(shared ? 192 : 160, (6 * nt * nt + 31) / 32 * 32));
  const size_t smem = std::max((size_t)corr_chunk(L.nb) * 12 * nt * sizeof(cplx_t<R>),
                               (size_t)threads * (shared ? 4 : 1) * sizeof(double2));
  auto kernel = shared ? corrections_kernel<R, true> : corrections_kernel<R, false>;
  cudaError_t e = allow_smem(kernel);
  if (e != cudaSuccess) return e;
  const int copies = corrections_copies(C, n_out);
  kernel<<<dim3(C.nsig + 2 * L.N + 2, copies), threads, smem, s>>>(
      L, C, rec, xw, plan, reinterpret_cast<double2*>(corr), C.elems * copies, xi);
  ++g_launches;
  return cudaGetLastError();
}

cudaError_t corrections_finish(const Layout& L, int n_out, double* corr, double* xi, cudaStream_t s) {
  const CorrLayout C = CorrLayout::make(L.N, L.nb);
  const int copies = corrections_copies(C, n_out);
  for (int o = 0; o < n_out; o += 32768) {
    const int n = std::min(32768, n_out - o);
    corrections_sum<<<dim3((unsigned)((C.elems + 255) / 256), n), 256, 0, s>>>(
        C, copies, C.elems * copies, reinterpret_cast<double2*>(corr) + (size_t)o * C.elems * copies,
        xi ? xi + (size_t)o * 6 * L.nb : nullptr);
    ++g_launches;
  }
  return cudaGetLastError();
}

template cudaError_t corrections_wave<float>(const Layout&, const float2*, const float2*, const WavePlan&, int, double*,
                                             bool, cudaStream_t);
template cudaError_t corrections_wave<double>(const Layout&, const double2*, const double2*, const WavePlan&, int,
                                              double*, bool, cudaStream_t);

}  // namespace ext4pcf
