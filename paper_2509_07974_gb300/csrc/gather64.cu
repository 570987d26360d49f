// FP64 neighbour gather: the records of gather.cu with positions and arithmetic in double.
//
// One CTA (8 warps) per centre:
//   (a) the rows of cells that can hold partners are contiguous ranges of the cell-sorted
//       catalogue (found by one warp, a row per lane); the CTA streams them, keeps pairs
//       with Theta_lo^2 <= r^2 < Theta_hi^2, and buckets them by radial bin into a
//       shared-memory chunk (stable order, so the summation order is deterministic).  Chunks
//       hold up to `cap` candidates; long neighbour lists take several chunks.
//   (b) the work of a chunk is split into items (bin, power block): block k holds the powers
//       m in [k*mb, k*mb+mb) of u = e^{i phi}.  The warps take the items in turn, outer
//       bins first.  For an item each lane walks pairs of the bin, raises u to the block's
//       first power (u^mb is stored per pair) and steps through the block by recurrence in
//       registers, accumulating seven real weights times u^m: Re x, Im x, Re x^2, Im x^2, w,
//       |x|^2, w^2.  The complex sums x u^{+-m} and x^2 u^{+-m} follow from the first four.
//       The 32 lanes' partial sums are combined by a transposed butterfly (each lane ends
//       with V/32 totals) and added to the centre's record in shared memory; no two items
//       of a chunk share a record entry.
//   (c) the record is written to the wave buffer (or added to it, for the later passes of the
//       tree approximation).
// The bin decision r^2 = dx*dx + dy*dy is evaluated with two rounded products and one rounded
// sum, as the FP64 definition reads.  The FP64 pipe (16 clocks a warp instruction and SM) bounds
// it: eight warps keep it full, so the registers go to blocks of six powers, whose set-up per pair
// and block (the first power, the weights) is paid half as often as with three.  1000 centres of
// 28000 pairs at n_max = 20: 69.5 -> 46.2 ms (846 multiply-adds a pair alone take 37.6 ms).
#include <algorithm>

#include "common.cuh"
#include "gather_common.cuh"

namespace ext4pcf {

namespace {

constexpr int kThreads = 256;
constexpr int kMB = 6;  // powers per block
constexpr int kWarps = kThreads / 32;
constexpr unsigned kFull = 0xFFFFFFFFu;

// Bucketed pairs in shared memory, structure of arrays: uv = (u_re, u_im, v_re, v_im) with
// u = e^{i phi}, v = u^mb; x = w gamma_c; w
struct __align__(16) Dbl4 { double x, y, z, w; };

// sums of an item (14 per power, 10 triple terms), rounded up to whole lanes
constexpr int V = (14 * kMB + 10 + 31) / 32 * 32;

// u^e for 0 <= e < 32 by binary powering, unrolled (e is uniform across the warp)
template <typename R>
__device__ __forceinline__ void cpow5(R br, R bi, int e, R& pr, R& pi) {
  pr = R(1); pi = R(0);
#pragma unroll
  for (int bit = 0; bit < 5; ++bit) {
    if (e & (1 << bit)) { R t = pr * br - pi * bi; pi = pr * bi + pi * br; pr = t; }
    if (e >> (bit + 1)) { R t = br * br - bi * bi; bi = R(2) * br * bi; br = t; }
  }
}

// transposed butterfly: after the call lane l holds in a[0..V/32) the warp totals of the
// original slots j + base(l), base(l) = sum_k bit_k(l) * V / 2^(5-k)
template <typename R, int V, int OFF>
__device__ __forceinline__ void rt_step(R* a, int lane) {
  constexpr int H = V / 2;
  const bool up = (lane & OFF) != 0;
#pragma unroll
  for (int j = 0; j < H; ++j) {
    R send = up ? a[j] : a[j + H];
    R keep = up ? a[j + H] : a[j];
    a[j] = keep + __shfl_xor_sync(kFull, send, OFF);
  }
}
template <typename R, int V>
__device__ __forceinline__ void reduce_transpose(R* a, int lane) {
  rt_step<R, V, 16>(a, lane);
  rt_step<R, V / 2, 8>(a, lane);
  rt_step<R, V / 4, 4>(a, lane);
  rt_step<R, V / 8, 2>(a, lane);
  rt_step<R, V / 16, 1>(a, lane);
}


// v^k for the block index k (uniform across the warp): the shortest product chain for
// k < 8 as straight-line code behind one uniform branch, binary powering beyond
__device__ __forceinline__ void vpow_block(double vr, double vi, int k, double2& P) {
  const double2 v = make_double2(vr, vi);
  switch (k) {
    case 0: P = make_double2(1.0, 0.0); return;
    case 1: P = v; return;
    case 2: P = cmul(v, v); return;
    case 3: P = cmul(cmul(v, v), v); return;
    case 4: { const double2 v2 = cmul(v, v); P = cmul(v2, v2); return; }
    case 5: { const double2 v2 = cmul(v, v); P = cmul(cmul(v2, v2), v); return; }
    case 6: { const double2 v2 = cmul(v, v); P = cmul(cmul(v2, v2), v2); return; }
    case 7: { const double2 v2 = cmul(v, v); P = cmul(cmul(cmul(v2, v2), v2), v); return; }
    default: cpow5<double>(vr, vi, k, P.x, P.y); return;
  }
}

// sums of one item, one pair per lane and iteration: a[0, 14 kMB) the powers of block k, 14 each,
// then the triple terms of its share of the bin
__device__ __forceinline__ void accumulate(double* a, const Dbl4* __restrict__ euv, const double2* __restrict__ ex,
                                           const double* __restrict__ ew, int s0, int s1, int lane, int k, int mb) {
  for (int e = s0 + lane; e < s1; e += 32) {
    const Dbl4 q = euv[e];
    const double2 xx = ex[e];
    const double w = ew[e];
    double2 P;
    vpow_block(q.z, q.w, k, P);
    const double wt[7] = {xx.x, xx.y, xx.x * xx.x - xx.y * xx.y, 2.0 * xx.x * xx.y, w, xx.x * xx.x + xx.y * xx.y,
                          w * w};
#pragma unroll
    for (int t = 0; t < kMB; ++t) {
      if (t >= mb) break;
#pragma unroll
      for (int j = 0; j < 7; ++j) {
        a[14 * t + 2 * j] += wt[j] * P.x;
        a[14 * t + 2 * j + 1] += wt[j] * P.y;
      }
      if (t + 1 < kMB) P = make_double2(P.x * q.x - P.y * q.y, P.x * q.y + P.y * q.x);
    }
  }
  if (k != 0) return;
  // x^3 u^-8, x^3 u^-4, x^2 x^* u^-4, x^2 x^*, w^3, with the first block
  double* tr = a + 14 * kMB;
  for (int e = s0 + lane; e < s1; e += 32) {
    const Dbl4 q = euv[e];
    const double2 xx = ex[e];
    const double w = ew[e];
    const double ur = q.x, ui = q.y, xr = xx.x, xi = xx.y;
    const double x2r = xr * xr - xi * xi, x2i = 2.0 * xr * xi, xa = xr * xr + xi * xi;
    const double u2r = ur * ur - ui * ui, u2i = 2.0 * ur * ui;
    const double u4r = u2r * u2r - u2i * u2i, u4i = 2.0 * u2r * u2i;
    const double u8r = u4r * u4r - u4i * u4i, u8i = 2.0 * u4r * u4i;
    const double x3r = x2r * xr - x2i * xi, x3i = x2r * xi + x2i * xr;
    const double xcr = xa * xr, xci = xa * xi;  // x^2 x^* = |x|^2 x
    tr[0] += x3r * u8r + x3i * u8i;  // x3 * conj(u8)
    tr[1] += x3i * u8r - x3r * u8i;
    tr[2] += x3r * u4r + x3i * u4i;
    tr[3] += x3i * u4r - x3r * u4i;
    tr[4] += xcr * u4r + xci * u4i;
    tr[5] += xci * u4r - xcr * u4i;
    tr[6] += xcr;
    tr[7] += xci;
    tr[8] += (w * w) * w;
  }
}

__global__ void __launch_bounds__(kThreads, 1)
gather64_kernel(const GatherArgs args, double2* __restrict__ rec, double2* __restrict__ xw) {
  using R = double;
  using Cx = double2;
  extern __shared__ __align__(16) unsigned char smem[];
  const SortedCat& cat = args.cat;
  const Layout L = args.L;
  const int nb = args.bins.nb, cap = args.cap, mb = args.mb, nblk = args.nblk;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  Dbl4* euv = reinterpret_cast<Dbl4*>(smem);
  Cx* ex = reinterpret_cast<Cx*>(euv + cap);
  R* ew = reinterpret_cast<R*>(ex + cap);
  double* e2 = reinterpret_cast<double*>(ew + cap);
  int* off = reinterpret_cast<int*>(e2 + 65);  // [65] bin offsets of the chunk
  int* wcnt = off + 65;                          // [warps][64] per-warp bin counts / positions
  int* rstart = wcnt + kWarps * 64;
  int* rpre = rstart + kMaxRows;
  int* misc = rpre + kMaxRows + 1;  // rows, candidates, work items taken
  int* fidx = misc + 8;             // [nblk][V] where the reduced slots of each power block go
  signed char* cbin = reinterpret_cast<signed char*>(fidx + nblk * V);  // bin of each candidate
  Cx* accs = reinterpret_cast<Cx*>((reinterpret_cast<uintptr_t>(cbin + cap) + 15) & ~(uintptr_t)15);

  for (int b = tid; b <= nb; b += kThreads) e2[b] = args.bins.e2[b];
  for (int k = tid; k < kWarps * 64; k += kThreads) wcnt[k] = 0;
  // Reduced slot s of power block k (slot order of the accumulation: 14 per power, then the
  // 10 triple terms) goes to the record's index fidx[k][s] + 2b for bin b (every array of the
  // record is [multipole][bin]); -1: nowhere
  for (int i = tid; i < nblk * V; i += kThreads) {
    const int k = i / V, slot = i % V, m0 = k * mb;
    int f = -1;
    if (slot < 14 * kMB) {
      const int t = slot / 14, q = slot % 14, m = m0 + t;
      int idx = -1;
      if (t < mb) {
        switch (q >> 1) {
          case 0: if (m <= 2 * L.N - 1) idx = L.G(m, 0); break;
          case 1: if (m >= 1 && m <= 2 * L.N + 3) idx = L.G(-m, 0); break;
          case 2: if (m <= 2 * L.N - 2) idx = L.XX(m, 0); break;
          case 3: if (m >= 1 && -m <= 2 * L.N - 2 && m <= 2 * L.N + 6) idx = L.XX(-m, 0); break;
          case 4: if (m <= 2 * L.N) idx = L.W(m, 0); break;
          case 5: if (m <= 2 * L.N + 2) idx = L.XA(m, 0); break;
          default: if (m <= 2 * L.N) idx = L.WW(m, 0); break;
        }
      }
      f = idx >= 0 ? 2 * idx + (slot & 1) : -1;
    } else if (slot < 14 * kMB + 10) {
      f = k == 0 ? 2 * L.TR((slot - 14 * kMB) >> 1, 0) + (slot & 1) : -1;
    }
    fidx[i] = f;
  }
  // the reduced slots this lane holds after the transposed butterfly: base + [0, V/32)
  const int rbase = (lane & 16 ? V / 2 : 0) + (lane & 8 ? V / 4 : 0) + (lane & 4 ? V / 8 : 0) +
                    (lane & 2 ? V / 16 : 0) + (lane & 1 ? V / 32 : 0);
  const double rmax = args.bins.rmax * (1.0 + 1e-9) + 1e-12;

  for (int c = blockIdx.x; c < args.plan.total; c += gridDim.x) {
    // the record's segment: its catalogue's grid and centre (padding records are skipped)
    int j = 0;
    const int si = seg_of(args.plan, c, &j);
    if (si < 0 || j >= seg_live(args.plan.seg[si])) continue;  // uniform over the block
    const WaveSeg& sg = args.plan.seg[si];
    const GridGeom gm = *sg.geom;
    const double gx0 = gm.x0, gy0 = gm.y0, cell = gm.cell;
    const int gncx = gm.ncx, gncy = gm.ncy;
    const int pi = sg.centres[sg.w0 + j];
    const double pxi = args.cen.px[pi], pyi = args.cen.py[pi];
    if (warp == 0) {
      // the rows of cells within rmax of the centre, one per lane (cells are at least rmax / 16
      // wide, so there are at most 34), kept in row order when they hold galaxies
      const double xc = pxi - gx0, yc = pyi - gy0;
      const int cy0 = max((int)floor((yc - rmax) / cell), 0);
      const int cy1 = min((int)floor((yc + rmax) / cell), gncy - 1);
      int nr = 0, tot = 0;
      for (int cyb = cy0; cyb <= cy1; cyb += 32) {
        const int cy = cyb + lane;
        int a = 0, len = 0;
        if (cy <= cy1) {
          const double lo = cy * cell, hi = lo + cell;
          const double gap = fmax(0.0, fmax(lo - yc, yc - hi));
          if (gap <= rmax) {
            const double hw = sqrt(fmax(0.0, rmax * rmax - gap * gap));
            const int cx0 = max((int)floor((xc - hw) / cell), 0);
            const int cx1 = min((int)floor((xc + hw) / cell), gncx - 1);
            if (cx0 <= cx1) {
              a = sg.cell_start[cy * gncx + cx0];
              len = max(sg.cell_start[cy * gncx + cx1 + 1] - a, 0);
            }
          }
        }
        const unsigned ok = __ballot_sync(kFull, len > 0);
        const int pos = nr + __popc(ok & ((1u << lane) - 1u));
        const bool keep = len > 0 && pos < kMaxRows;
        int inc = keep ? len : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(kFull, inc, o);
          if (lane >= o) inc += v;
        }
        if (keep) {
          rstart[pos] = a;
          rpre[pos] = tot + inc - len;
        }
        nr = min(nr + __popc(ok), kMaxRows);
        tot += __shfl_sync(kFull, inc, 31);
      }
      if (lane == 0) {
        rpre[nr] = tot;
        misc[0] = nr; misc[1] = tot;
      }
    }
    // the record collects in shared memory
    Cx* dst = rec + (size_t)c * L.rec;
    R* accf = reinterpret_cast<R*>(accs);
    for (int k = tid; k < L.rec; k += kThreads) accs[k] = cmk<Cx>(R(0), R(0));
    __syncthreads();
    const int nr = misc[0], total = misc[1];
    unsigned long long pairs_here = 0;

    for (int cpos = 0; cpos < total;) {
      // ---- classification and stable bucketing by bin of the next cap candidates
      const int cend = min(total, cpos + cap);
      if (tid == 0) misc[2] = 0;  // work items of this chunk taken so far (read after the barriers below)
      bucket_chunk<R, kWarps>(cat, rstart, rpre, nr, cpos, cend, pxi, pyi, make_float4(0.f, 0.f, 0.f, 0.f), e2, nullptr,
                              nullptr, BinLookup{}, nb, cbin, wcnt, off, [&](int dst, R ur, R ui, int q) {
                                R vr, vi;
                                cpow5<R>(ur, ui, mb, vr, vi);
                                euv[dst] = Dbl4{ur, ui, vr, vi};
                                ex[dst] = make_double2(cat.xr[q], cat.xi[q]);
                                ew[dst] = cat.w[q];
                              });
      // ---- pass 3: the work items (bin, power block) of the chunk, outer bins (the fuller
      // ones) first, each taken by the next free warp; an item's sums go straight into the
      // record, whose entries no other item of the chunk touches
      const int nitems = nb * nblk;
      int item = 0;
      if (lane == 0) item = atomicAdd(&misc[2], 1);
      item = __shfl_sync(kFull, item, 0);
      while (item < nitems) {
        // the warp's next item is requested now and used at the end of this one
        int next = 0;
        if (lane == 0) next = atomicAdd(&misc[2], 1);
        const int b = nb - 1 - item / nblk, k = item % nblk;
        const int s0 = off[b], s1 = off[b + 1];
        if (s0 < s1) {
          R a[V];
#pragma unroll
          for (int j = 0; j < V; ++j) a[j] = R(0);
          accumulate(a, euv, ex, ew, s0, s1, lane, k, mb);
          // the item's record entries (their current values load while the lanes reduce)
          int f[V / 32];
          R cur[V / 32];
#pragma unroll
          for (int j = 0; j < V / 32; ++j) {
            f[j] = fidx[k * V + rbase + j];
            cur[j] = f[j] >= 0 ? accf[f[j] + 2 * b] : R(0);
          }
          // with R = sum Re(x) u^m = (a0, a1) and I = sum Im(x) u^m = (a2, a3):
          //   sum x u^m = (a0 - a3, a1 + a2),  sum x conj(u^m) = (a0 + a3, a2 - a1)
#pragma unroll
          for (int t = 0; t < kMB; ++t) {
#pragma unroll
            for (int q = 0; q < 8; q += 4) {
              const R r0 = a[14 * t + q], r1 = a[14 * t + q + 1], i0 = a[14 * t + q + 2], i1 = a[14 * t + q + 3];
              a[14 * t + q] = r0 - i1;
              a[14 * t + q + 1] = r1 + i0;
              a[14 * t + q + 2] = r0 + i1;
              a[14 * t + q + 3] = i0 - r1;
            }
          }
          reduce_transpose<R, V>(a, lane);
#pragma unroll
          for (int j = 0; j < V / 32; ++j) {
            if (f[j] >= 0) accf[f[j] + 2 * b] = cur[j] + a[j];
          }
        }
        item = __shfl_sync(kFull, next, 0);
      }
      pairs_here += (unsigned long long)off[nb];
      cpos = cend;
      __syncthreads();
    }
    __syncthreads();
    if (args.accumulate) {
      for (int k = tid; k < L.rec; k += kThreads) dst[k] = cadd(dst[k], accs[k]);
    } else {
      for (int k = tid; k < L.rec; k += kThreads) dst[k] = accs[k];
    }
    if (tid == 0 && !args.accumulate) {
      xw[2 * (size_t)c] = make_double2(args.cen.xr[pi], args.cen.xi[pi]);
      xw[2 * (size_t)c + 1] = make_double2(args.cen.w[pi], 0.0);
    }
    if (tid == 0) {
      atomicAdd(args.pair_count, pairs_here);
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t gather_wave64(const SortedCat& cat, const SortedCat& cen, const Bins& bins, const Layout& L,
                          const WavePlan& plan, bool accumulate, double2* rec, double2* xw,
                          unsigned long long* pair_count, cudaStream_t s) {
  if (plan.total <= 0) return cudaSuccess;
  GatherArgs a;
  a.cat = cat; a.cen = cen; a.accumulate = accumulate ? 1 : 0;
  a.bins = bins; a.L = L; a.plan = plan; a.pair_count = pair_count;
  const int npow = L.max_pow + 1;
  const int nblk = (npow + kMB - 1) / kMB;  // the warps take (bin, block) items in turn
  a.mb = (npow + nblk - 1) / nblk;
  a.nblk = (npow + a.mb - 1) / a.mb;
  constexpr size_t per_pair = sizeof(Dbl4) + sizeof(double2) + sizeof(double) + 1;
  const size_t budget = 227 * 1024;
  // records past the limits of the header are refused: those that did not fit with the tables of
  // three-power blocks
  const int nblk3 = (npow + 2) / 3;
  const size_t common = (size_t)L.rec * sizeof(double2) + 16 + 65 * sizeof(double);
  const size_t refused = common + 130 * sizeof(float) + (65 + kWarps * 64 + 2 * kMaxRows + 1 + 8 +
                                                         (size_t)nblk3 * 64) * sizeof(int) + 256 + 64;
  const size_t fixed = common + (65 + kWarps * 64 + 2 * kMaxRows + 1 + 8 + (size_t)a.nblk * V) * sizeof(int) + 64;
  if (std::max(refused, fixed) + per_pair * kThreads > budget) return cudaErrorInvalidConfiguration;
  int cap = (int)((budget - fixed) / per_pair) / kThreads * kThreads;
  if (cap > 8192) cap = 8192;
  a.cap = cap;
  const size_t smem = fixed + (size_t)cap * per_pair;
  cudaError_t e = allow_smem(gather64_kernel);
  if (e != cudaSuccess) return e;
  gather64_kernel<<<plan.total, kThreads, smem, s>>>(a, rec, xw);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace ext4pcf
