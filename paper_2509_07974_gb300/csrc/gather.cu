// FP32 neighbour gather: for each centre galaxy i of a wave, the spin-weighted multipoles
//   G_n(theta_i, Theta) = sum_j x_j e^{i n phi_ij},   x_j = w_j gamma_c,j
// of its neighbours in every radial bin, plus W_n and the quantities that the
// multiple-counting corrections need (paper Eq. 4PCFUpsilon0 ff., Table tab:4PCFMCCorr).
//
// One CTA (8 warps) per centre:
//   (a) the rows of cells that can hold partners are contiguous ranges of the cell-sorted
//       catalogue (found by one warp, a row per lane); the CTA streams them, keeps pairs
//       with Theta_lo^2 <= r^2 < Theta_hi^2, and buckets them by radial bin into a
//       shared-memory chunk (stable order, so the summation order is deterministic).  Chunks
//       hold up to `cap` candidates; long neighbour lists take several chunks.
//   (b) the work of a chunk is split into items (bin, power block): block k holds the powers
//       m in [k*mb, k*mb+mb) of u = e^{i phi_ij}.  The warps take the items in turn, outer
//       bins first.  For an item each lane walks pairs of the bin, raises u to the block's
//       first power (u^mb is stored per pair) and steps through the block by recurrence in
//       registers, accumulating seven real weights times u^m: Re x, Im x, Re x^2, Im x^2, w,
//       |x|^2, w^2.  The complex sums x u^{+-m} and x^2 u^{+-m} follow from the first four.
//       The 32 lanes' partial sums are combined by a transposed butterfly (each lane ends
//       with V/32 totals) and added to the centre's record in shared memory; no two items
//       of a chunk share a record entry.
//   (c) the triple terms, split over the power blocks in FP32, are summed in block order,
//       and the record is written to the wave buffer (or added to it, for the later passes
//       of the tree approximation).
// Positions are cell-anchored floats (cell offset exact, in-cell offset rounded), so dx is accurate
// to ~1e-7 of the cell size; pairs whose r^2 lies within a few rounding errors of a bin edge are
// re-decided from the double positions.  (gather64.cu: the FP64 form; gather_sector.cu: dense
// catalogues, from where on is said there.)
#include "common.cuh"
#include "gather_common.cuh"

namespace ext4pcf {

namespace {

constexpr int kThreads = 256;
constexpr int kMB = 6;  // powers per block
constexpr int kWarps = kThreads / 32;
constexpr unsigned kFull = 0xFFFFFFFFu;

// Bucketed pairs in shared memory, structure of arrays: uv = (u_re, u_im, v_re, v_im) with
// u = e^{i phi}, v = u^mb; x = w gamma_c; w.  28 bytes per pair in FP32.

// sums of an item (14 per power, 10 triple terms), rounded up to whole lanes
constexpr int V = (14 * kMB + 10 + 31) / 32 * 32;

// u^e for 0 <= e < 32 by binary powering, unrolled (e is uniform across the warp)
__device__ __forceinline__ void cpow5(float br, float bi, int e, float& pr, float& pi) {
  pr = 1.f; pi = 0.f;
#pragma unroll
  for (int bit = 0; bit < 5; ++bit) {
    if (e & (1 << bit)) { float t = pr * br - pi * bi; pi = pr * bi + pi * br; pr = t; }
    if (e >> (bit + 1)) { float t = br * br - bi * bi; bi = 2.f * br * bi; br = t; }
  }
}

// transposed butterfly: after the call lane l holds in a[0..V/32) the warp totals of the
// original slots j + base(l), base(l) = sum_k bit_k(l) * V / 2^(5-k)
template <int W, int OFF>
__device__ __forceinline__ void rt_step(float* a, int lane) {
  constexpr int H = W / 2;
  const bool up = (lane & OFF) != 0;
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const float send = up ? a[j] : a[j + H];
    const float keep = up ? a[j + H] : a[j];
    a[j] = keep + __shfl_xor_sync(kFull, send, OFF);
  }
}
__device__ __forceinline__ void reduce_transpose(float* a, int lane) {
  rt_step<V, 16>(a, lane);
  rt_step<V / 2, 8>(a, lane);
  rt_step<V / 4, 4>(a, lane);
  rt_step<V / 8, 2>(a, lane);
  rt_step<V / 16, 1>(a, lane);
}


// v^k for the block index k (uniform across the warp): the shortest product chain for
// k < 8 as straight-line code behind one uniform branch, binary powering beyond
__device__ __forceinline__ float2 cmul_f(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ void vpow_block(float vr, float vi, int k, float2& P) {
  const float2 v = make_float2(vr, vi);
  switch (k) {
    case 0: P = make_float2(1.f, 0.f); return;
    case 1: P = v; return;
    case 2: P = cmul_f(v, v); return;
    case 3: P = cmul_f(cmul_f(v, v), v); return;
    case 4: { const float2 v2 = cmul_f(v, v); P = cmul_f(v2, v2); return; }
    case 5: { const float2 v2 = cmul_f(v, v); P = cmul_f(cmul_f(v2, v2), v); return; }
    case 6: { const float2 v2 = cmul_f(v, v); P = cmul_f(cmul_f(v2, v2), v2); return; }
    case 7: { const float2 v2 = cmul_f(v, v); P = cmul_f(cmul_f(cmul_f(v2, v2), v2), v); return; }
    default: cpow5(vr, vi, k, P.x, P.y); return;
  }
}

// The sums of one item, one pair per lane and iteration, with packed pairs: every (Re, Im)
// accumulator pair takes one two-lane fused multiply-add per pair of the bin (each lane rounds like
// a scalar FFMA), and the power recurrence u^{m+1} = u^m u runs on the pair (Re, Im) as one packed
// multiply and one packed multiply-add.  Fills a[0, 14 kMB) power by power, then the triple terms.
__device__ __forceinline__ void accumulate(float* a, const float4* __restrict__ euv, const float2* __restrict__ ex,
                                           const float* __restrict__ ew, int s0, int s1, int lane, int k, int mb,
                                           int tr_nsub) {
  constexpr int MB = kMB;
  float2 acc[7 * MB];
#pragma unroll
  for (int j = 0; j < 7 * MB; ++j) acc[j] = make_float2(0.f, 0.f);
  for (int e = s0 + lane; e < s1; e += 32) {
    const float4 q = euv[e];
    const float2 xx = ex[e];
    const float w = ew[e];
    float2 P;
    vpow_block(q.z, q.w, k, P);
    const float2 U = make_float2(q.x, q.y), Us = make_float2(-q.y, q.x);
    const float wt[7] = {xx.x, xx.y, xx.x * xx.x - xx.y * xx.y, 2.f * xx.x * xx.y, w,
                         xx.x * xx.x + xx.y * xx.y, w * w};
    auto step = [&](int t) {
#pragma unroll
      for (int qq = 0; qq < 7; ++qq) acc[7 * t + qq] = __ffma2_rn(make_float2(wt[qq], wt[qq]), P, acc[7 * t + qq]);
      P = __ffma2_rn(make_float2(P.x, P.x), U, __fmul2_rn(make_float2(P.y, P.y), Us));
    };
    if (mb == MB) {
#pragma unroll
      for (int t = 0; t < MB; ++t) step(t);
    } else {
#pragma unroll
      for (int t = 0; t < MB; ++t)
        if (t < mb) step(t);
    }
  }
#pragma unroll
  for (int j = 0; j < 7 * MB; ++j) { a[2 * j] = acc[j].x; a[2 * j + 1] = acc[j].y; }
  // x^3 u^-8, x^3 u^-4, x^2 x^* u^-4, x^2 x^*, w^3: a pass of its own (so that these sums
  // hold no registers in the power loop), shared by the tr_nsub power blocks of the bin:
  // block k takes the 32-pair groups k, k + tr_nsub, ...  The caller adds the blocks'
  // partial sums in a fixed order.
  float tr[10];
#pragma unroll
  for (int j = 0; j < 10; ++j) tr[j] = 0.f;
  {
    for (int e = s0 + lane + 32 * k; e < s1; e += 32 * tr_nsub) {
      const float4 q = euv[e];
      const float2 xx = ex[e];
      const float w = ew[e];
      const float ur = q.x, ui = q.y, xr = xx.x, xi = xx.y;
      const float x2r = xr * xr - xi * xi, x2i = 2.f * xr * xi, xa = xr * xr + xi * xi;
      float u2r = ur * ur - ui * ui, u2i = 2.f * ur * ui;
      float u4r = u2r * u2r - u2i * u2i, u4i = 2.f * u2r * u2i;
      float u8r = u4r * u4r - u4i * u4i, u8i = 2.f * u4r * u4i;
      float x3r = x2r * xr - x2i * xi, x3i = x2r * xi + x2i * xr;
      float xcr = xa * xr, xci = xa * xi;  // x^2 x^* = |x|^2 x
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
#pragma unroll
  for (int j = 0; j < 10; ++j) a[14 * MB + j] = tr[j];
}

// two CTAs of 8 warps per SM: 6 powers per block keep the accumulators within 128 registers, and
// each CTA gets half of the shared memory
__global__ void __launch_bounds__(kThreads, 2)
gather_kernel(const GatherArgs args, float2* __restrict__ rec, float2* __restrict__ xw) {
  extern __shared__ __align__(16) unsigned char smem[];
  const SortedCat& cat = args.cat;
  const Layout L = args.L;
  const int nb = args.bins.nb, cap = args.cap, mb = args.mb, nblk = args.nblk;
  // Nothing for a block past a masked wave's centres, nor for one of a dense catalogue, which is
  // gather_sector's.  (A block per centre all the same: the hardware's order balances them better than
  // strides over fewer blocks, 7.6 against 7.8 ms for 24001 centres.)
  {
    int j = 0;
    const int si = seg_of(args.plan, blockIdx.x, &j);
    if (si < 0 || j >= seg_live(args.plan.seg[si])) return;
    if (args.dense_min > 0.f && mean_candidates(args.plan.seg[si], (float)args.bins.rmax) >= args.dense_min) return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  float4* euv = reinterpret_cast<float4*>(smem);
  float2* ex = reinterpret_cast<float2*>(euv + cap);
  float* ew = reinterpret_cast<float*>(ex + cap);
  double* e2 = reinterpret_cast<double*>(ew + cap);
  float* e2f = reinterpret_cast<float*>(e2 + 65);
  float* win = e2f + 65;
  int* off = reinterpret_cast<int*>(win + 65);  // [65] bin offsets of the chunk
  int* wcnt = off + 65;                          // [warps][64] per-warp bin counts / positions
  int* rstart = wcnt + kWarps * 64;
  int* rpre = rstart + kMaxRows;
  int* misc = rpre + kMaxRows + 1;  // rows, candidates, work items taken
  int* fidx = misc + 8;             // [nblk][V] where the reduced slots of each power block go
  // partial sums of the split triple terms: trs [nb][nblk][10]
  float* trs = reinterpret_cast<float*>(fidx + nblk * V);
  unsigned char* btab = reinterpret_cast<unsigned char*>(trs + nb * nblk * 10);  // [256]
  signed char* cbin = reinterpret_cast<signed char*>(btab + 256);  // bin of each candidate
  float2* accs = reinterpret_cast<float2*>((reinterpret_cast<uintptr_t>(cbin + cap) + 15) & ~(uintptr_t)15);

  for (int b = tid; b <= nb; b += kThreads) {
    e2[b] = args.bins.e2[b]; e2f[b] = args.bins.e2f[b];
  }
  for (int k = tid; k < kWarps * 64; k += kThreads) wcnt[k] = 0;
  // the lookup table of the FP32 bin decision
  BinLookup lk;
  lk.tab = btab;
  lk.base = __float_as_uint(args.bins.e2f[0]);
  lk.shift = 0;
  while (((__float_as_uint(args.bins.e2f[nb]) - lk.base) >> lk.shift) >= 256u) ++lk.shift;
  lk.out_lo = lk.out_hi = 0.f;  // set per chunk from the rounding windows
  for (int i = tid; i < 256; i += kThreads) {
    const float v = __uint_as_float(lk.base + ((unsigned)i << lk.shift));
    int b = 0;
    while (b + 1 < nb && args.bins.e2f[b + 1] <= v) ++b;
    btab[i] = (unsigned char)b;
  }
  // Reduced slot s of power block k (slot order of the accumulation: 14 per power, then the
  // 10 triple terms) goes to the record's float index fidx[k][s] + 2b for bin b (every array
  // of the record is [multipole][bin]); <= -2: triple-term slot -2 - fidx of trs; -1: nowhere
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
      f = -2 - (slot - 14 * kMB);
    }
    fidx[i] = f;
  }
  // the reduced slots this lane holds after the transposed butterfly: base + [0, V/32)
  const int rbase = (lane & 16 ? V / 2 : 0) + (lane & 8 ? V / 4 : 0) + (lane & 4 ? V / 8 : 0) +
                    (lane & 2 ? V / 16 : 0) + (lane & 1 ? V / 32 : 0);
  const double rmax = args.bins.rmax * (1.0 + 1e-9) + 1e-12;
  double cell_w = -1.0;  // cell side the rounding windows were computed for

  for (int c = blockIdx.x; c < args.plan.total; c += gridDim.x) {
    // the record's segment: its catalogue's grid and centre (padding records are skipped)
    int j = 0;
    const int si = seg_of(args.plan, c, &j);
    if (si < 0 || j >= seg_live(args.plan.seg[si])) continue;  // uniform over the block
    const WaveSeg& sg = args.plan.seg[si];
    const GridGeom gm = *sg.geom;
    const double gx0 = gm.x0, gy0 = gm.y0, cell = gm.cell;
    const int gncx = gm.ncx, gncy = gm.ncy;
    if (cell != cell_w) {
      __syncthreads();
      for (int b = tid; b <= nb; b += kThreads) {
        // rounding window of the float bin decision: |dx| carries ~2 ulp of max(cell, r)
        const double e = sqrt(args.bins.e2[b]);
        const double err = 4.0 * 1.2e-7 * (cell + e);
        win[b] = (float)(2.0 * e * err + err * err);
      }
      cell_w = cell;
    }
    const int pi = sg.centres[sg.w0 + j];
    const double pxi = args.cen.px[pi], pyi = args.cen.py[pi];
    // the centre in the neighbours' grid frame: cell corner and offset as float, by the
    // arithmetic that builds the neighbours' (cell corner, offset) pairs
    const int ccx = min(max((int)floor((pxi - gx0) * gm.inv_cell), 0), gncx - 1);
    const int ccy = min(max((int)floor((pyi - gy0) * gm.inv_cell), 0), gncy - 1);
    const float4 Pi = make_float4((float)ccx * gm.cellf, (float)ccy * gm.cellf,
                                  (float)((pxi - gx0) - (double)ccx * cell), (float)((pyi - gy0) - (double)ccy * cell));
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
    float2* dst = rec + (size_t)c * L.rec;
    float* accf = reinterpret_cast<float*>(accs);
    for (int k = tid; k < L.rec; k += kThreads) accs[k] = make_float2(0.f, 0.f);
    for (int i = tid; i < nb * nblk * 10; i += kThreads) trs[i] = 0.f;
    __syncthreads();
    const int nr = misc[0], total = misc[1];
    unsigned long long pairs_here = 0;

    for (int cpos = 0; cpos < total;) {
      // ---- classification and stable bucketing by bin of the next cap candidates
      const int cend = min(total, cpos + cap);
      if (tid == 0) misc[2] = 0;  // work items of this chunk taken so far (read after the barriers below)
      bucket_chunk<float, kWarps>(cat, rstart, rpre, nr, cpos, cend, pxi, pyi, Pi, e2, e2f, win, lk, nb, cbin, wcnt,
                                  off, [&](int dst, float ur, float ui, int q) {
                                    float xr, xi, ww, vr, vi;
                                    Pair<float>::load_x(cat, q, xr, xi, ww);
                                    cpow5(ur, ui, mb, vr, vi);
                                    euv[dst] = make_float4(ur, ui, vr, vi);
                                    ex[dst] = make_float2(xr, xi);
                                    ew[dst] = ww;
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
          float a[V];
#pragma unroll
          for (int j = 0; j < V; ++j) a[j] = 0.f;
          accumulate(a, euv, ex, ew, s0, s1, lane, k, mb, nblk);
          // the item's record entries (their current values load while the lanes reduce)
          int f[V / 32];
          float cur[V / 32];
#pragma unroll
          for (int j = 0; j < V / 32; ++j) {
            f[j] = fidx[k * V + rbase + j];
            cur[j] = f[j] >= 0 ? accf[f[j] + 2 * b] : 0.f;
          }
          // with R = sum Re(x) u^m = (a0, a1) and I = sum Im(x) u^m = (a2, a3):
          //   sum x u^m = (a0 - a3, a1 + a2),  sum x conj(u^m) = (a0 + a3, a2 - a1)
#pragma unroll
          for (int t = 0; t < kMB; ++t) {
#pragma unroll
            for (int q = 0; q < 8; q += 4) {
              const float r0 = a[14 * t + q], r1 = a[14 * t + q + 1], i0 = a[14 * t + q + 2], i1 = a[14 * t + q + 3];
              a[14 * t + q] = r0 - i1;
              a[14 * t + q + 1] = r1 + i0;
              a[14 * t + q + 2] = r0 + i1;
              a[14 * t + q + 3] = i0 - r1;
            }
          }
          reduce_transpose(a, lane);
#pragma unroll
          for (int j = 0; j < V / 32; ++j) {
            if (f[j] >= 0) accf[f[j] + 2 * b] = cur[j] + a[j];
            else if (f[j] <= -2) trs[(b * nblk + k) * 10 + (-2 - f[j])] += a[j];
          }
        }
        item = __shfl_sync(kFull, next, 0);
      }
      pairs_here += (unsigned long long)off[nb];
      cpos = cend;
      __syncthreads();
    }
    // triple terms: the power blocks' sums, in block order
    for (int i = tid; i < nb * 10; i += kThreads) {
      const int b = i / 10, q = i % 10;
      float sum = 0.f;
      for (int k = 0; k < nblk; ++k) sum += trs[(b * nblk + k) * 10 + q];
      accf[2 * L.TR(q >> 1, b) + (q & 1)] += sum;
    }
    __syncthreads();
    if (args.accumulate) {
      for (int k = tid; k < L.rec; k += kThreads) dst[k] = cadd(dst[k], accs[k]);
    } else {
      for (int k = tid; k < L.rec; k += kThreads) dst[k] = accs[k];
    }
    if (tid == 0 && !args.accumulate) {
      float xr, xi, ww;
      Pair<float>::load_x(args.cen, pi, xr, xi, ww);
      xw[2 * (size_t)c] = make_float2(xr, xi);
      xw[2 * (size_t)c + 1] = make_float2(ww, 0.f);
    }
    if (tid == 0) {
      atomicAdd(args.pair_count, pairs_here);
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t gather_wave32(const SortedCat& cat, const SortedCat& cen, const Bins& bins, const Layout& L,
                          const WavePlan& plan, bool accumulate, float2* rec, float2* xw,
                          unsigned long long* pair_count, cudaStream_t s) {
  if (plan.total <= 0) return cudaSuccess;
  GatherArgs a;
  a.cat = cat; a.cen = cen; a.accumulate = accumulate ? 1 : 0;
  a.bins = bins; a.L = L; a.plan = plan; a.pair_count = pair_count;
  const int npow = L.max_pow + 1;
  const int nblk = (npow + kMB - 1) / kMB;  // the warps take (bin, block) items in turn
  a.mb = (npow + nblk - 1) / nblk;
  a.nblk = (npow + a.mb - 1) / a.mb;
  const size_t fixed = (size_t)L.rec * sizeof(float2) + 16 + 65 * sizeof(double) + 130 * sizeof(float) +
                       (65 + kWarps * 64 + 2 * kMaxRows + 1 + 8 + (size_t)a.nblk * V) * sizeof(int) + 256 +
                       64 + (size_t)bins.nb * a.nblk * 10 * sizeof(float);
  const size_t budget = 113 * 1024;
  constexpr size_t per_pair = sizeof(float4) + sizeof(float2) + sizeof(float) + 1;
  if (fixed + per_pair * kThreads > budget) return cudaErrorInvalidConfiguration;
  int cap = (int)((budget - fixed) / per_pair) / kThreads * kThreads;
  if (cap > 8192) cap = 8192;
  a.cap = cap;
  const size_t smem = fixed + (size_t)cap * per_pair;
  cudaError_t e = allow_smem(gather_kernel);
  if (e != cudaSuccess) return e;
  a.dense_min = 0.f;
  e = gather_sector(cat, cen, bins, L, plan, accumulate, a.mb, a.nblk, rec, xw, pair_count, s, &a.dense_min);
  if (e != cudaSuccess) return e;
  gather_kernel<<<plan.total, kThreads, smem, s>>>(a, rec, xw);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace ext4pcf
