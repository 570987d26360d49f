// FP32 neighbour gather of dense catalogues: the records of gather.cu, from angular sectors.
//
// A sum over a bin's pairs of weights times u^n, u = e^{i phi}, costs 14 multiply-adds a pair and
// power when it is taken power by power.  With the circle cut into 64 sectors about the angles
// phi_c and phi = phi_c + delta (Jacobi-Anger, t = delta / delta_max in [-1, 1]),
//   e^{i n phi} = e^{i n phi_c} [J_0(n delta_max) + 2 sum_{k>0} i^k J_k(n delta_max) T_k(t)],
// the pairs only enter through the moments sum weight T_k(t), k < K, of each sector: 7 K real
// multiply-adds a pair.  The 64-point transform over the sectors and the sum over k are done once
// per centre and bin.  K = 12 keeps every power <= 46 to 3e-8, K = 16 every power <= 86.
//
// One CTA (12 warps of 168 registers, one CTA per SM: the moments take a third of its shared memory)
// takes centres in turn:
//   (a) rows of cells as in gather.cu (found by one warp while the others finish the centre before);
//       3840 candidates at a time are classified, five groups of a warp at once, and bucketed by (bin,
//       sector) in a stable order, so the summation order is deterministic;
//   (b) items (bin, eight of its sectors): four lanes per sector walk its pairs, 7 K + 9 sums in
//       registers, which are then added to the bin's moments in shared memory.  At most four bins, the
//       widest, have sectors; the pairs of the others, few, are set aside and summed power by power;
//   (c) at the end the moments become the record's entries, in place.
// Measured: 8192 centres with 28000 candidates each, n_max = 20, 11.1 -> 8.0 ms; 256 centres of four
// patches, n_max = 30, three passes of the tree approximation, 7.6 -> 3.6 ms.  The records' error
// against 64 bits stays (7.1e-8 -> 6.9e-8 of the largest; 100000 galaxies, 7 bins, n_max = 15).  No
// unit is saturated: with three warps to a scheduler the latencies of (a), the unequal sectors
// of (b) and the barriers between them are what is left.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "gather_common.cuh"

namespace ext4pcf {

namespace {

constexpr int kThreads = 384;
constexpr int kWarps = kThreads / 32;
constexpr int kG = 10;                 // candidates per lane and chunk
constexpr int kCap = kThreads * kG;    // candidates per chunk
constexpr int kDefer = 1024;           // pairs of the bins without sectors kept over the chunks
constexpr int kSec = 64;               // sectors
constexpr int kSlots = 4;              // bins with sectors, at most
constexpr int kKeys = kSlots * kSec + 32;
constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kMB = 6;                 // powers per block of the bins without sectors
constexpr int V = (14 * kMB + 10 + 31) / 32 * 32;
static_assert(kKeys <= kThreads, "one thread per bucket");
// |delta| <= half a sector and the error of the sector's choice (0.0015)
constexpr double kDeltaMax = 3.14159265358979323846 / kSec * 1.035;

struct SectorArgs {
  GatherArgs g;
  int slots;        // bins with sectors that fit
  float share[32];  // part of the candidates that a bin expects
  float coef[87 * 16];  // [power][K]: J_0, 2 J_k of power * kDeltaMax
};

// the sector of (dx, dy): the arctangent to 0.0015 (Rajan et al. 2006), in units of a sector
__device__ __forceinline__ int sector_of(float dx, float dy) {
  const float ax = fabsf(dx), ay = fabsf(dy);
  const float a = __fdividef(fminf(ax, ay), fmaxf(ax, ay));
  float f = a * (8.f + (1.f - a) * (2.492494f + 0.675326f * a));
  if (ay > ax) f = 16.f - f;
  if (dx < 0.f) f = 32.f - f;
  if (dy < 0.f) f = -f;
  return __float2int_rn(f) & (kSec - 1);
}

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// rows of a bin's moments: 7 k + weight, then nine triple sums (x^3 e^{-8 i delta}, x^3 e^{-4 i delta},
// x |x|^2 e^{-4 i delta}, x |x|^2, w^3) and three empty ones
template <int K>
constexpr int kMomRows = 7 * K + 12;

// column of sector c in row r of the moments: the rows that a warp adds to at once on different banks
__device__ __forceinline__ int mom_col(int c, int r) { return (c + 16 * (r & 1) + 8 * (r >> 1 & 1)) & (kSec - 1); }

// Moments of one (bin, eight sectors): four lanes to a sector, each every fourth of its pairs.  U_k = T_k
// (-1)^{k/2} obeys U_{k+1} = -+ 2 t U_k + U_{k-1} (no subtraction, which the packed multiply-add
// lacks; the signs cancel those of i^k in the transform); both halves of a packed pair hold the same
// U_k.  Also the triple sums, with e^{-4 i delta} from its series.
template <int K>
__device__ __forceinline__ void sector_item(const float4* __restrict__ pairs, const int* __restrict__ koff, int key0,
                                            int part, int lane, float* __restrict__ mom) {
  const int sec = 8 * part + (lane & 7), sub = lane >> 3;
  const int e1 = koff[key0 + sec + 1];
  float2 ax[K], aq[K], aw[K];
  float aww[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    ax[k] = aq[k] = aw[k] = make_float2(0.f, 0.f);
    aww[k] = 0.f;
  }
  float tr[9];
#pragma unroll
  for (int j = 0; j < 9; ++j) tr[j] = 0.f;
  for (int e = koff[key0 + sec] + sub; e < e1; e += 4) {
    const float4 p = pairs[e];
    const float t = p.x, xr = p.y, xi = p.z, w = p.w;
    const float2 X = make_float2(xr, xi);
    const float2 Q = make_float2(xr * xr - xi * xi, 2.f * xr * xi);
    const float xa = xr * xr + xi * xi, ww = w * w;
    const float2 Wa = make_float2(w, xa);
    const float2 cp = make_float2(2.f * t, 2.f * t), cn = make_float2(-2.f * t, -2.f * t);
    float2 a = make_float2(1.f, 1.f), b = make_float2(t, t);
    ax[0] = __fadd2_rn(ax[0], X);
    aq[0] = __fadd2_rn(aq[0], Q);
    aw[0] = __fadd2_rn(aw[0], Wa);
    aww[0] += ww;
#pragma unroll
    for (int k = 1; k < K; ++k) {
      ax[k] = __ffma2_rn(X, b, ax[k]);
      aq[k] = __ffma2_rn(Q, b, aq[k]);
      aw[k] = __ffma2_rn(Wa, b, aw[k]);
      aww[k] += ww * b.x;
      const float2 n = __ffma2_rn(k & 1 ? cn : cp, b, a);
      a = b;
      b = n;
    }
    const float y = (float)(4.0 * kDeltaMax) * t, y2 = y * y;
    const float s4 = y * (1.f + y2 * (-1.f / 6.f + y2 * (1.f / 120.f)));
    const float c4 = 1.f + y2 * (-0.5f + y2 * (1.f / 24.f - y2 * (1.f / 720.f)));
    // x e^{-4 i delta}, times x^2, times e^{-4 i delta} again
    const float br = xr * c4 + xi * s4, bi = xi * c4 - xr * s4;
    const float cr = Q.x * br - Q.y * bi, ci = Q.x * bi + Q.y * br;
    tr[0] += cr * c4 + ci * s4;
    tr[1] += ci * c4 - cr * s4;
    tr[2] += cr;
    tr[3] += ci;
    tr[4] += xa * br;
    tr[5] += xa * bi;
    tr[6] += xa * xr;
    tr[7] += xa * xi;
    tr[8] += ww * w;
  }
  __syncwarp();
  // the four lanes of a sector: of the rows the lower half of the warp takes the even ones, the upper
  // half the odd ones, and the halves' halves again
  float r[kMomRows<K>];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    r[7 * k] = ax[k].x; r[7 * k + 1] = ax[k].y; r[7 * k + 2] = aq[k].x; r[7 * k + 3] = aq[k].y;
    r[7 * k + 4] = aw[k].x; r[7 * k + 5] = aw[k].y; r[7 * k + 6] = aww[k];
  }
#pragma unroll
  for (int j = 0; j < 12; ++j) r[7 * K + j] = j < 9 ? tr[j] : 0.f;
  const int up = lane >> 4;
#pragma unroll
  for (int j = 0; j < kMomRows<K>; j += 2) {
    const float send = up ? r[j] : r[j + 1];
    const float keep = up ? r[j + 1] : r[j];
    r[j / 2] = keep + __shfl_xor_sync(kFull, send, 16);
  }
  const int up2 = lane >> 3 & 1;
#pragma unroll
  for (int j = 0; j < kMomRows<K> / 2; j += 2) {
    const float send = up2 ? r[j] : r[j + 1];
    const float keep = up2 ? r[j + 1] : r[j];
    r[j / 2] = keep + __shfl_xor_sync(kFull, send, 8);
  }
  const int row = 2 * up2 + up;
#pragma unroll
  for (int j = 0; j < kMomRows<K> / 4; ++j) mom[(4 * j + row) * kSec + mom_col(sec, row)] += r[j];
}

template <int W, int OFF>
__device__ __forceinline__ void fold(float* a, int lane) {
  const bool up = (lane & OFF) != 0;
#pragma unroll
  for (int j = 0; j < W / 2; ++j) {
    const float send = up ? a[j] : a[j + W / 2];
    const float keep = up ? a[j + W / 2] : a[j];
    a[j] = keep + __shfl_xor_sync(kFull, send, OFF);
  }
}

// One (bin, block of powers) without sectors: pairs (u, catalogue position), as in gather.cu.
__device__ __forceinline__ void direct_item(const SortedCat& cat, const float4* __restrict__ pairs, int s0, int s1,
                                            int lane, int k, int mb, int nblk, int b, const int* __restrict__ fidx,
                                            float* __restrict__ accf, float* __restrict__ tr_out) {
  float2 acc[7 * kMB];
#pragma unroll
  for (int j = 0; j < 7 * kMB; ++j) acc[j] = make_float2(0.f, 0.f);
  float tr[9];
#pragma unroll
  for (int j = 0; j < 9; ++j) tr[j] = 0.f;
  for (int e = s0 + lane, g = 0; e < s1; e += 32, ++g) {
    const float4 p = pairs[e];
    const float4 sh = cat.s4[__float_as_int(p.z)];
    const float xr = sh.x, xi = sh.y, w = sh.z;
    const float2 U = make_float2(p.x, p.y), Us = make_float2(-p.y, p.x);
    float2 P = make_float2(1.f, 0.f), B = U;
    for (int n = k * mb; n > 0; n >>= 1) {  // u^{k mb}, uniform across the warp
      if (n & 1) P = cmulf(P, B);
      B = cmulf(B, B);
    }
    const float x2r = xr * xr - xi * xi, x2i = 2.f * xr * xi, xa = xr * xr + xi * xi;
    const float wt[7] = {xr, xi, x2r, x2i, w, xa, w * w};
#pragma unroll
    for (int t = 0; t < kMB; ++t) {
      if (t < mb) {
#pragma unroll
        for (int q = 0; q < 7; ++q) acc[7 * t + q] = __ffma2_rn(make_float2(wt[q], wt[q]), P, acc[7 * t + q]);
        P = __ffma2_rn(make_float2(P.x, P.x), U, __fmul2_rn(make_float2(P.y, P.y), Us));
      }
    }
    if (g % nblk == k) {  // the triple sums, split over the power blocks
      const float2 u2 = cmulf(U, U), u4 = cmulf(u2, u2), u8 = cmulf(u4, u4);
      const float x3r = x2r * xr - x2i * xi, x3i = x2r * xi + x2i * xr, cr = xa * xr, ci = xa * xi;
      tr[0] += x3r * u8.x + x3i * u8.y;
      tr[1] += x3i * u8.x - x3r * u8.y;
      tr[2] += x3r * u4.x + x3i * u4.y;
      tr[3] += x3i * u4.x - x3r * u4.y;
      tr[4] += cr * u4.x + ci * u4.y;
      tr[5] += ci * u4.x - cr * u4.y;
      tr[6] += cr;
      tr[7] += ci;
      tr[8] += (w * w) * w;
    }
  }
  __syncwarp();
  float a[V];
#pragma unroll
  for (int j = 0; j < V; ++j) a[j] = 0.f;
#pragma unroll
  for (int t = 0; t < kMB; ++t) {
#pragma unroll
    for (int q = 0; q < 4; q += 2) {  // x and x^2: sums with u^m and with its conjugate
      const float2 R = acc[7 * t + q], I = acc[7 * t + q + 1];
      a[14 * t + 2 * q] = R.x - I.y;
      a[14 * t + 2 * q + 1] = R.y + I.x;
      a[14 * t + 2 * q + 2] = R.x + I.y;
      a[14 * t + 2 * q + 3] = I.x - R.y;
    }
#pragma unroll
    for (int q = 4; q < 7; ++q) {
      a[14 * t + 2 * q] = acc[7 * t + q].x;
      a[14 * t + 2 * q + 1] = acc[7 * t + q].y;
    }
  }
#pragma unroll
  for (int j = 0; j < 9; ++j) a[14 * kMB + j] = tr[j];
  // transposed butterfly: lane l ends with slots base(l) + [0, V / 32)
  fold<V, 16>(a, lane);
  fold<V / 2, 8>(a, lane);
  fold<V / 4, 4>(a, lane);
  fold<V / 8, 2>(a, lane);
  fold<V / 16, 1>(a, lane);
  const int base = (lane & 16 ? V / 2 : 0) + (lane & 8 ? V / 4 : 0) + (lane & 4 ? V / 8 : 0) +
                   (lane & 2 ? V / 16 : 0) + (lane & 1 ? V / 32 : 0);
#pragma unroll
  for (int j = 0; j < V / 32; ++j) {
    const int f = fidx[k * V + base + j];
    if (f >= 0) accf[f + 2 * b] += a[j];
    else if (f <= -2) tr_out[-2 - f] += a[j];
  }
}

// The moments of one bin -> F_k(n) = sum_c e^{i n phi_c} moment_k(c), n = 0..32, in place: row r becomes
// (Re F(0), F(32), Re F(1), Im F(1), ...).  Lane n takes power n; even and odd n, and c against -c, are
// folded first, so an output is 17 multiply-adds.  Four rows at a time, the folded values through a
// small scratch of the warp.
__device__ __forceinline__ void sector_rows(float* __restrict__ m, int row, float4* __restrict__ scr, int lane,
                                            const float* cs, const float* sn) {
  float pe[4], qe[4], po[4], qo[4];
  const bool self = lane == 0 || lane == 16;
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const float x0 = m[h * kSec + mom_col(lane, row + h)];
    const float x1 = m[h * kSec + mom_col(lane + 32, row + h)];
    const float e = x0 + x1, o = x0 - x1;
    const float eP = __shfl_sync(kFull, e, (32 - lane) & 31), oP = __shfl_sync(kFull, o, (32 - lane) & 31);
    pe[h] = self ? e : e + eP;
    qe[h] = self ? 0.f : e - eP;
    po[h] = lane == 0 ? o : lane == 16 ? 0.f : o - oP;
    qo[h] = lane == 0 ? 0.f : lane == 16 ? o : o + oP;
  }
  if (lane <= 16) {
    scr[4 * lane] = make_float4(pe[0], pe[1], pe[2], pe[3]);
    scr[4 * lane + 1] = make_float4(po[0], po[1], po[2], po[3]);
    scr[4 * lane + 2] = make_float4(qe[0], qe[1], qe[2], qe[3]);
    scr[4 * lane + 3] = make_float4(qo[0], qo[1], qo[2], qo[3]);
  }
  __syncwarp();
  float2 out[4];
#pragma unroll
  for (int h = 0; h < 4; ++h) out[h] = make_float2(0.f, 0.f);
  const int qi = lane == 0 ? 0 : 2 + (lane & 1);  // lane 0: F(32) from the even sums
#pragma unroll
  for (int c = 0; c <= 16; ++c) {
    const float4 f = scr[4 * c + (lane & 1)], g = scr[4 * c + qi];
    out[0].x += f.x * cs[c]; out[0].y += g.x * sn[c];
    out[1].x += f.y * cs[c]; out[1].y += g.y * sn[c];
    out[2].x += f.z * cs[c]; out[2].y += g.z * sn[c];
    out[3].x += f.w * cs[c]; out[3].y += g.w * sn[c];
  }
#pragma unroll
  for (int h = 0; h < 4; ++h) reinterpret_cast<float2*>(m + h * kSec)[lane] = out[h];
  __syncwarp();
}

template <int K>
__global__ void __launch_bounds__(kThreads, 1)
gather_sector_kernel(const __grid_constant__ SectorArgs args, float2* __restrict__ rec, float2* __restrict__ xw) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int kRows = kMomRows<K>;
  const GatherArgs& ga = args.g;
  const SortedCat& cat = ga.cat;
  const Layout L = ga.L;
  const int nb = ga.bins.nb, mb = ga.mb, nblk = ga.nblk;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;

  float4* pairs = reinterpret_cast<float4*>(smem);                     // [kCap]
  float* mom = reinterpret_cast<float*>(pairs + kCap);                 // [slots][kRows][kSec]
  float* accf = mom + (size_t)args.slots * kRows * kSec;               // the record
  float4* cpos4 = reinterpret_cast<float4*>(accf + 2 * ((L.rec + 1) & ~1));  // the centre: in its cell,
  double* cxy = reinterpret_cast<double*>(cpos4 + 1);                  // [2] and in double
  double* e2 = cxy + 2;                                                // [65]
  float4* uc = reinterpret_cast<float4*>(e2 + 66);                     // [kSec] e^{i phi_c}, and what its
                                                                       // rounding left
  float* e2f = reinterpret_cast<float*>(uc + kSec);                   // [65]
  float* win = e2f + 65;                                               // [65]
  float2* safe = reinterpret_cast<float2*>(win + 65);                  // [32] bins less their rounding windows
  float* trs = reinterpret_cast<float*>(safe + 32);                    // [nb][nblk][10]
  float* coef = trs + nb * nblk * 10;                                   // [max_pow + 1][K]
  int* fidx = reinterpret_cast<int*>(coef + (L.max_pow + 1) * K);      // [nblk][V]
  int* rstart = fidx + nblk * V;
  int* rpre = rstart + kMaxRows;
  int* misc = rpre + kMaxRows + 1;  // rows, candidates, bins with sectors (count, mask), items taken
  int* kb = misc + 8;               // [32] first bucket of each bin
  int* orders = kb + 32;            // [2][32] (in turns) the bins with sectors, then those without, outer first
  int* wsum = orders + 64;          // [kWarps]
  int* koff = wsum + kWarps;        // [kKeys + 1]
  int* defer = koff + kKeys + 1;    // [kDefer]
  unsigned short* cnt = reinterpret_cast<unsigned short*>(defer + kDefer);  // [kWarps][kKeys]
  unsigned char* btab = reinterpret_cast<unsigned char*>(cnt + kWarps * kKeys);  // [256]

  // ---- nothing to do unless one of the block's centres is in a dense catalogue
  auto mine = [&](int c) {
    int j = 0;
    const int si = seg_of(ga.plan, c, &j);
    return si >= 0 && j < seg_live(ga.plan.seg[si]) &&
           mean_candidates(ga.plan.seg[si], (float)ga.bins.rmax) >= ga.dense_min;
  };
  int c = blockIdx.x;
  while (c < ga.plan.total && !mine(c)) c += gridDim.x;
  if (c >= ga.plan.total) return;

  for (int b = tid; b <= nb; b += kThreads) { e2[b] = ga.bins.e2[b]; e2f[b] = ga.bins.e2f[b]; }
  BinLookup lk;
  lk.tab = btab;
  lk.base = __float_as_uint(ga.bins.e2f[0]);
  lk.shift = 0;
  while (((__float_as_uint(ga.bins.e2f[nb]) - lk.base) >> lk.shift) >= 256u) ++lk.shift;
  for (int i = tid; i < 256; i += kThreads) {
    const float v = __uint_as_float(lk.base + ((unsigned)i << lk.shift));
    int b = 0;
    while (b + 1 < nb && ga.bins.e2f[b + 1] <= v) ++b;
    btab[i] = (unsigned char)b;
  }
  for (int i = tid; i < kSec; i += kThreads) {
    double sn, cs;
    sincospi(i * (2.0 / kSec), &sn, &cs);
    uc[i] = make_float4((float)cs, (float)sn, (float)(cs - (double)(float)cs), (float)(sn - (double)(float)sn));
  }
  for (int i = tid; i < (L.max_pow + 1) * K; i += kThreads) coef[i] = args.coef[i];
  for (int i = tid; i < nblk * V; i += kThreads) {  // as in gather.cu
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
    } else if (slot < 14 * kMB + 9) {
      f = -2 - (slot - 14 * kMB);
    }
    fidx[i] = f;
  }
  for (int i = tid; i < kWarps * kKeys; i += kThreads) cnt[i] = 0;
  const double rmax = ga.bins.rmax * (1.0 + 1e-9) + 1e-12;
  double cell_w = -1.0;  // cell side the rounding windows were computed for

  // warp 0: the centre in the neighbours' grid frame (gather.cu), the rows of cells within rmax of it
  // and the bins that get sectors
  auto find_rows = [&](int c, int flip) {
    int j = 0;
    const WaveSeg& sg = ga.plan.seg[seg_of(ga.plan, c, &j)];
    const GridGeom gm = *sg.geom;
    const double gx0 = gm.x0, gy0 = gm.y0, cell = gm.cell;
    const int gncx = gm.ncx, gncy = gm.ncy;
    const int pi = sg.centres[sg.w0 + j];
    int* order = orders + 32 * flip;
    const double pxi = ga.cen.px[pi], pyi = ga.cen.py[pi];
    if (lane == 0) {
      const int ccx = min(max((int)floor((pxi - gx0) * gm.inv_cell), 0), gncx - 1);
      const int ccy = min(max((int)floor((pyi - gy0) * gm.inv_cell), 0), gncy - 1);
      *cpos4 = make_float4((float)ccx * gm.cellf, (float)ccy * gm.cellf, (float)((pxi - gx0) - (double)ccx * cell),
                           (float)((pyi - gy0) - (double)ccy * cell));
      cxy[0] = pxi;
      cxy[1] = pyi;
    }
    // the rows of cells within rmax of the centre (gather.cu)
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
      const int pos = nr + __popc(ok & lt);
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
    // bins with sectors: those that expect at least 256 pairs, the outer ones first
    const bool want = lane < nb && tot * args.share[lane] >= 256.f;
    const unsigned wanted = __ballot_sync(kFull, want);
    const bool big = want && __popc(wanted >> lane) <= args.slots;
    const unsigned bigs = __ballot_sync(kFull, big);
    // buckets: bin by bin for those with sectors, after one bucket of all the others; the others'
    // own when it is their turn
    const unsigned rest = ~bigs & (nb < 32 ? (1u << nb) - 1u : kFull);
    if (lane < nb) {
      order[big ? __popc(bigs >> lane) - 1 : __popc(bigs) + __popc(rest >> lane) - 1] = lane;
      kb[lane] = big ? 1 + kSec * (__popc(bigs >> lane) - 1) : __popc(rest >> lane) - 1;
    }
    if (lane == 0) {
      rpre[nr] = tot;
      misc[0] = nr; misc[1] = tot; misc[2] = __popc(bigs); misc[3] = (int)bigs;
    }
  };
  auto next_mine = [&](int c) {
    while (c < ga.plan.total && !mine(c)) c += gridDim.x;
    return c;
  };
  const int first = c;
  int flip = 0;
  for (int cn; c < ga.plan.total; c = cn, flip ^= 1) {
    cn = next_mine(c + gridDim.x);
    int j = 0;
    const WaveSeg& sg = ga.plan.seg[seg_of(ga.plan, c, &j)];
    const double cell = sg.geom->cell;
    __syncthreads();
    if (cell != cell_w) {
      for (int b = tid; b <= nb; b += kThreads) {
        // rounding window of the float bin decision: |dx| carries ~2 ulp of max(cell, r)
        const double e = sqrt(ga.bins.e2[b]);
        const double err = 4.0 * 1.2e-7 * (cell + e);
        win[b] = (float)(2.0 * e * err + err * err);
      }
      cell_w = cell;
    }
    if (warp == 0 && c == first) find_rows(c, flip);
    const int pi = sg.centres[sg.w0 + j];
    const int* order = orders + 32 * flip;
    for (int k = tid; k < 2 * L.rec; k += kThreads) accf[k] = 0.f;
    for (int i = tid; i < nb * nblk * 10; i += kThreads) trs[i] = 0.f;
    for (int i = tid; i < args.slots * kRows * kSec / 4; i += kThreads)
      reinterpret_cast<float4*>(mom)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    if (tid < nb)
      safe[tid] = make_float2((e2f[tid] + win[tid]) * 1.0000003f, (e2f[tid + 1] - win[tid + 1]) * 0.9999997f);
    const int nr = misc[0], total = misc[1], nbig = misc[2];
    const unsigned bigs = (unsigned)misc[3];
    const float4 Pi = *cpos4;
    lk.out_lo = e2f[0] - win[0];
    lk.out_hi = e2f[nb] + win[nb];
    __syncthreads();
    unsigned long long pairs_here = 0;

    // Rounds: the chunks of candidates (mode 0), which leave the pairs of bins without sectors in a list;
    // that list (mode 1), when it is nearly full and at the end; a chunk again whose pairs the list had
    // no room for (mode 2: only they count).
    const int nchunks = (total + kCap - 1) / kCap, nsmall = nb - nbig;
    int ndefer = 0, mode = 0, few_before = 0;
    for (int ch = 0;;) {
      if (mode != 2) {
        if (ndefer > 0 && (ch == nchunks || ndefer + few_before * 3 / 2 > kDefer)) mode = 1;
        else if (ch < nchunks) mode = 0;
        else break;
      }
      const int nkeys = mode == 0 ? 1 + kSec * nbig : nsmall;
      // ---- classification: per candidate its bucket and rank in the warp's part of the bucket, its
      // position and t, kept where the pairs go later.  A chunk takes every nchunks-th group of 32
      // candidates (a stretch of rows would lie in a few sectors only); this warp's groups: [g0, g1).
      const int ngroups = mode == 1 ? (ndefer + 31) / 32 : ((total + 31) / 32 - ch + nchunks - 1) / nchunks;
      const int per = (ngroups + kWarps - 1) / kWarps;
      const int g0 = warp * per, g1 = min(ngroups, g0 + per);
      const int gstep = mode == 1 ? 1 : nchunks, gfirst = mode == 1 ? 0 : ch, tend = mode == 1 ? ndefer : total;
      int r = 0;
      if (mode != 1) {
        const int first = (g0 * nchunks + ch) * 32;
        int hi = nr;
        while (hi - r > 1) {
          const int mid = (r + hi) >> 1;
          if (first >= rpre[mid]) r = mid; else hi = mid;
        }
      }
      unsigned short* wc = cnt + warp * kKeys;
      // (the lanes of a bucket, a bit each)
      unsigned* same = reinterpret_cast<unsigned*>(pairs) + warp * kKeys;
      unsigned* ckr = reinterpret_cast<unsigned*>(pairs) + kWarps * kKeys;  // [kCap]
      float* ct = reinterpret_cast<float*>(ckr + kCap);                     // [kCap]
      int* cq = reinterpret_cast<int*>(ct + kCap);                          // [kCap]
      static_assert((kWarps * kKeys + 3 * kCap) * 4 <= kCap * (int)sizeof(float4), "the pairs' memory");
      for (int k = lane; k < nkeys; k += 32) same[k] = 0;
      __syncwarp();
      constexpr int kB = 5;  // groups of a warp on their way at once
#pragma unroll 1
      for (int ga0 = g0; ga0 < g1; ga0 += kB) {
        float4 Qs[kB];
        int qs[kB], bs[kB];
        float ds[kB];
        int sc[kB];
#pragma unroll
        for (int h = 0; h < kB; ++h) {
          const int t = ((ga0 + h) * gstep + gfirst) * 32 + lane;
          qs[h] = -1;
          Qs[h] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (ga0 + h < g1 && t < tend) {
            if (mode == 1) {
              qs[h] = defer[t];
            } else {
              while (r + 1 < nr && t >= rpre[r + 1]) ++r;
              qs[h] = rstart[r] + (t - rpre[r]);
            }
            Qs[h] = cat.p4[qs[h]];
          }
        }
        bool odd = false;  // some decision is within a rounding window
#pragma unroll
        for (int h = 0; h < kB; ++h) {
          const float dx = (Qs[h].x - Pi.x) + (Qs[h].z - Pi.z);
          const float dy = (Qs[h].y - Pi.y) + (Qs[h].w - Pi.w);
          const float r2 = dx * dx + dy * dy;
          int b = lk.tab[min((__float_as_uint(r2) - lk.base) >> lk.shift, 255u)];
          b += b + 1 < nb && r2 >= e2f[b + 1];
          const float2 sf = safe[b];
          const bool in = qs[h] >= 0 && r2 >= lk.out_lo && r2 < lk.out_hi;
          const bool sure = r2 >= sf.x && r2 < sf.y;
          bs[h] = in ? (sure ? b : -2) : -1;
          odd |= bs[h] == -2;
          sc[h] = sector_of(dx, dy);
          const float4 cc = uc[sc[h]];
          // sin delta, then delta / delta_max
          const float sd = ((dy * cc.x - dx * cc.y) + (dy * cc.z - dx * cc.w)) * rsqrtf(r2);
          const float s2 = sd * sd;
          ds[h] = sd * ((float)(1.0 / kDeltaMax) +
                        s2 * ((float)(1.0 / 6.0 / kDeltaMax) + s2 * (float)(3.0 / 40.0 / kDeltaMax)));
        }
        if (odd) {
#pragma unroll
          for (int h = 0; h < kB; ++h)
            if (bs[h] == -2) {
              const float dx = (Qs[h].x - Pi.x) + (Qs[h].z - Pi.z);
              const float dy = (Qs[h].y - Pi.y) + (Qs[h].w - Pi.w);
              bs[h] = Pair<float>::bin(cat, qs[h], cxy[0], cxy[1], dx * dx + dy * dy, e2, e2f, win, lk, nb);
            }
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < kB; ++h) {
          if (ga0 + h >= g1) break;  // uniform
          const bool big = bs[h] >= 0 && (bigs >> bs[h] & 1);
          int key = -1;
          if (bs[h] >= 0) {
            const int k0 = kb[bs[h]];
            key = mode == 0 ? (big ? k0 + sc[h] : 0) : (big ? -1 : k0);
          }
          if (key >= 0) atomicOr(&same[key], 1u << lane);
          __syncwarp();
          const unsigned peers = key >= 0 ? same[key] : 0, old = key >= 0 ? wc[key] : 0;
          __syncwarp();
          if (key >= 0 && (peers & lt) == 0) {
            wc[key] = (unsigned short)(old + __popc(peers));
            same[key] = 0;
          }
          __syncwarp();
          const int i = (ga0 + h) * 32 + lane;
          ckr[i] = key >= 0 ? (unsigned)key << 16 | (old + __popc(peers & lt)) : kFull;
          ct[i] = ds[h];
          cq[i] = max(qs[h], 0);
        }
      }
      if (tid == 0) misc[4] = 0;
      __syncthreads();
      // ---- bucket offsets, and every warp's first position in each bucket
      {
        int tot = 0;
        if (tid < nkeys)
#pragma unroll
          for (int w = 0; w < kWarps; ++w) tot += cnt[w * kKeys + tid];
        int inc = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(kFull, inc, o);
          if (lane >= o) inc += v;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        int pos = inc - tot;
        for (int w = 0; w < warp; ++w) pos += wsum[w];
        if (tid < nkeys) {
          koff[tid] = pos;
          if (tid == nkeys - 1) koff[nkeys] = pos + tot;
#pragma unroll
          for (int w = 0; w < kWarps; ++w) {
            const int n = cnt[w * kKeys + tid];
            cnt[w * kKeys + tid] = (unsigned short)pos;
            pos += n;
          }
        }
      }
      unsigned kr[kG];
      float ts[kG];
      int qs[kG];
#pragma unroll
      for (int g = 0; g < kG; ++g) {
        const int i = (g0 + g) * 32 + lane;
        const bool in = g0 + g < g1;
        kr[g] = in ? ckr[i] : kFull;
        ts[g] = in ? ct[i] : 0.f;
        qs[g] = in ? cq[i] : 0;
      }
      __syncthreads();
      // ---- the pairs to their places
      const int few = mode == 0 ? koff[1] : 0;  // those of bins without sectors
      const bool room = ndefer + few <= kDefer;
      if (mode == 0) {
#pragma unroll
        for (int g0b = 0; g0b < kG; g0b += kG / 2) {
          float4 sh[kG / 2];
#pragma unroll
          for (int g = 0; g < kG / 2; ++g) sh[g] = cat.s4[qs[g0b + g]];
#pragma unroll
          for (int g = 0; g < kG / 2; ++g) {
            const unsigned k = kr[g0b + g];
            if (k != kFull) {
              const int pos = wc[k >> 16] + (k & 0xFFFFu);
              if (k >> 16) pairs[pos] = make_float4(ts[g0b + g], sh[g].x, sh[g].y, sh[g].z);
              else if (room) defer[ndefer + pos] = qs[g0b + g];
            }
          }
        }
      } else {
#pragma unroll
        for (int g = 0; g < kG; ++g)
          if (kr[g] != kFull) {
            float ur, ui;
            Pair<float>::direction(cat, qs[g], 0.0, 0.0, Pi, ur, ui);
            pairs[wc[kr[g] >> 16] + (kr[g] & 0xFFFFu)] = make_float4(ur, ui, __int_as_float(qs[g]), 0.f);
          }
      }
      __syncthreads();
      for (int i = lane; i < nkeys; i += 32) wc[i] = 0;  // for the next round
      if (mode == 0) pairs_here += (unsigned long long)koff[nkeys];
      // ---- items, each taken by the next free warp: eight sectors of a bin (quarters of the bins took
      // 7% more of the whole: fewer items, and lanes less evenly filled), (bin, power block) of the
      // bins without
      const int nitems = mode == 0 ? 8 * nbig : nsmall * nblk;
      for (int item = warp; item < nitems;) {
        int next = 0;  // asked for now, used at the end
        if (lane == 0) next = kWarps + atomicAdd(&misc[4], 1);
        if (mode == 0) {
          const int slot = item >> 3, part = item & 7, key0 = 1 + kSec * slot;
          if (koff[key0 + 8 * part] < koff[key0 + 8 * part + 8])
            sector_item<K>(pairs, koff, key0, part, lane, mom + (size_t)slot * kRows * kSec);
        } else {
          const int i = item / nblk, b = order[nbig + i], k = item % nblk;
          if (koff[i] < koff[i + 1])
            direct_item(cat, pairs, koff[i], koff[i + 1], lane, k, mb, nblk, b, fidx, accf, trs + (b * nblk + k) * 10);
        }
        item = __shfl_sync(kFull, next, 0);
      }
      if (mode == 0) few_before = few;
      if (mode == 0 && room) ndefer += few;
      if (mode == 1) ndefer = 0;
      const bool again = mode == 0 && !room;
      if (!again) ch += mode != 1;
      mode = again ? 2 : 0;
      __syncthreads();
    }
    if (warp == 0 && cn < ga.plan.total) find_rows(cn, flip ^ 1);
    // ---- moments to sums over the sectors, one warp four rows at a time (the pairs' memory is free)
    {
      float cs[17], sn[17];
#pragma unroll
      for (int i = 0; i <= 16; ++i) {
        const float4 u = uc[lane * i & (kSec - 1)];
        cs[i] = u.x;
        sn[i] = u.y;
        if (lane == 0) sn[i] = i & 1 ? -1.f : 1.f;  // its imaginary place holds F(32)
      }
      float4* scr = pairs + warp * 68;
      constexpr int kPairs = 7 * K / 2;
      const int np = nbig * kPairs;
      // (warp 0 is busy with the next centre's rows)
      for (int p = 2 * (warp - 1); p >= 0 && p < np; p += 2 * (kWarps - 1)) {
        const int row = 2 * (p % kPairs);
        sector_rows(mom + ((size_t)(p / kPairs) * kRows + row) * kSec, row, scr, lane, cs, sn);
      }
      // the triple sums: each sector's times e^{-8 i phi_c}, e^{-4 i phi_c}
      if (warp > 0 && warp <= nbig) {
        const float* m = mom + ((size_t)(warp - 1) * kRows + 7 * K) * kSec;
        float v[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) v[j] = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int sec = lane + 32 * h;
          float s4, c4, s8, c8, t[9];
          sincospif(sec * (1.f / 8.f), &s4, &c4);
          sincospif(sec * (1.f / 4.f), &s8, &c8);
#pragma unroll
          for (int j = 0; j < 9; ++j) t[j] = m[j * kSec + mom_col(sec, 7 * K + j)];
          v[0] += t[0] * c8 + t[1] * s8;
          v[1] += t[1] * c8 - t[0] * s8;
          v[2] += t[2] * c4 + t[3] * s4;
          v[3] += t[3] * c4 - t[2] * s4;
          v[4] += t[4] * c4 + t[5] * s4;
          v[5] += t[5] * c4 - t[4] * s4;
          v[6] += t[6];
          v[7] += t[7];
          v[8] += t[8];
        }
#pragma unroll
        for (int j = 0; j < 9; ++j) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_xor_sync(kFull, v[j], o);
          if (lane == 0) trs[order[warp - 1] * nblk * 10 + j] = v[j];
        }
      }
    }
    __syncthreads();
    // ---- sums over k: the record's entries of the bins with sectors
    for (int i = tid; i < nbig * (L.max_pow + 1) * 5; i += kThreads) {
      const int task = i % 5, n = i / 5 % (L.max_pow + 1), slot = i / 5 / (L.max_pow + 1), b = order[slot];
      const float* m0 = mom + (size_t)slot * kRows * kSec;
      const int mm = n & (kSec - 1), mf = mm > 32 ? kSec - mm : mm;
      const float cj = mm > 32 ? -1.f : 1.f;
      auto sum = [&](int q) {
        float2 s = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const float* row = m0 + (7 * k + q) * kSec;
          float2 f = mf == 32 ? make_float2(row[1], 0.f) : reinterpret_cast<const float2*>(row)[mf];
          if (mf == 0) f.y = 0.f;
          f.y *= cj;
          const float a = coef[n * K + k];
          if (k & 1) { s.x -= a * f.y; s.y += a * f.x; }
          else { s.x += a * f.x; s.y += a * f.y; }
        }
        return s;
      };
      float2* acc = reinterpret_cast<float2*>(accf);
      if (task < 2) {
        const float2 R = sum(2 * task), I = sum(2 * task + 1);
        const float2 up = make_float2(R.x - I.y, R.y + I.x), dn = make_float2(R.x + I.y, I.x - R.y);
        if (task == 0) {
          if (n <= 2 * L.N - 1) acc[L.G(n, b)] = up;
          if (n >= 1 && n <= 2 * L.N + 3) acc[L.G(-n, b)] = dn;
        } else {
          if (n <= 2 * L.N - 2) acc[L.XX(n, b)] = up;
          if (n >= 1 && -n <= 2 * L.N - 2 && n <= 2 * L.N + 6) acc[L.XX(-n, b)] = dn;
        }
      } else if (task == 2) {
        if (n <= 2 * L.N) acc[L.W(n, b)] = sum(4);
      } else if (task == 3) {
        if (n <= 2 * L.N + 2) acc[L.XA(n, b)] = sum(5);
      } else {
        if (n <= 2 * L.N) acc[L.WW(n, b)] = sum(6);
      }
    }
    // triple terms: the parts' sums in order
    for (int i = tid; i < nb * 10; i += kThreads) {
      const int b = i / 10, q = i % 10;
      float sum = 0.f;
      for (int k = 0; k < nblk; ++k) sum += trs[(b * nblk + k) * 10 + q];
      accf[2 * L.TR(q >> 1, b) + (q & 1)] += sum;
    }
    __syncthreads();
    float2* dst = rec + (size_t)c * L.rec;
    const float2* accs = reinterpret_cast<const float2*>(accf);
    if (ga.accumulate) {
      for (int k = tid; k < L.rec; k += kThreads) dst[k] = cadd(dst[k], accs[k]);
    } else {
      for (int k = tid; k < L.rec; k += kThreads) dst[k] = accs[k];
    }
    if (tid == 0) {
      if (!ga.accumulate) {
        float xr, xi, ww;
        Pair<float>::load_x(ga.cen, pi, xr, xi, ww);
        xw[2 * (size_t)c] = make_float2(xr, xi);
        xw[2 * (size_t)c + 1] = make_float2(ww, 0.f);
      }
    }
    if (tid == 0) {
      atomicAdd(ga.pair_count, pairs_here);
      atomicAdd(ga.pair_count + 1, 1ull);  // centres of this kernel
    }
  }
}

// J_0, 2 J_1, ..., 2 J_{K-1} at 0 <= z < 5 by downward recurrence (Miller), normalised with
// J_0 + 2 sum J_{2k} = 1
void jacobi_anger(double z, int K, float* out) {
  if (z == 0.0) {
    for (int k = 0; k < K; ++k) out[k] = k ? 0.f : 1.f;
    return;
  }
  double f[33], sum = 0.0;
  f[32] = 0.0;
  f[31] = 1e-60;
  for (int k = 31; k > 0; --k) f[k - 1] = 2.0 * k / z * f[k] - f[k + 1];
  for (int k = 0; k < 32; k += 2) sum += k ? 2.0 * f[k] : f[k];
  for (int k = 0; k < K; ++k) out[k] = (float)((k ? 2.0 : 1.0) * f[k] / sum);
}

template <int K>
cudaError_t launch(SectorArgs& a, size_t smem, float2* rec, float2* xw, cudaStream_t s) {
  for (int n = 0; n <= a.g.L.max_pow; ++n) jacobi_anger(n * kDeltaMax, K, a.coef + n * K);
  cudaError_t e = allow_smem(gather_sector_kernel<K>);
  if (e != cudaSuccess) return e;
  gather_sector_kernel<K><<<std::min(a.g.plan.total, device_sms()), kThreads, smem, s>>>(a, rec, xw);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace

cudaError_t gather_sector(const SortedCat& cat, const SortedCat& cen, const Bins& bins, const Layout& L,
                          const WavePlan& plan, bool accumulate, int mb, int nblk, float2* rec, float2* xw,
                          unsigned long long* pair_count, cudaStream_t s, float* dense_min) {
  *dense_min = 0.f;
  const int K = L.max_pow <= 46 ? 12 : 16;
  SectorArgs a;
  GatherArgs& g = a.g;
  g.cat = cat; g.cen = cen; g.bins = bins; g.L = L; g.plan = plan; g.accumulate = accumulate ? 1 : 0;
  g.mb = mb; g.nblk = nblk; g.pair_count = pair_count;
  const size_t fixed = (size_t)kCap * sizeof(float4) + 2 * ((g.L.rec + 1) & ~1) * sizeof(float) + sizeof(float4) +
                       68 * sizeof(double) +
                       2 * kSec * sizeof(float2) + 195 * sizeof(float) +
                       (size_t)g.bins.nb * g.nblk * 10 * sizeof(float) +
                       (size_t)(g.L.max_pow + 1) * K * sizeof(float) +
                       ((size_t)g.nblk * V + 2 * kMaxRows + 1 + 8 + 32 + 64 + kWarps + kKeys + 1 + kDefer) * sizeof(int) +
                       (size_t)kWarps * kKeys * sizeof(unsigned short) + 256 + 16;
  const size_t slot = (size_t)(7 * K + 12) * kSec * sizeof(float), budget = 227 * 1024;
  if (fixed + 2 * slot > budget) return cudaSuccess;
  a.slots = (int)std::min<size_t>(kSlots, (budget - fixed) / slot);
  const double rm2 = g.bins.rmax * g.bins.rmax;
  double rest = 0.0, covered = 0.0;  // parts of the candidates in bins that get no sectors, in any bin
  int sectored = 0;
  for (int b = 31; b >= 0; --b) {
    const double part = b < g.bins.nb ? (g.bins.e2[b + 1] - g.bins.e2[b]) / rm2 : 0.0;
    a.share[b] = (float)(0.9 * part);
    covered += part;
    if (part > 0.0 && ++sectored > a.slots) rest += part;
  }
  sectored = std::min(sectored, a.slots);
  // Which catalogues.  Clocks per centre, measured on few bins beside the sectored ones: gather.cu 6.4 +
  // 0.165 powers a candidate; here 9.6 and 27 for each in a bin without sectors, and 25000 a centre for
  // the moments' transform and the like.  At ten bins from 0.5 to 40 the line is 6670 candidates at
  // n_max = 20 and 4230 at 30; at most four bins 27000 at n_max = 9, 42000 at 8, 94300 at 7, and no catalogue
  // below.  Records of 1216 centres just past it, gather.cu and here: 0.541, 0.526 ms (n_max = 20, 4 bins),
  // 1.98, 1.84 ms (8, 4), 4.23, 3.74 ms (7, 4).
  const int npow = L.max_pow + 1;
  const double gain = 6.4 + 0.165 * npow - (9.6 + 27.0 * rest);
  if (gain <= 0.0) return cudaSuccess;
  // Raised, or no catalogue, where by a second fit (916 cases: n_max 7 to 40, 1 to 16 bins, outer to inner radius 2
  // to 80; rms 5%) gather.cu is the faster one at the line: narrow bins leave many pairs without sectors,
  // whose sums cost by the power block (n_max = 40, ten bins to a twentieth of the radius, two of them sectored,
  // 8450 candidates: 1.39 ms there, 1.64 ms here), and many powers or few pairs among the candidates move
  // it up.
  const double there = 0.98 * (4.3 + covered * nblk * (mb == kMB ? 1.5 : 2.1));
  const double here = 5.0 + 0.2 * K * covered + 0.47 * sectored + rest * (25.0 + 4.3 * nblk);
  if (here >= there) return cudaSuccess;
  const double once = 29700.0 + 300.0 * L.nb * nblk + 6.8 * sectored * K * npow - 0.98 * (13800.0 + 420.0 * L.nb * nblk);
  const double least = std::max(25000.0 / gain, once / (there - here));
  if (cat.n < least) return cudaSuccess;
  g.dense_min = *dense_min = (float)least;
  const size_t smem = fixed + a.slots * slot;
  return K == 12 ? launch<12>(a, smem, rec, xw, s) : launch<16>(a, smem, rec, xw, s);
}

}  // namespace ext4pcf
