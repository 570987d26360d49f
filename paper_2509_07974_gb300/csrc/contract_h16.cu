// Split-FP16 tensor-core contraction of a wave (tcgen05 kind::f16, sm_103a).
//
// The GEMM runs over the independent sums of basis.cuh: for fixed sg the row products
// G_a(b2) G_{sg-a}(b3), b2 <= b3, are multiplied with the columns x G_{-sg-8}(b1), x^* G_{-sg-4}(b1),
// x G_{sg+4}^*(b1) and x^* G_sg^*(b1) (families F0..F3; W rows with the column w W_{-sg}), K running
// over the centres.  Every row product serves four families, so 1655 tiles of 128 rows (n_max = 20,
// 10 bins) hold what took 5572 tiles with a row type per component.  Forming the rows on the CUDA
// cores is the larger part of the work.  One wave of 8192 centres at these sizes: 6.5 -> 2.24 ms
// (3300 clocks per 64-centre stage of a tile; by count of its accesses shared memory is busy for about 2750
// of them: row products read 1024 wavefronts, the columns' embedding moves 480, the MMAs read 480
// and the bulk copies write 480).  The data are arranged for the producers:
//  * Power-of-two row scales.  A pre-pass finds the largest |component| of every row of the
//    wave array and the transpose writes each row times 2^k, its largest component in
//    [2^6, 2^7).  A product of two rows is then below 2^15, inside the fp16 range, with no
//    per-value scaling in the kernel; the epilogue takes out the exact factor in FP64.
//  * Planar staging.  Per 16 centres a G or W row holds their 16 real parts, then their 16
//    imaginary parts (128 bytes), so that two centres' real (or imaginary) parts form one 64-bit
//    register pair and the complex products run on the packed f32x2 pipe.  The column rows
//    (x G, x^* G, w W) are split into fp16 hi and lo by the transpose: real hi | imaginary hi |
//    real lo | imaginary lo, 64 centres each.
//  * Stage-major wave array.  The array is laid out [stage of 64 centres][row][512 bytes]; in
//    the G and W rows the 16-byte chunks of every 128-byte quarter are XOR-permuted by the row
//    index mod 8 (the 128-byte swizzle, applied by the transpose).  The rows a work item needs
//    for one stage are six contiguous ranges, fetched with six plain bulk copies
//    (cp.async.bulk) instead of one tensor box per 8 rows and 16 centres: the copy engine's
//    per-request cost, not bandwidth, bounded the boxed staging.  Eight lanes reading eight
//    consecutive rows at the same logical chunk hit eight different bank groups.
//  * K order.  In every group of 8 centres (one MMA, K = 16 halves) K = 0..7 holds the real
//    and K = 8..15 the imaginary parts.
//  * 64-centre stages and ring counters without divisions: each producer thread forms 16
//    values of its row per stage between two barrier crossings; two warps of their own write
//    the columns' real embedding (the B operand).
// Precision: every operand is split into fp16 hi + lo (22 significant bits) and the MMAs
// accumulate hi*lo + lo*hi + hi*hi in FP32 over one stage; the stage's partial sums are
// promoted into FP32 registers while the next stage runs, and the epilogue adds them into the
// FP64 reduced array.
// Every wait is bounded by a clock budget; on expiry the kernel records an error code, runs to
// its end, waits for its own MMAs and copies and frees its TMEM.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "basis.cuh"
#include "tc_ptx.cuh"

namespace ext4pcf {

namespace {

constexpr int kHCentres = 64;                        // centres per stage
constexpr int kHProducerWarps = 16;
constexpr int kHColumnWarps = 2;
constexpr int kHWarpMma = kHProducerWarps + kHColumnWarps, kHWarpLoad = kHWarpMma + 1;
constexpr int kHThreads = (kHWarpLoad + 1) * 32;
constexpr int kHArrivals = kHProducerWarps + kHColumnWarps;
constexpr int kHACols = 128;                         // TMEM columns per A slot: 64 hi + 64 lo
constexpr int kHMaxSlots = 3;                        // A (TMEM) and B (shared) ring depth at most
constexpr int kHMaxIn = 4;                           // staged-input ring depth at most
constexpr uint32_t kHTmemCols = 512;
constexpr int kHScaleTop = 6;                        // rows scaled into [2^6, 2^7)

// exponent k of the row scale 2^k for a row whose largest |component| has the float bits m
__host__ __device__ __forceinline__ int h_scale_exp(unsigned mbits) {
#ifdef __CUDA_ARCH__
  const float m = __uint_as_float(mbits);
  if (!(m > 0.f)) return 0;
  const int k = kHScaleTop - ilogbf(m);
  return k < -100 ? -100 : (k > 100 ? 100 : k);
#else
  (void)mbits;
  return 0;
#endif
}
__device__ __forceinline__ float h_pow2f(int k) { return __int_as_float((127 + k) << 23); }
__device__ __forceinline__ double h_pow2d(int k) { return __longlong_as_double((long long)(1023 + k) << 52); }

// Rows of the transposed wave array:
//   [0, w)       G_m(bin), m in [-2N-3, 2N-1]
//   [w, xg)      W_m(bin), m in [-2N, 2N]
//   [xg, xcg)    x G_m(bin)       (column rows, split into fp16 hi and lo)
//   [xcg, ww)    x^* G_m(bin)
//   [ww, rows)   w W_m(bin), m in [0, 2N]
struct HRows {
  int w, xg, xcg, ww, rows;
  __host__ __device__ static HRows make(const Layout& L) {
    HRows r;
    r.w = L.nG * L.nb;
    r.xg = r.w + (4 * L.N + 1) * L.nb;
    r.xcg = r.xg + L.nG * L.nb;
    r.ww = r.xcg + L.nG * L.nb;
    r.rows = r.ww + L.nW * L.nb;
    return r;
  }
};
// value of row r at one centre (rc: the centre's record, x = w gamma, w)
__device__ __forceinline__ float2 hwave_value(const Layout& L, const HRows& R, const float2* __restrict__ rc, float2 x,
                                              float w, int r) {
  const int nb = L.nb;
  if (r < R.w) return rc[L.oG + r];
  if (r < R.xg) {
    const int m = (r - R.w) / nb - 2 * L.N, b = (r - R.w) % nb;
    float2 f = rc[L.W(m >= 0 ? m : -m, b)];
    if (m < 0) f.y = -f.y;
    return f;
  }
  if (r >= R.ww) {
    const float2 f = rc[L.oW + (r - R.ww)];
    return make_float2(w * f.x, w * f.y);
  }
  if (r >= R.xcg) x.y = -x.y;
  const float2 f = rc[L.oG + (r >= R.xcg ? r - R.xcg : r - R.xg)];
  return make_float2(x.x * f.x - x.y * f.y, x.x * f.y + x.y * f.x);
}

// largest |component| of every row over the wave's centres: 32 rows x 128 centres per block
// (records of the wave's live centres only: padding records are never read)
__global__ void __launch_bounds__(256) hwave_rowmax_kernel(const Layout L, const float2* __restrict__ rec,
                                                           const float2* __restrict__ xw, const WavePlan plan,
                                                           const HRows R, unsigned* __restrict__ rowmax) {
  __shared__ float part[8][33];
  const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 128;
  if (c0 >= plan.total) return;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, r = r0 + tx;
  float m = 0.f;
  if (r < R.rows) {
    for (int k = 0; k < 16; ++k) {
      const int c = c0 + ty + 8 * k;
      int j = 0;
      const int si = c < plan.total ? seg_of(plan, c, &j) : -1;
      if (si >= 0 && j < seg_live(plan.seg[si])) {
        const float2 v = hwave_value(L, R, rec + (size_t)c * L.rec, xw[2 * (size_t)c], xw[2 * (size_t)c + 1].x, r);
        m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
      }
    }
  }
  part[ty][tx] = m;
  __syncthreads();
  if (ty == 0 && r < R.rows) {
    for (int k = 1; k < 8; ++k) m = fmaxf(m, part[k][tx]);
    if (m > 0.f) atomicMax(&rowmax[r], __float_as_uint(m));  // non-negative floats order as integers
  }
}

// The transposed, scaled wave array, stage-major: record c of row r sits in stage c / 64, in the
// 512 bytes of row r there.  G and W rows: float q * 32 + ((k ^ (r % 8)) * 4) + c % 4 with
// q = (c % 64) / 16 the quarter and k = (c % 16) / 4 (real part) or 4 + (c % 16) / 4 (imaginary
// part) the logical 16-byte chunk.  Column rows: half c % 64 of each of the four planes real hi,
// imaginary hi, real lo, imaginary lo.
// Padding records (between segments, past a segment's live centres, past the wave up to a
// multiple of 64) are written as zeros.
__global__ void __launch_bounds__(256) hwave_transpose_kernel(const Layout L, const float2* __restrict__ rec,
                                                              const float2* __restrict__ xw, const WavePlan plan,
                                                              const HRows R, const unsigned* __restrict__ rowmax,
                                                              float* __restrict__ out) {
  __shared__ float2 tile[32][33];
  const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  const int Tp = (plan.total + kHCentres - 1) / kHCentres * kHCentres;
  if (c0 >= Tp) return;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int c = c0 + ty + 8 * k, r = r0 + tx;
    float2 v = make_float2(0.f, 0.f);
    int j = 0;
    const int si = c < plan.total ? seg_of(plan, c, &j) : -1;
    if (si >= 0 && j < seg_live(plan.seg[si]) && r < R.rows)
      v = hwave_value(L, R, rec + (size_t)c * L.rec, xw[2 * (size_t)c], xw[2 * (size_t)c + 1].x, r);
    tile[ty + 8 * k][tx] = v;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int r = r0 + ty + 8 * k, c = c0 + tx;
    if (r >= R.rows) continue;
    const float sc = h_pow2f(h_scale_exp(rowmax[r]));
    float2 v = tile[tx][ty + 8 * k];
    v.x *= sc;
    v.y *= sc;
    float* row = out + ((size_t)(c >> 6) * R.rows + r) * 128;
    if (r >= R.xg) {
      __half* h = reinterpret_cast<__half*>(row) + (c & 63);
      const __half xh = __float2half_rn(v.x), yh = __float2half_rn(v.y);
      h[0] = xh;
      h[64] = yh;
      h[128] = __float2half_rn(v.x - __half2float(xh));
      h[192] = __float2half_rn(v.y - __half2float(yh));
    } else {
      const int q = (c & 63) >> 4, kre = (c & 15) >> 2, sw = r & 7;
      float* o = row + q * 32 + (c & 3);
      o[(kre ^ sw) * 4] = v.x;
      o[((4 + kre) ^ sw) * 4] = v.y;
    }
  }
}

struct HArgs {
  Layout L;
  HRows R;
  WavePlan plan;      // the wave's segments (a segment starts at a stage boundary)
  double2* red;       // reduced outputs, one array (basis.cuh) per slot
  size_t red_stride;  // complex elements per slot
  size_t red_w;       // first W element
  int npairs;
  const int4* items;  // kind | group << 1 | (first a of sg + 128) << 8 | rows << 16, sg, first row, row base
  int n_items;
  int ncomp;          // families per X item: 4, or 2 in two groups (F0, F2 and F1, F3)
  const unsigned* rowmax;  // largest |component| per row (float bits): the row scales
  const float* wave;  // the stage-major wave array
  int in_stages;      // staged-input ring depth
  int stage_rows;     // rows per staged stage
  int npad_max;       // rows of a B tile
  long long timeout;
  int* status;
};

// Geometry of one work item: the staged blocks (first rows of the wave array, rows) and where they
// sit in a staged stage, packed one after the other: the G_a (W_a) rows, the G_{sg-a} rows, then nb
// rows per column family
struct HGeo {
  bool w;
  int sg, row0, nrows, alo, base;
  int a1, a2, m1;   // the tile's a range, and the first index of the second block
  int blk2, blk3;   // first rows of the wave array
  int len;          // rows of each of the two blocks
  int nfam;         // column families
};
__device__ __forceinline__ HGeo hgeo(const HArgs& a, int4 item) {
  const int nb = a.L.nb, N = a.L.N;
  HGeo g;
  g.w = (item.x & 1) != 0;
  g.sg = item.y;
  g.row0 = item.z;
  g.base = item.w;
  g.alo = ((item.x >> 8) & 0xFF) - 128;
  g.nrows = item.x >> 16;
  g.a1 = g.alo + g.row0 / a.npairs;
  g.a2 = g.alo + (g.row0 + g.nrows - 1) / a.npairs;
  g.m1 = g.sg - g.a2;
  g.len = (g.a2 - g.a1 + 1) * nb;
  const int first = g.w ? a.R.w + 2 * N * nb : (2 * N + 3) * nb;  // the row of index 0
  g.blk2 = first + g.a1 * nb;
  g.blk3 = first + g.m1 * nb;
  g.nfam = g.w ? 1 : a.ncomp;
  return g;
}
// family of column group j of an item, and its first row in the wave array; an index outside
// the record (a family that no component reads at this sg) is clamped into it: its sums are finite
// and never read
__device__ __forceinline__ int hfam(const HArgs& a, int4 item, int j) {
  return a.ncomp == 4 ? j : ((item.x >> 1) & 0x7F) + 2 * j;
}
__device__ __forceinline__ int hcol_row(const HArgs& a, int4 item, int j) {
  const int nb = a.L.nb, N = a.L.N;
  if (item.x & 1) return a.R.ww - item.y * nb;
  const int q = hfam(a, item, j);
  const int m = min(max(basis_col_index(q, item.y), -2 * N - 3), 2 * N - 1);
  // x G^* = (x^* G)^*, x^* G^* = (x G)^*: the conjugated families read the other array
  const bool xc = basis_centre_conj(q) != basis_col_conj(q);
  return (xc ? a.R.xcg : a.R.xg) + (m + 2 * N + 3) * nb;
}

// packed FP32x2 arithmetic on register pairs (x in the low word)
__device__ __forceinline__ unsigned long long f2mul(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long f2fma(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long f2sub(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// fp16 hi/lo split of a pair: hi = (fp16(a), fp16(b)) with a in the low half, lo the same of
// the exact residuals a - hi_a, b - hi_b (formed by one mixed-precision FMA each)
__device__ __forceinline__ void split_h2(unsigned long long v, uint32_t& hi, uint32_t& lo) {
  asm("{\n .reg .f32 a, b, r0, r1;\n .reg .b16 h0, h1, m1;\n"
      " mov.b64 {a, b}, %2;\n"
      " cvt.rn.f16x2.f32 %0, b, a;\n"
      " mov.b32 {h0, h1}, %0;\n"
      " mov.b16 m1, 0xBC00;\n"
      " fma.rn.f32.f16 r0, h0, m1, a;\n"
      " fma.rn.f32.f16 r1, h1, m1, b;\n"
      " cvt.rn.f16x2.f32 %1, r1, r0;\n}\n"
      : "=r"(hi), "=r"(lo)
      : "l"(v));
}
// 16 bytes of shared memory as two register pairs
__device__ __forceinline__ void lds_2x64(uint32_t addr, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
}
// The products of one row for 8 centres (group h of the thread's 16): G_a at PB, G_{sg-a} at PC
// (shared addresses of the rows in the staged stage, swizzle term folded in: chunk c is at
// P ^ (c << 4)).  Writes hi / lo words 0..7: four pairs of real parts, then four pairs of
// imaginary parts.  One 16-byte chunk (four centres) at a time.
__device__ __forceinline__ void kr_group(uint32_t PB, uint32_t PC, int h, uint32_t* hi, uint32_t* lo) {
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const uint32_t re_off = (uint32_t)(2 * h + c) << 4, im_off = (uint32_t)(4 + 2 * h + c) << 4;
    unsigned long long xr[2], xi[2], cr[2], ci[2];
    lds_2x64(PB ^ re_off, xr[0], xr[1]);
    lds_2x64(PB ^ im_off, xi[0], xi[1]);
    lds_2x64(PC ^ re_off, cr[0], cr[1]);
    lds_2x64(PC ^ im_off, ci[0], ci[1]);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      split_h2(f2sub(f2mul(xr[p], cr[p]), f2mul(xi[p], ci[p])), hi[2 * c + p], lo[2 * c + p]);
      split_h2(f2fma(xr[p], ci[p], f2mul(xi[p], cr[p])), hi[4 + 2 * c + p], lo[4 + 2 * c + p]);
    }
  }
}
__device__ __forceinline__ uint4 lds_128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts_128(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// CW columns of this thread's TMEM lane
template <int CW>
__device__ __forceinline__ void tmem_ld_cols(uint32_t ta, uint32_t* v) {
  static_assert(CW == 16 || CW == 20 || CW == 24, "columns per quarter");
  tmem_ld16(ta, v);
  if (CW == 20) tmem_ld4(ta + 16, v + 16);
  if (CW == 24) tmem_ld8(ta + 16, v + 16);
}

// Warp roles: warps 0..15 form the A operand (row products, TMEM); warps 16 and 17 the B operand
// (shared memory) of each stage; warp 18 issues the MMAs (one thread); warp 19 stages each
// stage's rows of the wave array with bulk copies (one thread).  Rings and their mbarriers
// (counts in brackets):
//   staged input  in_full [1 + copied bytes] / in_empty [18 forming warps]
//   A and B       ab_full [18 forming warps] / ab_empty [1, tcgen05.commit]
//   partial sums  dfull [1, tcgen05.commit] / dempty [16 producer warps]
// CW: D columns per producer quarter (4 CW in all); SLOTS: A/B ring depth, what the
// 512 TMEM columns leave next to two D buffers.
template <int CW, int SLOTS>
__global__ void __launch_bounds__(kHThreads, 1)
contract_h16_kernel(const __grid_constant__ HArgs args) {
  constexpr int kDStride = CW == 16 ? 64 : 96, kABase = 2 * kDStride;
  static_assert(4 * CW <= kDStride && kABase + SLOTS * kHACols <= (int)kHTmemCols, "TMEM columns");
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sm = smem_raw + ((1024 - (saddr(smem_raw) & 1023)) & 1023);
  const Layout L = args.L;
  const int nb = L.nb, npairs = args.npairs;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t atom_bytes = (uint32_t)args.npad_max * 128u;  // one 128-byte-wide K-atom of a B tile
  const uint32_t bslot_bytes = 4u * atom_bytes;                  // hi tile (2 atoms) | lo tile (2 atoms)
  const uint32_t in_bytes = (uint32_t)args.stage_rows * 512u;    // one staged stage: rows of 512 bytes
  const int S_in = args.in_stages;
  unsigned char* in_base = sm + SLOTS * bslot_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(in_base + (size_t)S_in * in_bytes);
  uint64_t* in_full = bars;
  uint64_t* in_empty = in_full + kHMaxIn;
  uint64_t* ab_full = in_empty + kHMaxIn;
  uint64_t* ab_empty = ab_full + kHMaxSlots;
  uint64_t* dfull = ab_empty + kHMaxSlots;  // [2]
  uint64_t* dempty = dfull + 2;             // [2]
  uint64_t* drain = dempty + 2;             // [1]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tmem_slot)),
                 "r"(kHTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int k = 0; k < S_in; ++k) {
      mbar_init(&in_full[k], 1);
      mbar_init(&in_empty[k], kHArrivals);
    }
    for (int k = 0; k < SLOTS; ++k) {
      mbar_init(&ab_full[k], kHArrivals);
      mbar_init(&ab_empty[k], 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(&dfull[k], 1);
      mbar_init(&dempty[k], kHProducerWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const long long budget = args.timeout;
  int err = 0;
  // bounded wait on an mbarrier phase; the first wait of the CTA that runs out of its budget
  // raises the abort flag, after which every wait gives up at once
  auto wait = [&](uint64_t* b, uint32_t parity) -> bool {
    if (*abort_flag) {
      err = 1;
      return false;
    }
    if (mbar_try(b, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try(b, parity)) {
      if (*abort_flag || clock64() - t0 > budget) {
        *abort_flag = 1;
        err = 1;
        return false;
      }
    }
    return true;
  };

  if (warp < kHProducerWarps) {
    // ---------------------------------------------------------------------- producers
    const int grp = warp & 3, qq = warp >> 2;  // TMEM lane group; 16-centre quarter of a stage
    const uint32_t in_addr = saddr(in_base);
    int islot = 0, aslot = 0;
    uint32_t iph = 0, aph = 0;
    long long gs = 0;  // partial sums (stages) so far
    for (int it = blockIdx.x; it < args.n_items; it += gridDim.x) {
      const int4 item = args.items[it];
      const HGeo g = hgeo(args, item);
      const int ncols = 2 * g.nfam * nb, npad = (ncols + 15) & ~15;
      const int rl = grp * 32 + lane;  // tile row = TMEM lane
      const bool row_ok = rl < g.nrows;
      const int rr = g.row0 + (row_ok ? rl : 0);
      const int av = g.alo + rr / npairs;
      int b2, b3;
      basis_pair(rr % npairs, nb, b2, b3);
      // this row's two factors, quarter qq, in a staged stage, with the swizzle term of their
      // rows in the wave array folded in (chunk c at P ^ (c << 4))
      const int e2 = (av - g.a1) * nb + b2, e3 = (g.sg - av - g.m1) * nb + b3;
      const int r2 = g.blk2 + e2, r3 = g.blk3 + e3;
      const uint32_t x2 = (uint32_t)e2 * 512u + qq * 128u + ((uint32_t)(r2 & 7) << 4);
      const uint32_t x3 = (uint32_t)(g.len + e3) * 512u + qq * 128u + ((uint32_t)(r3 & 7) << 4);
      float accD[CW];  // FP32 sums of the promoted partials: this row, CW columns
      const bool has_cols = qq * CW < npad;
      // Software pipeline over the stages (k = this stage):
      //  * the partial sum of stage k - 2 is taken out of TMEM at the start of this stage: its MMAs
      //    were signalled in the middle of stage k - 1;
      //  * the rows of stage k - 1 were stored into TMEM at the end of the previous iteration;
      //    their completion is awaited (and the MMA warp signalled) only after the first half
      //    of this stage's rows is formed, so the store latency is hidden behind that work.
      // The MMAs of stage k - 1 thus start one iteration late; the wait for the slot of stage k
      // comes after the first half of its rows, when the MMAs of stage k - SLOTS are done.
      auto promote = [&](long long gg) {
        const int buf = (int)(gg & 1);
        wait(&dfull[buf], (uint32_t)((gg >> 1) & 1));
        tc_fence_after();
        if (has_cols) {
          uint32_t v[CW];
          tmem_ld_cols<CW>(tmem + ((uint32_t)(grp * 32) << 16) + buf * kDStride + qq * CW, v);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < CW; ++j) accD[j] += __uint_as_float(v[j]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&dempty[buf]);
      };
      auto publish = [&](int slot) {  // the rows (TMEM) of a slot are complete
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&ab_full[slot]);
      };
      // the wave's segments in order, runs of consecutive segments with the same output slot
      // accumulated together (the patches of one survey form one run): one pipeline drain and
      // one epilogue per run
      for (int si = 0; si < args.plan.nseg;) {
      const int slot = args.plan.seg[si].slot;
      int nstage = 0;
      for (; si < args.plan.nseg && args.plan.seg[si].slot == slot; ++si)
        nstage += (seg_live(args.plan.seg[si]) + kHCentres - 1) / kHCentres;
#pragma unroll
      for (int j = 0; j < CW; ++j) accD[j] = 0.f;
      int prev_slot = 0;
      for (int k = 0; k < nstage; ++k) {
        if (k >= 2) promote(gs + k - 2);
        wait(&in_full[islot], iph);
        const uint32_t st = in_addr + (uint32_t)islot * in_bytes;
        // A operand (TMEM): this row's products for the warp's 16 centres, in two groups of 8;
        // the previous stage is published between them
        const uint32_t PB = st + x2, PC = st + x3;
        const uint32_t acol = tmem + ((uint32_t)(grp * 32) << 16) + kABase + aslot * kHACols + qq * 16;
        {
          uint32_t hi[8], lo[8];
          kr_group(PB, PC, 0, hi, lo);
          if (k >= 1) publish(prev_slot);
          wait(&ab_empty[aslot], aph ^ 1u);
          tc_fence_after();
          tmem_st8(acol, hi);
          tmem_st8(acol + 64, lo);
        }
        {
          uint32_t hi[8], lo[8];
          kr_group(PB, PC, 1, hi, lo);
          // every value this warp loaded from the staged stage has been used: it can be refilled
          __syncwarp();
          if (lane == 0) mbar_arrive(&in_empty[islot]);
          tmem_st8(acol + 8, hi);
          tmem_st8(acol + 64 + 8, lo);
        }
        prev_slot = aslot;
        if (++islot == S_in) { islot = 0; iph ^= 1u; }
        if (++aslot == SLOTS) { aslot = 0; aph ^= 1u; }
      }
      // drain the pipeline: the last stage's rows, then the last two partial sums
      if (nstage >= 1) publish(prev_slot);
      for (long long gg = gs + (nstage >= 2 ? nstage - 2 : 0); gg < gs + nstage; ++gg) promote(gg);
      gs += nstage;
      // ---------------------------------------------------------------- epilogue
      if (row_ok && has_cols && nstage > 0) {  // (an empty run adds nothing)
        const int kr = h_scale_exp(args.rowmax[r2]) + h_scale_exp(args.rowmax[r3]);
        const size_t row = (size_t)g.base + (av - g.alo), pr = rr % npairs;
        double2* out = args.red + (size_t)slot * args.red_stride;
        out += g.w ? args.red_w + row * nb * npairs + pr : row * 4 * nb * npairs + pr;
#pragma unroll
        for (int j = 0; j < CW; j += 2) {
          const int v = (qq * CW + j) >> 1;
          if (2 * v < ncols) {
            const int f = v / nb, b1 = v - f * nb;
            const double unscale = h_pow2d(-(kr + h_scale_exp(args.rowmax[hcol_row(args, item, f) + b1])));
            double2* p = out + (size_t)(g.w ? b1 : hfam(args, item, f) * nb + b1) * npairs;
            double2 d = *p;
            d.x += (double)accD[j] * unscale;
            d.y += (double)accD[j + 1] * unscale;
            *p = d;
          }
        }
      }
      }  // runs of segments
    }
  } else if (warp < kHWarpMma) {
    // ---------------------------------------------------------------------- B operand
    // The real embedding of the columns, fp16 hi and lo tiles: for column value A = (A_r, A_i)
    // tile row 2 v (real output) holds A_r at the real and -A_i at the imaginary K, row 2 v + 1
    // (imaginary output) A_i and A_r; a conjugated column has A_i of the other sign.  A lane takes
    // 8 centres (one 16-byte chunk each of A_r and A_i, hi and lo) of column pair v: eight
    // 16-byte stores, the lanes of the upper K-atom taking A_r and A_i in the other order, so that
    // the eight lanes of a phase hit eight different bank groups.
    const uint32_t in_addr = saddr(in_base), b_addr = saddr(sm);
    int islot = 0, aslot = 0;
    uint32_t iph = 0, aph = 0;
    for (int it = blockIdx.x; it < args.n_items; it += gridDim.x) {
      const int4 item = args.items[it];
      const HGeo g = hgeo(args, item);
      // lane: centre chunk q of column pairs v0, v0 + 8, ...
      const int t0 = (warp - kHProducerWarps) * 32 + lane, v0 = t0 >> 3, q = t0 & 7;
      const int npair = g.nfam * nb;
      const bool up = q >= 4;  // upper K-atom
      const uint32_t src0 = (uint32_t)(2 * g.len + v0) * 512u + q * 16u + (up ? 128u : 0u);
      const uint32_t n7 = (2u * v0) & 7u;
      const uint32_t dst0 = (uint32_t)(q >> 2) * atom_bytes + ((2u * v0) >> 3) * 1024u + n7 * 128u +
                            (((uint32_t)(2 * (q & 3)) ^ n7) << 4) + (up ? 16u : 0u);
      // (n7 is even: the row below differs in the lowest chunk bit and the row only)
      const uint32_t dst1 = (uint32_t)(q >> 2) * atom_bytes + ((2u * v0) >> 3) * 1024u + (n7 + 1u) * 128u +
                            ((((uint32_t)(2 * (q & 3)) ^ (n7 + 1u)) << 4) ^ (up ? 16u : 0u));
      uint32_t conj = 0;  // bit i: column pair v0 + 8 i belongs to a conjugated family
      for (int v = v0, i = 0; v < npair; v += 8, ++i)
        if (!g.w && basis_col_conj(hfam(args, item, v / nb))) conj |= 1u << i;
      for (int si = 0; si < args.plan.nseg; ++si) {
        const int nstage = (seg_live(args.plan.seg[si]) + kHCentres - 1) / kHCentres;
        for (int k = 0; k < nstage; ++k) {
          wait(&in_full[islot], iph);
          wait(&ab_empty[aslot], aph ^ 1u);
          uint32_t src = in_addr + (uint32_t)islot * in_bytes + src0;
          uint32_t d = b_addr + (uint32_t)aslot * bslot_bytes;
          uint32_t cbits = conj;
          for (int v = v0; v < npair; v += 8, src += 8 * 512u, d += 2048u, cbits >>= 1) {
            // sign of the imaginary part in row 2 v; row 2 v + 1 has the other one
            const uint32_t s0 = cbits & 1u ? 0u : 0x80008000u, s1 = s0 ^ 0x80008000u;
            const uint32_t mx0 = up ? s0 : 0u, my0 = up ? 0u : s0, mx1 = up ? s1 : 0u, my1 = up ? 0u : s1;
#pragma unroll
            for (int h = 0; h < 2; ++h) {  // hi, lo
              // x: the real part (lower K-atom) or the imaginary part (upper), y: the other
              const uint4 x = lds_128(src + h * 256u), y = lds_128((src ^ 128u) + h * 256u);
              const uint32_t e = d + dst0 + h * 2u * atom_bytes, f = d + dst1 + h * 2u * atom_bytes;
              sts_128(e, make_uint4(x.x ^ mx0, x.y ^ mx0, x.z ^ mx0, x.w ^ mx0));
              sts_128(e ^ 16u, make_uint4(y.x ^ my0, y.y ^ my0, y.z ^ my0, y.w ^ my0));
              sts_128(f, make_uint4(y.x ^ my1, y.y ^ my1, y.z ^ my1, y.w ^ my1));
              sts_128(f ^ 16u, make_uint4(x.x ^ mx1, x.y ^ mx1, x.z ^ mx1, x.w ^ mx1));
            }
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(&in_empty[islot]);
            mbar_arrive(&ab_full[aslot]);
          }
          if (++islot == S_in) { islot = 0; iph ^= 1u; }
          if (++aslot == SLOTS) { aslot = 0; aph ^= 1u; }
        }
      }
    }
  } else if (warp == kHWarpMma) {
    // ---------------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      const uint64_t dbase = desc_sw128(saddr(sm));
      int aslot = 0;
      uint32_t aph = 0;
      long long gs = 0;
      for (int it = blockIdx.x; it < args.n_items; it += gridDim.x) {
        const HGeo g = hgeo(args, args.items[it]);
        const int npad = (2 * g.nfam * nb + 15) / 16 * 16;
        const uint32_t id = idesc(0u, npad);  // fp16 A and B, FP32 D
        for (int si = 0; si < args.plan.nseg; ++si) {
        const int nstage = (seg_live(args.plan.seg[si]) + kHCentres - 1) / kHCentres;
        for (int k = 0; k < nstage; ++k, ++gs) {
          const int buf = (int)(gs & 1);
          if (gs >= 2) wait(&dempty[buf], (uint32_t)(((gs >> 1) - 1) & 1));
          wait(&ab_full[aslot], aph);
          tc_fence_after();
          const uint32_t d = tmem + buf * kDStride;
          const uint32_t ah = tmem + kABase + aslot * kHACols, al = ah + 64;
          // descriptor of the slot's hi tile: start-address field (address / 16) plus the
          // offset / 16 (no carry: shared addresses stay below 2^18)
          const uint64_t db = dbase + (uint64_t)((aslot * bslot_bytes) >> 4);
          const uint64_t dl = (uint64_t)((2 * atom_bytes) >> 4);
          // the two small terms of every K step first, while the sum is small: the unit cuts each
          // addition to the sum's last bit, so the order leaves 8 such cuts at full size, not 24
#pragma unroll
          for (int q = 0; q < 8; ++q) {  // K = 16 halves = 8 centres per MMA
            const uint64_t bh = db + (uint64_t)((((q >> 2) * atom_bytes) + (q & 3) * 32) >> 4);
            mma_f16(d, ah + q * 8, bh + dl, id, q > 0 ? 1u : 0u);
            mma_f16(d, al + q * 8, bh, id, 1u);
          }
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const uint64_t bh = db + (uint64_t)((((q >> 2) * atom_bytes) + (q & 3) * 32) >> 4);
            mma_f16(d, ah + q * 8, bh, id, 1u);
          }
          mma_commit(&ab_empty[aslot]);
          mma_commit(&dfull[buf]);
          if (++aslot == SLOTS) { aslot = 0; aph ^= 1u; }
        }
        }  // segments
      }
      // every MMA of this CTA has completed before the TMEM is released (also when a wait
      // above gave up); an MMA always finishes, so this bound is generous
      mma_commit(drain);
      if (!mbar_wait(drain, 0u, 4000000000LL)) err = 1;
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------------- bulk-copy loader
    // One thread: per stage the blocks of the item, each a contiguous range of the
    // stage-major wave array, copied with one cp.async.bulk each.
    if (lane == 0) {
      int islot = 0;
      uint32_t iph = 0;
      int last[kHMaxIn];  // parity of the last phase issued per slot (-1: none)
      for (int k = 0; k < kHMaxIn; ++k) last[k] = -1;
      for (int it = blockIdx.x; it < args.n_items; it += gridDim.x) {
        const int4 item = args.items[it];
        const HGeo g = hgeo(args, item);
        int blk[6], n = 2 + g.nfam;
        blk[0] = g.blk2;
        blk[1] = g.blk3;
        for (int j = 0; j < g.nfam; ++j) blk[2 + j] = hcol_row(args, item, j);
        const int rows = 2 * g.len + g.nfam * nb;
        bool ok = rows <= args.stage_rows;
        for (int b = 0; b < n; ++b) {
          const int len = b < 2 ? g.len : nb;
          ok = ok && blk[b] >= 0 && blk[b] + len <= args.R.rows;
        }
        if (!ok) {  // never for the supported shapes
          *abort_flag = 1;
          err = 1;
        }
        for (int si = 0; si < args.plan.nseg; ++si) {
        const WaveSeg& sgm = args.plan.seg[si];
        const int nstage = (seg_live(sgm) + kHCentres - 1) / kHCentres, kst0 = sgm.off / kHCentres;
        for (int k = 0; k < nstage; ++k) {
          wait(&in_empty[islot], iph ^ 1u);
          if (!*abort_flag) {  // nothing more is copied once the CTA gives up
            last[islot] = (int)iph;
            mbar_expect_tx(&in_full[islot], (uint32_t)rows * 512u);
            unsigned char* st = in_base + (size_t)islot * in_bytes;
            const float* src = args.wave + (size_t)(kst0 + k) * args.R.rows * 128;
            for (int b = 0; b < n; ++b) {
              const int len = b < 2 ? g.len : nb;
              bulk_load(st, src + (size_t)blk[b] * 128, (uint32_t)len * 512u, &in_full[islot]);
              st += len * 512;
            }
          }
          if (++islot == S_in) { islot = 0; iph ^= 1u; }
        }
        }  // segments
      }
      // every copy has landed before the shared memory is given up: the phases of a slot
      // complete in order, so its last issued phase covers the earlier ones
      for (int k = 0; k < S_in; ++k)
        if (last[k] >= 0 && !mbar_wait(&in_full[k], (uint32_t)last[k], 4000000000LL)) err = 1;
    }
    __syncwarp();
  }
  if (err) atomicExch(args.status, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kHTmemCols) : "memory");
}

// families per X item: four while their columns fit a D buffer of 96, two in two groups beyond
int h_ncomp(int nb) { return nb <= 12 ? 4 : 2; }
int h_npad_max(int nb) { return (2 * h_ncomp(nb) * nb + 15) / 16 * 16; }
// D columns per producer quarter and A/B slots next to the two D buffers
int h_cw(int nb) { return h_npad_max(nb) <= 64 ? 16 : h_npad_max(nb) <= 80 ? 20 : 24; }
int h_slots(int nb) { return h_cw(nb) == 16 ? 3 : 2; }
// rows per tile: one TMEM lane each; half of them for a single bin, whose rows all have an a of
// their own (staged blocks of 128 rows each would not fit twice)
int h_tile_rows(int nb) { return nb == 1 ? 64 : 128; }
// rows per staged stage: two blocks of at most the tile's a values (+2 where tiles cut through
// the pairs of an a) and the column rows
int h_stage_rows(int nb) {
  const int np = nb * (nb + 1) / 2;
  const int av = np == 1 ? h_tile_rows(nb) : h_tile_rows(nb) / np + 2;
  return 2 * av * nb + h_ncomp(nb) * nb;
}
size_t h_fixed_smem(int nb) { return (size_t)h_slots(nb) * 4 * h_npad_max(nb) * 128 + 1024 + 512; }
int h_in_stages(int nb) {
  const size_t per = (size_t)h_stage_rows(nb) * 512;
  const size_t room = 227 * 1024 - h_fixed_smem(nb);
  int k = (int)(room / per);
  if (k > kHMaxIn) k = kHMaxIn;
  return k >= 2 ? k : 0;
}
size_t h_smem_bytes(int nb) { return h_fixed_smem(nb) + (size_t)h_in_stages(nb) * h_stage_rows(nb) * 512; }

template <int CW, int SLOTS>
cudaError_t launch_h16(const HArgs& a, int sms, size_t smem, cudaStream_t s) {
  cudaError_t e = allow_smem(contract_h16_kernel<CW, SLOTS>);
  if (e != cudaSuccess) return e;
  contract_h16_kernel<CW, SLOTS><<<sms, kHThreads, smem, s>>>(a);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace

int h16_wave_rows(const Layout& L) { return HRows::make(L).rows; }
static int h16_wave_pitch(int T) { return (T + kHCentres - 1) / kHCentres * kHCentres; }

bool h16_supported(const Layout& L) { return L.nb >= 1 && L.nb <= 16 && h_in_stages(L.nb) >= 2; }
size_t contract_h16_wave_bytes(const Layout& L, int T) {
  return (size_t)h16_wave_rows(L) * h16_wave_pitch(T) * sizeof(float2);
}
size_t contract_h16_rowmax_bytes(const Layout& L) { return (size_t)h16_wave_rows(L) * sizeof(unsigned); }

// work items: tiles of the rows of one sg (a by a, the pairs of an a side by side)
void h16_build_items(const Basis& B, std::vector<int4>& items) {
  items.clear();
  const int tile = h_tile_rows(B.nb), groups = 4 / h_ncomp(B.nb);
  for (int g = 0; g < groups; ++g)
    for (int q = 0; q < B.nsg; ++q) {
      const int rows = B.xlen[q] * B.npairs;
      for (int r = 0; r < rows; r += tile)
        items.push_back(make_int4((g << 1) | ((B.xlo[q] + 128) << 8) | (std::min(tile, rows - r) << 16), B.sg0 + q, r,
                                  B.xbase[q]));
    }
  for (int t = 0; t <= 2 * B.N; ++t) {
    const int rows = B.wlen(t) * B.npairs;
    for (int r = 0; r < rows; r += tile)
      items.push_back(make_int4(1 | ((128 - B.N) << 8) | (std::min(tile, rows - r) << 16), -t, r, B.wbase(t)));
  }
}

cudaError_t contract_wave_h16(const Layout& L, const Basis& B, const float2* rec, const float2* xw,
                              const WavePlan& plan, double* red, const int4* items, int n_items, float2* wave,
                              unsigned* rowmax, int* status, long long timeout, cudaStream_t s) {
  if (plan.total <= 0 || plan.nseg <= 0) return cudaSuccess;
  for (int i = 0; i < plan.nseg; ++i)  // segments start at stage boundaries
    if (plan.seg[i].off % kHCentres != 0) return cudaErrorInvalidValue;
  const HRows R = HRows::make(L);
  const int rows = R.rows, pitch = h16_wave_pitch(plan.total);
  cudaError_t e = cudaMemsetAsync(rowmax, 0, (size_t)rows * sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  hwave_rowmax_kernel<<<dim3((rows + 31) / 32, (plan.total + 127) / 128), 256, 0, s>>>(L, rec, xw, plan, R, rowmax);
  hwave_transpose_kernel<<<dim3((rows + 31) / 32, pitch / 32), 256, 0, s>>>(L, rec, xw, plan, R, rowmax,
                                                                          reinterpret_cast<float*>(wave));
  g_launches += 2;
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  HArgs a;
  a.L = L; a.R = R; a.plan = plan;
  a.red = reinterpret_cast<double2*>(red); a.red_stride = B.elems(); a.red_w = B.woff();
  a.npairs = B.npairs;
  a.items = items; a.n_items = n_items;
  a.ncomp = h_ncomp(L.nb);
  a.rowmax = rowmax;
  a.wave = reinterpret_cast<const float*>(wave);
  a.in_stages = h_in_stages(L.nb);
  a.stage_rows = h_stage_rows(L.nb);
  a.npad_max = h_npad_max(L.nb);
  a.timeout = timeout; a.status = status;
  if (a.in_stages < 2) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = h_smem_bytes(L.nb);
  if (h_cw(L.nb) == 16) return launch_h16<16, 3>(a, sms, smem, s);
  if (h_cw(L.nb) == 20) return launch_h16<20, 2>(a, sms, smem, s);
  return launch_h16<24, 2>(a, sms, smem, s);
}

}  // namespace ext4pcf
