// FP64 transforms of the multipoles:
//  * real space (paper Eq. Multipole2RealConversion): for each component and radial-bin
//    triple, the angular density (2 pi)^-2 sum_n Upsilon_n e^{i n2 phi12 + i n3 phi13} is
//    integrated over n_phi x n_phi uniform angular bins, as a separable two-stage sum;
//    Gamma = Upsilon / N per bin (Eq. 4PCF_quadrupletestimator);
//  * fourth-order aperture measures (Eq. 4PCF2M4) for the filter of Eq. CrittendenQ, whose
//    aperture-centre integral is done in closed form: with vt_0 = 0, vt_1 = t1,
//    vt_2 = t2 e^{i phi12}, vt_3 = t3 e^{i phi13}, d_a = vt_a - (vt_1+vt_2+vt_3)/4,
//      F_mu = 2 pi t1 t2 t3 e^{i ph_mu} (4 pi theta^4)^-4 exp(-sum|d_a|^2 / 2theta^2) J_mu,
//      J_mu = sum_p P_p R_p pi p! (theta^2/2)^{p+1},
//    P(z^*) = prod over unconjugated apertures (z^* + d_a^*)^2, R(z) = prod over conjugated
//    apertures (z + d_a)^2, ph_mu = 2 sum_a s_a zeta_a of the x-projection (s = +-1).
#include <algorithm>
#include <mutex>

#include "common.cuh"

namespace ext4pcf {

namespace {

constexpr double kPi = 3.14159265358979323846;

// (1/2pi) * integral of e^{i n phi} over angular bin p of n_phi uniform bins
__global__ void angle_table(int N, int nphi, double2* E) {
  const int nn = 2 * N + 1;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nn * nphi; k += gridDim.x * blockDim.x) {
    const int t = k / nphi, p = k % nphi, n = t - N;
    const double lo = 2.0 * kPi * p / nphi, hi = 2.0 * kPi * (p + 1) / nphi;
    double re, im;
    if (n == 0) {
      re = (hi - lo) / (2.0 * kPi);
      im = 0.0;
    } else {
      double sh, ch, sl, cl;
      sincos(n * hi, &sh, &ch);
      sincos(n * lo, &sl, &cl);
      // (e^{in hi} - e^{in lo}) / (i n) / (2 pi)
      re = (sh - sl) / (n * 2.0 * kPi);
      im = -(ch - cl) / (n * 2.0 * kPi);
    }
    E[k] = make_double2(re, im);
  }
}

// What real_space_kernel writes: the angular-bin counts of the normalisation, their reciprocals (see
// recip_of), Upsilon / N added into gamma, or Upsilon times the reciprocals of N.
enum RealOut { kCounts, kRecips, kGammaAdd, kGammaTimes };

// One reciprocal per angular bin serves the eight components (a division is ten FP64 operations).  A
// count whose reciprocal could leave the normal range, 0, infinities and NaN stay as they are: the
// magnitude tells the two apart.
constexpr double kRecipMax = 0x1p960, kRecipMin = 0x1p-960;
__device__ __forceinline__ bool is_recip(double v) { return fabs(v) >= kRecipMin && fabs(v) <= kRecipMax; }
__device__ __forceinline__ double recip_of(double count) { return is_recip(count) ? 1.0 / count : count; }

// One block per (component, radial triple): the separable sum over n3, then n2, of
// Upsilon_n E_n2(p) E_n3(q).  E_-n = E_n^*, and the bin p' = n_phi - 1 - p mirrors p: E_n(p') =
// E_n(p)^*.  With A_n = u_n + u_-n and B_n = u_n - u_-n a sum over n is
//   u_0 E_0 + sum_{n>0} A_n Re E_n(p) + i B_n Im E_n(p)   at p, and with - i at p':
// four FP64 multiply-adds for two n at two bins where the plain sum takes sixteen.  The FP64 pipe (2
// multiply-adds per clock and SM) bounds it; shared memory and the table are far from their limits,
// so a thread simply owns one (row or bin q, bin p) at a time.  1000 triples, n_max = 20, 129
// angular bins, nine components: 95 -> 15.6 ms.
constexpr int kRealThreads = 512;
template <RealOut OUT>
__global__ void __launch_bounds__(kRealThreads, 2)
real_space_kernel(const double2* __restrict__ ups, int nb, int N, int nphi, const double2* __restrict__ E, int tri0,
                  int ntri, const double* __restrict__ norm_in, double* __restrict__ norm_out,
                  double2* __restrict__ gam_out, size_t gam_mu_stride) {
  constexpr bool kNorm = OUT == kCounts || OUT == kRecips;
  extern __shared__ double2 sm[];
  const int nn = 2 * N + 1, half = (nphi + 1) / 2;
  const int mu = kNorm ? 8 : (int)(blockIdx.x / ntri);
  const int lt = (int)(blockIdx.x % ntri), tri = tri0 + lt;
  const size_t nb3 = (size_t)nb * nb * nb;
  double2* U = sm;                 // [nn][nn]
  double2* T1 = sm + nn * nn;      // [nn][nphi]
  for (int k = threadIdx.x; k < nn * nn; k += blockDim.x) U[k] = ups[((size_t)mu * nn * nn + k) * nb3 + tri];
  __syncthreads();
  // (A_n, B_n) in the places of (u_n, u_-n)
  for (int k = threadIdx.x; k < nn * N; k += blockDim.x) {
    double2& hi = U[(k / N) * nn + N + 1 + k % N];
    double2& lo = U[(k / N) * nn + N - 1 - k % N];
    const double2 u = hi, v = lo;
    hi = make_double2(u.x + v.x, u.y + v.y);
    lo = make_double2(u.x - v.x, u.y - v.y);
  }
  __syncthreads();
  const double e0 = 1.0 / nphi;  // E_0
  for (int k = threadIdx.x; k < nn * half; k += blockDim.x) {
    const int a2 = k / half, q = k - a2 * half;
    const double2* u = U + a2 * nn + N;
    double sx = u[0].x * e0, sy = u[0].y * e0, dx = 0, dy = 0;
    for (int n = 1; n <= N; ++n) {
      const double2 e = E[(N + n) * nphi + q], A = u[n], B = u[-n];
      sx += A.x * e.x;
      sy += A.y * e.x;
      dx += B.x * e.y;
      dy += B.y * e.y;
    }
    T1[a2 * nphi + q] = make_double2(sx - dy, sy + dx);
    if (q != nphi - 1 - q) T1[a2 * nphi + nphi - 1 - q] = make_double2(sx + dy, sy - dx);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < N * nphi; k += blockDim.x) {
    const int n = 1 + k / nphi, q = k % nphi;
    double2& hi = T1[(N + n) * nphi + q];
    double2& lo = T1[(N - n) * nphi + q];
    const double2 u = hi, v = lo;
    hi = make_double2(u.x + v.x, u.y + v.y);
    lo = make_double2(u.x - v.x, u.y - v.y);
  }
  __syncthreads();
  const size_t nph2 = (size_t)nphi * nphi;
  for (int k = threadIdx.x; k < half * nphi; k += blockDim.x) {
    const int p = k / nphi, q = k - p * nphi;
    const double2* t = T1 + N * nphi + q;
    double sx = t[0].x * e0, sy = t[0].y * e0, dx = 0, dy = 0;
    for (int n = 1; n <= N; ++n) {
      const double2 e = E[(N + n) * nphi + p], A = t[n * nphi], B = t[-n * nphi];
      sx += A.x * e.x;
      dy += B.y * e.y;
      if (!kNorm) {
        sy += A.y * e.x;
        dx += B.x * e.y;
      }
    }
#pragma unroll
    for (int m = 0; m < 2; ++m) {  // p, and its mirror
      const int pm = m ? nphi - 1 - p : p;
      if (m && pm == p) break;
      const double re = m ? sx + dy : sx - dy, im = m ? sy - dx : sy + dx;
      const size_t o = (size_t)lt * nph2 + (size_t)pm * nphi + q;
      if (OUT == kCounts) {
        norm_out[o] = re;
      } else if (OUT == kRecips) {
        norm_out[o] = recip_of(re);
      } else {
        const double nv = norm_in[o];
        double2* g = gam_out + (size_t)mu * gam_mu_stride + o;
        if (OUT == kGammaTimes) {
          *g = is_recip(nv) ? make_double2(re * nv, im * nv)
                            : nv != 0.0 ? make_double2(re / nv, im / nv) : make_double2(0, 0);
        } else if (nv != 0.0) {
          double2 v = *g;
          v.x += re / nv;
          v.y += im / nv;
          *g = v;
        }
      }
    }
  }
}

__global__ void add_arrays(double* __restrict__ dst, const double* __restrict__ src, size_t n) {
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x)
    dst[k] += src[k];
}

struct Map4Args {
  int nb, nphi, n_ap, tri0, ntri;
  double tb[32];   // representative radius per bin
  double vol[32];  // A_b / tb
  double ap[64];
};

__constant__ signed char kBeta[8][4] = {{0, 0, 0, 0}, {1, 0, 0, 0}, {0, 1, 0, 0}, {0, 0, 1, 0},
                                        {0, 0, 0, 1}, {1, 1, 0, 0}, {1, 0, 1, 0}, {1, 0, 0, 1}};

__device__ __forceinline__ double2 cm(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// e^{-sum|d|^2 / 2 theta^2} is a product of three functions of one angle each: with
// sum|d|^2 = (3/4) sum t^2 - (1/2) (t1 t2 cos p12 + t1 t3 cos p13 + t2 t3 cos(p12 - p13)) and
// cos = 1 - 2 sin^2(./2) every exponent stays <= 0.  Tables [triple][3][nphi][n_ap], the constant
// factor in the first; the third by (p - q) mod nphi: 3 nphi exponentials a radius, not nphi^2.
__global__ void map4_tables(const Map4Args a, double* __restrict__ tab) {
  const int per = 3 * a.nphi * a.n_ap;
  const int lt = blockIdx.x, tri = a.tri0 + lt, nb = a.nb;
  const double t1 = a.tb[tri / (nb * nb)], t2 = a.tb[(tri / nb) % nb], t3 = a.tb[tri % nb];
  const double dphi = 2.0 * kPi / a.nphi;
  const double base = 0.75 * (t1 * t1 + t2 * t2 + t3 * t3) - 0.5 * (t1 * t2 + t1 * t3 + t2 * t3);
  for (int k = threadIdx.x; k < per; k += blockDim.x) {
    const int w = k / (a.nphi * a.n_ap), p = (k / a.n_ap) % a.nphi, ia = k % a.n_ap;
    const double sh = sin(0.5 * (w == 2 ? p : p + 0.5) * dphi);
    const double tt = w == 0 ? t1 * t2 : w == 1 ? t1 * t3 : t2 * t3;
    const double x = tt * sh * sh + (w == 0 ? base : 0.0);
    const double th = a.ap[ia];
    tab[(size_t)lt * per + k] = exp(-x / (2.0 * th * th));
  }
}

// e^{i phi} at the middle of every angular bin
__global__ void map4_turns(int nphi, double2* __restrict__ turn) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nphi) return;
  double sn, cs;
  sincos((p + 0.5) * (2.0 * kPi / nphi), &sn, &cs);
  turn[p] = make_double2(cs, sn);
}

// The aperture integral of one radial triple over a slice of the angular bins.  The integrand is
// Gamma_mu times C_{mu,t} = geo e^{i ph_mu} P_t R_t (t <= min(deg P, deg R): 0 for mu = 0, 2 for one
// conjugated aperture, 4 for two: 28 coefficients) times the exponential and, at the end, the
// radius' factor of t.  Mirroring both angles conjugates the d_a and so every C, and leaves the
// exponential: the bins k and n_phi^2 - 1 - k are taken together,
//   Gamma C + Gamma' C^* = (Gamma + Gamma') Re C + i (Gamma - Gamma') Im C.
// Tiles of kM4Bins such pairs: one thread a pair forms all 28 coefficients (the products of the
// d_a shared by the components; sum d_a = 0 gives half of them), then a thread per coefficient and
// group of radii folds the tile into its sums.  FP64 multiply-adds bound it: 56 a pair and radius
// for the sums, about 500 a pair for the coefficients.  1000 triples, 129 angular bins, 24 radii:
// 198 -> 29.3 ms.
constexpr int kM4Bins = 128;    // bin pairs per tile
constexpr int kM4Row = kM4Bins + 1;  // a column of coefficients falls on different banks
constexpr int kM4Coef = 28;     // (mu, t)
constexpr int kM4Groups = 8;    // threads per coefficient
constexpr int kM4Threads = kM4Coef * kM4Groups;
constexpr int kM4Radii = 8;     // radii per thread: 64 / kM4Groups
// first coefficient of component mu
__host__ __device__ constexpr int m4_first(int mu) { return mu == 0 ? 0 : mu < 5 ? 1 + 3 * (mu - 1) : 13 + 5 * (mu - 5); }
static_assert(m4_first(8) == kM4Coef, "coefficients");

__device__ __forceinline__ double2 conj2(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sc2(double s, double2 a) { return make_double2(s * a.x, s * a.y); }

__global__ void __launch_bounds__(kM4Threads, 2) map4_kernel(const Map4Args a, const double2* __restrict__ gam,
                                                          size_t gam_mu_stride, const double* __restrict__ tab,
                                                          const double2* __restrict__ turn, int nsplit,
                                                          double2* __restrict__ partial) {
  extern __shared__ double2 m4s[];
  double2* coef = m4s;                                             // [kM4Coef][kM4Row]
  double* exs = reinterpret_cast<double*>(coef + kM4Coef * kM4Row);  // [n_ap][kM4Bins]
  const int nphi = a.nphi, n_ap = a.n_ap, nb = a.nb, tid = threadIdx.x;
  const long long nph2 = (long long)nphi * nphi, halfn = (nph2 + 1) / 2;
  const int lt = blockIdx.x / nsplit, split = blockIdx.x % nsplit, tri = a.tri0 + lt;
  const int b1 = tri / (nb * nb), b2 = (tri / nb) % nb, b3 = tri % nb;
  const double t1 = a.tb[b1], t2 = a.tb[b2], t3 = a.tb[b3];
  const double dphi = 2.0 * kPi / nphi;
  const double geo = 2.0 * kPi * t1 * t2 * t3 * a.vol[b1] * a.vol[b2] * a.vol[b3] * dphi * dphi;
  const double* tb = tab + (size_t)lt * 3 * nphi * n_ap;
  const long long kbeg = halfn * split / nsplit, kend = halfn * (split + 1) / nsplit;
  // this thread's coefficient, radii and (few radii) part of every tile
  const int c = tid % kM4Coef, grp = tid / kM4Coef;
  const int lanes = min(kM4Groups, n_ap), parts = kM4Groups / lanes, part = grp / lanes, ia0 = grp % lanes;
  const bool sums = part < parts;
  double2 acc[kM4Radii];
#pragma unroll
  for (int r = 0; r < kM4Radii; ++r) acc[r] = make_double2(0, 0);
  for (long long k0 = kbeg; k0 < kend; k0 += kM4Bins) {
    const int nk = (int)min((long long)kM4Bins, kend - k0);
    __syncthreads();  // the previous tile is done with
    if (tid < nk) {
      const long long k = k0 + tid, km = nph2 - 1 - k;
      const int p = (int)(k / nphi), q = (int)(k % nphi);
      const double2 e2 = turn[p], e3 = turn[q];
      // the neighbours' places less a quarter of their sum: d_0 .. d_3, and their conjugates u_a
      const double2 v2 = sc2(t2, e2), v3 = sc2(t3, e3);
      const double2 cen = make_double2(0.25 * (t1 + v2.x + v3.x), 0.25 * (v2.y + v3.y));
      const double2 d[4] = {make_double2(-cen.x, -cen.y), make_double2(t1 - cen.x, -cen.y),
                            make_double2(v2.x - cen.x, v2.y - cen.y), make_double2(v3.x - cen.x, v3.y - cen.y)};
      // products of two: q01 .. q23 of the d_a (those of the u_a are their conjugates)
      const double2 q01 = cm(d[0], d[1]), q02 = cm(d[0], d[2]), q03 = cm(d[0], d[3]), q12 = cm(d[1], d[2]),
                    q13 = cm(d[1], d[3]), q23 = cm(d[2], d[3]);
      // phases e^{i ph_mu}, from e^{2 i p12}, e^{i p13}, e^{3 i p13}, with the geometric factor
      const double2 e22 = sc2(geo, cm(e2, e2)), e33 = cm(cm(e3, e3), e3);
      const double2 f23 = cm(e22, e33), f21 = cm(e22, e3), f2m1 = cm(e22, conj2(e3)), f2m3 = cm(e22, conj2(e33));
      auto put = [&](int mu, int t, double2 C) {
        // (Gamma + Gamma') Re C + i (Gamma - Gamma') Im C; the middle bin is its own mirror
        const double2 g = gam[(size_t)mu * gam_mu_stride + (size_t)lt * nph2 + k];
        const double2 h = km != k ? gam[(size_t)mu * gam_mu_stride + (size_t)lt * nph2 + km] : make_double2(0, 0);
        const double sx = g.x + h.x, sy = g.y + h.y, dx = g.x - h.x, dy = g.y - h.y;
        coef[(m4_first(mu) + t) * kM4Row + tid] = make_double2(sx * C.x - dy * C.y, sy * C.x + dx * C.y);
      };
      {  // mu = 0: (u_0 u_1 u_2 u_3)^2
        const double2 P = conj2(cm(q01, q23));
        put(0, 0, cm(f23, cm(P, P)));
      }
      // one conjugated aperture c, the others' u: E_0 = their product, E_1 their products of two, E_2
      // their sum = -u_c; P = (E_0^2, 2 E_0 E_1, E_1^2 + 2 E_0 E_2), R = (d_c^2, 2 d_c, 1)
      auto one = [&](int mu, double2 dc, double2 pa, double2 pb, double2 pc, double2 third, double2 ph) {
        const double2 E0 = conj2(cm(pa, third)), E1 = conj2(add2(add2(pa, pb), pc));
        const double2 E0d = cm(E0, dc);
        put(mu, 0, cm(ph, cm(E0d, E0d)));
        put(mu, 1, sc2(4.0, cm(ph, cm(E0d, E1))));
        const double2 w = cm(E0, conj2(dc)), s = cm(E1, E1);
        put(mu, 2, cm(ph, make_double2(s.x - 2.0 * w.x, s.y - 2.0 * w.y)));
      };
      one(1, d[0], q12, q13, q23, d[3], f21);
      one(2, d[1], q02, q03, q23, d[3], f23);
      one(3, d[2], q01, q03, q13, d[3], conj2(f2m3));
      one(4, d[3], q01, q02, q12, d[2], f2m1);
      // two conjugated: p = u_a u_b, s = u_a + u_b, p' = d_c d_e, s' = d_c + d_e = -s^*:
      // P R = (p p')^2, 4 p p' s s', (s^2 + 2 p)(s'^2 + 2 p'), 4 s s', 1
      auto two = [&](int mu, double2 pu, double2 s, double2 pd, double2 ph) {
        const double2 pp = cm(pu, pd);
        const double ss = -(s.x * s.x + s.y * s.y);  // s s'
        put(mu, 0, cm(ph, cm(pp, pp)));
        put(mu, 1, sc2(4.0 * ss, cm(ph, pp)));
        const double2 s2 = cm(s, s), x = make_double2(s2.x + 2.0 * pu.x, s2.y + 2.0 * pu.y),
                      y = make_double2(s2.x + 2.0 * pd.x, -s2.y + 2.0 * pd.y);  // s'^2 = (s^2)^*
        put(mu, 2, cm(ph, cm(x, y)));
        put(mu, 3, sc2(4.0 * ss, ph));
        put(mu, 4, ph);
      };
      two(5, conj2(q23), conj2(add2(d[2], d[3])), q01, f21);
      two(6, conj2(q13), conj2(add2(d[1], d[3])), q02, conj2(f2m1));
      two(7, conj2(q12), conj2(add2(d[1], d[2])), q03, f2m3);
    }
    // exponentials of the tile, zero past its end
    for (int w = tid; w < kM4Bins * n_ap; w += kM4Threads) {
      const int ia = w / kM4Bins, j = w % kM4Bins;
      double e = 0.0;
      if (j < nk) {
        const long long k = k0 + j;
        const int p = (int)(k / nphi), q = (int)(k % nphi), pq = p >= q ? p - q : p - q + nphi;
        e = tb[p * n_ap + ia] * tb[(nphi + q) * n_ap + ia] * tb[(2 * nphi + pq) * n_ap + ia];
      }
      exs[ia * kM4Bins + j] = e;
    }
    __syncthreads();
    if (sums) {
      const int j0 = nk * part / parts, j1 = nk * (part + 1) / parts;
#pragma unroll
      for (int r = 0; r < kM4Radii; ++r) {
        const int ia = ia0 + r * lanes;
        if (ia >= n_ap) break;
        double2 s = acc[r];
        const double2* cf = coef + c * kM4Row;
        const double* ex = exs + ia * kM4Bins;
        for (int j = j0; j < j1; ++j) {
          s.x += cf[j].x * ex[j];
          s.y += cf[j].y * ex[j];
        }
        acc[r] = s;
      }
    }
  }
  // the radius' factors pi t! h^{t+1} / (4 pi theta^4)^4, then the sum over t and parts
  __syncthreads();
  double2* tot = m4s;  // [parts][n_ap][kM4Coef]
#pragma unroll
  for (int r = 0; r < kM4Radii; ++r) {
    const int ia = ia0 + r * lanes;
    if (!sums || ia >= n_ap) break;
    const int t = c == 0 ? 0 : c < 13 ? (c - 1) % 3 : (c - 13) % 5;
    const double th2 = a.ap[ia] * a.ap[ia], h = 0.5 * th2, q0 = 4.0 * kPi * th2 * th2;
    double f = kPi * h / (q0 * q0 * q0 * q0);
    for (int i = 1; i <= t; ++i) f *= i * h;
    tot[((size_t)part * n_ap + ia) * kM4Coef + c] = sc2(f, acc[r]);
  }
  __syncthreads();
  for (int w = tid; w < 8 * n_ap; w += kM4Threads) {
    const int ia = w / 8, mu = w % 8;
    double2 s = make_double2(0, 0);
    for (int pt = 0; pt < parts; ++pt)
      for (int i = m4_first(mu); i < m4_first(mu + 1); ++i) s = add2(s, tot[((size_t)pt * n_ap + ia) * kM4Coef + i]);
    partial[(((size_t)tri * nsplit + split) * n_ap + ia) * 8 + mu] = s;
  }
}

}  // namespace

namespace {
template <RealOut OUT>
cudaError_t launch_real(int blocks, size_t smem, cudaStream_t s, const double2* U, int nb, int N, int nphi,
                        const double2* E, int tri0, int ntri, const double* norm_in, double* norm_out, double2* gam,
                        size_t stride) {
  cudaError_t e = allow_smem(real_space_kernel<OUT>);
  if (e != cudaSuccess) return e;
  real_space_kernel<OUT><<<blocks, kRealThreads, smem, s>>>(U, nb, N, nphi, E, tri0, ntri, norm_in, norm_out, gam,
                                                            stride);
  ++g_launches;
  return cudaGetLastError();
}
}  // namespace

cudaError_t real_space(const double* ups, int nb, int N, int nphi, double* gamma, double* norm,
                       double* scratch_norm, double* E_scratch, cudaStream_t s) {
  const int nn = 2 * N + 1;
  const int ntri = nb * nb * nb;
  angle_table<<<64, 256, 0, s>>>(N, nphi, reinterpret_cast<double2*>(E_scratch));
  const size_t smem = (size_t)(nn * nn + nn * nphi) * sizeof(double2);
  const double2* U = reinterpret_cast<const double2*>(ups);
  const double2* E = reinterpret_cast<const double2*>(E_scratch);
  const size_t stride = (size_t)ntri * nphi * nphi;
  cudaError_t e = launch_real<kCounts>(ntri, smem, s, U, nb, N, nphi, E, 0, ntri, nullptr, scratch_norm, nullptr, 0);
  if (e != cudaSuccess) return e;
  e = launch_real<kGammaAdd>(8 * ntri, smem, s, U, nb, N, nphi, E, 0, ntri, scratch_norm, nullptr,
                             reinterpret_cast<double2*>(gamma), stride);
  if (e != cudaSuccess) return e;
  add_arrays<<<1024, 256, 0, s>>>(norm, scratch_norm, stride);
  return cudaGetLastError();
}

size_t real_space_smem(int N, int nphi) {
  const int nn = 2 * N + 1;
  return (size_t)(nn * nn + nn * nphi) * sizeof(double2);
}

// bytes of scratch next to the Gamma chunk: e^{i phi} per bin and the exponential tables of a chunk
size_t map4_table_bytes(int chunk_tri, int nphi, int n_ap) {
  return (size_t)nphi * sizeof(double2) + (size_t)chunk_tri * 3 * nphi * n_ap * sizeof(double);
}

// Radial triples of one chunk: 256 MB of Gamma and tables, and whole rounds of two blocks per SM of
// real_space_kernel (8 blocks a triple) where that leaves at least one.
int map4_chunk(int ntri, int nphi, int n_ap, int sms) {
  const size_t per = (size_t)nphi * nphi * 8 * sizeof(double2) + (size_t)3 * nphi * n_ap * sizeof(double);
  const size_t fit = std::max<size_t>(1, (size_t)(256u << 20) / per);
  if (fit >= (size_t)ntri) return ntri;
  const size_t round = std::max(1, 2 * sms / 8);
  return fit < round ? (int)fit : (int)(fit / round * round);
}

// Aperture measures: triples processed in chunks; returns per-(triple, slice, aperture)
// partial sums in `partial` [ntri][nsplit][n_ap][8] complex, the angular bins of each
// triple split into nsplit slices: 8 as the real-space blocks of the triple, more for a small chunk.
int map4_nsplit(int chunk_tri, int ntri, int n_ap, int sms) {
  int ns = std::max(8, (4 * sms + chunk_tri - 1) / chunk_tri);
  const size_t cap = (size_t)(256u << 20) / ((size_t)ntri * n_ap * 8 * 16);
  if ((size_t)ns > cap) ns = (int)cap;
  return ns < 1 ? 1 : (ns > 16 ? 16 : ns);
}

cudaError_t map4_partials(const double* ups, const double* edges_host, int nb, int N, int nphi,
                          const double* ap_host, int n_ap, double* E_scratch, double* norm_chunk,
                          double* gam_chunk, double* tables, int chunk_tri, int nsplit, double* partial,
                          cudaStream_t s) {
  const int nn = 2 * N + 1;
  const int ntri = nb * nb * nb;
  angle_table<<<64, 256, 0, s>>>(N, nphi, reinterpret_cast<double2*>(E_scratch));
  ++g_launches;
  const size_t smem = (size_t)(nn * nn + nn * nphi) * sizeof(double2);
  const size_t smem4 = kM4Coef * kM4Row * sizeof(double2) + kM4Bins * (size_t)n_ap * sizeof(double);
  // (the sums at the end, [parts][n_ap][kM4Coef] with parts n_ap <= 8 or parts = 1, fit in it)
  static_assert(kM4Groups <= kM4Bins && 64 <= kM4Bins, "sums");
  cudaError_t e = allow_smem(map4_kernel);
  if (e != cudaSuccess) return e;
  Map4Args a;
  a.nb = nb; a.nphi = nphi; a.n_ap = n_ap;
  for (int b = 0; b < nb; ++b) {
    const double lo = edges_host[b], hi = edges_host[b + 1];
    a.tb[b] = (2.0 / 3.0) * (hi * hi * hi - lo * lo * lo) / (hi * hi - lo * lo);
    a.vol[b] = 0.5 * (hi * hi - lo * lo) / a.tb[b];
  }
  for (int k = 0; k < n_ap; ++k) a.ap[k] = ap_host[k];
  const double2* U = reinterpret_cast<const double2*>(ups);
  const double2* E = reinterpret_cast<const double2*>(E_scratch);
  double2* turn = reinterpret_cast<double2*>(tables);
  double* tab = tables + 2 * (size_t)nphi;
  double2* gam = reinterpret_cast<double2*>(gam_chunk);
  const size_t nph2 = (size_t)nphi * nphi;
  map4_turns<<<(nphi + 127) / 128, 128, 0, s>>>(nphi, turn);
  ++g_launches;
  for (int t0 = 0; t0 < ntri; t0 += chunk_tri) {
    const int nt = min(chunk_tri, ntri - t0);
    const size_t stride = (size_t)nt * nph2;
    e = launch_real<kRecips>(nt, smem, s, U, nb, N, nphi, E, t0, nt, nullptr, norm_chunk, nullptr, 0);
    if (e != cudaSuccess) return e;
    e = launch_real<kGammaTimes>(8 * nt, smem, s, U, nb, N, nphi, E, t0, nt, norm_chunk, nullptr, gam, stride);
    if (e != cudaSuccess) return e;
    a.tri0 = t0; a.ntri = nt;
    map4_tables<<<nt, 256, 0, s>>>(a, tab);
    map4_kernel<<<nt * nsplit, kM4Threads, smem4, s>>>(a, gam, stride, tab, turn, nsplit,
                                                       reinterpret_cast<double2*>(partial));
    g_launches += 2;
  }
  return cudaGetLastError();
}

namespace {

// Sum the partials over triples and slices (fixed order), then the E/B split and the
// Gaussian part.
constexpr int kM4FinThreads = 512;
__global__ void __launch_bounds__(kM4FinThreads) map4_finish(const double2* __restrict__ partial, int nunits, int n_ap,
                            const double* __restrict__ xipm, const double* __restrict__ tb,
                            const double* __restrict__ area, int nb, const double* __restrict__ ap,
                            double* __restrict__ m4, double* __restrict__ eb, double* __restrict__ disc) {
  const int ia = blockIdx.x;
  __shared__ double2 mm[8];
  __shared__ double2 D[16];
  __shared__ double2 run[kM4FinThreads];
  {  // thread (stretch of the units, component), then the stretches in order
    const int mu = threadIdx.x % 8, st = threadIdx.x / 8, ns = kM4FinThreads / 8;
    const int u0 = (int)((long long)nunits * st / ns), u1 = (int)((long long)nunits * (st + 1) / ns);
    double re = 0, im = 0;
    for (int t = u0; t < u1; ++t) {
      const double2 v = partial[((size_t)t * n_ap + ia) * 8 + mu];
      re += v.x; im += v.y;
    }
    run[threadIdx.x] = make_double2(re, im);
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    double re = 0, im = 0;
    for (int st = 0; st < kM4FinThreads / 8; ++st) {
      const double2 v = run[8 * st + threadIdx.x];
      re += v.x; im += v.y;
    }
    mm[threadIdx.x] = make_double2(re, im);
    m4[16 * ia + 2 * threadIdx.x] = re;
    m4[16 * ia + 2 * threadIdx.x + 1] = im;
  }
  __syncthreads();
  // all 16 conjugation patterns: the 8 computed ones and their complex conjugates
  if (threadIdx.x == 0) {
    for (int mu = 0; mu < 8; ++mu) {
      int code = 0, ccode = 0;
      for (int j = 0; j < 4; ++j) { code = 2 * code + kBeta[mu][j]; ccode = 2 * ccode + (1 - kBeta[mu][j]); }
      D[code] = mm[mu];
      D[ccode] = make_double2(mm[mu].x, -mm[mu].y);
    }
  }
  __syncthreads();
  // component c: bits of the label "t/x" for apertures 0..3 in the order of
  // Eq. 4PCF_rawcomponents (x = 1)
  const unsigned char lab[16] = {0x0, 0x8, 0x4, 0x2, 0x1, 0x3, 0x5, 0x6, 0x9, 0xA, 0xC, 0x7, 0xB, 0xD, 0xE, 0xF};
  if (threadIdx.x < 16) {
    const int c = threadIdx.x;
    double re = 0;
    for (int code = 0; code < 16; ++code) {
      // coefficient prod_a (t: 1/2; x: unconj -i/2, conj +i/2)
      double cr = 1, ci = 0;
      for (int j = 0; j < 4; ++j) {
        const bool isx = (lab[c] >> (3 - j)) & 1;
        const bool cj = (code >> (3 - j)) & 1;
        double fr, fi;
        if (!isx) { fr = 0.5; fi = 0; } else { fr = 0; fi = cj ? 0.5 : -0.5; }
        const double nr = cr * fr - ci * fi;
        ci = cr * fi + ci * fr;
        cr = nr;
      }
      re += cr * D[code].x - ci * D[code].y;
    }
    eb[16 * ia + c] = re;
  }
  __syncthreads();
  if (disc && xipm) {
    if (threadIdx.x == 0) {
      const double th = ap[ia];
      double Ar = 0, Ai = 0, Bp = 0;
      for (int b = 0; b < nb; ++b) {
        // xi_+ = sum x^* G_0 / sum w W_0, xi_- = sum x G_-4 / sum w W_0
        const double den = xipm[6 * b + 4];
        if (den == 0.0) continue;
        const double x = tb[b] / th, g = exp(-0.25 * x * x);
        const double Tp = (x * x * x * x - 16.0 * x * x + 32.0) / 128.0 * g;
        const double Tm = x * x * x * x / 128.0 * g;
        Bp += xipm[6 * b] / den * Tp * area[b] / (th * th);
        Ar += xipm[6 * b + 2] / den * Tm * area[b] / (th * th);
        Ai += xipm[6 * b + 3] / den * Tm * area[b] / (th * th);
      }
      for (int code = 0; code < 16; ++code) {
        int be[4];
        for (int j = 0; j < 4; ++j) be[j] = (code >> (3 - j)) & 1;
        double2 pr[4][4];
        for (int x = 0; x < 4; ++x)
          for (int y = 0; y < 4; ++y)
            pr[x][y] = (be[x] == be[y]) ? make_double2(Ar, be[x] ? -Ai : Ai) : make_double2(Bp, 0.0);
        const double2 a1 = cm(pr[0][1], pr[2][3]), a2 = cm(pr[0][2], pr[1][3]), a3 = cm(pr[0][3], pr[1][2]);
        D[code] = make_double2(a1.x + a2.x + a3.x, a1.y + a2.y + a3.y);
      }
    }
    __syncthreads();
    if (threadIdx.x < 16) {
      const int c = threadIdx.x;
      double re = 0;
      for (int code = 0; code < 16; ++code) {
        double cr = 1, ci = 0;
        for (int j = 0; j < 4; ++j) {
          const bool isx = (lab[c] >> (3 - j)) & 1;
          const bool cj = (code >> (3 - j)) & 1;
          double fr, fi;
          if (!isx) { fr = 0.5; fi = 0; } else { fr = 0; fi = cj ? 0.5 : -0.5; }
          const double nr = cr * fr - ci * fi;
          ci = cr * fi + ci * fr;
          cr = nr;
        }
        re += cr * D[code].x - ci * D[code].y;
      }
      disc[16 * ia + c] = re;
    }
  }
}

}  // namespace

cudaError_t map4_finish_launch(const double* partial, int ntri, int n_ap, const double* d_xipm,
                               const double* d_tb, const double* d_area, int nb, const double* d_ap,
                               double* d_m4, double* d_eb, double* d_disc, cudaStream_t s) {
  map4_finish<<<n_ap, kM4FinThreads, 0, s>>>(reinterpret_cast<const double2*>(partial), ntri, n_ap, d_xipm, d_tb,
                                  d_area, nb, d_ap, d_m4, d_eb, d_disc);
  ++g_launches;
  return cudaGetLastError();
}


// ---------------------------------------------------------------------------------------
// Real-space transform that allocates nothing.
//
// Some callers cannot call cudaMalloc: code running while a CUDA graph is being captured
// with a relaxed allocator policy, plug-ins whose host application owns all device memory,
// and real-time loops that must not block in the allocator.  For them this entry point
// keeps its scratch (the angular-bin table and the per-bin normalisation counts) in one
// file-scope device array of kStaticScratchBytes, held by every GPU that loads the library
// until the process exits.  Its address is looked up once per device with
// cudaGetSymbolAddress (the host symbol is only a stand-in and must not be passed to a
// kernel).  Every call shares the array: calls that overlap on the GPU race.  Both scratch
// regions are fully overwritten by each call before they are read, so nothing needs to be
// cleared.
// ---------------------------------------------------------------------------------------
namespace {
constexpr size_t kStaticScratchBytes = 16u << 20;  // 16 MiB
__device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

std::mutex g_static_mutex;
void* g_static_ptr[64] = {};

// address of the static scratch on the current device (set-up on first use per device)
cudaError_t static_scratch_ptr(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return e;
    g_static_ptr[dev] = p;
  }
  *out = g_static_ptr[dev];
  return cudaSuccess;
}

bool device_resident(const void* p) {
  if (!p) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}
}  // namespace

size_t real_space_smem(int N, int nphi);
cudaError_t real_space(const double* ups, int nb, int N, int nphi, double* gamma, double* norm,
                       double* scratch_norm, double* E_scratch, cudaStream_t s);

}  // namespace ext4pcf

extern "C" EXT4PCF_API int ext4pcf_to_real_space_noalloc(const double* upsilon, int n_bins, int n_max,
                                                         int n_phi, double* gamma, double* norm,
                                                         void* stream) {
  using namespace ext4pcf;
  if (!upsilon || !gamma || !norm) return EXT4PCF_E_INVALID_ARG;
  if (n_bins < 1 || n_bins > 32 || n_max < 0 || n_max > 40 || n_phi < 1 || n_phi > 1024)
    return EXT4PCF_E_INVALID_ARG;
  const size_t table_bytes = (size_t)(2 * n_max + 1) * n_phi * 16;
  const size_t norm_bytes = (size_t)n_bins * n_bins * n_bins * n_phi * n_phi * 8;
  const size_t table_off = (norm_bytes + 255) / 256 * 256;
  if (table_off + table_bytes > kStaticScratchBytes) return EXT4PCF_E_UNSUPPORTED;
  if (real_space_smem(n_max, n_phi) > 227 * 1024) return EXT4PCF_E_UNSUPPORTED;
  if (!device_resident(upsilon) || !device_resident(gamma) || !device_resident(norm))
    return EXT4PCF_E_INVALID_ARG;
  void* base = nullptr;
  if (static_scratch_ptr(&base) != cudaSuccess) return EXT4PCF_E_CUDA;
  unsigned char* b = static_cast<unsigned char*>(base);
  cudaError_t e = real_space(upsilon, n_bins, n_max, n_phi, gamma, norm, reinterpret_cast<double*>(b),
                             reinterpret_cast<double*>(b + table_off), static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? EXT4PCF_OK : EXT4PCF_E_CUDA;
}
