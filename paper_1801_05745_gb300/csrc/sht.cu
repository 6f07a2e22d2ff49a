// Spherical-harmonic analysis of a HEALPix RING map and its angular power
// spectrum (the full-sky C_l of Sec. 3.2, whose covariance over realisations
// Eq. 10-11 estimates):
//   a_lm = (4 pi / N_pix) sum_p map_p Y*_lm(theta_p, phi_p),  0 <= m <= l <= lmax,
//   C_l  = (|a_l0|^2 + 2 sum_{m>0} |a_lm|^2) / (2l + 1),
// evaluated ring by ring in FP64, with the long sums and recurrences in
// double-float (pairs of FP32, about 48 bits) on the FP32 pipe:
//   k_sht_tables     : the 8 Nside unit roots e^{-2 pi i j / (8 Nside)} and the
//                      one-dimensional tables from which every recurrence
//                      coefficient and normalisation is a product.
//   k_ring_transform : per ring, F_m = sum_j map_j e^{-i m phi_j}
//                      = e^{-i m phi_0} X_{m mod n}, X the ring's DFT
//                      (sht_ring.cu); F stored m-major.
//   k_lmm            : lambda_mm(z) of every north/south ring pair for every m,
//                      as mantissa x 2^exponent (no underflow near the poles).
//   k_legendre       : per (m, chunk of ring pairs) the recurrence over l of
//                      rescaled Legendre functions, the pair's even/odd
//                      combination of F, and a block reduction over the pairs
//                      -> a_lm (or partial a_lm of a chunk).
//   k_alm_sum        : a_lm from the chunk partials.
//   k_alm2cl         : C_l.
// a_lm is stored m-major (index m (2 lmax + 1 - m) / 2 + l) as FP64 (re, im).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sht_common.cuh"

namespace ufc {

constexpr int kLegChunkL = 64;         // l values per round (two barriers, or one): 32 cost
                                       // 1.5% more

// v * f, the exact product of the high parts plus the cross terms (not
// renormalised); nv = -v.h
__device__ __forceinline__ dfx dfx_mul_raw(dfx v, dfx f) {
  const u64 p = x2_mul(v.h, f.h);
  u64 e = x2_fma(v.h, f.h, x2_neg(p));
  e = x2_fma(v.h, f.l, e);
  return {p, x2_fma(v.l, f.h, e)};
}
// acc += v * f, the low part not renormalised; nv = -v.h (the product is
// formed negated, so that its error is one fused multiply-add without a
// sign change, and subtracted)
__device__ __forceinline__ void dfx_mac(dfx& acc, dfx v, u64 nv, dfx f) {
  const u64 pn = x2_mul(nv, f.h);
  u64 e = x2_fma(v.h, f.h, pn);
  e = x2_fma(v.h, f.l, e);
  e = x2_fma(v.l, f.h, e);
  const u64 s = x2_sub(acc.h, pn);
  const u64 bb = x2_sub(s, acc.h);
  const u64 er = x2_sub(x2_sub(acc.h, x2_sub(s, bb)), x2_add(pn, bb));
  acc.h = s;
  acc.l = x2_add(acc.l, x2_add(er, e));
}
// One step of the Legendre recurrence: (v2, v1) <- (v1, (a z) v1 + v2) with z
// a whole number (the ring heights times 3 N^2; a carries the division);
// nv = -v1.h.  18 packed operations.
__device__ __forceinline__ void leg_step(dfx& v1, dfx& v2, u64 nv, dfx a, u64 z) {
  dfx c;
  c.h = x2_mul(a.h, z);
  c.l = x2_fma(a.l, z, x2_fma(a.h, z, x2_neg(c.h)));
  const u64 pn = x2_mul(c.h, nv);
  u64 e = x2_fma(c.h, v1.h, pn);
  e = x2_fma(c.h, v1.l, e);
  e = x2_fma(c.l, v1.h, e);
  const u64 s = x2_sub(v2.h, pn);
  const u64 bb = x2_sub(s, v2.h);
  const u64 er = x2_sub(x2_sub(v2.h, x2_sub(s, bb)), x2_add(pn, bb));
  const u64 lo = x2_add(er, x2_add(e, v2.l));
  v2 = v1;
  v1.h = x2_add(s, lo);
  v1.l = x2_add(lo, x2_sub(s, v1.h));
}

// ------------------------------------------------------ Legendre tables --
// z lambda_lm = eps_{l+1} lambda_{l+1,m} + eps_l lambda_{l-1,m} with
// eps_l^2 = (l^2 - m^2) / (4 l^2 - 1).  Written for lambda_lm = alpha_l q_l
// with alpha_m = alpha_{m+1} = 1 and alpha_{l+1} = -alpha_{l-1} eps_l / eps_{l+1}
// the recurrence has one coefficient instead of two,
//   q_{l+1} = a_l z q_l + q_{l-1},  a_l = alpha_l / (eps_{l+1} alpha_{l+1}),
// (two products and one sum in double-float instead of three and one; the
// rescaling by alpha_l is one FP64 product per a_lm).  The products telescope:
// with w(k) = (2k-1)!!/(2k)!!, W_k = w(k), V_k = 1 / ((2k+1) w(k)) and
// k = floor((l - m) / 2),
//   l - m even: alpha_l^2 = W_k W_{m+k} (2l+1) / (W_m (2m+1)),
//   l - m odd : alpha_l^2 = V_k V_{m+k} (2l+1) W_m (2m+1) / (2m+3),
//   |a_l| = sqrt(2m+3) alpha_l^2,
// so alpha and a are products of one-dimensional tables (SW = sqrt(W),
// SV = sqrt(V), SL_l = sqrt(2l+1)) and no FP64 division or square root is
// left per (l, m).  alpha has the sign + + - - of (l - m) mod 4, a that of
// + - + -.  The ring heights are whole numbers over 3 N^2 (z = 1 - i^2 / (3 N^2)
// in the caps, 2 N (2N - i) / (3 N^2) in the belt, all below 2^22), so they
// enter the recurrence exactly as one FP32 number and a is divided by 3 N^2.
// Also lambda_mm = (-1)^m sqrt((2m+1) w(m) / (4 pi)) sin^m(theta).
struct ShtTables {
  const float4* roots;     // [8 N] e^{-2 pi i j / (8N)}
  const double* sw;        // [lmax + 2] sqrt(w(k))
  const double* sv;        // [lmax + 2] sqrt(V_k)
  const double* sl;        // [lmax + 2] sqrt(2 l + 1)
  const double* cm;        // [lmax + 2] (-1)^m sqrt((2m+1) w(m) / (4 pi))
  const float4* pair;      // [2 N] (3 N^2 z, z, sin(theta), 0) of the northern rings
  double inv_z;            // 1 / (3 N^2)
};
constexpr int kShtTab = 4 * kShtMaxNside + 2;     // entries of the one-dimensional tables

// w(k) = Gamma(k + 1/2) / (sqrt(pi) Gamma(k + 1)): exact below 24 (binomial
// C(2k, k) / 4^k, integers under 2^53), above by the asymptotic series of
// Gamma(x + 1/4) / Gamma(x + 3/4), x = k + 1/4, in 1/x^2 (from the Bernoulli
// polynomials at 1/4; the first term left out is below 2^-75 at x = 24).
struct Binomials { double c[24]; };             // C(2k, k)
constexpr Binomials make_binomials() {
  Binomials b{};
  long long c = 1;
  for (int k = 0; k < 24; ++k) {
    b.c[k] = (double)c;
    c = c * (2 * (2 * k + 1)) / (k + 1);
  }
  return b;
}
__constant__ const Binomials kBinom = make_binomials();
__device__ __forceinline__ double sht_w(int k) {
  if (k < 24) return ldexp(kBinom.c[k], -2 * k);
  const double x = (double)k + 0.25, y = 1.0 / (x * x);
  double p = 7426362705.0 / 1099511627776.0;
  p = fma(p, y, -20898423.0 / 8589934592.0);
  p = fma(p, y, 180323.0 / 134217728.0);
  p = fma(p, y, -671.0 / 524288.0);
  p = fma(p, y, 21.0 / 8192.0);
  p = fma(p, y, -1.0 / 64.0);
  const double r = 0.56418958354775628695 / sqrt(x);      // 1 / sqrt(pi x)
  return fma(p * y, r, r);
}

// All tables of one call.  Unit roots e^{-2 pi i j / (8N)}, j < 8N, as double-float
// complex numbers (FP64 sincospi, split once).  Every power-of-two ring (n = 4N, or
// n = 4i with i a power of two) has n | 8N: its FFT twiddles are T[k 8N/n] and the
// phase of its first pixel, e^{-i m phi_0} with phi_0 = pi/n, is T[m 4N/n mod 8N].
// Each FP64 chain has threads of its own (the kernel is latency: one thread per index
// with all of them, and the binomials of w by a loop of divisions, took 21 us at Nside
// 64, 8 now).
__global__ void __launch_bounds__(64)
k_sht_tables(int32_t N, int32_t lmax, float4* __restrict__ T, double* __restrict__ tab,
             float4* __restrict__ pair, double* __restrict__ sin_d, int* __restrict__ bad) {
  const int n8 = 8 * N, nl = (lmax + 2 + 31) / 32 * 32;              // (whole warps per part)
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j == 0) *bad = 0;
  if (j < n8) {
    double sn, cs;
    sincospi(-2.0 * (double)j / (double)n8, &sn, &cs);
    T[j] = cdf_pack(df_from_d(cs), df_from_d(sn));
    return;
  }
  j -= n8;
  if (j < 2 * N) {
    const Ring g = ring_geom(N, j);
    const int i = j + 1;                                             // (whole numbers below 2^22)
    pair[j] = make_float4((float)(i < N ? 3 * N * N - i * i : 2 * N * (2 * N - i)), (float)g.z,
                          (float)g.s, 0.f);
    sin_d[j] = g.s;
    return;
  }
  j -= 2 * N;
  const int part = j / nl;
  j -= part * nl;
  if (part > 3 || j >= lmax + 2) return;
  const double l2 = 2.0 * j + 1.0;
  if (part == 2) {
    tab[2 * kShtTab + j] = sqrt(l2);
    return;
  }
  const double w = sht_w(j);
  if (part == 0) tab[j] = sqrt(w);
  else if (part == 1) tab[kShtTab + j] = sqrt(1.0 / (l2 * w));
  else {
    const double c = sqrt(l2 * w * 0.079577471545947667884);         // 1 / (4 pi)
    tab[3 * kShtTab + j] = (j & 1) ? -c : c;
  }
}

// Per-order factors of alpha and a, formed once per block (a division per
// coefficient instead kept the FP64 pipe 9 to 13% busy).
struct OrderConst { double even, odd, step; };
__device__ __forceinline__ OrderConst order_const(const ShtTables& t, int m) {
  const double m0 = t.sw[m] * t.sl[m], s1 = t.sl[m + 1];
  return {1.0 / m0, m0 / s1, s1 * t.inv_z};
}
// alpha_l, with the sign + + - - of (l - m) mod 4.
__device__ __forceinline__ double sht_alpha(const ShtTables& t, int l, int m, OrderConst oc) {
  const int d = l - m, k = d >> 1;
  const double a = (d & 1) ? t.sv[k] * t.sv[m + k] * t.sl[l] * oc.odd
                           : t.sw[k] * t.sw[m + k] * t.sl[l] * oc.even;
  return (d & 2) ? -a : a;
}

// True when |lambda_lm| < 2^-128 for every l <= lmax on the ring with cos and
// sin of the colatitude (c, s), and on every ring nearer the pole: m lies above
// the turning point (lmax + 1/2) sin(theta) and the phase integral
//   S = int sqrt(m^2 / sin^2 - L^2) dtheta  from theta to the turning point
//     = m ln((m c + D) / (s R)) - L ln((L c + D) / R),
// L = lmax + 1/2, D = sqrt(m^2 - L^2 s^2), R = sqrt(L^2 - m^2), of the
// exponentially small side exceeds 130 ln 2 (against the recurrence over all
// orders at lmax 11 to 4096, -log2 of the largest |lambda_lm| is above
// S / ln 2 - 2).
__device__ __forceinline__ bool leg_negligible(int lmax, int m, float c, float s) {
  const float L = (float)lmax + 0.5f, fm = (float)m, Ls = L * s;
  if (!(fm > Ls)) return false;
  const float D = sqrtf((fm - Ls) * (fm + Ls)), R = sqrtf((L - fm) * (L + fm));
  return fm * logf((fm * c + D) / (s * R)) - L * logf((L * c + D) / R) > 130.0f * 0.69314718f;
}

// lambda_mm = cm_m sin(theta)^m of every ring pair p (north ring p) for
// m = 0..lmax, as mu * 2^ex with the mantissa mu a double-float of magnitude
// in [1/2, 1).  Each thread owns one pair and a run of `run` orders; it
// starts from sin(theta)^{m0} by repeated squaring, as (mantissa in [1/2, 1),
// binary exponent) so that nothing underflows, and steps through its run by
// products with sin(theta).  Long runs share the squarings, short ones the
// chip: 64 orders fill it at Nside 1024 (0.09 ms), and small maps take the
// longest run that still gives every SM a block.
//
// Bound by the FP64 pipe: per coefficient two products and the split, six
// instructions of it; exponents, the range test and the widening of the high part
// are integer operations on the bits, and sin(theta) comes from the tables.  (With
// frexp, an FP64 comparison and ring_geom per thread 69 us at Nside 512, lmax 1535,
// and 14 us at Nside 64, lmax 150; now 37 and 8.)
struct MantExp { double m; int e; };
// x > 0 (normal) as mantissa in [1/2, 1) and exponent
__device__ __forceinline__ MantExp me_split(double x) {
  const int hi = __double2hiint(x);
  return {__hiloint2double((hi & 0x000FFFFF) | 0x3FE00000, __double2loint(x)), (hi >> 20) - 1022};
}
__device__ __forceinline__ MantExp me_mul(MantExp a, MantExp b) {
  const MantExp r = me_split(a.m * b.m);
  return {r.m, a.e + b.e + r.e};
}
// double-float of |x| in [1/2, 1): the high part is a normal FP32 number
__device__ __forceinline__ float2 split_unit(double x) {
  const float h = __double2float_rn(x);
  const unsigned b = __float_as_uint(h);
  const double hd = __hiloint2double(
      (int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20))), (int)(b << 29));
  return make_float2(h, __double2float_rn(x - hd));
}
__global__ void __launch_bounds__(256)
k_lmm(int32_t lmax, int32_t npairs, int32_t run, const double* __restrict__ cm,
      const double* __restrict__ sin_d, float2* __restrict__ mu, int32_t* __restrict__ ex) {
  const int nrun = lmax / run + 1;
  const int64_t total = (int64_t)npairs * nrun;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int p = int(t % npairs), j = int(t / npairs);
    const double sn = sin_d[p];                 // in (0, 1]
    const int m0 = run * j, mend = min(lmax, m0 + run - 1);
    MantExp r{0.5, 1};                          // 1
    MantExp b = me_split(sn);
    for (int k = m0; k; k >>= 1) {              // s^{m0}
      if (k & 1) r = me_mul(r, b);
      b = me_mul(b, b);
    }
    double v = r.m;
    int e = r.e;
    for (int m = m0; m <= mend; ++m) {
      if (m > m0) {
        v *= sn;
        if (__double2hiint(v) < 0x20B00000) { v *= 0x1p500; e -= 500; }   // below 2^-500
      }
      const double c = cm[m] * v;               // (of either sign, never 0)
      const int hi = __double2hiint(c);
      mu[(size_t)m * npairs + p] = split_unit(
          __hiloint2double((hi & (int)0x800FFFFF) | 0x3FE00000, __double2loint(c)));
      ex[(size_t)m * npairs + p] = e + ((hi >> 20) & 0x7FF) - 1022;
    }
  }
}

__device__ __forceinline__ double warp_sum_dd(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
  return v;
}

// Coefficients of one round of degrees, duplicated for
// the packed instructions (h, h, l, l); 0 above lmax.  One thread per degree.
__device__ __forceinline__ float4 leg_coef(const ShtTables& t, int l, int lmax, int m,
                                           OrderConst oc) {
  if (l >= lmax) return make_float4(0.f, 0.f, 0.f, 0.f);   // (the step from lmax is not used)
  const double al = sht_alpha(t, l, m, oc);
  const double a = oc.step * al * al;
  const dfl f = df_from_d(((l - m) & 1) ? -a : a);
  return make_float4(f.h, f.h, f.l, f.l);
}
__device__ __forceinline__ dfx dfx_of(float4 v) { return {x2_pack(v.x, v.y), x2_pack(v.z, v.w)}; }

constexpr float kLegBig = 0x1p30f;     // mantissas are brought below this every 4 steps
constexpr int kLegMinExp = -120;       // terms of pairs at or below this exponent are left out

// Block (chunk, m): NT threads, each with G groups of two adjacent ring pairs
// in packed double-float; group g of the block covers the pairs from
// chunk 2 G NT + 2 g NT, a warp 64 adjacent ones of them.  Pair p is the north
// ring p and the south ring 4N - 2 - p (the equator ring, p = 2N - 1, is its
// own mirror); lambda_lm(-z) = (-1)^(l+m) lambda_lm(z), so the pair
// contributes lambda_lm(z_p) (F_north +- F_south).  q_l = v 2^e with the
// mantissa v brought below 2^30 every 4 steps (a step grows it by less than
// |a z| + 1 < 2^8, so |v| < 2^62 throughout), the factor 2^e folded into the
// pair's F while e > -120 (below, the pair's terms are under 2^-58 |F| and are
// left out until e grows; F is folded anew from memory whenever e changes).
//
// What bounds it: the FP32 pipe (18 packed operations for the recurrence and
// 12 for each of the two sums per degree and pair of ring pairs).  Work that
// contributes nothing is left out by warps: a group whose lambda_lm stay
// below 2^-128 up to lmax (leg_negligible: orders above the turning point,
// 16% of the (l, m, pair) triples at Nside 1024, lmax 3071) is never started,
// and a group none of whose pairs has reached e > -120 runs the recurrence
// only.  Groups are numbered from the pole, so the last group of a warp is
// active whenever any is; it starts the degree's sums and the others add.
// The sums of 4 degrees over a thread's two halves and 4 lanes are folded
// together (each exchange halves the number of degrees a lane holds: 7
// complex sums instead of 16), then the block adds the groups of 4 lanes
// through shared memory.  Everything in double-float (FP64 only for the
// block's result: an FP64 instruction costs the FP32 pipe's time for about 64).
// Output: alm (nchunk = 1) or part[chunk], with the factor alpha_l w.
//
// Measured at Nside 1024, lmax 3071 (9.7e9 triples): 13.0 ms; in rounds of 32
// degrees and with a division per coefficient 13.4 ms with G = 2 and
// 128 threads, 4 blocks per SM (128 registers); G = 4 with 128 threads and 2
// blocks 16.6 ms, G = 2 with 256 threads and 2 blocks 14.2 ms, with 64 threads
// and 8 blocks 13.6 ms: 16 warps per SM hide the recurrence's chain of
// dependent operations, fewer do not (FMA pipe 55% busy at 8 warps).  The
// previous kernel (four scalar pairs per thread, two recurrence coefficients
// per degree, every pair from l = m on) took 27.4 ms.  Error of a_lm against
// FP64 at Nside 512, lmax 1535: 4e-13 (9e-11 before, from F folded at 2^e
// near 2^-120 and scaled up from there).
template <int G, int NT, int MB>
__global__ void __launch_bounds__(NT, MB)
k_legendre(const float4* __restrict__ F, const float2* __restrict__ mu,
           const int32_t* __restrict__ ex, ShtTables tb, int32_t lmax, int32_t nrings,
           int32_t npairs, int64_t nalm, double w, double2* __restrict__ out) {
  constexpr int NW = NT / 32;
  __shared__ float4 cs[2][kLegChunkL];
  // sums of 4 adjacent lanes (re.h, re.l, im.h, im.l): 8 per warp
  __shared__ float4 red[NT / 4][kLegChunkL];
  __shared__ float4 red2[NW][kLegChunkL];                 // partials of the warps
  __shared__ int live_s[NW];
  const int chunk = blockIdx.x, m = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned full = 0xFFFFFFFFu;
  const size_t base = (size_t)m * (2 * lmax + 1 - m) / 2;  // index of (l = 0, m)
  double2* dst = out + (size_t)chunk * nalm + base;
  const OrderConst oc = order_const(tb, m);
  // the block's most equatorial pair decides whether there is any work
  const int p_hi = min((chunk + 1) * 2 * G * NT, npairs) - 1;
  {
    const float4 t = tb.pair[p_hi];
    if (leg_negligible(lmax, m, t.y, t.z)) {
      for (int l = m + threadIdx.x; l <= lmax; l += NT) dst[l] = make_double2(0.0, 0.0);
      return;
    }
  }
  u64 z[G];
  dfx v1[G], v2[G], E[G][2], O[G][2];
  int e[G][2], pp[G];
  bool alive[G], act[G];                                  // (uniform over the warp)
  // component k of pair p of group g: (F_north +- F_south) 2^e, or 0 below 2^-120
  auto fold = [&](int p, int ee, dfl* f) {
    if (ee <= kLegMinExp) {
      f[0] = f[1] = f[2] = f[3] = dfl{0.f, 0.f};
      return;
    }
    const float4 fn = F[(size_t)m * nrings + p];
    const int ps = nrings - 1 - p;
    const float4 fs = ps != p ? F[(size_t)m * nrings + ps] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float sc = __int_as_float((ee + 127) << 23);    // 2^ee, -120 < ee < 128
    const float4 a = cdf_add(fn, fs), b = cdf_sub(fn, fs);
    f[0] = df_scale(dfl{a.x, a.y}, sc);
    f[1] = df_scale(dfl{a.z, a.w}, sc);
    f[2] = df_scale(dfl{b.x, b.y}, sc);
    f[3] = df_scale(dfl{b.z, b.w}, sc);
  };
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int first = chunk * 2 * G * NT + 2 * g * NT + warp * 64;   // the warp's first pair
    const int last = min(first + 63, npairs - 1);
    alive[g] = false;
    if (first < npairs) {
      const float4 t = tb.pair[last];
      alive[g] = !leg_negligible(lmax, m, t.y, t.z);
    }
    pp[g] = first + 2 * lane;
    const bool have = alive[g] && pp[g] < npairs;                    // (npairs is even)
    dfl f0[4], f1[4];
    f0[0] = f0[1] = f0[2] = f0[3] = dfl{0.f, 0.f};
    f1[0] = f1[1] = f1[2] = f1[3] = dfl{0.f, 0.f};
    float2 q0 = make_float2(0.f, 0.f), q1 = q0;
    float z0 = 0.f, z1 = 0.f;
    e[g][0] = e[g][1] = -100000;
    if (have) {
      z0 = tb.pair[pp[g]].x;
      z1 = tb.pair[pp[g] + 1].x;
      const size_t at = (size_t)m * npairs + pp[g];
      q0 = mu[at];
      q1 = mu[at + 1];
      e[g][0] = ex[at];
      e[g][1] = ex[at + 1];
      fold(pp[g], e[g][0], f0);
      fold(pp[g] + 1, e[g][1], f1);
    }
    z[g] = x2_pack(z0, z1);
    v1[g] = dfx_set(dfl{q0.x, q0.y}, dfl{q1.x, q1.y});
    v2[g] = dfx{0ull, 0ull};
    E[g][0] = dfx_set(f0[0], f1[0]);
    E[g][1] = dfx_set(f0[1], f1[1]);
    O[g][0] = dfx_set(f0[2], f1[2]);
    O[g][1] = dfx_set(f0[3], f1[3]);
    act[g] = __any_sync(full, max(e[g][0], e[g][1]) > kLegMinExp);
  }
#pragma unroll
  for (int g = 1; g < G; ++g) act[g] |= act[g - 1];
  if (lane == 0) live_s[warp] = alive[G - 1];
  // brings the mantissas of group g below 2^30 (rare beyond the growing part)
  auto rescale = [&](int g) {
    float2 a = x2_get(v1[g].h), b = x2_get(v2[g].h);
    float m0_ = fmaxf(fabsf(a.x), fabsf(b.x)), m1_ = fmaxf(fabsf(a.y), fabsf(b.y));
    if (fmaxf(m0_, m1_) > kLegBig) {
      float s0 = 1.f, s1 = 1.f;
      const int o0 = e[g][0], o1 = e[g][1];
      while (m0_ > kLegBig) { m0_ *= 0x1p-30f; s0 *= 0x1p-30f; e[g][0] += 30; }
      while (m1_ > kLegBig) { m1_ *= 0x1p-30f; s1 *= 0x1p-30f; e[g][1] += 30; }
      const u64 sc = x2_pack(s0, s1);                     // powers of two: exact
      v1[g].h = x2_mul(v1[g].h, sc);
      v1[g].l = x2_mul(v1[g].l, sc);
      v2[g].h = x2_mul(v2[g].h, sc);
      v2[g].l = x2_mul(v2[g].l, sc);
      dfl f[4];
      auto put = [&](dfx& d, dfl x, bool hi) {
        const float2 h = x2_get(d.h), l = x2_get(d.l);
        d.h = hi ? x2_pack(h.x, x.h) : x2_pack(x.h, h.y);
        d.l = hi ? x2_pack(l.x, x.l) : x2_pack(x.l, l.y);
      };
      if (e[g][0] != o0) {
        fold(pp[g], e[g][0], f);
        put(E[g][0], f[0], false);
        put(E[g][1], f[1], false);
        put(O[g][0], f[2], false);
        put(O[g][1], f[3], false);
      }
      if (e[g][1] != o1) {
        fold(pp[g] + 1, e[g][1], f);
        put(E[g][0], f[0], true);
        put(E[g][1], f[1], true);
        put(O[g][0], f[2], true);
        put(O[g][1], f[3], true);
      }
    }
  };
  if (threadIdx.x < kLegChunkL)
    cs[0][threadIdx.x] = leg_coef(tb, m + threadIdx.x, lmax, m, oc);
  __syncthreads();
  int buf = 0;
  for (int l0 = m; l0 <= lmax; l0 += kLegChunkL, buf ^= 1) {
    const int cnt = min(kLegChunkL, lmax + 1 - l0);
    if (alive[G - 1]) {
#pragma unroll 1
      for (int t = 0; t < cnt; t += 4) {                  // degrees l0 + t .. + 3: even, odd, ...
        const float4* ct = &cs[buf][t];
        float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
        const int d = ((lane & 1) << 1) | ((lane >> 1) & 1);   // the degree this lane ends with
        if (act[G - 1]) {
          dfx cr[4], ci[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            constexpr int g = G - 1;
            const u64 nv = x2_neg(v1[g].h);
            cr[j] = dfx_mul_raw(v1[g], (j & 1) ? O[g][0] : E[g][0]);
            ci[j] = dfx_mul_raw(v1[g], (j & 1) ? O[g][1] : E[g][1]);
            leg_step(v1[g], v2[g], nv, dfx_of(ct[j]), z[g]);
          }
          rescale(G - 1);
#pragma unroll
          for (int g = G - 2; g >= 0; --g) {
            if (act[g]) {
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const u64 nv = x2_neg(v1[g].h);
                dfx_mac(cr[j], v1[g], nv, (j & 1) ? O[g][0] : E[g][0]);
                dfx_mac(ci[j], v1[g], nv, (j & 1) ? O[g][1] : E[g][1]);
                leg_step(v1[g], v2[g], nv, dfx_of(ct[j]), z[g]);
              }
              rescale(g);
            } else if (alive[g]) {
#pragma unroll
              for (int j = 0; j < 4; ++j) leg_step(v1[g], v2[g], x2_neg(v1[g].h), dfx_of(ct[j]), z[g]);
              rescale(g);
              act[g] = __any_sync(full, max(e[g][0], e[g][1]) > kLegMinExp);
            }
          }
          // halves: (degree 0, 1) and (2, 3) side by side
          auto halves = [](dfx a, dfx b) {
            const float2 ah = x2_get(a.h), al = x2_get(a.l), bh = x2_get(b.h), bl = x2_get(b.l);
            return dfx_add_raw(dfx{x2_pack(ah.x, bh.x), x2_pack(al.x, bl.x)},
                               dfx{x2_pack(ah.y, bh.y), x2_pack(al.y, bl.y)});
          };
          const dfx r01 = halves(cr[0], cr[1]), r23 = halves(cr[2], cr[3]);
          const dfx i01 = halves(ci[0], ci[1]), i23 = halves(ci[2], ci[3]);
          // lanes differing in bit 0: even lanes keep degrees 0 and 1
          const bool b0 = lane & 1, b1 = lane & 2;
          auto swap1 = [&](dfx lo, dfx hi) {
            const dfx keep = b0 ? hi : lo, send = b0 ? lo : hi;
            return dfx_add_raw(keep, dfx{__shfl_xor_sync(full, send.h, 1), __shfl_xor_sync(full, send.l, 1)});
          };
          const dfx sr = swap1(r01, r23), si = swap1(i01, i23);
          // lanes differing in bit 1: one degree each, real and imaginary side by side
          const float2 rh = x2_get(sr.h), rl = x2_get(sr.l), ih = x2_get(si.h), il = x2_get(si.l);
          const dfx lo{x2_pack(rh.x, ih.x), x2_pack(rl.x, il.x)};
          const dfx hi{x2_pack(rh.y, ih.y), x2_pack(rl.y, il.y)};
          const dfx keep = b1 ? hi : lo, send = b1 ? lo : hi;
          const dfx s = dfx_add_raw(keep, dfx{__shfl_xor_sync(full, send.h, 2),
                                              __shfl_xor_sync(full, send.l, 2)});
          const float2 fh = x2_get(s.h), fl = x2_get(s.l);
          r = make_float4(fh.x, fl.x, fh.y, fl.y);
        } else {
#pragma unroll
          for (int g = 0; g < G; ++g)
            if (alive[g]) {
#pragma unroll
              for (int j = 0; j < 4; ++j) leg_step(v1[g], v2[g], x2_neg(v1[g].h), dfx_of(ct[j]), z[g]);
              rescale(g);
              act[g] = __any_sync(full, max(e[g][0], e[g][1]) > kLegMinExp);
            }
        }
#pragma unroll
        for (int g = 1; g < G; ++g) act[g] |= act[g - 1];
        red[warp * 8 + (lane >> 2)][t + d] = r;
      }
    }
    if (threadIdx.x < kLegChunkL)                         // the next round's coefficients
      cs[buf ^ 1][threadIdx.x] = leg_coef(tb, l0 + kLegChunkL + threadIdx.x, lmax, m, oc);
    __syncthreads();
    // the group sums of each degree: warp j adds rows j, j + NW, ...
    // (lane t: conflict-free rows), then the warps' partials per degree
#pragma unroll
    for (int t = lane; t < kLegChunkL; t += 32) {
      if (t >= cnt) break;
      dfl sr{0.f, 0.f}, si{0.f, 0.f};
      for (int row = warp; row < NT / 4; row += NW) {
        if (!live_s[row >> 3]) continue;                  // (uniform)
        const float4 v = red[row][t];
        sr = df_add(sr, dfl{v.x, v.y});
        si = df_add(si, dfl{v.z, v.w});
      }
      red2[warp][t] = make_float4(sr.h, sr.l, si.h, si.l);
    }
    __syncthreads();
    if (threadIdx.x < cnt) {
      const int t = threadIdx.x, l = l0 + t;
      dfl sr{0.f, 0.f}, si{0.f, 0.f};
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        const float4 v = red2[k][t];
        sr = df_add(sr, dfl{v.x, v.y});
        si = df_add(si, dfl{v.z, v.w});
      }
      const double f = w * sht_alpha(tb, l, m, oc);
      dst[l] = make_double2(f * df_to_d(sr), f * df_to_d(si));
    }
  }
}

__global__ void k_alm_sum(const double2* __restrict__ part, int nchunk, int64_t nalm,
                          double2* __restrict__ alm) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nalm;
       i += (int64_t)gridDim.x * blockDim.x) {
    double sr = 0.0, si = 0.0;
    for (int c = 0; c < nchunk; ++c) {
      const double2 v = part[(size_t)c * nalm + i];
      sr += v.x;
      si += v.y;
    }
    alm[i] = make_double2(sr, si);
  }
}

// One warp per degree l: lane k adds the orders m = k, k + 32, ... (their
// loads in flight together), then a fixed shuffle tree.
__global__ void k_alm2cl(const double2* __restrict__ alm, int32_t lmax, double* __restrict__ cl) {
  const int l = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (l > lmax) return;                        // (uniform over the warp)
  double s = 0.0;
  for (int m = lane; m <= l; m += 32) {
    const double2 a = alm[(size_t)m * (2 * lmax + 1 - m) / 2 + l];
    const double q = a.x * a.x + a.y * a.y;
    s += m == 0 ? q : 2.0 * q;
  }
  s = warp_sum_dd(s);
  if (lane == 0) cl[l] = s / (2.0 * l + 1.0);
}

// ------------------------------------------------------------ synthesis --
// map_p = sum_l sum_{m>=0} (2 - delta_m0) Re(a_lm Y_lm(theta_p, phi_p)), the
// real field with a_l,-m = (-1)^m conj(a_lm), ring by ring:
//   k_legendre_synth : G_m(ring) = sum_l a_lm lambda_lm(z_ring), per (m, ring
//                      pair) with the even/odd split of the mirror rings;
//   k_ring_synth     : map_j = sum_{|m| <= lmax} G_m e^{i m phi_j}, folding
//                      m onto the ring's n frequencies and an inverse DFT
//                      (sht_ring.cu).
//
// k_legendre_synth: block (chunk, m), a thread two adjacent ring pairs in
// packed double-float, the recurrence and the exponents as in k_legendre; the
// sums over l stay in the thread (in units of 2^e, rescaled with the
// mantissas: terms 2^-30 below the current scale may lose bits, they are
// negligible), so nothing is reduced across threads.  A warp whose pairs are
// all negligible up to lmax (leg_negligible) writes zeros, and none of its
// terms is formed before one of its pairs has e > -120.  These terms are 0 for
// finite coefficients only, so one that is not finite sets *bad, with which
// k_ring_synth makes every pixel a NaN: the sums of the equator's pair, which
// leaves nothing out, are NaNs then.  (The imaginary part of order 0 does not
// enter the map.  A test of every coefficient by every block, or by the equator's
// thread at the end, made this kernel up to 12% slower at Nside 128.)  Bound by the FP32
// pipe: 18 + 24 packed operations per degree and pair of ring pairs (FMA pipe
// 71% busy).  Nside 512, lmax 1535: 1.47 ms with blocks of 128 threads, 1.51 with
// 256 or 64 (2.96 ms before the one-coefficient recurrence and the packed pairs).
template <int NT>
__global__ void __launch_bounds__(NT)
k_legendre_synth(const double2* __restrict__ alm, const float2* __restrict__ mu,
                 const int32_t* __restrict__ ex, ShtTables tb, int32_t lmax, int32_t nrings,
                 int32_t npairs, float4* __restrict__ G, int* __restrict__ bad) {
  __shared__ float4 cs[2][kLegChunkL];
  __shared__ float4 as[2][kLegChunkL][2];                 // alpha_l a_lm: real, imaginary
  const int chunk = blockIdx.x, m = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned full = 0xFFFFFFFFu;
  const size_t base = (size_t)m * (2 * lmax + 1 - m) / 2;
  const OrderConst oc = order_const(tb, m);
  const int first = chunk * 2 * NT + warp * 64;           // the warp's first pair
  const int p = first + 2 * lane;
  const bool have = p < npairs;                           // (npairs is even)
  bool alive = false;
  if (first < npairs) {
    const float4 t = tb.pair[min(first + 63, npairs - 1)];
    alive = !leg_negligible(lmax, m, t.y, t.z);
  }
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  {
    const float4 t = tb.pair[min((chunk + 1) * 2 * NT, npairs) - 1];   // the block's last pair
    if (leg_negligible(lmax, m, t.y, t.z)) {
      if (have)
        for (int k = 0; k < 2; ++k) {
          G[(size_t)m * nrings + p + k] = zero;
          G[(size_t)m * nrings + (nrings - 1 - p - k)] = zero;
        }
      return;
    }
  }
  u64 z = 0ull;
  dfx v1{0ull, 0ull}, v2{0ull, 0ull};
  dfx ge[2] = {{0ull, 0ull}, {0ull, 0ull}}, go[2] = {{0ull, 0ull}, {0ull, 0ull}};
  int e0 = -100000, e1 = -100000;
  if (have && alive) {
    const size_t at = (size_t)m * npairs + p;
    const float2 q0 = mu[at], q1 = mu[at + 1];
    z = x2_pack(tb.pair[p].x, tb.pair[p + 1].x);
    v1 = dfx_set(dfl{q0.x, q0.y}, dfl{q1.x, q1.y});
    e0 = ex[at];
    e1 = ex[at + 1];
  }
  bool act = __any_sync(full, max(e0, e1) > kLegMinExp);
  auto load = [&](int b, int l0) {                        // one round's coefficients
    for (int t = threadIdx.x; t < 2 * kLegChunkL; t += NT) {
      const int l = l0 + (t & (kLegChunkL - 1));
      if (t < kLegChunkL) {
        cs[b][t] = leg_coef(tb, l, lmax, m, oc);
      } else {
        float4 re = zero, im = zero;
        if (l <= lmax) {
          const double2 a = alm[base + l];
          const double f = sht_alpha(tb, l, m, oc);
          const dfl x = df_from_d(f * a.x), y = df_from_d(f * a.y);
          re = make_float4(x.h, x.h, x.l, x.l);
          im = make_float4(y.h, y.h, y.l, y.l);
        }
        as[b][l - l0][0] = re;
        as[b][l - l0][1] = im;
      }
    }
  };
  load(0, m);
  __syncthreads();
  int buf = 0;
  for (int l0 = m; l0 <= lmax; l0 += kLegChunkL, buf ^= 1) {
    const int cnt = min(kLegChunkL, lmax + 1 - l0);
    if (l0 + kLegChunkL <= lmax) load(buf ^ 1, l0 + kLegChunkL);
    if (alive) {
#pragma unroll 1
      for (int t = 0; t < cnt; t += 4) {                  // degrees l0 + t .. + 3: even, odd, ...
        if (act) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {                   // (coefficients above lmax are 0)
            const u64 nv = x2_neg(v1.h);
            dfx* s = (j & 1) ? go : ge;
            dfx_mac(s[0], v1, nv, dfx_of(as[buf][t + j][0]));
            dfx_mac(s[1], v1, nv, dfx_of(as[buf][t + j][1]));
            leg_step(v1, v2, nv, dfx_of(cs[buf][t + j]), z);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) leg_step(v1, v2, x2_neg(v1.h), dfx_of(cs[buf][t + j]), z);
        }
        const float2 a = x2_get(v1.h), b = x2_get(v2.h);
        float m0_ = fmaxf(fabsf(a.x), fabsf(b.x)), m1_ = fmaxf(fabsf(a.y), fabsf(b.y));
        if (fmaxf(m0_, m1_) > kLegBig) {
          float s0 = 1.f, s1 = 1.f;
          while (m0_ > kLegBig) { m0_ *= 0x1p-30f; s0 *= 0x1p-30f; e0 += 30; }
          while (m1_ > kLegBig) { m1_ *= 0x1p-30f; s1 *= 0x1p-30f; e1 += 30; }
          const u64 sc = x2_pack(s0, s1);
          auto down = [&](dfx& d) { d.h = x2_mul(d.h, sc); d.l = x2_mul(d.l, sc); };
          down(v1);
          down(v2);
          down(ge[0]);
          down(ge[1]);
          down(go[0]);
          down(go[1]);
        }
        if (!act) act = __any_sync(full, max(e0, e1) > kLegMinExp);
      }
    }
    __syncthreads();
  }
  if (!have) return;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int ee = k ? e1 : e0, r = p + k, ps = nrings - 1 - r;
    const float sc = ee > kLegMinExp ? __int_as_float((ee + 127) << 23) : 0.f;
    auto part = [&](dfx d) {
      const float2 h = x2_get(d.h), l = x2_get(d.l);
      return df_scale(k ? df_norm(h.y, l.y) : df_norm(h.x, l.x), sc);
    };
    const float4 ev = cdf_pack(part(ge[0]), part(ge[1])), od = cdf_pack(part(go[0]), part(go[1]));
    const float4 sum = cdf_add(ev, od);
    G[(size_t)m * nrings + r] = sum;
    if (ps == r && (isnan(sum.x) || (m && isnan(sum.z)))) *bad = 1;   // (the equator)
    if (ps != r) G[(size_t)m * nrings + ps] = cdf_sub(ev, od);
  }
}

// a_lm b_l with the Gaussian beam b_l = exp(-l(l+1) sigma^2 / 2).  A thread
// takes one degree and every gridDim.y-th order, so that the FP64 exponential
// (and the index of a coefficient) is not formed per coefficient: 92 us at lmax
// 1535 when it was, for 38 MB of traffic.  Consecutive threads take consecutive
// coefficients of one order.
__global__ void __launch_bounds__(256)
k_alm_beam(const double2* __restrict__ in, int32_t lmax, double sigma,
           double2* __restrict__ out) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l > lmax) return;
  const double b = exp(-0.5 * (double)l * (l + 1) * sigma * sigma);
  for (int m = blockIdx.y; m <= l; m += gridDim.y) {
    const size_t i = (size_t)m * (2 * lmax + 1 - m) / 2 + l;
    const double2 a = in[i];
    out[i] = make_double2(a.x * b, a.y * b);
  }
}

// Band powers: out[b] = mean of C_l over l in [lmin + b dl, lmin + (b+1) dl).
__global__ void k_cl_bin(const double* __restrict__ cl, int32_t lmin, int32_t dl, int32_t nbins,
                         double* __restrict__ out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nbins) return;
  double s = 0.0;
  for (int l = lmin + b * dl; l < lmin + (b + 1) * dl; ++l) s += cl[l];
  out[b] = s / dl;
}

// ------------------------------------------------------------------ host --

// Workspace of the transforms: the tables, then the ring coefficients
// (F or G), the seeds lambda_mm and, with several chunks of ring pairs, the
// partial a_lm; every piece 256-byte aligned.
struct ShtSpace {
  ShtTables tb;
  float4* ring;        // [lmax + 1][4N - 1]
  float2* mu;          // [lmax + 1][2N]
  int32_t* ex;
  double2* part;       // [nchunk][nalm]
  int* bad;            // synthesis: a coefficient is not finite (cleared with the tables)
};
static ufc_status sht_space(ufc_ctx* c, int nside, int lmax, int nchunk, ShtSpace& o) {
  const size_t nrings = 4 * (size_t)nside - 1, npairs = 2 * (size_t)nside;
  const size_t nalm = (size_t)(lmax + 1) * (lmax + 2) / 2;
  size_t at = 0;
  auto piece = [&](size_t bytes) { const size_t r = at; at += (bytes + 255) / 256 * 256; return r; };
  const size_t o_roots = piece((size_t)8 * nside * sizeof(float4));
  const size_t o_tab = piece((size_t)4 * kShtTab * sizeof(double));
  const size_t o_pair = piece(npairs * sizeof(float4));
  const size_t o_sin = piece(npairs * sizeof(double));
  const size_t o_ring = piece((size_t)(lmax + 1) * nrings * sizeof(float4));
  const size_t o_mu = piece((size_t)(lmax + 1) * npairs * sizeof(float2));
  const size_t o_ex = piece((size_t)(lmax + 1) * npairs * sizeof(int32_t));
  const size_t o_part = piece(nchunk > 1 ? nchunk * nalm * sizeof(double2) : 0);
  const size_t o_bad = piece(sizeof(int));
  char* ws = (char*)ws_get(c, kSlotSht, at);
  if (!ws) return UFC_ERR_ALLOC;
  float4* roots = reinterpret_cast<float4*>(ws + o_roots);
  double* tab = reinterpret_cast<double*>(ws + o_tab);
  float4* pair = reinterpret_cast<float4*>(ws + o_pair);
  double* sin_d = reinterpret_cast<double*>(ws + o_sin);
  o.tb = ShtTables{roots, tab, tab + kShtTab, tab + 2 * kShtTab, tab + 3 * kShtTab, pair,
                   1.0 / (3.0 * (double)nside * (double)nside)};
  o.ring = reinterpret_cast<float4*>(ws + o_ring);
  o.mu = reinterpret_cast<float2*>(ws + o_mu);
  o.ex = reinterpret_cast<int32_t*>(ws + o_ex);
  o.part = reinterpret_cast<double2*>(ws + o_part);
  o.bad = reinterpret_cast<int*>(ws + o_bad);
  {
    ProfScope ps_(c, "k_sht_tables");
    const int n = 10 * nside + 4 * ((lmax + 2 + 31) / 32 * 32);
    k_sht_tables<<<(n + 63) / 64, 64, 0, c->stream>>>(nside, lmax, roots, tab, pair,
                                                        sin_d, o.bad);
  }
  {
    ProfScope ps_(c, "k_lmm");
    int run = 64;                           // orders per thread: see k_lmm
    while (run > 4 && (int64_t)npairs * (lmax / run + 1) < 256ll * c->num_sms) run /= 2;
    const int64_t lt = (int64_t)npairs * (lmax / run + 1);
    k_lmm<<<(int)std::min<int64_t>((lt + 255) / 256, 8 * c->num_sms), 256, 0, c->stream>>>(
        lmax, (int)npairs, run, o.tb.cm, sin_d, o.mu, o.ex);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

ufc_status run_map2alm(ufc_ctx* c, const float* map, int nside, int lmax, double* alm_out) {
  if (!map || !alm_out) return set_err(c, UFC_ERR_ARG, "map_dev and alm_dev are required");
  if (nside < 1 || nside > kShtMaxNside || (nside & (nside - 1)))
    return set_err(c, UFC_ERR_UNSUPPORTED, "map2alm needs a power-of-two nside <= %d", kShtMaxNside);
  if (lmax < 0 || lmax > 4 * nside)
    return set_err(c, UFC_ERR_ARG, "lmax must be in [0, 4 nside]");
  if ((reinterpret_cast<uintptr_t>(alm_out) & 15))
    return set_err(c, UFC_ERR_ARG, "alm_dev must be 16-byte aligned");
  const int nrings = 4 * nside - 1, npairs = 2 * nside;
  const int64_t nalm = (int64_t)(lmax + 1) * (lmax + 2) / 2;
  // ring pairs per block: 512 (two groups per thread), or all of a small map's
  const int per_block = npairs > 256 ? 512 : (npairs > 128 ? 256 : 128);
  const int nchunk = (npairs + per_block - 1) / per_block;
  ShtSpace sp;
  const ufc_status s = sht_space(c, nside, lmax, nchunk, sp);
  if (s) return s;
  const ufc_status sr = launch_ring_transform(c, map, sp.tb.roots, nside, lmax, sp.ring);
  if (sr) return sr;
  double2* alm = reinterpret_cast<double2*>(alm_out);
  {
    ProfScope ps_(c, "k_legendre");
    const dim3 grid(nchunk, lmax + 1);
    const double w = 4.0 * M_PI / (12.0 * (double)nside * nside);
    double2* out = nchunk > 1 ? sp.part : alm;
#define UFC_LEG(G, NT, MB)                                                                        \
  k_legendre<G, NT, MB><<<grid, NT, 0, c->stream>>>(sp.ring, sp.mu, sp.ex, sp.tb, lmax, nrings,   \
                                                    npairs, nalm, w, out)
    if (per_block == 512) UFC_LEG(2, 128, 4);
    else if (per_block == 256) UFC_LEG(1, 128, 1);
    else UFC_LEG(1, 64, 1);
#undef UFC_LEG
  }
  if (nchunk > 1) {
    ProfScope ps_(c, "k_alm_sum");
    k_alm_sum<<<2 * c->num_sms, 256, 0, c->stream>>>(sp.part, nchunk, nalm, alm);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

ufc_status run_cl_bin(ufc_ctx* c, const double* cl, int lmax, int lmin, int dl, int nbins,
                      double* out) {
  if (!cl || !out) return set_err(c, UFC_ERR_ARG, "cl_dev and out_dev are required");
  if (lmin < 0 || dl < 1 || nbins < 1 || (int64_t)lmin + (int64_t)nbins * dl > (int64_t)lmax + 1)
    return set_err(c, UFC_ERR_ARG, "bins [lmin, lmin + nbins dl) must lie in [0, lmax]");
  ProfScope ps_(c, "k_cl_bin");
  k_cl_bin<<<(nbins + 255) / 256, 256, 0, c->stream>>>(cl, lmin, dl, nbins, out);
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

ufc_status run_alm2map(ufc_ctx* c, const double* alm, int nside, int lmax, float* map) {
  if (!alm || !map) return set_err(c, UFC_ERR_ARG, "alm_dev and map_dev are required");
  if (nside < 1 || nside > kShtMaxNside || (nside & (nside - 1)))
    return set_err(c, UFC_ERR_UNSUPPORTED, "alm2map needs a power-of-two nside <= %d", kShtMaxNside);
  if (lmax < 0 || lmax > 4 * nside) return set_err(c, UFC_ERR_ARG, "lmax must be in [0, 4 nside]");
  if ((reinterpret_cast<uintptr_t>(alm) & 15))
    return set_err(c, UFC_ERR_ARG, "alm_dev must be 16-byte aligned");
  const int nrings = 4 * nside - 1, npairs = 2 * nside;
  ShtSpace sp;
  const ufc_status s = sht_space(c, nside, lmax, 1, sp);
  if (s) return s;
  {
    ProfScope ps_(c, "k_legendre_synth");
    const int nt = npairs > 128 ? 128 : 64;
    const dim3 grid((npairs + 2 * nt - 1) / (2 * nt), lmax + 1);
#define UFC_SYN(NT)                                                                                \
  k_legendre_synth<NT><<<grid, NT, 0, c->stream>>>(reinterpret_cast<const double2*>(alm), sp.mu,   \
                                                   sp.ex, sp.tb, lmax, nrings, npairs, sp.ring, \
                                                   sp.bad)
    if (nt == 128) UFC_SYN(128);
    else UFC_SYN(64);
#undef UFC_SYN
  }
  UFC_CUDA(c, cudaGetLastError());
  return launch_ring_synth(c, sp.ring, sp.tb.roots, nside, lmax, sp.bad, map);
}

ufc_status run_alm_beam(ufc_ctx* c, const double* in, int lmax, double sigma, double* out) {
  if (!in || !out) return set_err(c, UFC_ERR_ARG, "alm_in_dev and alm_out_dev are required");
  if (lmax < 0 || !(sigma >= 0.0) || !std::isfinite(sigma))
    return set_err(c, UFC_ERR_ARG, "lmax >= 0 and a finite sigma >= 0 are required");
  if ((reinterpret_cast<uintptr_t>(in) & 15) || (reinterpret_cast<uintptr_t>(out) & 15))
    return set_err(c, UFC_ERR_ARG, "a_lm buffers must be 16-byte aligned");
  ProfScope ps_(c, "k_alm_beam");
  const int nl = lmax / 256 + 1;                       // blocks of 256 degrees
  const int slices = std::min(lmax + 1, std::max(1, 8 * c->num_sms / nl));
  k_alm_beam<<<dim3(nl, slices), 256, 0, c->stream>>>(reinterpret_cast<const double2*>(in), lmax,
                                                      sigma, reinterpret_cast<double2*>(out));
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

ufc_status run_alm2cl(ufc_ctx* c, const double* alm, int lmax, double* cl) {
  if (!alm || !cl) return set_err(c, UFC_ERR_ARG, "alm_dev and cl_dev are required");
  if (lmax < 0) return set_err(c, UFC_ERR_ARG, "lmax must be >= 0");
  if ((reinterpret_cast<uintptr_t>(alm) & 15))
    return set_err(c, UFC_ERR_ARG, "alm_dev must be 16-byte aligned");
  ProfScope ps_(c, "k_alm2cl");
  k_alm2cl<<<(lmax + 8) / 8, 256, 0, c->stream>>>(reinterpret_cast<const double2*>(alm), lmax,
                                                        cl);
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

}  // namespace ufc
