// kappa map (Eq. 6), moments (Eq. 12-13), PDF (Sec. 3.3), adjoint sums, and
// the Welford covariance over realisations (Eq. 10-11).
//
// GB300 runs FP64 at ~1/64 of FP32, so the per-pixel sums over shells are
// carried in double-float (pairs of FP32, ~2^-44 relative) and converted to
// FP64 only per thread or per block.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "ctx.h"
#include "direct.cuh"
#include "packed.cuh"
#include "pixel.cuh"

namespace ufc {

// ------------------------------------------------------------ helpers -----
struct f2 { float h, l; };

__device__ __forceinline__ f2 f2_two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ f2 f2_norm(float h, float l) {
  float s = __fadd_rn(h, l);
  return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
// acc += (a_h + a_l) * n, n an exactly representable count.
__device__ __forceinline__ void f2_mac(f2& acc, float ah, float al, float n) {
  float ph = __fmul_rn(ah, n);
  float pe = __fmaf_rn(ah, n, -ph);
  f2 s = f2_two_sum(acc.h, ph);
  acc.h = s.h;
  acc.l = __fadd_rn(acc.l, __fadd_rn(s.l, __fmaf_rn(al, n, pe)));
}
__device__ __forceinline__ f2 f2_add(f2 x, f2 y) {
  f2 s = f2_two_sum(x.h, y.h);
  return f2_norm(s.h, __fadd_rn(s.l, __fadd_rn(x.l, y.l)));
}
__device__ __forceinline__ f2 f2_mul(f2 x, f2 y) {
  float p = __fmul_rn(x.h, y.h);
  float e = __fmaf_rn(x.h, y.h, -p);
  e = __fmaf_rn(x.h, y.l, __fmaf_rn(x.l, y.h, e));
  return f2_norm(p, e);
}
__device__ __forceinline__ double f2_to_d(f2 x) { return double(x.h) + double(x.l); }

__device__ __forceinline__ double warp_sum_d(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
  return v;
}
// Sum of v[0], v[stride], ..., v[(n - 1) stride] by one warp in a fixed
// order: lane l adds elements l, l + 32, ... in turn, then a butterfly; every
// lane ends with the same value (each pairwise sum is formed by both lanes).
__device__ __forceinline__ double warp_sum_fixed(const double* v, int n, int stride) {
  double s = 0.0;
  for (int i = threadIdx.x & 31; i < n; i += 32) s += __ldcg(v + (size_t)i * stride);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  return s;
}

// Block sum of a double in fixed order (lane order, then warp order).
template <int NT>
__device__ __forceinline__ double block_sum_d(double v, double* sh) {
  v = warp_sum_d(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < NT / 32; ++i) t += sh[i];
  return t;   // valid in thread 0
}

// Clears the PDF that the moment pass after this kernel adds to and its count of
// finished blocks (block 0; pdf may be NULL: no moment pass).  One launch less
// than a memset between the two passes.
struct MomentOut {
  unsigned long long* pdf;
  int npdf;
  unsigned int* ticket;      // beside the pass's partial sums
};
__device__ __forceinline__ void clear_pdf(const MomentOut& o) {
  if (!o.pdf || blockIdx.x != 0) return;
  for (int i = threadIdx.x; i < o.npdf; i += blockDim.x) o.pdf[i] = 0ull;
  if (threadIdx.x == 0 && o.ticket) *o.ticket = 0u;
}

struct Coef {
  float ah[kMaxShells];
  float al[kMaxShells];
  float ch, cl;        // C as double-float
  int32_t nshell;
  int32_t npix;
};

// ------------------------------------------------- kappa + adjoint sums ---
// kappa_p = sum_b A_b n_bp - C is accumulated in double-float over the
// shells in order.  The adjoint needs per-shell sums S1_b = sum_p e_p n_bp,
// S2_b = sum_p e_p^2 n_bp, T_b = sum_p g_p n_bp, N_b = sum_p n_bp and global
// sums P_k = sum_p e_p^k (k = 1..3), Q = sum_p g_p of the unrounded map e;
// e, e^2 and g are quantised to pairs of integers and multiplied by the
// counts in exact integer arithmetic.
constexpr int kKT = 256;   // threads of the scalar-load kappa kernel

// round(x) as int for |x| < 2^22, and the rounded value as float (the FP32
// magic-number form of pixel.cuh: no conversion instruction, which GB300
// executes on its narrow FP64 pipe)
__device__ __forceinline__ int32_t round_fast(float x, float& xr) {
  const float r = __fadd_rn(x, kMagic);
  xr = __fsub_rn(r, kMagic);
  return __float_as_int(r) - kMagicBits;
}
// 2^s as float for s in [-126, 127]
__device__ __forceinline__ float pow2f(int s) { return __int_as_float((127 + s) << 23); }
// floor(log2(x)) of a normal float x > 0
__device__ __forceinline__ int ilog2f(float x) { return ((__float_as_int(x) >> 23) & 0xFF) - 127; }

// Splits v (double-float, |v| 2^s < 2^22) into two integers with
// v 2^s = hi + lo 2^-22 to within 2^-23: hi = round(v.h 2^s), lo the rounded
// remainder (|remainder| <= 3/4, so |lo| < 2^22).
__device__ __forceinline__ void quant2(f2 v, int s, int& hi, int& lo) {
  const float sc = pow2f(s);
  const float a = __fmul_rn(v.h, sc);
  float ar;
  hi = round_fast(a, ar);
  const float rem = __fadd_rn(__fsub_rn(a, ar), __fmul_rn(v.l, sc));   // a - ar is exact
  float dummy;
  lo = round_fast(__fmul_rn(rem, 4194304.0f), dummy);                  // 2^22
}

// 128-bit two's-complement fixed-point accumulator (integer operations only).
struct I128 { unsigned long long lo; long long hi; };
__device__ __forceinline__ void i128_add(I128& acc, I128 v) {
  const unsigned long long nlo = acc.lo + v.lo;
  acc.hi += v.hi + (nlo < acc.lo ? 1ll : 0ll);
  acc.lo = nlo;
}
// v * 2^sh rounded to the nearest whole number, |sh| < 128 (the adjoint's flush
// passes kFrac - s - 22 with the scale s from 8, a maximum below 2^14, to 120).
__device__ __forceinline__ I128 i128_shift(I128 v, int sh) {
  if (sh < 0) i128_add(v, sh > -65 ? I128{1ull << (-sh - 1), 0ll} : I128{0ull, 1ll << (-sh - 65)});
  if (sh >= 64) return {0ull, (long long)(v.lo << (sh - 64))};
  if (sh > 0) return {v.lo << sh, (long long)((unsigned long long)v.hi << sh | v.lo >> (64 - sh))};
  if (sh == 0) return v;
  if (sh > -64) return {v.lo >> -sh | (unsigned long long)v.hi << (64 + sh), v.hi >> -sh};
  return {(unsigned long long)(v.hi >> (-sh - 64)), v.hi >> 63};
}
// v[0] + 2^8 v[1] + 2^16 v[2] + 2^-22 (the same of v[3 .. 5]), times 2^22: exact.
__device__ __forceinline__ I128 i128_digits(const long long* v) {
  I128 r{0ull, 0ll};
#pragma unroll
  for (int k = 0; k < 6; ++k)
    i128_add(r, i128_shift(I128{(unsigned long long)v[k], v[k] >> 63}, k < 3 ? 22 + 8 * k : 8 * (k - 3)));
  return r;
}
// (by the magnitude: a small negative value has 64 high and many low bits set, and
// converted as it is would keep 2^-53 of 2^64, not of itself)
__device__ __forceinline__ double i128_to_d(I128 a, int frac_bits) {
  const bool neg = a.hi < 0;
  if (neg) a = I128{0ull - a.lo, (long long)(0ull - (unsigned long long)a.hi - (a.lo ? 1ull : 0ull))};
  const double m = (double)(unsigned long long)a.hi * 18446744073709551616.0 + (double)a.lo;
  return ldexp(neg ? -m : m, -frac_bits);
}
// Fractional bits of the adjoint sums S1 (e n), S2 (e^2 n), T (g n); with
// |e|, |g| < 2^14 and |e|^2 < 2^28 every sum fits the 128-bit range.
constexpr int kFrac1 = 72, kFrac2 = 56, kFrac3 = 72;
struct AdjRow { I128 s[3]; long long n; long long pad_; };

// Forward pass with scalar loads, for a kappa buffer that is not 16-byte
// aligned.
__global__ void __launch_bounds__(kKT)
k_kappa_plain(const int32_t* __restrict__ counts, Coef cf, float* __restrict__ kappa,
              double* __restrict__ ksum_part, MomentOut mo) {
  clear_pdf(mo);
  __shared__ float ah_s[kMaxShells], al_s[kMaxShells];
  __shared__ double red[kKT / 32];
  const int S = cf.nshell;
  for (int i = threadIdx.x; i < S; i += blockDim.x) { ah_s[i] = cf.ah[i]; al_s[i] = cf.al[i]; }
  __syncthreads();
  f2 ks{0.f, 0.f};
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < cf.npix; p += gridDim.x * blockDim.x) {
    f2 acc{0.f, 0.f};
#pragma unroll 8
    for (int b = 0; b < S; ++b)
      f2_mac(acc, ah_s[b], al_s[b], float(__ldcs(counts + (size_t)b * cf.npix + p)));
    f2 e = f2_add(f2_norm(acc.h, acc.l), f2{-cf.ch, -cf.cl});
    const float kf = __fadd_rn(e.h, e.l);
    kappa[p] = kf;
    ks = f2_add(ks, f2{kf, 0.f});
  }
  const double t = block_sum_d<kKT>(f2_to_d(ks), red);
  if (threadIdx.x == 0) ksum_part[blockIdx.x] = t;
}

// Forward pass with vector loads: each thread owns 4 adjacent pixels at a time
// and reads every shell row of them as one 16-byte streaming load.  Four rows
// are in flight in registers: a row's register is loaded with the row four
// further on, or with the thread's next pixels, as soon as its counts are taken,
// so the loads never drain at the end of a map column.  The sums are
// double-float, the shells in order, two pixels side by side in the packed FP32
// instructions.  Bound by the counts' read: 60 shells at Nside 1024 take 466 us,
// 6.6 TB/s or 97% of the copy rate (scalar arithmetic with loads eight rows at a
// time: 555 us).  Other depths: 3 rows with five
// blocks per SM 509, 6 rows (spills) 481, 8 rows with three blocks 479.  Needs
// 16-byte aligned counts and kappa (12 nside^2 is a multiple of 4).
constexpr int kKV = 256, kKRows = 4;
__device__ __forceinline__ float kappa_round(f2 a, f2 mc) {
  const f2 e = f2_add(f2_norm(a.h, a.l), mc);   // e = acc - C (unrounded)
  return __fadd_rn(e.h, e.l);
}
__device__ __forceinline__ int kappa_rows(int S) { return (S + kKRows - 1) / kKRows * kKRows; }
// a += A n for two pixels: n as FP32 numbers below 2^23 (fb: 0x4B000000 | n, that
// is 2^23 + n), the operations of f2_mac
__device__ __forceinline__ void kappa_mac(dfx& a, u64 ah, u64 al, u64 fb) {
  const u64 two23 = x2_pack(8388608.0f, 8388608.0f);
  const u64 f = x2_sub(fb, two23);
  const u64 pn = x2_mul(ah, x2_sub(two23, fb));              // -A_h n
  const u64 pe = x2_fma(ah, f, pn);
  const u64 sm = x2_sub(a.h, pn), bb = x2_sub(sm, a.h);
  const u64 er = x2_sub(x2_sub(a.h, x2_sub(sm, bb)), x2_add(pn, bb));
  a.h = sm;
  a.l = x2_add(a.l, x2_add(er, x2_fma(al, f, pe)));
}
__device__ __forceinline__ u64 kappa_bits(int n0, int n1) {
  return x2_pack(__int_as_float(n0 | 0x4B000000), __int_as_float(n1 | 0x4B000000));
}
// out(g, a) with the unnormalised sums a[4] of the pixels 4 g .. 4 g + 3, for the
// groups of block vb of a grid of nb blocks of kKV threads.  cs[kappa_rows(S)]:
// (A_h, A_h, A_l, A_l) per shell, 0 above the last.
template <class Out>
__device__ __forceinline__ void kappa_stream(const int32_t* __restrict__ counts, const float4* cs,
                                             int S, int npix, int vb, int nb, Out&& out) {
  const int ng = npix >> 2, step = nb * kKV, rows = kappa_rows(S);
  const size_t stride = (size_t)npix * 4;
  const int4* c4 = reinterpret_cast<const int4*>(counts);
  auto load = [](const char* q) { return __ldcs(reinterpret_cast<const int4*>(q)); };
  int g = vb * kKV + (int)threadIdx.x;
  if (g >= ng) return;
  int4 v[kKRows];
  const char* q0 = reinterpret_cast<const char*>(c4 + g);
#pragma unroll
  for (int u = 0; u < kKRows; ++u) v[u] = u < S ? load(q0 + u * stride) : make_int4(0, 0, 0, 0);
  for (; g < ng; g += step) {
    dfx a0{0ull, 0ull}, a1{0ull, 0ull};
    unsigned nor = 0u;
    const char* q = reinterpret_cast<const char*>(c4 + g);
#pragma unroll 1
    for (int b0 = 0; b0 < rows; b0 += kKRows) {
      const bool more = b0 + kKRows < rows;                  // else the next pixels' first rows
      const int nb0 = more ? b0 + kKRows : 0;
      const bool in = more || g + step < ng;
      q = more ? q + kKRows * stride : reinterpret_cast<const char*>(c4 + g + step);
      auto take = [&](int u, auto&& next) {
        const int4 n = v[u];
        v[u] = next(u);
        nor |= (unsigned)(n.x | n.y) | (unsigned)(n.z | n.w);
        const float4 c = cs[b0 + u];
        const u64 ah = x2_pack(c.x, c.y), al = x2_pack(c.z, c.w);
        kappa_mac(a0, ah, al, kappa_bits(n.x, n.y));
        kappa_mac(a1, ah, al, kappa_bits(n.z, n.w));
      };
      if (in && nb0 + kKRows <= S) {
#pragma unroll
        for (int u = 0; u < kKRows; ++u) take(u, [&](int k) { return load(q + k * stride); });
      } else {
#pragma unroll
        for (int u = 0; u < kKRows; ++u)
          take(u, [&](int k) {
            return in && nb0 + k < S ? load(q + k * stride) : make_int4(0, 0, 0, 0);
          });
      }
    }
    f2 a[4];
    {
      const float2 h0 = x2_get(a0.h), l0 = x2_get(a0.l), h1 = x2_get(a1.h), l1 = x2_get(a1.l);
      a[0] = f2{h0.x, l0.x};
      a[1] = f2{h0.y, l0.y};
      a[2] = f2{h1.x, l1.x};
      a[3] = f2{h1.y, l1.y};
    }
    if (nor & 0xFF800000u) {               // rare: counts of 2^23 and more, or negative
      a[0] = a[1] = a[2] = a[3] = f2{0.f, 0.f};
      for (int b = 0; b < S; ++b) {
        const int4 n = c4[(size_t)b * ng + g];
        const float4 c = cs[b];
        f2_mac(a[0], c.x, c.z, float(n.x));
        f2_mac(a[1], c.x, c.z, float(n.y));
        f2_mac(a[2], c.x, c.z, float(n.z));
        f2_mac(a[3], c.x, c.z, float(n.w));
      }
    }
    out(g, a);
  }
}
// cs from the coefficients (every thread of the block; ends with a barrier)
template <class Get>
__device__ __forceinline__ void kappa_coef(float4* cs, int S, Get&& get) {
  for (int i = threadIdx.x; i < kappa_rows(S); i += blockDim.x) {
    const float2 a = i < S ? get(i) : make_float2(0.f, 0.f);
    cs[i] = make_float4(a.x, a.x, a.y, a.y);
  }
  __syncthreads();
}
// One block's share of the vector-load forward pass (every thread of the block
// calls it); returns the block's sum of the FP32 kappa values, valid in thread 0.
__device__ __forceinline__ double kappa_vec_block(const int32_t* __restrict__ counts,
                                                  const float4* cs, int S, int npix, f2 mc,
                                                  float* __restrict__ kappa, int vb, int nb,
                                                  double* red) {
  f2 ks{0.f, 0.f};
  kappa_stream(counts, cs, S, npix, vb, nb, [&](int g, const f2 (&a)[4]) {
    const float4 kv = make_float4(kappa_round(a[0], mc), kappa_round(a[1], mc),
                                  kappa_round(a[2], mc), kappa_round(a[3], mc));
    reinterpret_cast<float4*>(kappa)[g] = kv;
    ks = f2_add(ks, f2_add(f2_two_sum(kv.x, kv.y), f2_two_sum(kv.z, kv.w)));
  });
  return block_sum_d<kKV>(f2_to_d(ks), red);
}

__global__ void __launch_bounds__(kKV, 4)
k_kappa_vec(const int32_t* __restrict__ counts, const __grid_constant__ Coef cf,
            float* __restrict__ kappa, double* __restrict__ ksum_part, MomentOut mo) {
  clear_pdf(mo);
  __shared__ float4 cs[kMaxShells];
  __shared__ double red[kKV / 32];
  kappa_coef(cs, cf.nshell, [&](int i) { return make_float2(cf.ah[i], cf.al[i]); });
  const double t = kappa_vec_block(counts, cs, cf.nshell, cf.npix, f2{-cf.ch, -cf.cl}, kappa,
                                   blockIdx.x, gridDim.x, red);
  if (threadIdx.x == 0) ksum_part[blockIdx.x] = t;
}

// ----------------------------------------- subvolume partial sums -----
// Sec. 2.4 processes subvolumes independently and combines their maps; kappa
// is linear in the counts, so a subvolume contributes its partial sum
// e_p = sum_b A_b n_bp (no -C) and the map is kappa_p = (sum over
// subvolumes of e_p) - C.  The partial is accumulated in double-float over
// the shells in order, as the forward pass does, and stored as FP64 (the
// pair's sum), so that the subvolumes' partials add in FP64.
// An FP64 value as a double-float pair (h + l within 2^-48 relative).
__device__ __forceinline__ f2 d_to_f2(double v) {
  const float h = __double2float_rn(v);
  return {h, __double2float_rn(__dsub_rn(v, (double)h))};
}

__global__ void __launch_bounds__(kKV, 4)
k_kappa_partial(const int32_t* __restrict__ counts, const __grid_constant__ Coef cf,
                double* __restrict__ part) {
  __shared__ float4 cs[kMaxShells];
  kappa_coef(cs, cf.nshell, [&](int i) { return make_float2(cf.ah[i], cf.al[i]); });
  double2* o2 = reinterpret_cast<double2*>(part);
  kappa_stream(counts, cs, cf.nshell, cf.npix, blockIdx.x, gridDim.x,
               [&](int g, const f2 (&a)[4]) {
    o2[2 * g] = make_double2(f2_to_d(f2_norm(a[0].h, a[0].l)), f2_to_d(f2_norm(a[1].h, a[1].l)));
    o2[2 * g + 1] = make_double2(f2_to_d(f2_norm(a[2].h, a[2].l)),
                                 f2_to_d(f2_norm(a[3].h, a[3].l)));
  });
}

// The FP32 map from the summed partials: kappa_p = (E_p - C) in double-float
// (E_p split into a pair), rounded once to FP32, with the per-block sums of
// the map over the same grid and in the same order as k_kappa_vec, so that
// the moment pass treats it exactly as a map from the counts.
__global__ void __launch_bounds__(kKV)
k_kappa_finish(const double* __restrict__ part, float ch, float cl, int npix,
               float* __restrict__ kappa, double* __restrict__ ksum_part, MomentOut mo) {
  clear_pdf(mo);
  __shared__ double red[kKV / 32];
  const int ng = npix >> 2;
  const f2 mc{-ch, -cl};
  const double2* p2 = reinterpret_cast<const double2*>(part);
  f2 ks{0.f, 0.f};
  for (int g = blockIdx.x * kKV + threadIdx.x; g < ng; g += gridDim.x * kKV) {
    const double2 d01 = __ldcs(p2 + 2 * g), d23 = __ldcs(p2 + 2 * g + 1);
    const float4 kv = make_float4(kappa_round(d_to_f2(d01.x), mc), kappa_round(d_to_f2(d01.y), mc),
                                  kappa_round(d_to_f2(d23.x), mc), kappa_round(d_to_f2(d23.y), mc));
    reinterpret_cast<float4*>(kappa)[g] = kv;
    ks = f2_add(ks, f2_add(f2_two_sum(kv.x, kv.y), f2_two_sum(kv.z, kv.w)));
  }
  const double t = block_sum_d<kKV>(f2_to_d(ks), red);
  if (threadIdx.x == 0) ksum_part[blockIdx.x] = t;
}

// --------------------------------------------------------- adjoint -----
// One read of the counts (k_adj_main) in tiles of 2 NT pixels, two adjacent
// pixels per thread, a few blocks per SM so that one block's arithmetic overlaps
// another's loads.
//
// Bound by the latency that is left: 60 shells at Nside 1024 take 730 us for 3.0 GB
// read once (4.1 TB/s, 61% of the copy rate; 55% issue, DRAM 50%), with waits for
// loads and the barriers around phase 2; 140 shells at Nside 512 501 us (3.5 TB/s).
// Two reads with 64-bit integer multiply-adds took 1050 and 1330 us.  Counts of 256
// and more cost a tile a second read and product: 919 us for the counts of 2 x 1024^3
// binned particles (1050 in the two reads), 988 where every tile has them (1005).  A
// batch of 8 shells in flight while 8 are added (80 registers, three blocks per
// SM) against none: 930; 4 shells: 765; two blocks with 16: 830.  256-pixel tiles for
// every shell count: 780.  Phase 2's pixels split over idle warps: 875 (its sums take
// the shared memory that the loads in flight use as L1).
//
// Phase 1: e_p = sum_b A_b n_bp - C unrounded (double-float, the shells in order,
// the operations of the forward pass, two pixels side by side in packed
// registers), e_p^2, the power sums P1..P3 = sum_p e_p^k and Q = sum_p g_p, and
// the tile's maxima of |e|, e^2, |g|.  The counts' low bytes stay in shared
// memory.
//
// Quantisation: each quantity as two integers (quant2: 43 bits relative to the
// scale) with a power-of-two scale from the block's running maximum over the
// tiles it has seen; when a tile raises a maximum, the sums so far are first
// flushed at the old scale into the block's 128-bit fixed-point rows, each flush
// exactly or, where the map is so small that the rows end before its digits,
// rounded once to nearest.  Every pixel is therefore quantised at least as finely
// as a single scale from the global maxima would.
//
// Phase 2: the per-shell sums sum_p q_p n_bp are a matrix product, shells x
// pixels times pixels x quantities, on the tensor cores: the integers as signed
// 8-bit digits (three per integer, six per quantity, and one column of ones
// for N_b), the counts byte by byte, both exactly as FP16, and FP32 sums of
// products that stay whole numbers up to 2^24, which they hold exactly (1.6e7
// sums of random and of extreme digits up to 1.67e7 equal the integers on this
// GPU).  They are added to 64-bit sums in shared memory every few steps (with a
// bound of 2^22, four times as often: 759 us instead of 738 for 60 shells at Nside
// 1024, 790 instead of 737 where counts reach 100).  Counts of 256 and more take further passes
// over the tile (from L2) with their higher bytes, the last one signed.  (mma.sync:
// 16 or 24 columns are far too few for a tcgen05 tile to matter; the product
// takes 16 multiply-adds per count, a percent of the tensor cores' rate.)  With
// 64-bit integer multiply-adds in place of it, a warp per three shells, the
// counts were read a second time and phase 2 took as long as phase 1.
//
// With EXT, e comes from summed subvolume partials E_p (e = E_p - C, the same
// double-float subtraction as k_kappa_finish) and the counts, those of one
// subvolume, enter phase 2 only: the per-shell sums are then that subvolume's
// share, and they add over subvolumes.
// columns: digits of e and e^2 (6 each), ones, digits of g (6), padded to 8
__host__ __device__ constexpr int adj_cols(bool g) { return g ? 24 : 16; }
__host__ __device__ constexpr int adj_lda(int nt) { return 2 * nt + 32; }    // bytes per count row
__host__ __device__ constexpr int adj_ldb(int nt) { return 2 * nt + 32; }    // halves per column
// (row strides of 8 and 16 words modulo 32: the fragments' loads meet no bank
// conflict)
__host__ __device__ constexpr int adj_batch(int nt) { return nt < 256 ? 16 : 8; }  // shells a fetch
__host__ __device__ constexpr int adj_rows(int S) {               // whole batches, or pairs
  return (S + 15) / 16 * 16;
}
__host__ __device__ inline size_t adj_smem(int nt, int S, bool g) {
  const size_t mp = adj_rows(S), nc = adj_cols(g);
  return mp * adj_lda(nt) + nc * adj_ldb(nt) * 2 + mp * nc * 8 + (size_t)S * sizeof(AdjRow) +
         mp * sizeof(float4);
}

__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                        uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Two integers u < 1024 in the halves of w (0x6400 | u is the FP16 number
// 1024 + u), minus 1024 + off: exact.
__device__ __forceinline__ uint32_t half2_minus(uint32_t w, uint32_t bias) {
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(w), "r"(bias));
  return r;
}
constexpr uint32_t kHalf1024 = 0x64006400u;   // 1024, 1024
constexpr uint32_t kHalf1152 = 0x64806480u;   // 1152, 1152

template <bool USE_G, int NT, bool EXT>
__global__ void __launch_bounds__(NT, USE_G || NT < 256 ? 2 : 3)
k_adj_main(const int32_t* __restrict__ counts, const __grid_constant__ Coef cf,
           const float* __restrict__ g, double* __restrict__ rows_out,
           double* __restrict__ sumpart, unsigned long long* range_flag,
           float* __restrict__ kappa_out, double* __restrict__ ksum_out,
           const double* __restrict__ ext, MomentOut mo) {
  extern __shared__ __align__(16) uint8_t adj_sm[];
  constexpr int NW = NT / 32, P = 2 * NT, NC = adj_cols(USE_G);
  constexpr int LDA = adj_lda(NT), LDB = adj_ldb(NT);
  if (kappa_out) clear_pdf(mo);
  const int S = cf.nshell, npix = cf.npix, np2 = npix >> 1;
  const int mt_n = (S + 15) >> 4, mp = adj_rows(S);      // tiles of 16 shells; rows held
  uint8_t* An = adj_sm;                                      // [mp][LDA] a byte of the counts
  uint16_t* Bq = reinterpret_cast<uint16_t*>(An + (size_t)mp * LDA);            // [NC][LDB]
  long long* sums = reinterpret_cast<long long*>(Bq + (size_t)NC * LDB);        // [mp][NC]
  AdjRow* rows = reinterpret_cast<AdjRow*>(sums + (size_t)mp * NC);           // [S]
  float4* coef = reinterpret_cast<float4*>(rows + S);                           // [mp] A_b, twice
  __shared__ float mred[3][NW];
  __shared__ unsigned nred[NW];
  __shared__ double red[NW];
  const int tid = threadIdx.x, w = tid >> 5, ln = tid & 31;
  for (int i = tid; i < mp; i += NT)                         // 0 above the last shell
    coef[i] = i < S ? make_float4(cf.ah[i], cf.ah[i], cf.al[i], cf.al[i])
                    : make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = tid; i < S; i += NT) rows[i] = AdjRow{};
  for (int i = tid; i < mp * NC; i += NT) sums[i] = 0;
  // the column of ones, and zeros in the padding
  for (int i = tid; i < P / 2; i += NT) {
    reinterpret_cast<uint32_t*>(Bq + 12 * LDB)[i] = 0x3C003C00u;               // 1, 1
    for (int k = USE_G ? 19 : 13; k < NC; ++k) reinterpret_cast<uint32_t*>(Bq + k * LDB)[i] = 0u;
  }
  // running maxima of |e|, e^2, |g| over this block's tiles, in shared
  // memory: thread 0 updates them after a barrier that every thread's read
  // of them for the tile has passed
  __shared__ float Ms[3];
  if (tid == 0) Ms[0] = Ms[1] = Ms[2] = 0.f;
  auto scale = [](float M) { return M > 0.f ? min(120, 21 - ilog2f(M)) : 0; };
  // the 64-bit sums into the rows (thread t takes shells t, t + NT, ...)
  auto flush = [&](int s1, int s2, int s3) {
    for (int b = tid; b < S; b += NT) {
      AdjRow& row = rows[b];
      long long* v = sums + (size_t)b * NC;
      // (the digits put together before the shift, which rounds once per flush: with a
      // shift that drops bits for each digit, S2_b of a map near 1e-3 was 2 to 5 times
      // less exact, with one for each integer on the fewer blocks of a larger tile
      // 8e-15 at Nside 64, 40 shells)
      i128_add(row.s[0], i128_shift(i128_digits(v), kFrac1 - s1 - 22));
      i128_add(row.s[1], i128_shift(i128_digits(v + 6), kFrac2 - s2 - 22));
      if (USE_G) i128_add(row.s[2], i128_shift(i128_digits(v + 13), kFrac3 - s3 - 22));
      row.n += v[12];
      for (int k = 0; k < NC; ++k) v[k] = 0;
    }
  };
  // digits of the integers h0, h1 of the thread's two pixels into columns col,
  // col + 1, col + 2: h = d0 + 2^8 d1 + 2^16 d2, |d| <= 128
  auto digits = [&](int col, int h0, int h1) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      h0 += 128;
      h1 += 128;
      const uint32_t u = k < 2 ? (uint32_t)(h0 & 255) | (uint32_t)(h1 & 255) << 16
                               : (uint32_t)h0 | (uint32_t)h1 << 16;      // d2 + 128 in [0, 255]
      reinterpret_cast<uint32_t*>(Bq + (size_t)(col + k) * LDB)[tid] =
          half2_minus(u | kHalf1024, kHalf1152);
      h0 >>= 8;
      h1 >>= 8;
    }
  };
  // phase 2 with the byte plane in An (shift 8 plane; u_off 128 when its bytes
  // are signed), counts below `most` in it
  auto product = [&](int plane, bool sgn, unsigned most) {
    const int gq = ln >> 2, c = ln & 3;
    const uint32_t flip = sgn ? 0x80808080u : 0u, bias = sgn ? kHalf1152 : kHalf1024;
    const int steps = max(1, 4096 / (int)max(1u, min(most, 255u)));   // of 32 pixels per sum
    for (int mt = w; mt < mt_n; mt += NW) {
      const uint8_t* r0 = An + (size_t)(16 * mt + gq) * LDA + 8 * c;
      const uint8_t* r1 = r0 + 8 * LDA;
      long long* dst = sums + (size_t)(16 * mt + gq) * NC + 2 * c;
      for (int k0 = 0; k0 < P / 32; k0 += steps) {
        float acc[NC / 8][4];
#pragma unroll
        for (int j = 0; j < NC / 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
        const int k1 = min(k0 + steps, P / 32);
        for (int k = k0; k < k1; ++k) {
          uint2 x = *reinterpret_cast<const uint2*>(r0 + 32 * k);
          uint2 y = *reinterpret_cast<const uint2*>(r1 + 32 * k);
          x.x ^= flip; x.y ^= flip; y.x ^= flip; y.y ^= flip;
          // bytes 0, 1 and 2, 3 as FP16 pairs
          auto lo = [&](uint32_t v) { return half2_minus(__byte_perm(v, 0x64, 0x4140), bias); };
          auto hi = [&](uint32_t v) { return half2_minus(__byte_perm(v, 0x64, 0x4342), bias); };
          const uint32_t a0 = lo(x.x), a1 = lo(y.x), a2 = hi(x.x), a3 = hi(y.x);
          const uint32_t e0 = lo(x.y), e1 = lo(y.y), e2 = hi(x.y), e3 = hi(y.y);
#pragma unroll
          for (int j = 0; j < NC / 8; ++j) {
            const uint4 q = *reinterpret_cast<const uint4*>(Bq + (size_t)(8 * j + gq) * LDB +
                                                            32 * k + 8 * c);
            mma_f16(acc[j], a0, a1, a2, a3, q.x, q.y);
            mma_f16(acc[j], e0, e1, e2, e3, q.z, q.w);
          }
        }
#pragma unroll
        for (int j = 0; j < NC / 8; ++j) {
          auto add = [&](long long* p, float v) {
            *p += (long long)__float2int_rn(v) * (1ll << (8 * plane));
          };
          add(dst + 8 * j, acc[j][0]);
          add(dst + 8 * j + 1, acc[j][1]);
          add(dst + 8 * NC + 8 * j, acc[j][2]);
          add(dst + 8 * NC + 8 * j + 1, acc[j][3]);
        }
      }
    }
  };
  const f2 mc{-cf.ch, -cf.cl};
  const int ntile = (npix + P - 1) / P;
  // power sums: the tile's two pixels first, then into the running sums, of
  // which the threads of a narrow block (more tiles each) have two in turn, so
  // that none takes more than some tens of additions per million pixels
  constexpr int kA = NT < 256 ? 2 : 1;
  f2 pw[kA][4];
#pragma unroll
  for (int i = 0; i < 4 * kA; ++i) pw[i >> 2][i & 3] = f2{0.f, 0.f};
  f2 ks{0.f, 0.f};                         // this thread's sum of the FP32 map (kappa_out)
  // the counts in batches of kB shells, the next one's loads in flight while one
  // is added (in a second set of registers, or in the same one by one: the first
  // is faster in wide blocks, where the second spills at 80 registers, 750 against 800
  // us for 60 shells at Nside 1024; the second in narrow ones, 595 against 554 us
  // for 140 shells at Nside 512); the first batch of the next tile before phase 2
  constexpr int kB = adj_batch(NT);
  // (q: row b0 of the thread's pixels; whole tiles and batches without tests)
  const uint32_t stride = (uint32_t)npix * 4u;
  auto row = [&](const char* q, int u) {
    return reinterpret_cast<const int2*>(q + (size_t)stride * (uint32_t)u);
  };
  auto fetch = [&](int2* v, const char* q, int b0, int tile) {
    if ((tile + 1) * NT <= np2 && b0 + kB <= S) {            // (uniform)
#pragma unroll
      for (int u = 0; u < kB; ++u) v[u] = __ldg(row(q, u));
    } else {
      const bool in = tile * NT + tid < np2;
#pragma unroll
      for (int u = 0; u < kB; ++u)
        v[u] = in && b0 + u < S ? __ldg(row(q, u)) : make_int2(0, 0);
    }
  };
  const char* base = reinterpret_cast<const char*>(counts) + 8 * (size_t)tid;
  auto tile_at = [&](int tile) { return base + (size_t)tile * (8 * NT); };
  constexpr bool kTurn = NT < 256;
  int2 v0[kB], v1[kTurn ? 1 : kB];
  fetch(v0, tile_at(blockIdx.x), 0, blockIdx.x);
  __syncthreads();
  for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    // phase 1 (past the map's end: counts of 0)
    const int gi = tile * NT + tid;        // pair of pixels
    const bool have = gi < np2;
    const int2* src = reinterpret_cast<const int2*>(counts) + gi;
    uint8_t* arow = An + 2 * tid;
    dfx a{0ull, 0ull};
    unsigned nor = 0u;
    auto take = [&](int2 n, int b) {
      nor |= (unsigned)n.x | (unsigned)n.y;
      *reinterpret_cast<uint16_t*>(arow + (size_t)b * LDA) =
          (uint16_t)__byte_perm(n.x, n.y, 0x0040);
      if constexpr (!EXT) {                    // (counts of 2^23 and more: below)
        const float4 cb = coef[b];
        kappa_mac(a, x2_pack(cb.x, cb.y), x2_pack(cb.z, cb.w), kappa_bits(n.x, n.y));
      }
    };
    if constexpr (kTurn) {
      // a register takes the row kB further on as soon as its counts are used
      const char* q = tile_at(tile);
#pragma unroll 1
      for (int b0 = 0; b0 < mp; b0 += kB) {
        const bool more = b0 + kB < mp;                      // else the next tile's first batch
        const int nb0 = more ? b0 + kB : 0, nt = more ? tile : tile + (int)gridDim.x;
        q = more ? q + (size_t)stride * kB : tile_at(nt);
        if ((nt + 1) * NT <= np2 && nb0 + kB <= S) {         // (uniform)
#pragma unroll
          for (int u = 0; u < kB; ++u) {
            const int2 n = v0[u];
            v0[u] = __ldg(row(q, u));
            take(n, b0 + u);
          }
        } else {
          const bool in = nt * NT + tid < np2;
#pragma unroll
          for (int u = 0; u < kB; ++u) {
            const int2 n = v0[u];
            v0[u] = in && nb0 + u < S ? __ldg(row(q, u)) : make_int2(0, 0);
            take(n, b0 + u);
          }
        }
      }
    } else {
#pragma unroll 1
      for (int b0 = 0; b0 < mp; b0 += 2 * kB) {
        const char* q = tile_at(tile) + (size_t)stride * (uint32_t)b0;
        fetch(v1, q + (size_t)stride * kB, b0 + kB, tile);
#pragma unroll
        for (int u = 0; u < kB; ++u) take(v0[u], b0 + u);
        const bool more = b0 + 2 * kB < mp;                  // else the next tile's first batch
        const int nt = more ? tile : tile + (int)gridDim.x;
        fetch(v0, more ? q + (size_t)stride * (2 * kB) : tile_at(nt), more ? b0 + 2 * kB : 0, nt);
#pragma unroll
        for (int u = 0; u < kB; ++u) take(v1[u], b0 + kB + u);
      }
    }
    f2 av[2];
    {
      const float2 h = x2_get(a.h), l = x2_get(a.l);
      av[0] = f2{h.x, l.x};
      av[1] = f2{h.y, l.y};
    }
    if constexpr (EXT) {
      if (have) {
        const double2 d = reinterpret_cast<const double2*>(ext)[gi];
        av[0] = d_to_f2(d.x);
        av[1] = d_to_f2(d.y);
      }
    } else if (nor & 0xFF800000u) {        // rare: counts of 2^23 and more, or negative
      av[0] = av[1] = f2{0.f, 0.f};
      for (int b = 0; b < S; ++b) {
        const int2 n = src[(size_t)b * np2];
        f2_mac(av[0], coef[b].x, coef[b].z, float(n.x));
        f2_mac(av[1], coef[b].x, coef[b].z, float(n.y));
      }
    }
    const float2 gv = (USE_G && have) ? reinterpret_cast<const float2*>(g)[gi] : make_float2(0.f, 0.f);
    const float gs[2] = {gv.x, gv.y};
    f2 e[2], e2[2];
    float kv[2], t1 = 0.f, t2 = 0.f, t3 = 0.f;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      e[i] = f2_add(f2_norm(av[i].h, av[i].l), mc);
      kv[i] = __fadd_rn(e[i].h, e[i].l);       // the FP32 map, as the forward pass rounds it
      e2[i] = f2_mul(e[i], e[i]);
      if (!have) { e[i] = f2{0.f, 0.f}; e2[i] = f2{0.f, 0.f}; }
      t1 = fmaxf(t1, fabsf(e[i].h));
      t2 = fmaxf(t2, fabsf(e2[i].h));
      t3 = fmaxf(t3, fabsf(gs[i]));
    }
    if (have) {
      const f2 d[4] = {f2_add(e[0], e[1]), f2_add(e2[0], e2[1]),
                       f2_add(f2_mul(e2[0], e[0]), f2_mul(e2[1], e[1])), f2_two_sum(gs[0], gs[1])};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const f2 t = f2_add(pw[kA - 1][k], d[k]);
        if (kA > 1) pw[kA - 1][k] = pw[0][k];
        pw[0][k] = t;
      }
    }
    if (kappa_out && have) {                   // (uniform) the map itself, with its sum
      reinterpret_cast<float2*>(kappa_out)[gi] = make_float2(kv[0], kv[1]);
      ks = f2_add(ks, f2_two_sum(kv[0], kv[1]));
    }
    nor = __reduce_or_sync(0xFFFFFFFFu, nor);
    for (int o = 16; o > 0; o >>= 1) {
      t1 = fmaxf(t1, __shfl_xor_sync(0xFFFFFFFFu, t1, o));
      t2 = fmaxf(t2, __shfl_xor_sync(0xFFFFFFFFu, t2, o));
      t3 = fmaxf(t3, __shfl_xor_sync(0xFFFFFFFFu, t3, o));
    }
    if (ln == 0) { nred[w] = nor; mred[0][w] = t1; mred[1][w] = t2; mred[2][w] = t3; }
    __syncthreads();
    unsigned NOR = 0u;                         // every count <= NOR (as unsigned)
    float T1 = 0.f, T2 = 0.f, T3 = 0.f;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      NOR |= nred[i];
      T1 = fmaxf(T1, mred[0][i]);
      T2 = fmaxf(T2, mred[1][i]);
      T3 = fmaxf(T3, mred[2][i]);
    }
    const float M1 = Ms[0], M2 = Ms[1], M3 = Ms[2];
    const bool grow = T1 > M1 || T2 > M2 || T3 > M3;   // (uniform)
    const float N1 = fmaxf(M1, T1), N2 = fmaxf(M2, T2), N3 = fmaxf(M3, T3);
    const int s1 = scale(N1), s2 = scale(N2), s3 = scale(N3);
    if (grow) {
      if (tid == 0 && (N1 >= 16384.0f || N3 >= 16384.0f || N2 >= 268435456.0f))
        atomicAdd(range_flag, 1ull);
      // a maximum that stays below the next power of two leaves the scale as it is (a
      // flush costs as much as a tile: a map whose values rise along the rings paid one
      // per tile); before the first values there is nothing to flush
      const int o1 = scale(M1), o2 = scale(M2), o3 = scale(M3);
      if ((s1 != o1 || s2 != o2 || s3 != o3) && (M1 > 0.f || M2 > 0.f || M3 > 0.f))
        flush(o1, o2, o3);
    }
    {
      int h0, l0, h1, l1;
      quant2(e[0], s1, h0, l0);
      quant2(e[1], s1, h1, l1);
      digits(0, h0, h1);
      digits(3, l0, l1);
      quant2(e2[0], s2, h0, l0);
      quant2(e2[1], s2, h1, l1);
      digits(6, h0, h1);
      digits(9, l0, l1);
      if (USE_G) {
        quant2(f2{gs[0], 0.f}, s3, h0, l0);
        quant2(f2{gs[1], 0.f}, s3, h1, l1);
        digits(13, h0, h1);
        digits(16, l0, l1);
      }
    }
    __syncthreads();                       // bytes and digits complete; every thread has read Ms
    if (grow && tid == 0) { Ms[0] = N1; Ms[1] = N2; Ms[2] = N3; }
    // phase 2: the low bytes, then (rare) the higher ones
    product(0, false, NOR);
    for (int plane = 1; plane < 4 && NOR >> (8 * plane); ++plane) {
      __syncthreads();
      // (eight loads in flight, whole batches of rows without tests: 60 shells of counts
      // near 300 at Nside 1024, which need this everywhere, take 0.99 ms, 1.08 with a test
      // per row, 1.01 in the two reads with 64-bit multiply-adds that this form replaced)
      const unsigned sel = 0x0040u + 0x11u * plane;          // byte `plane` of both
      if (have) {
        const char* q = tile_at(tile);
        for (int b0 = 0; b0 < S; b0 += 8, q += 8 * (size_t)stride) {
          int2 n[8];
          if (b0 + 8 <= S) {
#pragma unroll
            for (int u = 0; u < 8; ++u) n[u] = __ldg(row(q, u));
          } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) n[u] = b0 + u < S ? __ldg(row(q, u)) : make_int2(0, 0);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u)
            *reinterpret_cast<uint16_t*>(arow + (size_t)(b0 + u) * LDA) =
                (uint16_t)__byte_perm(n[u].x, n[u].y, sel);
        }
      }
      __syncthreads();
      product(plane, plane == 3, plane == 3 ? 128u : NOR >> (8 * plane));
    }
    __syncthreads();                       // the next tile rewrites the bytes, digits and maxima
  }
  flush(scale(Ms[0]), scale(Ms[1]), scale(Ms[2]));
  double* dst = rows_out + (size_t)blockIdx.x * 4 * S;
  for (int b = tid; b < S; b += NT) {      // (this thread's own rows)
    dst[4 * b + 0] = i128_to_d(rows[b].s[0], kFrac1);
    dst[4 * b + 1] = i128_to_d(rows[b].s[1], kFrac2);
    dst[4 * b + 2] = USE_G ? i128_to_d(rows[b].s[2], kFrac3) : 0.0;
    dst[4 * b + 3] = (double)rows[b].n;
  }
  if (kappa_out) {                         // (uniform)
    const double vk = block_sum_d<NT>(f2_to_d(ks), red);
    if (tid == 0) ksum_out[blockIdx.x] = vk;
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double own = f2_to_d(pw[0][k]) + (kA > 1 ? f2_to_d(pw[kA - 1][k]) : 0.0);
    const double v = block_sum_d<NT>(own, red);
    if (tid == 0) sumpart[4 * blockIdx.x + k] = v;
  }
}

// out[k] = the sum of quantity k (4 S row entries, then 4 power sums) over the
// blocks of k_adj_main, one warp each in a fixed order; out[4 S + 4] = the range
// flag, which is cleared.
__global__ void __launch_bounds__(128)
k_adj_reduce(const double* __restrict__ rows, const double* __restrict__ sums, int S, int nblk,
             unsigned long long* range_flag, double* __restrict__ out) {
  const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (k == 0 && threadIdx.x == 0) {
    out[4 * S + 4] = (double)*range_flag;
    *range_flag = 0ull;
  }
  if (k >= 4 * S + 4) return;
  const double v = k < 4 * S ? warp_sum_fixed(rows + k, nblk, 4 * S)
                             : warp_sum_fixed(sums + (k - 4 * S), nblk, 4);
  if ((threadIdx.x & 31) == 0) out[k] = v;
}

// Per-block sums of an FP32 map (double-float per thread), the first pass of
// the moments of an arbitrary map (ufc_map_stats).  Needs a 16-byte aligned
// map of a multiple of 4 values.
__global__ void __launch_bounds__(kKV)
k_map_sum(const float* __restrict__ map, int npix, double* __restrict__ ksum_part, MomentOut mo) {
  clear_pdf(mo);
  __shared__ double red[kKV / 32];
  const int ng = npix >> 2;
  f2 ks{0.f, 0.f};
  for (int g = blockIdx.x * kKV + threadIdx.x; g < ng; g += gridDim.x * kKV) {
    const float4 v = reinterpret_cast<const float4*>(map)[g];
    ks = f2_add(ks, f2_add(f2_two_sum(v.x, v.y), f2_two_sum(v.z, v.w)));
  }
  const double t = block_sum_d<kKV>(f2_to_d(ks), red);
  if (threadIdx.x == 0) ksum_part[blockIdx.x] = t;
}

// ------------------------------------------------ moments + PDF pass -----
// Second pass over the FP32 map (L2-resident at these sizes): central
// power sums about the exact FP64 mean in double-float, and the PDF.
// PDF bin = floor((kappa - lo) * scale) in FP64; an FP32 estimate decides
// all but the values within a proven band of a bin edge.
constexpr int kMT = 256;
constexpr int kMaxBins = 4096;

struct PdfParam {
  double lo, hi, scale;     // scale = nbins / (hi - lo)
  float lo_f, scale_f, band;
  float lo_dn, lo_up, hi_dn, hi_up;   // FP32 brackets of lo and hi
  int32_t nbins;
};

// PDF slot of one FP32 value by the FP64 definition: floor((k - lo) * scale),
// under/overflow and NaN.  A call of its own: inlined, the compiler evaluates
// the FP64 expressions for every value (they have no side effects) and selects
// afterwards, and at GB300's FP64 rate that alone is 200 us for the 12.6 M
// pixels of Nside 1024.
__device__ __noinline__ int pdf_slot_exact(float k, double lo, double hi, double scale, int nbins) {
  if (isnan(k)) return nbins + 2;
  const double x = (double)k;
  if (x < lo) return nbins;
  if (x >= hi) return nbins + 1;
  const int b = (int)floor(__dmul_rn(__dsub_rn(x, lo), scale));
  return b >= nbins ? nbins - 1 : (b < 0 ? 0 : b);
}

// PDF slot of one FP32 value, decided in FP32 where the value lies outside
// the FP32 neighbours of lo and hi and farther than a proven band from every
// bin edge, else by the FP64 definition.
__device__ __forceinline__ int pdf_slot(float k, const PdfParam& pp) {
  const float x = (k - pp.lo_f) * pp.scale_f;
  float xr;
  int b = round_fast(x, xr);
  const float d = x - xr;                       // distance to the nearest edge, signed
  b = d < 0.f ? b - 1 : b;                      // floor
  const bool inside = k >= pp.lo_up && k < pp.hi_dn && fabsf(d) >= pp.band;
  if (inside) return min(max(b, 0), pp.nbins - 1);
  if (k < pp.lo_dn) return pp.nbins;
  if (k >= pp.hi_up) return pp.nbins + 1;
  return pdf_slot_exact(k, pp.lo, pp.hi, pp.scale, pp.nbins);
}

__device__ __forceinline__ float2 mean_pair(double mean) {
  const float h = (float)mean;
  return make_float2(h, (float)(mean - (double)h));
}
// One block's share of the moment pass: block vb of a grid of nb blocks of
// kMT threads (every thread calls it).  Central power sums about `mean` into
// out[0..2] (global; red holds 6 kMT / 32, 16-byte aligned); PDF counts into the shared histogram.  Two
// of a thread's pixels at a time, side by side in packed double-float.
__device__ __forceinline__ void moments_block(const float* __restrict__ kappa, int npix,
                                              float2 mean, const PdfParam& pp, int vb, int nb,
                                              unsigned int* hist, double* red, double* out) {
  const float mh = mean.x, ml = mean.y;
  const u64 nmh = x2_pack(-mh, -mh), nml = x2_pack(-ml, -ml);
  dfx a2{0ull, 0ull}, a3{0ull, 0ull}, a4{0ull, 0ull};
  // (the running sums are renormalised every four additions: low parts that grow
  // over hundreds lose bits of their own, 1e-11 of mu4 of a two-valued map of Nside
  // 4096, and each addition renormalised takes 5% longer)
  auto acc = [](dfx& a, dfx x) { a = dfx_add_raw(a, x); };
  auto norm_all = [&]() {
    a2 = dfx_norm(a2.h, a2.l);
    a3 = dfx_norm(a3.h, a3.l);
    a4 = dfx_norm(a4.h, a4.l);
  };
  auto add_pair = [&](float k0, float k1, bool both) {
    // d = (k - mh) - ml: two exact sums, renormalised
    const u64 k = x2_pack(k0, k1);
    const u64 s = x2_add(k, nmh), bb = x2_sub(s, k);
    const u64 e = x2_add(x2_sub(k, x2_sub(s, bb)), x2_sub(nmh, bb));
    dfx d = dfx_add_raw(dfx{s, e}, dfx{nml, 0ull});
    d = dfx_norm(d.h, d.l);
    if (!both) {                                       // (the second half counts as d = 0)
      d.h = x2_pack(x2_get(d.h).x, 0.f);
      d.l = x2_pack(x2_get(d.l).x, 0.f);
    }
    const dfx d2 = dfx_mul(d, d);
    acc(a2, d2);
    acc(a3, dfx_mul(d2, d));
    acc(a4, dfx_mul(d2, d2));
    atomicAdd(hist + pdf_slot(k0, pp), 1u);
    if (both) atomicAdd(hist + pdf_slot(k1, pp), 1u);
  };
  const int step = nb * kMT;
  int p = vb * kMT + threadIdx.x;
  if ((reinterpret_cast<uintptr_t>(kappa) & 15) == 0) {      // (12 nside^2 is a multiple of 4)
    // four adjacent pixels per load, the next load in flight
    const float4* k4 = reinterpret_cast<const float4*>(kappa);
    const int ng = npix >> 2;
    float4 v = p < ng ? k4[p] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int it = 0; p < ng; p += step, ++it) {
      const float4 w = v;
      if (p + step < ng) v = k4[p + step];
      add_pair(w.x, w.y, true);
      add_pair(w.z, w.w, true);
      if (it & 1) norm_all();
    }
  } else {
#pragma unroll 1
    for (int it = 0; p < npix; p += 2 * step, ++it) {
      const bool both = p < npix - step;
      const float k0 = kappa[p], k1 = both ? kappa[p + step] : k0;
      add_pair(k0, k1, both);
      if ((it & 3) == 3) norm_all();
    }
  }
  // Over the lanes in double-float, over the halves and warps in FP64 by the lanes of
  // one warp, in fixed orders.  (FP64 kept its pipe 79% busy in a batch of small maps when
  // it added the lanes, 74% when every warp converted its sums: 150 maps of Nside 64 took
  // 174 us, then 119, now 68.)
  const int w = threadIdx.x >> 5, ln = threadIdx.x & 31;
  float4* part = reinterpret_cast<float4*>(red);       // [3][kMT / 32]
  dfx q[3] = {a2, a3, a4};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    q[k] = dfx_norm(q[k].h, q[k].l);
    for (int o = 16; o > 0; o >>= 1) {
      const dfx r{__shfl_down_sync(0xFFFFFFFFu, q[k].h, o), __shfl_down_sync(0xFFFFFFFFu, q[k].l, o)};
      q[k] = dfx_add_raw(q[k], r);
      q[k] = dfx_norm(q[k].h, q[k].l);
    }
    const float2 h = x2_get(q[k].h), l = x2_get(q[k].l);
    if (ln == 0) part[kMT / 32 * k + w] = make_float4(h.x, l.x, h.y, l.y);
  }
  __syncthreads();
  static_assert(3 * kMT / 32 <= 32, "one warp adds the warps' sums");
  if (w == 0) {
    const float4 p = ln < 3 * kMT / 32 ? part[ln] : make_float4(0.f, 0.f, 0.f, 0.f);
    double v = ((double)p.x + (double)p.y) + ((double)p.z + (double)p.w);
    for (int o = kMT / 64; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    if (ln < 3 * kMT / 32 && ln % (kMT / 32) == 0) out[ln / (kMT / 32)] = v;
  }
}

// moments[10] from the partial sums, by a block of kMT threads (fixed orders:
// warp q sums quantity q; thread 0 writes).
__device__ __forceinline__ void moments_final_block(const double* ksum_part, int nksum,
                                                    const double* part, int npart, int npix,
                                                    double* red, double* m) {
  const int w = threadIdx.x >> 5;
  __syncthreads();
  if (w < 4) {
    // the mean as k_moments forms it, then the power sums
    const double s = w == 0 ? warp_sum_fixed(ksum_part, nksum, 1)
                            : warp_sum_fixed(part + (w - 1), npart, 3);
    if ((threadIdx.x & 31) == 0) red[w] = s;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double N = double(npix);
  const double mu2 = red[1] / N, mu3 = red[2] / N, mu4 = red[3] / N;
  m[0] = red[0] / N;
  m[1] = mu2;
  m[2] = mu3;
  m[3] = mu4;
  m[4] = mu3 / (mu2 * sqrt(mu2));
  m[5] = mu4 / (mu2 * mu2) - 3.0;
  m[6] = (N - 1.0) * mu2 / N;
  // Eq. 13 with every product and difference rounded on its own (explicit
  // intrinsics: no contraction can differ between the copies of this code)
  const double N3 = __dmul_rn(__dmul_rn(N, N), N);
  const double c1 = __ddiv_rn(__dmul_rn(N - 1.0, N - 1.0), N3);
  const double c2 = __ddiv_rn(__dmul_rn(N - 1.0, N - 3.0), N3);
  m[7] = __dsub_rn(__dmul_rn(c1, mu4), __dmul_rn(__dmul_rn(c2, mu2), mu2));
  m[8] = mu2 / m[7];
  m[9] = N;
}

// Blocks of the moment pass: 4 per SM (32 warps), no more than there are
// pixels for at four per thread (the loads a thread has in flight; a block of
// fewer pixels pays its prologue and its PDF's global atomics for little).  What
// bounds the pass is the latency of a pixel's chain (load, shared-memory histogram, double-float
// sums): with 2 blocks per SM and one pixel at a time it took 200 us for the
// 12.6 M pixels of Nside 1024, with four scalar loads in flight 59, with four
// pixels per load and the next load in flight 51 (6 blocks per SM 53, 8 55), 55 with the
// sums renormalised every four additions.
static int moments_grid(int num_sms, int npix) {
  return std::min(4 * num_sms, (npix + 4 * kMT - 1) / (4 * kMT));
}

// The last block to finish (ticket, cleared by the kernel before) turns the
// partial sums into the moments: one launch less, and nothing waits.
__global__ void __launch_bounds__(kMT)
k_moments(const float* __restrict__ kappa, int npix, const double* __restrict__ ksum_part,
          int nksum, PdfParam pp, double* __restrict__ part /*[grid][3]*/,
          unsigned long long* __restrict__ pdf /*[nbins+3]*/, double* __restrict__ m,
          unsigned int* __restrict__ ticket) {
  extern __shared__ unsigned int hist[];   // [nbins + 3]
  __shared__ __align__(16) double red[6 * kMT / 32];
  __shared__ float2 mean_s;                // the mean as a double-float
  __shared__ bool last_s;
  for (int i = threadIdx.x; i < pp.nbins + 3; i += blockDim.x) hist[i] = 0;
  if (threadIdx.x < 32) {
    const double s = warp_sum_fixed(ksum_part, nksum, 1);   // fixed order
    if (threadIdx.x == 0) mean_s = mean_pair(s / double(npix));
  }
  __syncthreads();
  moments_block(kappa, npix, mean_s, pp, blockIdx.x, gridDim.x, hist, red, part + 3 * blockIdx.x);
  if (threadIdx.x < 32) {
    __threadfence();                       // this block's sums before its ticket
    __syncwarp();
    if (threadIdx.x == 0) last_s = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < pp.nbins + 3; i += blockDim.x)
    if (hist[i]) atomicAdd(pdf + i, (unsigned long long)hist[i]);
  if (!last_s) return;
  __threadfence();                         // every block's sums are visible
  moments_final_block(ksum_part, nksum, part, gridDim.x, npix, red, m);
}

// Statistics vector of one map for the covariance (Eq. 10): the first six
// moments (mean, mu2, mu3, mu4, skew, kurtosis) then the PDF bins divided by
// the pixel count.
__global__ void k_stats_vector(const double* __restrict__ m, const unsigned long long* __restrict__ pdf,
                               int nbins, double* __restrict__ v) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 6 + nbins; i += gridDim.x * blockDim.x)
    v[i] = i < 6 ? m[i] : double(pdf[i - 6]) / m[9];
}

// ---------------------------------------------------------- Welford -----
// Welford update of st by the nvec vectors v [nvec][d] in order.  Element
// (i, j) of M2 takes the products dold_i dnew_j of the vectors as one chain of
// fused multiply-adds (dold = x - mean before, dnew = x - mean after), so the
// elements are independent given the deltas, and a component's deltas are one
// short chain (difference, mean += delta (1 / n), difference).  A block owns 16 x 16
// elements: its first 256 threads hold one each in a register, and one more
// warp forms the deltas of the block's 16 rows and 16 columns, run after run
// of kWfRun vectors into the other of two buffers while the run before is
// added.  (The chains are the same whatever the blocks: the result does not
// depend on how the vectors are split over calls.)  Every block reads the old
// mean and count, so they are written last: by a second launch, k_welford_mean,
// which forms the mean's chain once more.  The update then keeps nothing outside
// the caller's state: updates of different states may overlap on different
// streams, and a captured one allocates nothing.  The batched call, which has
// scratch of its own anyway, passes a place for the new mean and a count of
// finished blocks (0 at launch) instead, and the last block to finish copies the
// mean: 200 vectors' chain, formed again, takes some 20 us of latency.
//
// FP64 at 1/64 of the FP32 rate bounds it: one block of 1024 threads took 12 us
// for one vector of 206 components and 2 ms for 150 (the tail of a batched
// call); spread over 169 blocks they share the chip's FP64 pipes.
constexpr int kWfTile = 16;
constexpr int kWfThreads = kWfTile * kWfTile + 32;
constexpr int kWfRun = 16;
// One run of the chain of component `comp` by one warp (comp per lane, all lanes
// call it): vectors r0 .. r0 + kWfRun - 1, the mean m carried on, out(q, dold, dnew)
// for each.
template <class Out>
__device__ __forceinline__ void welford_run(const double* __restrict__ v, int nvec, int d, int comp,
                                            double n0, int r0, double& m, Out&& out) {
  // the run's values first (their loads in flight together) and 1 / n of
  // its vectors, one per lane; the chain is then three operations a vector
  const double rn = 1.0 / (n0 + double(r0 + ((int)threadIdx.x & (kWfRun - 1)) + 1));
  double x[kWfRun];
#pragma unroll
  for (int q = 0; q < kWfRun; ++q)
    x[q] = comp < d && r0 + q < nvec ? v[(size_t)(r0 + q) * d + comp] : 0.0;
#pragma unroll
  for (int q = 0; q < kWfRun; ++q) {
    const double r = __shfl_sync(0xFFFFFFFFu, rn, q);
    const double a = x[q] - m;
    const double mq = __fma_rn(a, r, m);
    if (r0 + q < nvec) m = mq;
    out(q, a, x[q] - mq);
  }
}

__global__ void __launch_bounds__(kWfThreads)
k_welford_update(const double* __restrict__ v, int nvec, int d, double* __restrict__ st,
                 double* __restrict__ mean_new, unsigned int* __restrict__ ticket) {
  __shared__ double dold[2][kWfRun][kWfTile], dnew[2][kWfRun][kWfTile];
  __shared__ bool last_s;
  double* mean = st + 1;
  double* M2 = st + 1 + d;
  const double n0 = st[0];
  const int i0 = blockIdx.y * kWfTile, j0 = blockIdx.x * kWfTile;
  const int t = threadIdx.x;
  const bool maker = t >= kWfTile * kWfTile;         // the warp that forms the deltas
  const int lane = t & 31;
  const int comp = (lane < kWfTile ? i0 : j0 - kWfTile) + lane;   // its component
  double m = maker && comp < d ? mean[comp] : 0.0;
  const int i = i0 + t / kWfTile, j = j0 + t % kWfTile;
  const bool mine = !maker && i < d && j < d;
  double acc = mine ? M2[(size_t)i * d + j] : 0.0;
  auto make = [&](int r0, int buf) {                 // (the maker warp)
    welford_run(v, nvec, d, comp, n0, r0, m, [&](int q, double a, double b) {
      if (lane < kWfTile) dold[buf][q][lane] = a;
      else dnew[buf][q][lane - kWfTile] = b;
    });
  };
  if (maker) make(0, 0);
  __syncthreads();
  for (int r0 = 0, buf = 0; r0 < nvec; r0 += kWfRun, buf ^= 1) {
    if (maker) {
      if (r0 + kWfRun < nvec) make(r0 + kWfRun, buf ^ 1);
    } else {
      const int nr = min(kWfRun, nvec - r0);
      for (int q = 0; q < nr; ++q)
        acc = __fma_rn(dold[buf][q][t / kWfTile], dnew[buf][q][t % kWfTile], acc);
    }
    __syncthreads();
  }
  if (mine) M2[(size_t)i * d + j] = acc;
  if (!mean_new) return;                             // (uniform) k_welford_mean follows
  if (maker && blockIdx.x == 0 && lane < kWfTile && comp < d) mean_new[comp] = m;
  __threadfence();                                   // the means before the ticket
  __syncthreads();
  if (t == 0) last_s = atomicAdd(ticket, 1u) == gridDim.x * gridDim.y - 1;
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  for (int k = t; k < d; k += kWfThreads) mean[k] = __ldcg(mean_new + k);
  if (t == 0) st[0] = n0 + double(nvec);
}

// The mean and the count after k_welford_update: one cluster, so that the count
// is written after every block has read it.
constexpr int kWfCluster = 8;
__global__ void __cluster_dims__(kWfCluster, 1, 1) __launch_bounds__(256)
k_welford_mean(const double* __restrict__ v, int nvec, int d, double* __restrict__ st) {
  const double n0 = st[0];
  const int lane = threadIdx.x & 31, nth = gridDim.x * blockDim.x;
  for (int c0 = blockIdx.x * blockDim.x + threadIdx.x - lane; c0 < d; c0 += nth) {
    const int comp = c0 + lane;
    double m = comp < d ? st[1 + comp] : 0.0;
    for (int r0 = 0; r0 < nvec; r0 += kWfRun)
      welford_run(v, nvec, d, comp, n0, r0, m, [](int, double, double) {});
    if (comp < d) st[1 + comp] = m;
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
  if (blockIdx.x == 0 && threadIdx.x == 0) st[0] = n0 + double(nvec);
}

// One vector into a state of up to kWfOne components (a map at a time) by one
// cluster in one launch: the operations of the two kernels above.  Such a caller is
// bound by the host, and a second launch costs it more than the arithmetic on 8 SMs:
// bin, kappa, vector and update of a map of Nside 64 take 104 us with one launch,
// 110 with two (medians of 12 processes each).
constexpr int kWfOne = 256, kWfOneThreads = 512;
__global__ void __cluster_dims__(kWfCluster, 1, 1) __launch_bounds__(kWfOneThreads)
k_welford_one(const double* __restrict__ v, int d, double* __restrict__ st) {
  __shared__ double dold[kWfOne], dnew[kWfOne], rn_s;
  constexpr int kV = 8;                              // elements in flight per thread
  const int t = threadIdx.x, step = kWfCluster * kWfOneThreads;
  const double n0 = st[0];
  double* M2 = st + 1 + d;
  double x = 0.0, m = 0.0;
  if (t < d) { x = v[t]; m = st[1 + t]; }
  int k = blockIdx.x * kWfOneThreads + t;
  double acc[kV];
#pragma unroll
  for (int u = 0; u < kV; ++u) acc[u] = k + u * step < d * d ? M2[k + u * step] : 0.0;
  if (t == 0) rn_s = 1.0 / (n0 + 1.0);
  __syncthreads();
  double mq = 0.0;
  if (t < d) {
    const double a = x - m;
    mq = __fma_rn(a, rn_s, m);
    dold[t] = a;
    dnew[t] = x - mq;
  }
  __syncthreads();
  for (; k < d * d; k += kV * step) {
#pragma unroll
    for (int u = 0; u < kV; ++u) {
      const int q = k + u * step;
      if (q < d * d) M2[q] = __fma_rn(dold[q / d], dnew[q % d], acc[u]);
      const int nq = q + kV * step;
      acc[u] = nq < d * d ? M2[nq] : 0.0;
    }
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
  if (blockIdx.x != 0) return;
  if (t < d) st[1 + t] = mq;
  if (t == 0) st[0] = n0 + 1.0;
}

__global__ void __launch_bounds__(1024)
k_welford_merge(double* __restrict__ a, const double* __restrict__ b, int d) {
  const double na = a[0], nb = b[0], n = na + nb;
  if (nb == 0.0) return;
  double* ma = a + 1;
  const double* mb = b + 1;
  double* Ma = a + 1 + d;
  const double* Mb = b + 1 + d;
  const double f = (n > 0.0) ? na * nb / n : 0.0;
  for (int k = threadIdx.x; k < d * d; k += blockDim.x) {
    const int i = k / d, j = k - i * d;
    Ma[k] += Mb[k] + (mb[i] - ma[i]) * (mb[j] - ma[j]) * f;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < d; i += blockDim.x) ma[i] += (mb[i] - ma[i]) * nb / n;
  __syncthreads();
  if (threadIdx.x == 0) a[0] = n;
}

__global__ void __launch_bounds__(1024)
k_welford_final(const double* __restrict__ st, int d, int ddof, double* __restrict__ mean,
                double* __restrict__ cov, double* __restrict__ corr) {
  const double n = st[0];
  const double den = n - double(ddof);
  for (int i = threadIdx.x; i < d; i += blockDim.x) mean[i] = st[1 + i];
  for (int k = threadIdx.x; k < d * d; k += blockDim.x) cov[k] = st[1 + d + k] / den;
  __syncthreads();
  for (int k = threadIdx.x; k < d * d; k += blockDim.x) {
    const int i = k / d, j = k - i * d;
    const double q = sqrt((st[1 + d + i * d + i] / den) * (st[1 + d + j * d + j] / den));
    corr[k] = q > 0.0 ? (st[1 + d + k] / den) / q : 0.0;
  }
}

// --------------------------------------------------------- batched maps --
// Realisations of small maps in one call (Sec. 3.2: statistics over many
// realisations), a launch per stage over all of them: the binning (k_direct,
// direct.cu, with one item per (realisation, box)), then the kappa maps, the
// moments with PDF and statistics vector, and the Welford update.  Blocks
// (x, r) of the kappa and moment stages do what block x of the one-at-a-time
// kernels does for realisation r (kappa_vec_block, moments_block with the same
// grids), so the results equal those calls bit for bit.  (One persistent
// kernel that binned one particle per thread with every stage inline, finished
// each realisation in one block and ran the Welford update in the last one took
// 6.1 ms for 150 realisations of 2 x 64^3 particles.)
struct BatchCoef {          // per realisation: C, then the coefficients [S]
  float2 c, a[1];
};
__host__ __device__ inline size_t batch_coef_stride(int S) {
  return ((size_t)(S + 1) * sizeof(float2) + 15) / 16 * 16;
}
struct BatchArgs {
  const char* coef;         // [nreal] BatchCoef, batch_coef_stride(S) apart
  int32_t S, npix;
  int32_t* counts;          // [nreal][S][npix]
  float* kappa;             // [nreal][npix]
  double* ksum;             // [nreal][gk]
  double* mpart;            // [nreal][3 gm]
  int32_t gk, gm;           // grids of the serial kappa and moment passes
  double* moments;          // [nreal][10]
  int64_t* pdf;             // [nreal][nbins + 3]
  double* stats;            // [nreal][d]
  int32_t nbins, d;
  unsigned int* done;       // [nreal] blocks of the moment pass finished (zero at launch)
};

__global__ void __launch_bounds__(kKV, 4)
k_batch_kappa(const __grid_constant__ BatchArgs ba) {
  __shared__ float4 cs[kMaxShells];
  __shared__ double red[kKV / 32];
  const int r = blockIdx.y, S = ba.S;
  clear_pdf(MomentOut{(unsigned long long*)ba.pdf + (size_t)(ba.nbins + 3) * r, ba.nbins + 3,
                      nullptr});
  const BatchCoef& cf = *reinterpret_cast<const BatchCoef*>(ba.coef + batch_coef_stride(S) * r);
  kappa_coef(cs, S, [&](int i) { return make_float2(cf.a[i].x, cf.a[i].y); });
  const double t = kappa_vec_block(ba.counts + (size_t)r * S * ba.npix, cs, S, ba.npix,
                                   f2{-cf.c.x, -cf.c.y}, ba.kappa + (size_t)r * ba.npix,
                                   blockIdx.x, ba.gk, red);
  if (threadIdx.x == 0) ba.ksum[(size_t)r * ba.gk + blockIdx.x] = t;
}

__global__ void __launch_bounds__(kMT)
k_batch_moments(const __grid_constant__ BatchArgs ba, const __grid_constant__ PdfParam pp) {
  extern __shared__ unsigned int hist[];   // [nbins + 3]
  __shared__ __align__(16) double red[6 * kMT / 32];
  __shared__ float2 mean_s;                // the mean as a double-float
  __shared__ bool last_s;
  const int r = blockIdx.y;
  const double* ks = ba.ksum + (size_t)r * ba.gk;
  double* mp = ba.mpart + (size_t)r * 3 * ba.gm;
  int64_t* pd = ba.pdf + (size_t)(ba.nbins + 3) * r;
  for (int i = threadIdx.x; i < ba.nbins + 3; i += blockDim.x) hist[i] = 0;
  if (threadIdx.x < 32) {
    const double s = warp_sum_fixed(ks, ba.gk, 1);          // fixed order, as k_moments
    if (threadIdx.x == 0) mean_s = mean_pair(s / double(ba.npix));
  }
  __syncthreads();
  moments_block(ba.kappa + (size_t)r * ba.npix, ba.npix, mean_s, pp, blockIdx.x, ba.gm, hist, red,
                mp + 3 * blockIdx.x);
  for (int i = threadIdx.x; i < ba.nbins + 3; i += blockDim.x)
    if (hist[i]) atomicAdd((unsigned long long*)pd + i, (unsigned long long)hist[i]);
  __threadfence();                         // sums and PDF before this block's count
  __syncthreads();
  if (threadIdx.x == 0) last_s = atomicAdd(ba.done + r, 1u) == (unsigned)(ba.gm - 1);
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  double* mo = ba.moments + 10 * (size_t)r;
  moments_final_block(ks, ba.gk, mp, ba.gm, ba.npix, red, mo);
  __syncthreads();
  double* v = ba.stats + (size_t)ba.d * r;
  for (int i = threadIdx.x; i < ba.d; i += blockDim.x)
    v[i] = i < 6 ? mo[i] : double(__ldcg(pd + i - 6)) / mo[9];
}

// ============================================================== host =====

// Index-check record of this translation unit (checked builds), read and
// cleared on the context stream.
cudaError_t take_checks_stats(CheckRec* out, cudaStream_t s) { return take_check_rec(out, s); }

static void make_coef(const double* A, double C, int S, int npix, Coef& cf) {
  std::memset(&cf, 0, sizeof cf);
  for (int b = 0; b < S; ++b) {
    cf.ah[b] = (float)A[b];
    cf.al[b] = (float)(A[b] - (double)cf.ah[b]);
  }
  cf.ch = (float)C;
  cf.cl = (float)(C - (double)cf.ch);
  cf.nshell = S;
  cf.npix = npix;
}

static ufc_status check_kappa_args(ufc_ctx* c, const int32_t* counts, int S, int nside,
                                   const double* A, double C) {
  if (!counts) return set_err(c, UFC_ERR_ARG, "counts_dev is NULL");
  if (S < 1 || S > kMaxShells) return set_err(c, UFC_ERR_ARG, "nshell must be in [1,%d]", kMaxShells);
  if (nside < 1 || nside > UFC_MAX_NSIDE || (nside & (nside - 1)))
    return set_err(c, UFC_ERR_ARG, "nside must be a power of two in [1,%d]", UFC_MAX_NSIDE);
  if ((int64_t)S * 12 * nside * nside >= (1ll << 31))
    return set_err(c, UFC_ERR_ARG, "nshell * 12 nside^2 must be < 2^31");
  if (!A) return set_err(c, UFC_ERR_ARG, "A is NULL");
  for (int b = 0; b < S; ++b)
    if (!std::isfinite(A[b])) return set_err(c, UFC_ERR_ARG, "A[%d] is not finite", b);
  if (!std::isfinite(C)) return set_err(c, UFC_ERR_ARG, "C is not finite");
  return UFC_OK;
}


// Forward kappa pass shared by ufc_kappa_stats and its allocation-free
// variant (identical results): grid blocks, one partial sum each in ksum.
static int kappa_fwd_grid(const ufc_ctx* c, int npix) {   // blocks with work only
  return std::min(8 * c->num_sms, (npix / 4 + kKV - 1) / kKV);
}
static ufc_status launch_kappa_fwd(ufc_ctx* c, const int32_t* counts, const Coef& cf,
                                   float* kappa, double* ksum, int grid, const MomentOut& mo) {
  if ((reinterpret_cast<uintptr_t>(kappa) & 15) == 0) {
    k_kappa_vec<<<grid, kKV, 0, c->stream>>>(counts, cf, kappa, ksum, mo);
  } else {
    k_kappa_plain<<<grid, kKT, 0, c->stream>>>(counts, cf, kappa, ksum, mo);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}


// Scratch of a map pass and the moment pass after it, in doubles: the block sums
// of `grid` blocks, three sums for each of `mgrid`, and the moment pass's count of
// finished blocks.  (Each pass's own, so that passes with different scratch may
// overlap on different streams.)
static size_t pass_doubles(int grid, int mgrid) { return (size_t)grid + 3 * (size_t)mgrid + 1; }
static MomentOut moment_out(double* mpart, int mgrid, int64_t* pdf, int nbins) {
  return MomentOut{reinterpret_cast<unsigned long long*>(pdf), nbins + 3,
                   reinterpret_cast<unsigned int*>(mpart + 3 * mgrid)};
}

// Moments and PDF of an FP32 map whose per-block sums (grid of them) are in
// ksum: the second pass over the map and the final reduction.
static PdfParam make_pdf_param(double lo, double hi, int nbins) {
  PdfParam pp;
  pp.lo = lo;
  pp.hi = hi;
  pp.scale = (double)nbins / (hi - lo);
  pp.lo_f = (float)lo;
  pp.scale_f = (float)pp.scale;
  pp.nbins = nbins;
  // |x_f - x_64| <= u |lo| s + 3u |x| + 2^-52 |x| (u = 2^-24) with x in
  // [0, nbins]; the band is twice that at x = nbins.  A range whose band
  // passes 1/4 sends every value through the FP64 expression.  (With a band
  // that held for |lo| s < 16 only, a range of +- 6 sigma in 200 bins took the
  // FP64 expression for every pixel: 200 us of the Nside-1024 map's moment
  // pass.)
  const double band = std::ldexp(1.0, -23) * (std::fabs(lo) * pp.scale + 3.0 * nbins + 4.0);
  pp.band = band < 0.25 ? (float)band : 2.0f;
  auto fdn = [](double v) { float f = (float)v; return (double)f > v ? nextafterf(f, -INFINITY) : f; };
  auto fup = [](double v) { float f = (float)v; return (double)f < v ? nextafterf(f, INFINITY) : f; };
  pp.lo_dn = fdn(lo);
  pp.lo_up = fup(lo);
  pp.hi_dn = fdn(hi);
  pp.hi_up = fup(hi);
  return pp;
}

// (the PDF and the count have been cleared by the kernel that wrote ksum)
static ufc_status launch_moments(ufc_ctx* c, const float* kmap, int npix, const double* ksum,
                                 int grid, double lo, double hi, int nbins, double* mpart,
                                 double* moments, int64_t* pdf, bool timed) {
  const PdfParam pp = make_pdf_param(lo, hi, nbins);
  const int smem = (nbins + 3) * 4;
  {
    ProfScope ps_(timed ? c : nullptr, "k_moments");
    const int mgrid = moments_grid(c->num_sms, npix);
    const MomentOut mo = moment_out(mpart, mgrid, pdf, nbins);
    k_moments<<<mgrid, kMT, smem, c->stream>>>(kmap, npix, ksum, grid, pp, mpart, mo.pdf, moments,
                                               mo.ticket);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

// Moments and PDF of any FP32 RING map (smoothed maps of Sec. 3.3).
ufc_status run_map_stats(ufc_ctx* c, const float* map, int nside, double lo, double hi,
                         int nbins, double* moments, int64_t* pdf) {
  if (!map || !moments || !pdf) return set_err(c, UFC_ERR_ARG, "map, moments and pdf are required");
  if (nside < 1 || nside > UFC_MAX_NSIDE || (nside & (nside - 1)))
    return set_err(c, UFC_ERR_ARG, "nside must be a power of two in [1,%d]", UFC_MAX_NSIDE);
  if (nbins < 1 || nbins > kMaxBins) return set_err(c, UFC_ERR_ARG, "nbins must be in [1,%d]", kMaxBins);
  if (!(hi > lo) || !std::isfinite(lo) || !std::isfinite(hi))
    return set_err(c, UFC_ERR_ARG, "PDF range needs finite lo < hi");
  if (reinterpret_cast<uintptr_t>(map) & 15) return set_err(c, UFC_ERR_ARG, "map_dev must be 16-byte aligned");
  const int npix = 12 * nside * nside;
  const int grid = kappa_fwd_grid(c, npix), mgrid = moments_grid(c->num_sms, npix);
  double* ksum = (double*)ws_get(c, kSlotPartials, pass_doubles(grid, mgrid) * 8);
  if (!ksum) return UFC_ERR_ALLOC;
  {
    ProfScope ps_(c, "k_map_sum");
    k_map_sum<<<grid, kKV, 0, c->stream>>>(map, npix, ksum,
                                           moment_out(ksum + grid, mgrid, pdf, nbins));
  }
  UFC_CUDA(c, cudaGetLastError());
  return launch_moments(c, map, npix, ksum, grid, lo, hi, nbins, ksum + grid, moments, pdf, true);
}

ufc_status run_kappa_stats(ufc_ctx* c, const int32_t* counts, int S, int nside,
                           const double* A, double C, double lo, double hi, int nbins,
                           float* kappa, double* moments, int64_t* pdf) {
  ufc_status s = check_kappa_args(c, counts, S, nside, A, C);
  if (s) return s;
  const int npix = 12 * nside * nside;
  const bool want_stats = moments || pdf;
  if (want_stats) {
    if (nbins < 1 || nbins > kMaxBins)
      return set_err(c, UFC_ERR_ARG, "nbins must be in [1,%d]", kMaxBins);
    if (!(hi > lo) || !std::isfinite(lo) || !std::isfinite(hi))
      return set_err(c, UFC_ERR_ARG, "PDF range needs finite lo < hi");
    if (!moments || !pdf)
      return set_err(c, UFC_ERR_ARG, "moments_dev and pdf_dev go together");
  }
  Coef cf;
  make_coef(A, C, S, npix, cf);
  if (reinterpret_cast<uintptr_t>(counts) & 15)
    return set_err(c, UFC_ERR_ARG, "counts_dev must be 16-byte aligned");
  const int grid = kappa_fwd_grid(c, npix);
  const int mgrid = moments_grid(c->num_sms, npix);
  double* ksum = (double*)ws_get(c, kSlotPartials, pass_doubles(grid, mgrid) * 8);
  if (!ksum) return UFC_ERR_ALLOC;
  double* mpart = ksum + grid;
  float* kmap = kappa;
  if (!kmap && want_stats) {
    kmap = (float*)ws_get(c, kSlotMisc, (size_t)npix * 4);
    if (!kmap) return UFC_ERR_ALLOC;
  }
  if (!kmap) return UFC_OK;   // nothing requested
  {
    ProfScope ps_(c, "k_kappa");
    s = launch_kappa_fwd(c, counts, cf, kmap, ksum, grid, moment_out(mpart, mgrid, pdf, nbins));
    if (s) return s;
  }
  if (!want_stats) return UFC_OK;
  return launch_moments(c, kmap, npix, ksum, grid, lo, hi, nbins, mpart, moments, pdf, true);
}

// The adjoint's device pass and its reduction to the sums
// out[4 b + k] (b < S: S1_b = sum_p e_p n_bp, S2_b = sum_p e_p^2 n_bp,
// T_b = sum_p g_p n_bp, N_b = sum_p n_bp) and out[4 S + k] (P1, P2, P3 =
// sum_p e_p^k, Q = sum_p g_p).  e is built from the counts with A (ext NULL)
// or taken from summed subvolume partials ext (e = ext - C).  With kappa
// (non-NULL) the same launch writes the FP32 map and its block sums and the
// moment pass gives moments and PDF.  Synchronises.
static ufc_status adjoint_sums(ufc_ctx* c, const int32_t* counts, int S, int nside,
                               const Coef& cf, const double* ext, const float* g, float* kappa,
                               double lo, double hi, int nbins, double* moments, int64_t* pdf,
                               double* out) {
  if (kappa) {
    if (!moments || !pdf) return set_err(c, UFC_ERR_ARG, "moments_dev and pdf_dev are required");
    if (reinterpret_cast<uintptr_t>(kappa) & 15)
      return set_err(c, UFC_ERR_ARG, "kappa_dev must be 16-byte aligned");
    if (nbins < 1 || nbins > kMaxBins)
      return set_err(c, UFC_ERR_ARG, "nbins must be in [1,%d]", kMaxBins);
    if (!(hi > lo) || !std::isfinite(lo) || !std::isfinite(hi))
      return set_err(c, UFC_ERR_ARG, "PDF range needs finite lo < hi");
  }
  if (reinterpret_cast<uintptr_t>(counts) & 15)
    return set_err(c, UFC_ERR_ARG, "counts_dev must be 16-byte aligned");
  if (g && (reinterpret_cast<uintptr_t>(g) & 15))
    return set_err(c, UFC_ERR_ARG, "g_dev must be 16-byte aligned");
  if (ext && (reinterpret_cast<uintptr_t>(ext) & 15))
    return set_err(c, UFC_ERR_ARG, "partial_dev must be 16-byte aligned");
  const int npix = 12 * nside * nside;
  // threads per block and blocks per SM: 512-pixel tiles where two blocks' shared
  // memory fits an SM (up to 128 shells, 96 with g), 256-pixel tiles above
  // (Nside 512, wide against narrow tiles: 100 shells 366 and 405 us, 128 shells
  // 421 and 451, 90 with g 349 and 397; 140 shells, one wide block per SM, 657
  // and 515)
  const size_t sm_bytes = (size_t)c->smem_optin;             // (per block; an SM holds 1 KB more)
  const bool wide = 2 * (adj_smem(256, S, g != nullptr) + 1024) <= sm_bytes + 1024;
  const int nt = wide ? 256 : 128;
  const size_t smem2 = adj_smem(nt, S, g != nullptr);
  const int per_sm = std::max(1, std::min(g || !wide ? 2 : 3, (int)((sm_bytes + 1024) / (smem2 + 1024))));
  const int grid2 = std::min(per_sm * c->num_sms, (npix + 2 * nt - 1) / (2 * nt));
  const size_t nrow = (size_t)grid2 * 4 * S, nsum = (size_t)grid2 * 4;
  const int mgrid = moments_grid(c->num_sms, npix);
  const size_t nmap = kappa ? pass_doubles(grid2, mgrid) : 0;   // map sums, moment partials
  const size_t nout = 4 * (size_t)S + 5;
  double* part = (double*)ws_get(c, kSlotPartials, (nrow + nsum + nmap + nout) * 8);
  if (!part) return UFC_ERR_ALLOC;
  double* rows = part;
  double* sums = part + nrow;
  double* ksum = sums + nsum;
  double* mpart = ksum + grid2;
  double* dout = part + nrow + nsum + nmap;
  BinCounters* bc = reinterpret_cast<BinCounters*>(c->counters);
  const MomentOut mo = moment_out(mpart, mgrid, pdf, nbins);     // (used with kappa only)
  {
    ProfScope ps_(c, "k_adj_main");
#define UFC_ADJ(G, NT_, X)                                                                        \
  do {                                                                                            \
    UFC_CUDA(c, cudaFuncSetAttribute(k_adj_main<G, NT_, X>,                                       \
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2));   \
    k_adj_main<G, NT_, X><<<grid2, NT_, smem2, c->stream>>>(                                      \
        counts, cf, g, rows, sums, &bc->range, kappa, ksum, ext, mo);                             \
  } while (0)
#define UFC_ADJ_X(G, NT_)                                                                         \
  do {                                                                                            \
    if (ext) UFC_ADJ(G, NT_, true);                                                               \
    else UFC_ADJ(G, NT_, false);                                                                  \
  } while (0)
    if (g && wide) UFC_ADJ_X(true, 256);
    else if (g) UFC_ADJ_X(true, 128);
    else if (wide) UFC_ADJ_X(false, 256);
    else UFC_ADJ_X(false, 128);
#undef UFC_ADJ_X
#undef UFC_ADJ
  }
  {
    ProfScope ps_(c, "k_adj_reduce");
    k_adj_reduce<<<(int)(nout + 3) / 4, 128, 0, c->stream>>>(rows, sums, S, grid2, &bc->range, dout);
  }
  UFC_CUDA(c, cudaGetLastError());
  if (kappa) {                             // moments and PDF of the map just written
    ufc_status s = launch_moments(c, kappa, npix, ksum, grid2, lo, hi, nbins, mpart, moments, pdf,
                                  true);
    if (s) return s;
  }
  double hp[4 * kMaxShells + 5];
  UFC_CUDA(c, cudaMemcpyAsync(hp, dout, nout * 8, cudaMemcpyDeviceToHost, c->stream));
  UFC_CUDA(c, cudaStreamSynchronize(c->stream));
  if (hp[4 * S + 4] != 0.0)
    return set_err(c, UFC_ERR_UNSUPPORTED,
                   "adjoint needs |kappa_p| < 2^14 and |g_p| < 2^14 (fixed-point range)");
  std::memcpy(out, hp, (4 * (size_t)S + 4) * 8);
  return UFC_OK;
}

// dL/dtheta from the adjoint sums (layout of adjoint_sums), host FP64.
void grad_from_sums(const double* sm, int S, int npix, double w_var, double w_skew,
                    const double* dA, const double* dC, double* grad, double* G, double* H) {
  // central moments of the unrounded map from the raw sums about 0
  const double N = npix;
  const double P1 = sm[4 * S], P2 = sm[4 * S + 1], P3 = sm[4 * S + 2], Q = sm[4 * S + 3];
  const double m1 = P1 / N, r2 = P2 / N, r3 = P3 / N;
  const double mu2 = r2 - m1 * m1;
  const double mu3 = r3 - 3.0 * m1 * r2 + 2.0 * m1 * m1 * m1;
  // G_b = sum_p gbar_p n_bp with
  //   dvar/dk_p  = 2 (k_p - m)/N
  //   dskew/dk_p = 3[(k_p - m)^2 - mu2] mu2^-3/2 / N - 3 mu3 mu2^-5/2 (k_p - m)/N
  std::vector<double> Gb(S);
  const double i32 = 1.0 / (mu2 * std::sqrt(mu2));
  const double i52 = i32 / mu2;
  for (int b = 0; b < S; ++b) {
    const double S1 = sm[4 * b], S2 = sm[4 * b + 1], T = sm[4 * b + 2], Nb = sm[4 * b + 3];
    const double c1 = S1 - m1 * Nb;                             // sum (k-m) n
    const double c2 = S2 - 2.0 * m1 * S1 + m1 * m1 * Nb;        // sum (k-m)^2 n
    const double gv = 2.0 * c1 / N;
    const double gs = 3.0 * (c2 - mu2 * Nb) * i32 / N - 3.0 * mu3 * i52 * c1 / N;
    Gb[b] = w_var * gv + w_skew * gs + T;
  }
  const double Hs = Q;   // var and skew are shift invariant: their H is 0
  for (int j = 0; j < 5; ++j) {
    double acc = 0.0;
    for (int b = 0; b < S; ++b) acc += dA[j * S + b] * Gb[b];
    grad[j] = acc - dC[j] * Hs;
  }
  if (G)
    for (int b = 0; b < S; ++b) G[b] = Gb[b];
  if (H) *H = Hs;
}

// Adjoint sums -> gradients (host FP64 assembly).  Synchronises.
// With kappa (non-NULL) the same launch also writes the FP32 map and its
// block sums, and the moment pass gives moments and PDF
// (ufc_kappa_stats_backward).
ufc_status run_kappa_backward_ex(ufc_ctx* c, const int32_t* counts, int S, int nside,
                                 const double* A, double C, double w_var, double w_skew,
                                 const float* g, const double* dA, const double* dC,
                                 double* grad, double* G, double* H, float* kappa, double lo,
                                 double hi, int nbins, double* moments, int64_t* pdf) {
  ufc_status s = check_kappa_args(c, counts, S, nside, A, C);
  if (s) return s;
  if (!grad) return set_err(c, UFC_ERR_ARG, "grad_theta is NULL");
  if (!dA || !dC) return set_err(c, UFC_ERR_ARG, "dA and dC are required");
  const int npix = 12 * nside * nside;
  Coef cf;
  make_coef(A, C, S, npix, cf);
  std::vector<double> sm(4 * (size_t)S + 4);
  s = adjoint_sums(c, counts, S, nside, cf, nullptr, g, kappa, lo, hi, nbins, moments, pdf,
                   sm.data());
  if (s) return s;
  grad_from_sums(sm.data(), S, npix, w_var, w_skew, dA, dC, grad, G, H);
  return UFC_OK;
}

// ---- subvolume partial sums (Sec. 2.4) --------------------------------------
ufc_status run_kappa_partial(ufc_ctx* c, const int32_t* counts, int S, int nside,
                             const double* A, double* partial) {
  ufc_status s = check_kappa_args(c, counts, S, nside, A, 0.0);
  if (s) return s;
  if (!partial) return set_err(c, UFC_ERR_ARG, "partial_dev is NULL");
  if ((reinterpret_cast<uintptr_t>(counts) & 15) || (reinterpret_cast<uintptr_t>(partial) & 15))
    return set_err(c, UFC_ERR_ARG, "counts_dev and partial_dev must be 16-byte aligned");
  const int npix = 12 * nside * nside;
  Coef cf;
  make_coef(A, 0.0, S, npix, cf);
  {
    ProfScope ps_(c, "k_kappa_partial");
    k_kappa_partial<<<kappa_fwd_grid(c, npix), kKV, 0, c->stream>>>(counts, cf, partial);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

static ufc_status check_partial_args(ufc_ctx* c, const double* partial, int nside, double C) {
  if (!partial) return set_err(c, UFC_ERR_ARG, "partial_dev is NULL");
  if (reinterpret_cast<uintptr_t>(partial) & 15)
    return set_err(c, UFC_ERR_ARG, "partial_dev must be 16-byte aligned");
  if (nside < 1 || nside > UFC_MAX_NSIDE || (nside & (nside - 1)))
    return set_err(c, UFC_ERR_ARG, "nside must be a power of two in [1,%d]", UFC_MAX_NSIDE);
  if (!std::isfinite(C)) return set_err(c, UFC_ERR_ARG, "C is not finite");
  return UFC_OK;
}

ufc_status run_kappa_stats_partial(ufc_ctx* c, const double* partial, int nside, double C,
                                   double lo, double hi, int nbins, float* kappa,
                                   double* moments, int64_t* pdf) {
  ufc_status s = check_partial_args(c, partial, nside, C);
  if (s) return s;
  if (!kappa || !moments || !pdf)
    return set_err(c, UFC_ERR_ARG, "kappa_dev, moments_dev and pdf_dev are required");
  if (reinterpret_cast<uintptr_t>(kappa) & 15)
    return set_err(c, UFC_ERR_ARG, "kappa_dev must be 16-byte aligned");
  if (nbins < 1 || nbins > kMaxBins)
    return set_err(c, UFC_ERR_ARG, "nbins must be in [1,%d]", kMaxBins);
  if (!(hi > lo) || !std::isfinite(lo) || !std::isfinite(hi))
    return set_err(c, UFC_ERR_ARG, "PDF range needs finite lo < hi");
  const int npix = 12 * nside * nside;
  const int grid = kappa_fwd_grid(c, npix), mgrid = moments_grid(c->num_sms, npix);
  double* ksum = (double*)ws_get(c, kSlotPartials, pass_doubles(grid, mgrid) * 8);
  if (!ksum) return UFC_ERR_ALLOC;
  const float ch = (float)C, cl = (float)(C - (double)ch);
  {
    ProfScope ps_(c, "k_kappa_finish");
    k_kappa_finish<<<grid, kKV, 0, c->stream>>>(partial, ch, cl, npix, kappa, ksum,
                                                moment_out(ksum + grid, mgrid, pdf, nbins));
  }
  UFC_CUDA(c, cudaGetLastError());
  return launch_moments(c, kappa, npix, ksum, grid, lo, hi, nbins, ksum + grid, moments, pdf, true);
}

ufc_status run_kappa_adjoint_sums(ufc_ctx* c, const int32_t* counts, int S, int nside,
                                  const double* partial, double C, const float* g, float* kappa,
                                  double lo, double hi, int nbins, double* moments, int64_t* pdf,
                                  double* sums) {
  ufc_status s = check_partial_args(c, partial, nside, C);
  if (s) return s;
  if (!counts) return set_err(c, UFC_ERR_ARG, "counts_dev is NULL");
  if (S < 1 || S > kMaxShells) return set_err(c, UFC_ERR_ARG, "nshell must be in [1,%d]", kMaxShells);
  if ((int64_t)S * 12 * nside * nside >= (1ll << 31))
    return set_err(c, UFC_ERR_ARG, "nshell * 12 nside^2 must be < 2^31");
  if (!sums) return set_err(c, UFC_ERR_ARG, "sums is NULL");
  const int npix = 12 * nside * nside;
  std::vector<double> zeros(S, 0.0);
  Coef cf;
  make_coef(zeros.data(), C, S, npix, cf);   // A unused: e comes from the partials
  return adjoint_sums(c, counts, S, nside, cf, partial, g, kappa, lo, hi, nbins, moments, pdf,
                      sums);
}

ufc_status run_kappa_backward(ufc_ctx* c, const int32_t* counts, int S, int nside,
                              const double* A, double C, double w_var, double w_skew,
                              const float* g, const double* dA, const double* dC,
                              double* grad, double* G, double* H) {
  return run_kappa_backward_ex(c, counts, S, nside, A, C, w_var, w_skew, g, dA, dC, grad, G, H,
                               nullptr, 0.0, 1.0, 1, nullptr, nullptr);
}

// ---- variant of ufc_kappa_stats that allocates nothing -------------------
// Its per-block partial sums and its count of finished blocks live in this
// file-scope device array instead of the context workspace.  Every GPU that loads the library holds the array
// (kNoAllocScratch doubles = 32 KB) until the process exits; all calls on a
// device share it, so calls that overlap on the GPU race on it.
constexpr int kNoAllocScratch = 4096;
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocScratch];

// Device address of g_noalloc_scratch, looked up once per device (with that
// device current) the first time the variant runs there.
static std::mutex g_noalloc_mu;
static double* g_noalloc_ptr[64] = {};

static ufc_status noalloc_scratch(ufc_ctx* c, double** out) {
  if (c->device < 0 || c->device >= 64)
    return set_err(c, UFC_ERR_UNSUPPORTED, "device index above 63");
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[c->device]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return set_err(c, UFC_ERR_CUDA, "cudaGetSymbolAddress of the scratch array failed: %s",
                     cudaGetErrorString(e));
    g_noalloc_ptr[c->device] = static_cast<double*>(p);
  }
  *out = g_noalloc_ptr[c->device];
  return UFC_OK;
}

ufc_status run_kappa_stats_noalloc(ufc_ctx* c, const int32_t* counts, int S, int nside,
                                   const double* A, double C, double lo, double hi, int nbins,
                                   float* kappa, double* moments, int64_t* pdf) {
  ufc_status s = check_kappa_args(c, counts, S, nside, A, C);
  if (s) return s;
  if (!kappa || !moments || !pdf)
    return set_err(c, UFC_ERR_ARG, "the no-allocation variant needs kappa_dev, moments_dev and pdf_dev");
  if (nbins < 1 || nbins > kMaxBins)
    return set_err(c, UFC_ERR_ARG, "nbins must be in [1,%d]", kMaxBins);
  if (!(hi > lo) || !std::isfinite(lo) || !std::isfinite(hi))
    return set_err(c, UFC_ERR_ARG, "PDF range needs finite lo < hi");
  if (reinterpret_cast<uintptr_t>(counts) & 15)
    return set_err(c, UFC_ERR_ARG, "counts_dev must be 16-byte aligned");
  const int npix = 12 * nside * nside;
  const int grid = kappa_fwd_grid(c, npix);
  const int mgrid = moments_grid(c->num_sms, npix);
  if (pass_doubles(grid, mgrid) > (size_t)kNoAllocScratch)
    return set_err(c, UFC_ERR_CAPACITY,
                   "scratch needs %zu doubles, the fixed array holds %d", pass_doubles(grid, mgrid),
                   kNoAllocScratch);
  double* ksum = nullptr;
  s = noalloc_scratch(c, &ksum);
  if (s) return s;
  double* mpart = ksum + grid;   // every slot is written before it is read, the count cleared
  Coef cf;
  make_coef(A, C, S, npix, cf);
  s = launch_kappa_fwd(c, counts, cf, kappa, ksum, grid, moment_out(mpart, mgrid, pdf, nbins));
  if (s) return s;
  // (no kernel-timing records here: recording them may allocate)
  return launch_moments(c, kappa, npix, ksum, grid, lo, hi, nbins, mpart, moments, pdf, false);
}

ufc_status run_stats_vector(ufc_ctx* c, const double* m, const int64_t* pdf, int nbins,
                            double* v) {
  if (!m || !pdf || !v || nbins < 1 || nbins > kMaxBins)
    return set_err(c, UFC_ERR_ARG, "stats_vector: bad arguments");
  {
    ProfScope ps_(c, "k_stats_vector");
    k_stats_vector<<<1, 256, 0, c->stream>>>(m, (const unsigned long long*)pdf, nbins, v);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

// mean_new [d] and ticket (0 when the launch runs): scratch that no other call
// uses meanwhile, or NULL both.
static ufc_status launch_welford(ufc_ctx* c, const double* v, int nvec, int d, double* st,
                                 double* mean_new, unsigned int* ticket) {
  if (!v || !st || nvec < 0 || d < 1 || d > 8192)
    return set_err(c, UFC_ERR_ARG, "welford_update: bad arguments");
  if (nvec == 0) return UFC_OK;
  if (nvec == 1 && d <= kWfOne) {
    ProfScope ps_(c, "k_welford_update");
    k_welford_one<<<kWfCluster, kWfOneThreads, 0, c->stream>>>(v, d, st);
    UFC_CUDA(c, cudaGetLastError());
    return UFC_OK;
  }
  {
    ProfScope ps_(c, "k_welford_update");
    const int g = (d + kWfTile - 1) / kWfTile;
    k_welford_update<<<dim3(g, g), kWfThreads, 0, c->stream>>>(v, nvec, d, st, mean_new, ticket);
  }
  if (!mean_new) {
    ProfScope ps_(c, "k_welford_mean");
    const int warps = (d + 32 * kWfCluster - 1) / (32 * kWfCluster);       // per block, at most 8
    k_welford_mean<<<kWfCluster, 32 * std::min(warps, 8), 0, c->stream>>>(v, nvec, d, st);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}
ufc_status run_welford_update(ufc_ctx* c, const double* v, int nvec, int d, double* st) {
  return launch_welford(c, v, nvec, d, st, nullptr, nullptr);
}
ufc_status run_welford_merge(ufc_ctx* c, double* a, const double* b, int d) {
  if (!a || !b || d < 1 || d > 8192) return set_err(c, UFC_ERR_ARG, "welford_merge: bad arguments");
  {
    ProfScope ps_(c, "k_welford_merge");
    k_welford_merge<<<1, 1024, 0, c->stream>>>(a, b, d);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}
ufc_status run_welford_finalize(ufc_ctx* c, const double* st, int d, int ddof, double* mean,
                                double* cov, double* corr) {
  if (!st || !mean || !cov || !corr || d < 1 || d > 8192 || ddof < 0)
    return set_err(c, UFC_ERR_ARG, "welford_finalize: bad arguments");
  {
    ProfScope ps_(c, "k_welford_final");
    k_welford_final<<<1, 1024, 0, c->stream>>>(st, d, ddof, mean, cov, corr);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

// ---- batched call: host side -------------------------------------------------
ufc_status batch_geometry(ufc_ctx* c, const double* chi, int nshell, const ufc_box* boxes,
                          int nbox, ShellTable& st, BoxGeom* bg);
void batch_bands(int nside, float smax, Bands& bd);

// Workspace of a batched call: per realisation a count map, a kappa map and the
// partial sums of the serial grids, then the items, the coefficients, the
// finished-block counters (one per realisation, one of the Welford update), the
// new Welford mean, and the binning's tables and counters: the call shares
// nothing with the binning, kappa and moment calls of its context (which may run
// on another stream meanwhile) and leaves ufc_bin_info as it was.
// A launch takes as many realisations as its grid has rows and the 17 bits of an
// item's number in an undecided image's entry allow.
constexpr int kBatchRows = 65535, kBatchItems = 1 << 17;
struct BatchSpace {
  size_t maps, kappa, part;                  // offsets in the map buffer
  size_t maps_bytes;
  size_t items, coef, done, mean, tab, cnt, up_bytes, desc_bytes;   // in the descriptor buffer
  int gk, gm;
};
static BatchSpace batch_space(const ufc_ctx* c, int nreal, int nbox, int S, int nside, int d) {
  const int npix = 12 * nside * nside;
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  BatchSpace o;
  o.gk = kappa_fwd_grid(c, npix);
  o.gm = moments_grid(c->num_sms, npix);
  o.maps = 0;
  o.kappa = up((size_t)nreal * S * npix * 4);
  o.part = o.kappa + up((size_t)nreal * npix * 4);
  o.maps_bytes = o.part + (size_t)nreal * (o.gk + 3 * o.gm) * 8;
  o.items = 0;
  o.coef = up((size_t)nreal * nbox * sizeof(DirectItem));
  o.up_bytes = o.coef + (size_t)nreal * batch_coef_stride(S);
  o.done = up(o.up_bytes);
  o.mean = up(o.done + (size_t)(nreal + 1) * 4);
  o.tab = up(o.mean + (size_t)d * 8);
  o.cnt = up(o.tab + sizeof(BinTables));
  o.desc_bytes = o.cnt + sizeof(BinCounters);
  return o;
}
// Whether the batched call of this shape runs stage by stage over all
// realisations.
bool batch_stages_ok(const ufc_ctx* c, int nreal, int nbox, int S, int nside, size_t max_bytes) {
  return nbox <= kBatchItems &&
         batch_space(c, nreal, nbox, S, nside, 0).maps_bytes <= max_bytes;
}

// A batched call over all realisations at once.  The items and coefficients
// are built in page-locked memory of the context and copied from there; the
// next call waits (on the host, for the copy only) before it overwrites them.
ufc_status run_batch_stages(ufc_ctx* c, int nreal, int nbox, const float* const* xyz,
                            const int64_t* n, const ufc_box* boxes, const double* chi, int S,
                            int nside, const double* A, const double* C, double lo, double hi,
                            int nbins, double* moments, int64_t* pdf, double* stats,
                            double* state) {
  cudaStreamCaptureStatus cs;
  UFC_CUDA(c, cudaStreamIsCapturing(c->stream, &cs));
  if (cs != cudaStreamCaptureStatusNone)
    return set_err(c, UFC_ERR_UNSUPPORTED, "ufc_batched_stats cannot be captured into a graph");
  const int npix = 12 * nside * nside, nitems = nreal * nbox;
  const BatchSpace sp = batch_space(c, nreal, nbox, S, nside, 6 + nbins);
  char* maps = (char*)ws_get(c, kSlotBatchMaps, sp.maps_bytes);
  char* desc = (char*)ws_get(c, kSlotBatchDesc, sp.desc_bytes);
  if (!maps || !desc) return UFC_ERR_ALLOC;
  if (!c->batch_ev) UFC_CUDA(c, cudaEventCreateWithFlags(&c->batch_ev, cudaEventDisableTiming));
  if (c->batch_host_cap < sp.up_bytes) {
    if (c->batch_host) {
      UFC_CUDA(c, cudaEventSynchronize(c->batch_ev));
      cudaFreeHost(c->batch_host);
      c->batch_host = nullptr;
      c->batch_host_cap = 0;
    }
    const size_t want = sp.up_bytes + sp.up_bytes / 8;
    if (cudaHostAlloc(&c->batch_host, want, cudaHostAllocDefault) != cudaSuccess) {
      cudaGetLastError();
      c->batch_host = nullptr;
      return set_err(c, UFC_ERR_ALLOC, "cudaHostAlloc of %zu bytes failed", want);
    }
    c->batch_host_cap = want;
  } else {
    UFC_CUDA(c, cudaEventSynchronize(c->batch_ev));    // the last call's copy has been made
  }
  char* host = static_cast<char*>(c->batch_host);
  DirectItem* items = reinterpret_cast<DirectItem*>(host + sp.items);
  DirectArgs a;
  std::memset(&a, 0, sizeof a);
  int64_t total = 0;
  for (int i = 0; i < nitems; ++i) {
    if (n[i] < 0) return set_err(c, UFC_ERR_ARG, "n[%d] < 0", i);
    if (n[i] > 0 && !xyz[i]) return set_err(c, UFC_ERR_ARG, "xyz[%d] is NULL", i);
    if (n[i] >= (1ll << 47)) return set_err(c, UFC_ERR_ARG, "n[%d] too large", i);
    if (n[i] > 0 && (reinterpret_cast<uintptr_t>(xyz[i]) & 3))
      return set_err(c, UFC_ERR_ARG, "xyz[%d] is not 4-byte aligned", i);
    total += n[i];
  }
  a.task = c->batch_chunk > 0 ? c->batch_chunk : direct_task(c, total);
  const int per = std::min(kBatchRows, kBatchItems / nbox);      // realisations per launch
  std::vector<int64_t> ntasks;                                   // of each launch
  std::vector<BoxGeom> bg(nbox);
  ShellTable st;
  float smax = 0.f;
  for (int r = 0; r < nreal; ++r) {
    if (r % per == 0) ntasks.push_back(0);
    const ufc_status s = batch_geometry(c, r == 0 ? chi : nullptr, S, boxes + (size_t)r * nbox, nbox,
                                        st, bg.data());
    if (s) return s;
    for (int k = 0; k < nbox; ++k) {
      const size_t i = (size_t)r * nbox + k;
      const BoxGeom& g = bg[k];
      DirectItem& d = items[i];
      smax = std::max(smax, g.smax);
      d.xyz = xyz[i];
      d.n = n[i];
      d.task0 = ntasks.back();
      d.counts = reinterpret_cast<int32_t*>(maps + sp.maps) + (size_t)r * S * npix;
      d.shell_lo = g.shell_lo;
      d.shell_hi = g.shell_hi;
      for (int ax = 0; ax < 3; ++ax) {
        d.shf[ax] = g.shf[ax][0];
        d.shlo[ax] = g.shlo[ax][0];
        d.sh64[ax] = g.sh64[ax][0];
      }
      ntasks.back() += (n[i] + a.task - 1) / a.task;
    }
    BatchCoef* cf = reinterpret_cast<BatchCoef*>(host + sp.coef + batch_coef_stride(S) * r);
    auto split = [](double x) {
      const float h = (float)x;
      return make_float2(h, (float)(x - (double)h));
    };
    for (int b = 0; b < S; ++b) cf->a[b] = split(A[(size_t)r * S + b]);
    cf->c = split(C[r]);
  }
  UFC_CUDA(c, cudaMemcpyAsync(desc, host, sp.up_bytes, cudaMemcpyHostToDevice, c->stream));
  UFC_CUDA(c, cudaEventRecord(c->batch_ev, c->stream));
  UFC_CUDA(c, cudaMemsetAsync(desc + sp.done, 0, (size_t)(nreal + 1) * 4, c->stream));
  // the bands of the largest shift of all the boxes
  batch_bands(nside, smax, a.bd);
  a.tab = reinterpret_cast<BinTables*>(desc + sp.tab);
  a.cnt = reinterpret_cast<BinCounters*>(desc + sp.cnt);
  ufc_status s = bin_prep(c, st, maps + sp.maps, sp.kappa, a.tab, a.cnt, &a.lut_scale);
  if (s) return s;
  a.N = nside;
  a.npix = npix;
  a.ncell = (int64_t)S * npix;
  double* const ksum = reinterpret_cast<double*>(maps + sp.part);
  unsigned int* const done = reinterpret_cast<unsigned int*>(desc + sp.done);
  for (int r0 = 0; r0 < nreal; r0 += per) {
    const int nr = std::min(per, nreal - r0);
    a.items = reinterpret_cast<const DirectItem*>(desc + sp.items) + (size_t)r0 * nbox;
    a.nitems = nr * nbox;
    a.ntasks = ntasks[r0 / per];
    s = launch_direct(c, a, c->batch_blocks_per_sm);
    if (s) return s;
    BatchArgs ba;
    ba.coef = desc + sp.coef + batch_coef_stride(S) * r0;
    ba.S = S;
    ba.npix = npix;
    ba.counts = reinterpret_cast<int32_t*>(maps + sp.maps) + (size_t)r0 * S * npix;
    ba.kappa = reinterpret_cast<float*>(maps + sp.kappa) + (size_t)r0 * npix;
    ba.ksum = ksum + (size_t)sp.gk * r0;
    ba.mpart = ksum + (size_t)sp.gk * nreal + (size_t)3 * sp.gm * r0;
    ba.gk = sp.gk;
    ba.gm = sp.gm;
    ba.moments = moments + (size_t)10 * r0;
    ba.pdf = pdf + (size_t)(nbins + 3) * r0;
    ba.stats = stats + (size_t)(6 + nbins) * r0;
    ba.nbins = nbins;
    ba.d = 6 + nbins;
    ba.done = done + r0;
    {
      ProfScope ps_(c, "k_batch_kappa");
      k_batch_kappa<<<dim3(sp.gk, nr), kKV, 0, c->stream>>>(ba);
    }
    {
      ProfScope ps_(c, "k_batch_moments");
      k_batch_moments<<<dim3(sp.gm, nr), kMT, (nbins + 3) * 4, c->stream>>>(
          ba, make_pdf_param(lo, hi, nbins));
    }
  }
  UFC_CUDA(c, cudaGetLastError());
  return launch_welford(c, stats, nreal, 6 + nbins, state, reinterpret_cast<double*>(desc + sp.mean),
                        done + nreal);
}

}  // namespace ufc

