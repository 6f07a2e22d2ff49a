// Ring transforms of the spherical-harmonic analysis and synthesis: the real
// DFT of every HEALPix ring, forward and inverse, in double-float on the FP32
// pipe.
//
// A ring of n = 4i pixels is taken as L = n/2 complex numbers z_j = x_{2j} +
// i x_{2j+1}; from their DFT Z, X_k = (Z_k + conj Z_{L-k}) / 2 - i w_n^k
// (Z_k - conj Z_{L-k}) / 2 for k <= L (w_n = e^{-2 pi i / n}), and back.
//  - n a power of two (every belt ring, and the cap rings with i a power of
//    two): one FFT of length L in shared memory.
//  - otherwise the length-2i DFT splits into two of length i, and those go
//    through a cyclic convolution of length M = 2^p >= 2i - 1 with the chirp
//    c_a = e^{-pi i a^2 / i} (Bluestein, 1970): D_k = c_k sum_a (x_a c_a)
//    conj(c_{k-a}).  Three forward FFTs (chirp and both halves) and two inverse
//    ones of length M <= 2048, where the direct length-i sums grew as i^2.
// The FFTs are decimation in frequency forward (natural order in, bit-reversed
// out) and decimation in time back, two radix-2 steps at a time, so no
// reordering pass is needed around the convolution.  Complex numbers sit in
// packed registers as (re, im) pairs of the high and of the low parts, 16
// bytes each in shared memory.
//
// What bounds them: the FP32 pipe and the shared-memory latency of 2 blocks of
// 16 warps per SM.  The 4095 rings of Nside 1024 take 0.49 ms forward (3.93 ms
// with direct length-i sums and full-length complex FFTs of the belt's real
// rings) and 0.59 back at lmax 3071, the 2047 of Nside 512 0.135 ms back at lmax
// 1535 (its column-wise reads of G, 16 bytes per row, are what is left there).
#include <algorithm>
#include <cmath>

#include "sht_common.cuh"

namespace ufc {

constexpr int kRingThreads = 512;

// ------------------------------------------------- packed complex numbers --
typedef dfx cx;                                   // h = (re.h, im.h), l = (re.l, im.l)
typedef ulonglong2 cxs;                           // the same in memory
__device__ __forceinline__ cx cx_ld(const cxs& v) { return {v.x, v.y}; }
__device__ __forceinline__ cxs cx_st(cx v) { return make_ulonglong2(v.h, v.l); }
// from and to the (re.h, re.l, im.h, im.l) layout of the tables and of F, G
__device__ __forceinline__ cx cx_of(float4 v) { return {x2_pack(v.x, v.z), x2_pack(v.y, v.w)}; }
__device__ __forceinline__ float4 cx_to4(cx v) {
  const float2 h = x2_get(v.h), l = x2_get(v.l);
  return make_float4(h.x, l.x, h.y, l.y);
}
__device__ __forceinline__ cx cx_add(cx a, cx b) {
  const dfx r = dfx_add_raw(a, b);
  return dfx_norm(r.h, r.l);
}
__device__ __forceinline__ cx cx_sub(cx a, cx b) {
  const u64 s = x2_sub(a.h, b.h);
  const u64 bb = x2_sub(s, a.h);                  // about -b
  const u64 er = x2_sub(x2_sub(a.h, x2_sub(s, bb)), x2_add(b.h, bb));
  return dfx_norm(s, x2_add(er, x2_sub(a.l, b.l)));
}
__device__ __forceinline__ cx cx_conj(cx a) {
  return {a.h ^ 0x8000000000000000ull, a.l ^ 0x8000000000000000ull};
}
__device__ __forceinline__ cx cx_real(cx a) { return {a.h & 0xFFFFFFFFull, a.l & 0xFFFFFFFFull}; }
__device__ __forceinline__ cx cx_times_i(cx a) {  // (re, im) -> (-im, re)
  const float2 h = x2_get(a.h), l = x2_get(a.l);
  return {x2_pack(-h.y, h.x), x2_pack(-l.y, l.x)};
}
__device__ __forceinline__ cx cx_scale(cx a, float p2) {   // by a power of two: exact
  const u64 s = x2_pack(p2, p2);
  return {x2_mul(a.h, s), x2_mul(a.l, s)};
}
__device__ __forceinline__ dfx cx_prod(dfx a, dfx b) {     // elementwise, not renormalised
  const u64 p = x2_mul(a.h, b.h);
  u64 e = x2_fma(a.h, b.h, x2_neg(p));
  e = x2_fma(a.h, b.l, e);
  return {p, x2_fma(a.l, b.h, e)};
}
// a w = (ar wr, ai wr) + (ai, ar) (-wi, wi)
__device__ __forceinline__ cx cx_mul(cx a, cx w) {
  const float2 ah = x2_get(a.h), al = x2_get(a.l), wh = x2_get(w.h), wl = x2_get(w.l);
  const dfx p = cx_prod(a, dfx{x2_pack(wh.x, wh.x), x2_pack(wl.x, wl.x)});
  const dfx q = cx_prod(dfx{x2_pack(ah.y, ah.x), x2_pack(al.y, al.x)},
                        dfx{x2_pack(-wh.y, wh.y), x2_pack(-wl.y, wl.y)});
  const dfx r = dfx_add_raw(p, q);
  return dfx_norm(r.h, r.l);
}

// ---------------------------------------------------------------- FFTs -----
// nb transforms of length 2^b (b >= 1), one after the other in x, by the whole
// block; twiddles e^{-2 pi i j / len} = T[j 8N / len] (conjugated with CONJ, for
// the unscaled inverse transform).  Every thread calls it; ends with a barrier.
template <bool CONJ>
__device__ __forceinline__ void fft_dif(cxs* x, int nb, int b, const float4* __restrict__ T, int N8) {
  const int M = 1 << b;
  auto tw = [&](int j, int lb) {
    const cx w = cx_of(__ldg(T + j * (N8 >> lb)));
    return CONJ ? cx_conj(w) : w;
  };
  int lb = b;
  if (b & 1) {
    const int half = M >> 1;
    for (int t = threadIdx.x; t < nb * half; t += kRingThreads) {
      const int j = t & (half - 1);
      cxs* p = x + ((t >> (b - 1)) << b) + j;
      const cx u = cx_ld(p[0]), v = cx_ld(p[half]);
      p[0] = cx_st(cx_add(u, v));
      p[half] = cx_st(cx_mul(cx_sub(u, v), tw(j, lb)));
    }
    __syncthreads();
    --lb;
  }
  // two steps at a time: y0 = (a + c) + (b + d), y2 = (a + c) - (b + d) in the
  // first half, y1, y3 = (a - c) -+ i (b - d) in the second, with their twiddles
  for (; lb >= 2; lb -= 2) {
    const int q = 1 << (lb - 2);
    for (int t = threadIdx.x; t < nb * (M >> 2); t += kRingThreads) {
      const int j = t & (q - 1);
      cxs* p = x + ((t >> (lb - 2)) << lb) + j;
      const cx a = cx_ld(p[0]), c = cx_ld(p[2 * q]), e = cx_ld(p[q]), d = cx_ld(p[3 * q]);
      const cx t0 = cx_add(a, c), t1 = cx_sub(a, c), t2 = cx_add(e, d);
      cx t3 = cx_times_i(cx_sub(e, d));             // i (b - d)
      if (CONJ) t3 = dfx{x2_neg(t3.h), x2_neg(t3.l)};
      const cx y1 = cx_sub(t1, t3), y3 = cx_add(t1, t3);
      p[0] = cx_st(cx_add(t0, t2));
      if (q > 1) {
        p[q] = cx_st(cx_mul(cx_sub(t0, t2), tw(2 * j, lb)));
        p[2 * q] = cx_st(cx_mul(y1, tw(j, lb)));
        p[3 * q] = cx_st(cx_mul(y3, tw(3 * j, lb)));
      } else {                                      // (the twiddles are 1)
        p[q] = cx_st(cx_sub(t0, t2));
        p[2 * q] = cx_st(y1);
        p[3 * q] = cx_st(y3);
      }
    }
    __syncthreads();
  }
}
// The inverse of fft_dif<false> times 2^b: bit-reversed in, natural order out.
__device__ __forceinline__ void fft_dit_inv(cxs* x, int nb, int b, const float4* __restrict__ T,
                                            int N8) {
  const int M = 1 << b;
  auto tw = [&](int j, int lb) { return cx_conj(cx_of(__ldg(T + j * (N8 >> lb)))); };
  const int top = b & ~1;
  for (int lb = 2; lb <= top; lb += 2) {
    const int q = 1 << (lb - 2);
    for (int t = threadIdx.x; t < nb * (M >> 2); t += kRingThreads) {
      const int j = t & (q - 1);
      cxs* p = x + ((t >> (lb - 2)) << lb) + j;
      cx y0 = cx_ld(p[0]), y2 = cx_ld(p[q]), y1 = cx_ld(p[2 * q]), y3 = cx_ld(p[3 * q]);
      if (q > 1) {
        y2 = cx_mul(y2, tw(2 * j, lb));
        y1 = cx_mul(y1, tw(j, lb));
        y3 = cx_mul(y3, tw(3 * j, lb));
      }
      const cx t0 = cx_add(y0, y2), t2 = cx_sub(y0, y2), t1 = cx_add(y1, y3);
      const cx t3 = cx_times_i(cx_sub(y1, y3));     // i (y1 - y3) = b - d, doubled
      p[0] = cx_st(cx_add(t0, t1));
      p[2 * q] = cx_st(cx_sub(t0, t1));
      p[q] = cx_st(cx_add(t2, t3));
      p[3 * q] = cx_st(cx_sub(t2, t3));
    }
    __syncthreads();
  }
  if (b & 1) {
    const int half = M >> 1;
    for (int t = threadIdx.x; t < nb * half; t += kRingThreads) {
      const int j = t & (half - 1);
      cxs* p = x + ((t >> (b - 1)) << b) + j;
      const cx u = cx_ld(p[0]), v = cx_mul(cx_ld(p[half]), tw(j, b));
      p[0] = cx_st(cx_add(u, v));
      p[half] = cx_st(cx_sub(u, v));
    }
    __syncthreads();
  }
}

__device__ __forceinline__ int log2_of(int v) { return 31 - __clz(v); }   // v a power of two
__device__ __forceinline__ int bit_rev(int k, int b) { return (int)(__brev((unsigned)k) >> (32 - b)); }

// Unit roots w_n^k of a ring of n = 4i pixels that is not a power of two: the
// first quarter k < i in shared memory, the rest by exact quadrant rotations
// (w_n^{k + i} = -i w_n^k).  k < 32 and the multiples of 32 by FP64 sincospi
// (split once), the others as the double-float product of two of these; wf[i] =
// w_{2n}.  (FP64 runs at 1/64 of the FP32 rate: with a sincospi per root, and w_2n
// and the ring's geometry by every thread, its pipe was 42% busy and the 2047 rings of
// Nside 512 took 380 us to synthesise, 324 without; the transform of Nside 64 24 us, 13
// now.)  Every thread calls it; ends with a barrier.
__device__ __forceinline__ void fill_quarter(float4* wf, int i) {
  const int nd = min(i, 32) + (i - 1) / 32;              // roots formed directly, then w_2n
  for (int t = threadIdx.x; t <= nd; t += kRingThreads) {
    const int k = t < 32 && t < i ? t : (t - min(i, 32) + 1) * 32;
    double sn, cs;
    sincospi(t == nd ? -0.25 / (double)i : -0.5 * (double)k / (double)i, &sn, &cs);
    wf[t == nd ? i : k] = cdf_pack(df_from_d(cs), df_from_d(sn));
  }
  __syncthreads();
  for (int k = 32 + threadIdx.x; k < i; k += kRingThreads)
    if (k & 31) wf[k] = cx_to4(cx_mul(cx_of(wf[k & ~31]), cx_of(wf[k & 31])));
  __syncthreads();
}
__device__ __forceinline__ cx quarter_root(const float4* wf, int i, int k) {   // 0 <= k < 4i
  int q = 0;
  if (k >= 2 * i) { k -= 2 * i; q = 2; }
  if (k >= i) { k -= i; ++q; }
  const float4 v = wf[k];
  const float4 r = (q & 1) ? make_float4(v.z, v.w, -v.x, -v.y) : v;            // times -i
  return cx_of((q & 2) ? make_float4(-r.x, -r.y, -r.z, -r.w) : r);
}
// c_a = e^{-pi i a^2 / i} = w_n^{2 (a^2 mod 2i)}
__device__ __forceinline__ cx chirp(const float4* wf, int i, int a) {
  return quarter_root(wf, i, 2 * ((a * a) % (2 * i)));
}
// e^{-i m phi_0} = w_{2n}^m (phi_0 = pi / n) of such a ring: w_n^{m/2}, times
// w_{2n} = h1 for odd m
__device__ __forceinline__ cx quarter_phase(const float4* wf, int i, int m, cx h1) {
  const cx p = quarter_root(wf, i, (m >> 1) % (4 * i));
  return (m & 1) ? cx_mul(p, h1) : p;
}
// First pixel and number of pixels of ring r, and whether its first pixel lies half a
// step from azimuth 0 (ring_geom, whole numbers only).
struct RingSpan { int32_t start, n; bool shifted; };
__device__ __forceinline__ RingSpan ring_span(int N, int r) {
  const int i = r + 1, k = 4 * N - i;
  if (i < N) return {2 * i * (i - 1), 4 * i, true};
  if (i <= 3 * N) return {2 * N * (N - 1) + 4 * N * (i - N), 4 * N, ((i - N + 1) & 1) != 0};
  return {12 * N * N - 2 * k * (k + 1), 4 * k, true};
}

// One block per ring.
__global__ void __launch_bounds__(kRingThreads, 2)
k_ring_transform(const float* __restrict__ map, const float4* __restrict__ T, int32_t N,
                 int32_t lmax, int32_t nrings, float4* __restrict__ F) {
  extern __shared__ __align__(16) cxs sh[];
  const int r = blockIdx.x;
  const RingSpan g = ring_span(N, r);
  const int n = g.n, L = n / 2, N8 = 8 * N;
  const float* px = map + g.start;
  // X_k from Z_k and Z_{L-k}
  auto real_dft = [](cx zk, cx zl, cx w) {
    const cx c = cx_conj(zl);
    const cx o = cx_mul(cx_sub(zk, c), w);                   // w_n^k (Z_k - conj Z_{L-k})
    return cx_scale(cx_sub(cx_add(zk, c), cx_times_i(o)), 0.5f);
  };
  if (is_pow2(n)) {
    cxs* Z = sh;                                             // [L]
    cxs* X = sh + L;                                         // [L + 1]
    const int b = log2_of(L), ts = N8 / n, ps = 4 * N / n;
    for (int j = threadIdx.x; j < L; j += kRingThreads)
      Z[j] = make_ulonglong2(x2_pack(__ldg(px + 2 * j), __ldg(px + 2 * j + 1)), 0ull);
    __syncthreads();
    fft_dif<false>(Z, 1, b, T, N8);
    for (int k = threadIdx.x; k <= L; k += kRingThreads)
      X[k] = cx_st(real_dft(cx_ld(Z[bit_rev(k & (L - 1), b)]),
                            cx_ld(Z[bit_rev((L - k) & (L - 1), b)]), cx_of(__ldg(T + k * ts))));
    __syncthreads();
    const bool shifted = g.shifted;                          // phi_0 = pi / n or 0
    for (int m = threadIdx.x; m <= lmax; m += kRingThreads) {
      const int k = m & (n - 1);
      cx v = k <= L ? cx_ld(X[k]) : cx_conj(cx_ld(X[n - k]));
      if (shifted) v = cx_mul(v, cx_of(__ldg(T + ((m * ps) & (N8 - 1)))));
      F[(size_t)m * nrings + r] = cx_to4(v);
    }
    return;
  }
  const int i = n / 4, b = 32 - __clz(2 * i - 2), M = 1 << b;   // M >= 2i - 1
  cxs* B = sh;                                               // chirp, then Z [2i]
  cxs* U = sh + M;                                           // even z, then X [2i + 1]
  cxs* V = sh + 2 * M;                                       // odd z
  float4* wf = reinterpret_cast<float4*>(sh + 3 * M);        // [i + 1]
  fill_quarter(wf, i);
  for (int a = threadIdx.x; a < M; a += kRingThreads) {
    cx u{0ull, 0ull}, v{0ull, 0ull}, c{0ull, 0ull};
    if (a < i) {
      c = chirp(wf, i, a);
      u = cx_mul(cx{x2_pack(__ldg(px + 4 * a), __ldg(px + 4 * a + 1)), 0ull}, c);
      v = cx_mul(cx{x2_pack(__ldg(px + 4 * a + 2), __ldg(px + 4 * a + 3)), 0ull}, c);
    } else if (a > M - i) {
      c = chirp(wf, i, M - a);
    }
    B[a] = cx_st(cx_conj(c));
    U[a] = cx_st(u);
    V[a] = cx_st(v);
  }
  __syncthreads();
  fft_dif<false>(sh, 3, b, T, N8);
  for (int a = threadIdx.x; a < M; a += kRingThreads) {
    const cx c = cx_ld(B[a]);
    U[a] = cx_st(cx_mul(cx_ld(U[a]), c));
    V[a] = cx_st(cx_mul(cx_ld(V[a]), c));
  }
  __syncthreads();
  fft_dit_inv(U, 2, b, T, N8);
  const float sc = 1.0f / (float)M;
  for (int k = threadIdx.x; k < i; k += kRingThreads) {
    const cx c = cx_scale(chirp(wf, i, k), sc);
    const cx e = cx_mul(cx_ld(U[k]), c);
    const cx o = cx_mul(cx_mul(cx_ld(V[k]), c), quarter_root(wf, i, 2 * k));   // times w_{2i}^k
    B[k] = cx_st(cx_add(e, o));
    B[k + i] = cx_st(cx_sub(e, o));
  }
  __syncthreads();
  for (int k = threadIdx.x; k <= L; k += kRingThreads)
    U[k] = cx_st(real_dft(cx_ld(B[k == L ? 0 : k]), cx_ld(B[k == 0 ? 0 : L - k]),
                          quarter_root(wf, i, k)));
  __syncthreads();
  const cx h1 = cx_of(wf[i]);
  for (int m = threadIdx.x; m <= lmax; m += kRingThreads) {
    const int k = m % n;
    const cx v = k <= L ? cx_ld(U[k]) : cx_conj(cx_ld(U[n - k]));
    F[(size_t)m * nrings + r] = cx_to4(cx_mul(v, quarter_phase(wf, i, m, h1)));
  }
}

// Complex numbers of shared memory that a ring with at least two threads per H_k
// (L + 1 <= kRingThreads / 2, that is i <= 127) uses: three buffers of M <= 256
// and i + 1 roots.
constexpr int kPartUsed = 3 * 256 + 128;
// One block per ring: H_k = sum over m = k mod n (0 <= m <= lmax) of
// G_m e^{i m phi_0} plus, for the negative frequencies, the conjugates of
// the terms with m = -k mod n (1 <= m <= lmax), for k <= L (H_{n-k} = conj
// H_k); then the inverse of the real DFT, map_j = sum_k H_k e^{2 pi i k j / n}:
// Z_k = E_k + i O_k with E_k = H_k + conj H_{L-k}, O_k = (H_k - conj H_{L-k})
// e^{2 pi i k / n}, and z = the inverse DFT of Z.  The terms of H_k are dealt to
// as many threads as a short ring leaves free, each adding its own in increasing
// m, and the parts added in order.  (One thread per H_k left the rings next to the
// poles, 3 to 9 sums of hundreds of dependent loads, as the tail of the kernel: 350
// us at Nside 512, lmax 1535, now 135.)
__global__ void __launch_bounds__(kRingThreads, 2)
k_ring_synth(const float4* __restrict__ G, const float4* __restrict__ T, int32_t N,
             int32_t lmax, int32_t nrings, int cap, const int* __restrict__ bad,
             float* __restrict__ map) {
  extern __shared__ __align__(16) cxs sh[];                  // [cap]
  const int r = blockIdx.x;
  const RingSpan g = ring_span(N, r);
  const int n = g.n, L = n / 2, N8 = 8 * N;
  const float off = *bad ? NAN : 0.f;                        // added to every pixel
  float* px = map + g.start;
  // (free below the last kRingThreads numbers where a ring deals out its terms:
  // it then uses at most kPartUsed of them, see ring_synth_cap)
  cxs* part_s = sh + (cap - kRingThreads);
  auto fold = [&](cxs* H, auto term) {                       // H_k, k <= L
    auto some = [&](int k, int p, int np) {                  // part p of np
      cx h{0ull, 0ull};
      for (int m = k + p * n; m <= lmax; m += np * n) h = cx_add(h, term(m));
      for (int m = (k ? n - k : n) + p * n; m <= lmax; m += np * n)
        h = cx_add(h, cx_conj(term(m)));
      return k ? h : cx_real(h);                             // (H_0: the conjugates cancel, and
    };                                                       // Im G_0 does not enter the map)
    const int np = kRingThreads / (L + 1);                   // (uniform)
    if (np < 2) {
      for (int k = threadIdx.x; k <= L; k += kRingThreads) H[k] = cx_st(some(k, 0, 1));
      return;
    }
    if (threadIdx.x < (L + 1) * np)
      part_s[threadIdx.x] = cx_st(some(threadIdx.x % (L + 1), threadIdx.x / (L + 1), np));
    __syncthreads();
    if (threadIdx.x <= L) {
      cx h = cx_ld(part_s[threadIdx.x]);
      for (int p = 1; p < np; ++p) h = cx_add(h, cx_ld(part_s[p * (L + 1) + threadIdx.x]));
      H[threadIdx.x] = cx_st(h);
    }
  };
  auto z_of = [](cx hk, cx hl, cx w) {                       // H_k, H_{L-k}, e^{2 pi i k / n}
    const cx c = cx_conj(hl);
    return cx_add(cx_add(hk, c), cx_times_i(cx_mul(cx_sub(hk, c), w)));
  };
  if (is_pow2(n)) {
    cxs* Z = sh;                                             // [L]
    cxs* H = sh + L;                                         // [L + 1]
    const int b = log2_of(L), ts = N8 / n, ps = 4 * N / n;
    const bool shifted = g.shifted;
    fold(H, [&](int m) {
      const cx v = cx_of(G[(size_t)m * nrings + r]);
      return shifted ? cx_mul(v, cx_conj(cx_of(__ldg(T + ((m * ps) & (N8 - 1)))))) : v;
    });
    __syncthreads();
    for (int k = threadIdx.x; k < L; k += kRingThreads)
      Z[k] = cx_st(z_of(cx_ld(H[k]), cx_ld(H[L - k]), cx_conj(cx_of(__ldg(T + k * ts)))));
    __syncthreads();
    fft_dif<true>(Z, 1, b, T, N8);
    for (int j = threadIdx.x; j < L; j += kRingThreads) {
      const cx v = cx_ld(Z[bit_rev(j, b)]);
      const float2 x = x2_get(x2_add(v.h, v.l));
      px[2 * j] = x.x + off;
      px[2 * j + 1] = x.y + off;
    }
    return;
  }
  // z_{2a} and z_{2a+1} as inverse DFTs of length i of Z_k + Z_{k+i} and
  // (Z_k - Z_{k+i}) e^{2 pi i k / (2i)}, by the conjugate chirp
  const int i = n / 4, b = 32 - __clz(2 * i - 2), M = 1 << b;
  cxs* B = sh;                                               // H [2i + 1], then the chirp
  cxs* U = sh + M;
  cxs* V = sh + 2 * M;
  float4* wf = reinterpret_cast<float4*>(sh + 3 * M);        // [i + 1]
  fill_quarter(wf, i);
  const cx h1 = cx_of(wf[i]);
  fold(B, [&](int m) {
    return cx_mul(cx_of(G[(size_t)m * nrings + r]), cx_conj(quarter_phase(wf, i, m, h1)));
  });
  __syncthreads();
  for (int k = threadIdx.x; k < M; k += kRingThreads) {
    cx u{0ull, 0ull}, v{0ull, 0ull};
    if (k < i) {
      const cx z0 = z_of(cx_ld(B[k]), cx_ld(B[L - k]), cx_conj(quarter_root(wf, i, k)));
      const cx z1 = z_of(cx_ld(B[k + i]), cx_ld(B[i - k]), cx_conj(quarter_root(wf, i, k + i)));
      const cx c = cx_conj(chirp(wf, i, k));
      u = cx_mul(cx_add(z0, z1), c);
      v = cx_mul(cx_mul(cx_sub(z0, z1), cx_conj(quarter_root(wf, i, 2 * k))), c);
    }
    U[k] = cx_st(u);
    V[k] = cx_st(v);
  }
  __syncthreads();
  for (int a = threadIdx.x; a < M; a += kRingThreads)
    B[a] = a < i ? cx_st(chirp(wf, i, a))
                 : (a > M - i ? cx_st(chirp(wf, i, M - a)) : make_ulonglong2(0ull, 0ull));
  __syncthreads();
  fft_dif<false>(sh, 3, b, T, N8);
  for (int a = threadIdx.x; a < M; a += kRingThreads) {
    const cx c = cx_ld(B[a]);
    U[a] = cx_st(cx_mul(cx_ld(U[a]), c));
    V[a] = cx_st(cx_mul(cx_ld(V[a]), c));
  }
  __syncthreads();
  fft_dit_inv(U, 2, b, T, N8);
  const float sc = 1.0f / (float)M;
  for (int a = threadIdx.x; a < i; a += kRingThreads) {
    const cx c = cx_scale(cx_conj(chirp(wf, i, a)), sc);
    const cx e = cx_mul(cx_ld(U[a]), c), o = cx_mul(cx_ld(V[a]), c);
    const float2 x = x2_get(x2_add(e.h, e.l)), y = x2_get(x2_add(o.h, o.l));
    px[4 * a] = x.x + off;
    px[4 * a + 1] = x.y + off;
    px[4 * a + 2] = y.x + off;
    px[4 * a + 3] = y.y + off;
  }
}

// Shared memory: three buffers of M <= 2N complex numbers and N roots (the
// belt rings' 4N + 1 complex numbers fit in that).
static int ring_cap(int nside) { return 7 * nside; }
// The synthesis' partial sums lie at the end of that: a map too small to hold them
// beside the buffers of the rings that deal out their terms has room for them
// behind.  (A buffer of their own kept the second block of Nside 1024 off an SM:
// 0.66 ms at lmax 3071, now 0.59.)
static int ring_synth_cap(int nside) {
  return std::max(ring_cap(nside), std::min(ring_cap(nside), kPartUsed) + kRingThreads);
}

ufc_status launch_ring_transform(ufc_ctx* c, const float* map, const float4* T, int nside, int lmax,
                                 float4* F) {
  const int smem = ring_cap(nside) * (int)sizeof(cxs), nrings = 4 * nside - 1;
  UFC_CUDA(c, cudaFuncSetAttribute(k_ring_transform, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   smem));
  {
    ProfScope ps_(c, "k_ring_transform");
    k_ring_transform<<<nrings, kRingThreads, smem, c->stream>>>(map, T, nside, lmax, nrings, F);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

ufc_status launch_ring_synth(ufc_ctx* c, const float4* G, const float4* T, int nside, int lmax,
                             const int* bad, float* map) {
  const int cap = ring_synth_cap(nside), smem = cap * (int)sizeof(cxs), nrings = 4 * nside - 1;
  UFC_CUDA(c, cudaFuncSetAttribute(k_ring_synth, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  {
    ProfScope ps_(c, "k_ring_synth");
    k_ring_synth<<<nrings, kRingThreads, smem, c->stream>>>(G, T, nside, lmax, nrings, cap, bad, map);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

}  // namespace ufc
