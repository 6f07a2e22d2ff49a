// Ring geometry and double-float arithmetic of the spherical-harmonic
// transforms (sht.cu: Legendre stages, sht_ring.cu: ring transforms).
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"
#include "ctx.h"
#include "packed.cuh"

namespace ufc {

constexpr int kShtMaxNside = 1024;     // shared memory of the ring transforms
struct Ring {
  int64_t start;   // first pixel
  int32_t n;       // pixels
  double z, s;     // cos and sin of the colatitude
};

// Ring r (0-based, north to south) of the RING scheme.
__host__ __device__ inline Ring ring_geom(int32_t N, int32_t r) {
  const int64_t npix = 12ll * N * N;
  const int32_t i = r + 1;
  Ring g;
  if (i < N) {
    g.n = 4 * i;
    g.start = 2ll * i * (i - 1);
    const double t = (double)((int64_t)i * i) / (3.0 * (double)((int64_t)N * N));
    g.z = 1.0 - t;
    g.s = sqrt(t * (2.0 - t));
  } else if (i <= 3 * N) {
    g.n = 4 * N;
    g.start = 2ll * N * (N - 1) + 4ll * N * (i - N);
    g.z = 4.0 / 3.0 - 2.0 * (double)i / (3.0 * (double)N);
    g.s = sqrt((1.0 - g.z) * (1.0 + g.z));
  } else {
    const int32_t k = 4 * N - i;
    g.n = 4 * k;
    g.start = npix - 2ll * k * (k + 1);
    const double t = (double)((int64_t)k * k) / (3.0 * (double)((int64_t)N * N));
    g.z = -(1.0 - t);
    g.s = sqrt(t * (2.0 - t));
  }
  return g;
}

__device__ __forceinline__ bool is_pow2(int v) { return (v & (v - 1)) == 0; }

// Double-float arithmetic on the FP32 pipe (GB300 runs FP64 at 1/64 of the
// FP32 rate): a value is h + l with |l| <= ulp(h)/2, about 48 bits.  Every
// step is a correctly rounded FP32 intrinsic, so that no contraction changes
// the error-free transformations (Dekker/Knuth two-sum, FMA two-product).
struct dfl { float h, l; };
__device__ __forceinline__ dfl df_from_d(double x) {
  const float h = __double2float_rn(x);
  return {h, __double2float_rn(x - (double)h)};
}
__device__ __forceinline__ double df_to_d(dfl a) { return (double)a.h + (double)a.l; }
// h + l with |h| >= |l| renormalised (fast two-sum)
__device__ __forceinline__ dfl df_norm(float h, float l) {
  const float s = __fadd_rn(h, l);
  return {s, __fadd_rn(l, __fsub_rn(h, s))};
}
// a + b (two-sum of the high parts)
__device__ __forceinline__ dfl df_add(dfl a, dfl b) {
  const float s = __fadd_rn(a.h, b.h);
  const float bb = __fsub_rn(s, a.h);
  const float err = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fsub_rn(b.h, bb));
  return df_norm(s, __fadd_rn(err, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ dfl df_scale(dfl a, float p2) { return {a.h * p2, a.l * p2}; }  // exact

// Complex numbers with double-float parts, (re.h, re.l, im.h, im.l) in a float4.
__device__ __forceinline__ float4 cdf_pack(dfl re, dfl im) { return make_float4(re.h, re.l, im.h, im.l); }
__device__ __forceinline__ float4 cdf_add(float4 a, float4 b) {
  return cdf_pack(df_add(dfl{a.x, a.y}, dfl{b.x, b.y}), df_add(dfl{a.z, a.w}, dfl{b.z, b.w}));
}
__device__ __forceinline__ float4 cdf_sub(float4 a, float4 b) {
  return cdf_pack(df_add(dfl{a.x, a.y}, dfl{-b.x, -b.y}), df_add(dfl{a.z, a.w}, dfl{-b.z, -b.w}));
}

__device__ __forceinline__ dfx dfx_set(dfl a, dfl b) { return {x2_pack(a.h, b.h), x2_pack(a.l, b.l)}; }

// sht_ring.cu: F_m of every ring of a map ([lmax + 1][4N - 1]), and the map of
// such coefficients (all NaN when *bad is set); T: the 8N unit roots
// e^{-2 pi i j / (8N)}.
ufc_status launch_ring_transform(ufc_ctx* c, const float* map, const float4* T, int nside, int lmax,
                                 float4* F);
ufc_status launch_ring_synth(ufc_ctx* c, const float4* G, const float4* T, int nside, int lmax,
                             const int* bad, float* map);

}  // namespace ufc
