// Device tables of a binning call and the direct (global-atomic) binning
// kernel, shared by bin.cu and the batched call of stats.cu.
#pragma once
#include "common.cuh"
#include "ctx.h"
#include "pixel.cuh"

namespace ufc {

// Shell lookup table over r^2.  Bin i holds the r2 values whose FP32
// v = fminf(r2 * scale, kLut - 1) rounds to i; its low 15 bits count the
// edges e certainly at or below every such r2 (hi2[e] <= the bin's lowest
// possible r2), and bit 15 is set unless the next edge is certainly above
// every such r2 (lo2[e0] > the bin's highest possible r2).  A clean bin
// gives the shell with one load; the others scan the edges (exact).
constexpr int kLutBits = 13;
constexpr int kLut = 1 << kLutBits;
constexpr uint16_t kLutScan = 0x8000;

// A block's copy of the table with one comparison per particle: the shell itself where a bin
// lies in one of the shells [lo, hi) for certain, kLutOut where it is outside for certain, and
// the flag kLutScan (with the edge to scan from in the low bits) for the other bins and for
// those of radii below the near guard.
constexpr uint32_t kLutOut = 0x4000u;
__device__ __forceinline__ void fill_lut_classified(uint16_t* lut, const uint16_t* src,
                                                    int near_bin, int lo, int hi) {
  auto conv = [&](uint32_t e, int bin) -> uint32_t {
    const uint32_t a = e - 1u;
    const uint32_t r = a - uint32_t(lo) < uint32_t(hi - lo) ? a : kLutOut;
    return (e & kLutScan) || bin <= near_bin ? e | kLutScan : r;
  };
  const uint4* s8 = reinterpret_cast<const uint4*>(src);
  uint4* d8 = reinterpret_cast<uint4*>(lut);
#pragma unroll 2
  for (int i = threadIdx.x; i < kLut / 8; i += blockDim.x) {
    const uint4 w = s8[i];
    auto two = [&](uint32_t e, int bin) {
      return conv(e & 0xFFFFu, bin) | conv(e >> 16, bin + 1) << 16;
    };
    d8[i] = make_uint4(two(w.x, 8 * i), two(w.y, 8 * i + 2), two(w.z, 8 * i + 4),
                       two(w.w, 8 * i + 6));
  }
}
// The bin of a squared radius (the nearest integer, exact).
__device__ __forceinline__ int lut_bin(float r2, float scale) {
  return __float_as_int(fminf(r2 * scale, float(kLut - 1)) + 8388608.0f) - 0x4B000000;
}

// Tables of one call in device memory, written by k_bin_prep.
struct BinTables {
  ShellTable st;
  float2 atab[kAtanTab + 1];                 // arctangent table of the refine stage
  alignas(16) uint16_t lut[kLut];
  int bounds[kMaxBoxes][8];                  // particle bounds of the boxes with images, empty
};

// One set of particles of the direct path: a box of a binning call, or a
// (realisation, box) of a batched one.
struct DirectItem {
  const float* xyz;
  int64_t n;
  int64_t task0;             // first task of this item (ascending over the items)
  int32_t* counts;           // count map [nshell][npix] of the item
  int32_t shell_lo, shell_hi;
  float shf[3], shlo[3];     // the box's shift split as in BoxGeom (without images)
  double sh64[3];
};

struct DirectArgs {
  DirectItem inl[kMaxBoxes];   // the items when `items` is NULL
  const DirectItem* items;
  int32_t nitems;
  int32_t task;                // particles per task (without images)
  int64_t ntasks;
  int32_t nslice;              // tasks per 32 particles (with images)
  float lut_scale;
  BinTables* tab;
  Bands bd;
  int32_t N, npix;
  int64_t ncell;               // cells of a count map (checked builds' bound)
  BinCounters* cnt;
};

// Tables of one call into `tab` (device), the counters `cnt` cleared and
// `zero_bytes` of `zero` (16-byte aligned, a multiple of 16; may be NULL) set
// to 0, by one launch on the context stream.
ufc_status bin_prep(ufc_ctx* c, const ShellTable& st, void* zero, size_t zero_bytes,
                    BinTables* tab, BinCounters* cnt, float* lut_scale);
// Empties the particle bounds of box `box` again.
ufc_status bin_prep_bounds(ufc_ctx* c, BinTables* tab, int box);
// The direct path over a.nitems items (a.tab, a.bd, a.N, a.npix, a.cnt, the
// items' task0 and a.ntasks set), `blocks` resident blocks per SM (0: 2).
ufc_status launch_direct(ufc_ctx* c, const DirectArgs& a, int blocks);
// The same for one box with periodic images (geometry g), item a.inl[0]; box
// numbers the call's boxes.
ufc_status launch_direct_images(ufc_ctx* c, DirectArgs a, const BoxGeom& g, int box);
// Particles per task for `total` particles in one call.
int direct_task(const ufc_ctx* c, int64_t total);

}  // namespace ufc
