// The direct path of the binning: particles to count maps that sit in L2, by
// global atomics, with every stage of the key (FP32, double-float, FP64) in one
// kernel.  Used for small maps, for periodic images and for batched calls.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <type_traits>

#include "direct.cuh"

namespace ufc {

// ------------------------------------------------------------------ tables --
// One thread per table entry, the shell edges copied to shared memory first.
// On the host the lookup table took 8192 bins x 2 FP64 divisions per call and
// went to each kernel as a 16 KB parameter.
__global__ void __launch_bounds__(256)
k_bin_prep(ShellTable st, float scale, BinTables* __restrict__ t,
           unsigned long long* __restrict__ cnt, int ncnt, int4* __restrict__ zero, int64_t nzero) {
  __shared__ float lo2_s[kMaxShells + 1], hi2_s[kMaxShells + 1];
  const int S = st.nshell;
  for (int i = threadIdx.x; i <= S; i += blockDim.x) {
    lo2_s[i] = st.lo2[i];
    hi2_s[i] = st.hi2[i];
  }
  __syncthreads();
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = gid; i < kLut; i += nth) {
    // r2 whose fminf(r2 * scale, kLut - 1) rounds to i has r2 * scale in
    // [i - 1/2, i + 1/2] up to the product's rounding (< 2^-11 here);
    // the range is widened by 2^-10
    const double sc = (double)scale;
    const double rlo = ((double)i - 0.5 - 0x1p-10) / sc;
    const double rhi = i == kLut - 1 ? (double)INFINITY : ((double)i + 0.5 + 0x1p-10) / sc;
    int a = 0, b = S + 1;                      // edges with hi2 <= rlo
    while (a < b) {
      const int m = (a + b) >> 1;
      if ((double)hi2_s[m] <= rlo) a = m + 1; else b = m;
    }
    const bool clean = a > S || (double)lo2_s[a] > rhi;
    t->lut[i] = (uint16_t)(a | (clean ? 0 : kLutScan));
  }
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&st);
  uint32_t* dst = reinterpret_cast<uint32_t*>(&t->st);
  for (int64_t i = gid; i < (int64_t)(sizeof(ShellTable) / 4); i += nth) dst[i] = src[i];
  if (blockIdx.x == gridDim.x - 1) fill_atan_table(t->atab);
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < ncnt; i += blockDim.x) cnt[i] = 0ull;
    for (int i = threadIdx.x; i < 8 * kMaxBoxes; i += blockDim.x)
      t->bounds[i / 8][i % 8] = 0x7F800000;              // +inf: no particle yet
  }
  for (int64_t i = gid; i < nzero; i += nth) zero[i] = make_int4(0, 0, 0, 0);
}

ufc_status bin_prep(ufc_ctx* c, const ShellTable& st, void* zero, size_t zero_bytes,
                    BinTables* tab, BinCounters* cnt, float* lut_scale) {
  // bins 0 .. kLut-2 cover [0, hi2[nshell]]
  const double top = std::max((double)st.hi2[st.nshell], 1e-30);
  *lut_scale = (float)std::min((kLut - 2) / top, 1e30);
  const int64_t nzero = zero ? (int64_t)(zero_bytes / 16) : 0;
  const int grid =
      std::max(c->num_sms, (int)std::min<int64_t>(8 * c->num_sms, (nzero + 255) / 256));
  {
    ProfScope ps_(c, "k_bin_prep");
    k_bin_prep<<<grid, 256, 0, c->stream>>>(st, *lut_scale, tab, (unsigned long long*)cnt,
                                            (int)(offsetof(BinCounters, timeouts) / 8), (int4*)zero,
                                            nzero);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

__global__ void k_clear_bounds(int* b) {
  if (threadIdx.x < 8) b[threadIdx.x] = 0x7F800000;
}
ufc_status bin_prep_bounds(ufc_ctx* c, BinTables* tab, int box) {
  k_clear_bounds<<<1, 32, 0, c->stream>>>(tab->bounds[box]);
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

// ------------------------------------------------------------ direct kernel --
constexpr int kDT = 384;                       // 12 warps, two blocks per SM
constexpr int kDWarps = kDT / 32;
constexpr int kDList = 64;                     // entries of one pending list
constexpr int kDUnd = 256;                     // undecided images waiting in a warp: at most 31
                                               // + 3 x 32 of a step + 2 x 32 of a drain
constexpr int kDMaxImg = kMaxImg1D * kMaxImg1D * kMaxImg1D;

struct DirectShared {
  float lo2[kMaxShells + 2], hi2[kMaxShells + 2];
  alignas(16) uint16_t lut[kLut];
  float4 lists[kDWarps][2][kDList];
  uint64_t und[kDWarps][kDUnd];
};
struct DirectImages {                          // after DirectShared, with images only
  float shf[3][kMaxImg1D], shlo[3][kMaxImg1D];
  int count;
  uint32_t mask[(kDMaxImg + 31) / 32];         // images kept, one bit each
  uint16_t list[kDMaxImg];                     // in increasing order, the same in every block:
                                               // the image's place per axis, 5 bits each
};

// Key of an image the FP32 stage left open: the double-float stage, then the
// FP64 procedure (exact set).  Out of line, so that its registers are not the
// fast stage's.
__device__ __noinline__ int2 key_late(const BinTables* t, int32_t lo, int32_t hi, int32_t N,
                                      int32_t npix, float3 p, float3 shf, float3 shlo,
                                      double3 sh64) {
  const int32_t key = key_refine(t->st.chih, t->st.chil, t->atab, lo, hi, N, npix, p.x, p.y, p.z,
                                 shf.x, shf.y, shf.z, shlo.x, shlo.y, shlo.z);
  if (key != kKeyUndecided) return make_int2(key, 0);
  return make_int2(key_exact(t->st, lo, hi, N, npix, p.x, p.y, p.z, sh64.x, sh64.y, sh64.z), 1);
}

// Each warp takes its tasks alone (task w, w + warps, ...), 32 particles at a
// time:
//   A: radius, shell (lookup table) and zone in FP32; belt and cap particles are
//      appended, with their observer-relative coordinates, to two pending
//      lists of the warp in shared memory (ballots), undecided ones to a third;
//   B: whenever a list holds 32 entries, the warp computes the pixels of the
//      newest 32 together and adds them to the item's count map (atomics in L2);
//   C: whenever 32 undecided images wait, their keys by the double-float and
//      FP64 stages, out of line.
// Without images (IMG false) a task is a.task particles of one item, read
// straight from global memory one group ahead (three loads per lane): at the
// direct path's sizes the particles' reads are not what bounds it.  With
// images a task is 32 particles, held in registers, times a slice of the
// box's image list: the images that can hold a particle inside the box's
// shells, from the bounds of the particles (k_direct_bounds).  The list is
// exact: x + shift and the FP32 r^2 are monotone in each coordinate, so r^2 of
// the nearest and farthest point of the bounds, formed by the same operations,
// brackets every particle's, and an image is left out only if that interval
// lies beyond the last edge or, clear of the observer, below the first.  Image
// 0 stays in the list for non-finite and overflowing coordinates, which count
// once per particle.
//
// What bounds it: without images the scattered atomics (150 realisations of 2 x 64^3
// particles: 106 G/s, 0.7 per SM and cycle; issue 44%, the particles' loads wait behind
// them, and neither loads two groups ahead nor the next task's particles fetched into L2
// changed that); with images the issue slots; at small sizes latency.  24 warps per SM (32
// of 64 registers spill: 940 against 775 us for the batched case then).
// Measured: 64^3 particles with four image layers (729 images, 10 shells, Nside 64) 1910 us
// with every image of every particle tested, in chunks of 3840 particles that left half of
// the SMs idle; 442 us with the image list; 288 us with one comparison per table entry, lists
// as stacks and the images' places per axis kept in the list (no divisions per step).  Two
// boxes of 64^3 in one launch of 20 us instead of two of 27, a late stage of 16 + 13 + 7 us
// and their queues; 150 realisations of 2 x 64^3 particles 743 us.
template <bool IMG>
__global__ void __launch_bounds__(kDT, 2)
k_direct(const __grid_constant__ DirectArgs a, const __grid_constant__ BoxGeom bg, int box) {
  extern __shared__ __align__(16) uint8_t dsm[];
  DirectShared& fs = *reinterpret_cast<DirectShared*>(dsm);
  DirectImages& im = *reinterpret_cast<DirectImages*>(dsm + sizeof(DirectShared));
  const unsigned full = 0xFFFFFFFFu;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const BinTables* tab = a.tab;
  const int S = tab->st.nshell;
  for (int i = threadIdx.x; i <= S; i += kDT) {
    fs.lo2[i] = tab->st.lo2[i];
    fs.hi2[i] = tab->st.hi2[i];
  }
  if (threadIdx.x == 0) fs.lo2[S + 1] = fs.hi2[S + 1] = INFINITY;
  // (all shells: the items of a launch have their own ranges)
  fill_lut_classified(fs.lut, tab->lut, lut_bin(a.bd.r2_min, a.lut_scale), 0, S);
  if (IMG) {
    const int n1 = 2 * bg.R + 1;
    for (int i = threadIdx.x; i < 3 * kMaxImg1D; i += kDT) {
      im.shf[i / kMaxImg1D][i % kMaxImg1D] = bg.shf[i / kMaxImg1D][i % kMaxImg1D];
      im.shlo[i / kMaxImg1D][i % kMaxImg1D] = bg.shlo[i / kMaxImg1D][i % kMaxImg1D];
    }
    __syncthreads();
    // bounds: ordered integers of min x, y, z and of -max x, y, z
    auto val = [&](int k) {
      const int o = tab->bounds[box][k];
      return __int_as_float(o >= 0 ? o : o ^ 0x7FFFFFFF);
    };
    const float b0[3] = {val(0), val(1), val(2)}, b1[3] = {-val(3), -val(4), -val(5)};
    const int nword = (bg.nimg + 31) >> 5;
    for (int w = warp; w < nword; w += kDWarps) {
      const int i = 32 * w + lane;
      const int id[3] = {i / (n1 * n1), (i / n1) % n1, i % n1};
      bool keep = i < bg.nimg;
      if (keep && i > 0) {
        float near[3], far[3];
        for (int k = 0; k < 3; ++k) {
          const float d0 = (b0[k] + im.shf[k][id[k]]) + im.shlo[k][id[k]];
          const float d1 = (b1[k] + im.shf[k][id[k]]) + im.shlo[k][id[k]];
          near[k] = d0 > 0.f ? d0 : (d1 < 0.f ? d1 : 0.f);
          far[k] = fmaxf(fabsf(d0), fabsf(d1));
        }
        const float r2n = fmaf(near[2], near[2], fmaf(near[1], near[1], near[0] * near[0]));
        const float r2f = fmaf(far[2], far[2], fmaf(far[1], far[1], far[0] * far[0]));
        keep = !(b0[0] > b1[0] || r2n >= fs.hi2[bg.shell_hi] ||
                 (r2f < fs.lo2[bg.shell_lo] && r2n >= a.bd.r2_min));
      }
      const unsigned m = __ballot_sync(full, keep);
      if (lane == 0) im.mask[w] = m;
    }
    __syncthreads();
    for (int w = warp; w < nword; w += kDWarps) {
      unsigned before = 0;
      for (int k = lane; k < w; k += 32) before += __popc(im.mask[k]);
      before = __reduce_add_sync(full, before);
      const unsigned m = im.mask[w];
      if (m >> lane & 1u) {
        const int i = 32 * w + lane;
        im.list[before + __popc(m & lt_mask)] =
            (uint16_t)(i / (n1 * n1) << 10 | (i / n1) % n1 << 5 | i % n1);
      }
      if (w == nword - 1 && lane == 0) im.count = before + __popc(m);
    }
  }
  __syncthreads();
  const int nimg = IMG ? im.count : 1;

  float4* list_eq = fs.lists[warp][0];
  float4* list_cap = fs.lists[warp][1];
  uint64_t* und = fs.und[warp];
  int ne = 0, nc = 0;                          // lengths of the two lists
  int hu = 0, nu = 0;                          // of the undecided images
  unsigned n_keyed = 0, n_invalid = 0, n_ref = 0, n_ex = 0;   // of this lane
  unsigned n_group = 0;                        // keys of the pixel stage (whole warp)
  const int64_t nw = (int64_t)gridDim.x * kDWarps;
  int it = -1;                                 // current item
  int32_t* cmap = nullptr;
  int lo = 0, hi = 0;
  float sx = 0.f, sy = 0.f, sz = 0.f, lx = 0.f, ly = 0.f, lz = 0.f;
  auto item = [&](int i) -> const DirectItem& { return a.items ? a.items[i] : a.inl[i]; };

  // C: `take` (<= 32) undecided images
  auto settle = [&](int take) {
    if (lane < take) {
      const uint64_t e = und[(hu + lane) & (kDUnd - 1)];
      const int tag = int(e >> 47);
      const int64_t p = qidx(e);
      const DirectItem& d = item(IMG ? 0 : tag);
      float3 f, l;
      double3 s;
      if (IMG) {
        const int n1 = 2 * bg.R + 1, ii = tag / (n1 * n1), jj = (tag / n1) % n1, kk = tag % n1;
        f = make_float3(bg.shf[0][ii], bg.shf[1][jj], bg.shf[2][kk]);
        l = make_float3(bg.shlo[0][ii], bg.shlo[1][jj], bg.shlo[2][kk]);
        s = make_double3(bg.sh64[0][ii], bg.sh64[1][jj], bg.sh64[2][kk]);
      } else {
        f = make_float3(d.shf[0], d.shf[1], d.shf[2]);
        l = make_float3(d.shlo[0], d.shlo[1], d.shlo[2]);
        s = make_double3(d.sh64[0], d.sh64[1], d.sh64[2]);
      }
      const float* q = d.xyz + 3 * p;
      const int2 k = key_late(tab, d.shell_lo, d.shell_hi, a.N, a.npix,
                              make_float3(__ldg(q), __ldg(q + 1), __ldg(q + 2)), f, l, s);
      ++n_ref;
      n_ex += k.y;
      n_invalid += k.x == kKeyInvalid;
      if (k.x >= 0) {
        ++n_keyed;
        if (UFC_IDX_OK(k.x, a.ncell, 2)) atomicAdd(d.counts + k.x, 1);
      }
    }
    hu = (hu + take) & (kDUnd - 1);
    nu -= take;
    __syncwarp();
  };
  auto image_tag = [&](uint32_t img) {         // the image's number, in an undecided entry
    const uint32_t n1 = uint32_t(2 * bg.R + 1);
    return uint64_t(((img >> 10) * n1 + ((img >> 5) & 31u)) * n1 + (img & 31u)) << 47;
  };
  auto push = [&](bool want, uint64_t e) {     // (the whole warp calls it)
    const unsigned m = __ballot_sync(full, want);
    if (want) und[(hu + nu + __popc(m & lt_mask)) & (kDUnd - 1)] = e;
    nu += __popc(m);
  };

#pragma unroll 1
  for (int64_t t = (int64_t)blockIdx.x * kDWarps + warp; t < a.ntasks; t += nw) {
    if (it < 0 || (!IMG && it + 1 < a.nitems && item(it + 1).task0 <= t)) {
      ++it;
      while (!IMG && it + 1 < a.nitems && item(it + 1).task0 <= t) ++it;
      const DirectItem& d = item(it);
      cmap = d.counts;
      lo = d.shell_lo;
      hi = d.shell_hi;
      if (!IMG) {
        sx = d.shf[0]; sy = d.shf[1]; sz = d.shf[2];
        lx = d.shlo[0]; ly = d.shlo[1]; lz = d.shlo[2];
      }
    }
    int64_t p0;                                // first particle of the task
    int cnt;                                   // particles
    int nsteps, i0 = 0;                        // groups of 32, or images from i0 on
    const DirectItem& ti = item(it);
    if (IMG) {
      const int64_t g = t / a.nslice;
      const int sl = int(t - g * a.nslice);
      p0 = 32 * g;
      cnt = int(min((int64_t)32, ti.n - p0));
      i0 = int((int64_t)nimg * sl / a.nslice);
      nsteps = int((int64_t)nimg * (sl + 1) / a.nslice) - i0;
    } else {
      p0 = (t - ti.task0) * a.task;
      cnt = int(min((int64_t)a.task, ti.n - p0));
      nsteps = (cnt + 31) >> 5;
    }
    // the late stage is called outside the loop over the steps, with nothing of
    // the fast stage in registers: once 32 images wait (or the task ends) the
    // lists are drained, and the loop starts again after the call
    int h = 0;
#pragma unroll 1
    do {
      float x = INFINITY, y = 0.f, z = 0.f;    // no particle: sorted out with the edge scans
      const int j0 = IMG ? lane : 32 * h + lane;
      const float* q = ti.xyz + 3 * (p0 + j0);
      if (j0 < cnt) { x = __ldg(q); y = __ldg(q + 1); z = __ldg(q + 2); }
#pragma unroll 1
      for (;;) {
        const bool tail = h == nsteps || nu >= 32;       // drains the lists
        if (!tail) {
          // ---- A
          uint32_t img = 0;                      // the image's place per axis
          float x1 = INFINITY, y1 = 0.f, z1 = 0.f;   // the next group's particle
          if (IMG) {
            img = im.list[i0 + h];
            const uint32_t ii = img >> 10, jj = (img >> 5) & 31u, kk = img & 31u;
            sx = im.shf[0][ii]; sy = im.shf[1][jj]; sz = im.shf[2][kk];
            lx = im.shlo[0][ii]; ly = im.shlo[1][jj]; lz = im.shlo[2][kk];
          } else {
            q += 96;
            if (32 * (h + 1) + lane < cnt) { x1 = __ldg(q); y1 = __ldg(q + 1); z1 = __ldg(q + 2); }
          }
          const float dx = (x + sx) + lx;
          const float dy = (y + sy) + ly;
          const float dz = (z + sz) + lz;
          const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
          uint32_t b = fs.lut[lut_bin(r2, a.lut_scale)];
          bool in = b - uint32_t(lo) < uint32_t(hi - lo), open = false;
          const bool fin = r2 <= 3.0e38f;                // false for NaN and overflow
          const bool scan = b >= kLutScan || !fin;
          if (__any_sync(full, scan)) {                  // rare: scan the edges
            if (scan) {
              in = false;
              const bool have = (IMG ? lane : 32 * h + lane) < cnt;
              // (non-finite or overflowing coordinates once per particle, with image 0)
              open = have && (fin ? !(r2 >= a.bd.r2_min)   // near the observer (r == 0 is invalid)
                                  : (!IMG || img == 0u));
              if (fin && !open) {
                int e = int(b & 0x7FFFu) - 1;
                for (;;) {                               // (ends at the +inf sentinel)
                  if (r2 < fs.lo2[e + 1]) break;
                  if (r2 < fs.hi2[e + 1]) { open = true; break; }
                  ++e;
                }
                in = !open && e >= lo && e < hi;
                b = uint32_t(e);
              }
            }
          }
          const float dz2 = dz * dz;
          const bool c2 = in && dz2 <= a.bd.z_eq2 * r2;
          const bool c3 = in && dz2 > a.bd.z_cap2 * r2;
          const bool c1 = open || (in && !c2 && !c3);
          // entry: coordinates, shell, and particle (offset, or lane and image)
          const uint32_t meta = b | (IMG ? uint32_t(lane) << 8 | img << 13
                                         : uint32_t(32 * h + lane) << 8);
          const float4 ent = make_float4(dx, dy, dz, __uint_as_float(meta));
          const unsigned meq = __ballot_sync(full, c2), mcap = __ballot_sync(full, c3);
          if (c2) list_eq[ne + __popc(meq & lt_mask)] = ent;
          if (c3) list_cap[nc + __popc(mcap & lt_mask)] = ent;
          ne += __popc(meq);
          nc += __popc(mcap);
          if (__any_sync(full, c1))
            push(c1, (IMG ? image_tag(img) : uint64_t(it) << 47) |
                         uint64_t(p0 + (IMG ? lane : 32 * h + lane)));
          if (!IMG) { x = x1; y = y1; z = z1; }
          ++h;
        }
        __syncwarp();
        // ---- B
        auto group_b = [&](auto zone_tag, int& len) {    // the newest 32 (or the rest)
          constexpr int ZONE = decltype(zone_tag)::value;
          const int take = min(len, 32);
          len -= take;
          const bool on = lane < take;           // (a lane without one reads an old entry)
          const float4 ent = (ZONE == 0 ? list_eq : list_cap)[len + lane];
          const float dx = ent.x, dy = ent.y, dz = ent.z;
          const uint32_t meta = __float_as_uint(ent.w);
          const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
          const float rinv = rsqrt_fast(r2);
          const float zz = dz * rinv;
          int32_t pix;
          if constexpr (ZONE == 0) pix = pixel_fast_eq(a.N, a.bd, dx, dy, zz);
          else pix = pixel_fast_cap(a.N, a.bd, dx, dy, dz, r2, rinv, zz);
          const bool ok = on && pix != kKeyUndecided;
          const int32_t key = int(meta & 255u) * a.npix + pix;
          if (ok && UFC_IDX_OK(key, a.ncell, 2)) atomicAdd(cmap + key, 1);
          const unsigned m = __ballot_sync(full, ok);
          n_group += __popc(m);
          if (m != full) {
            const uint64_t eu = IMG ? image_tag(meta >> 13) | uint64_t(p0 + ((meta >> 8) & 31u))
                                    : uint64_t(it) << 47 | uint64_t(p0 + (meta >> 8));
            push(on && !ok, eu);
          }
        };
        const int need = tail ? 1 : 32;
        if (ne >= need) group_b(std::integral_constant<int, 0>{}, ne);
        if (nc >= need) group_b(std::integral_constant<int, 1>{}, nc);
        __syncwarp();
        if (tail) break;
      }
      // ---- C: fewer than 32 stay, so that a step's pushes and the drain's fit
#pragma unroll 1
      while (nu >= 32) settle(32);
    } while (h < nsteps);
  }
  if (nu) settle(nu);
  n_keyed = __reduce_add_sync(full, n_keyed) + n_group;
  n_invalid = __reduce_add_sync(full, n_invalid);
  n_ref = __reduce_add_sync(full, n_ref);
  n_ex = __reduce_add_sync(full, n_ex);
  if (lane == 0) {
    if (n_keyed) atomicAdd(&a.cnt->keyed, (unsigned long long)n_keyed);
    if (n_invalid) atomicAdd(&a.cnt->invalid, (unsigned long long)n_invalid);
    if (n_ref) atomicAdd(&a.cnt->refined, (unsigned long long)n_ref);
    if (n_ex) atomicAdd(&a.cnt->exact, (unsigned long long)n_ex);
  }
}

// Bounds of the particles with finite coordinates: min x, y, z and min of
// -x, -y, -z as integers in the floats' order (b holds +inf before).
__global__ void __launch_bounds__(256)
k_direct_bounds(const float* __restrict__ xyz, int64_t n, int* __restrict__ b) {
  float m[6];
  for (int k = 0; k < 6; ++k) m[k] = INFINITY;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x) {
    const float v[3] = {__ldg(xyz + 3 * p), __ldg(xyz + 3 * p + 1), __ldg(xyz + 3 * p + 2)};
    if (isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]))
      for (int k = 0; k < 3; ++k) {
        m[k] = fminf(m[k], v[k]);
        m[k + 3] = fminf(m[k + 3], -v[k]);
      }
  }
  for (int k = 0; k < 6; ++k) {
    const int i = __float_as_int(m[k]);
    const int o = __reduce_min_sync(0xFFFFFFFFu, i >= 0 ? i : i ^ 0x7FFFFFFF);
    if ((threadIdx.x & 31) == 0 && o != 0x7F800000) atomicMin(b + k, o);
  }
}

// ---------------------------------------------------------------- host ------

// Index-check record of this translation unit (checked builds).
cudaError_t take_checks_direct(CheckRec* out, cudaStream_t s) { return take_check_rec(out, s); }

// Particles per task: enough tasks for every warp of the chip, at most 1024
// particles (the tasks in flight then cover few maps of a batched call, which
// stay in L2), at least 96 (the lists are drained at the end of a task, and a
// short task drains them part full).
int direct_task(const ufc_ctx* c, int64_t total) {
  const int64_t warps = 2ll * c->num_sms * kDWarps;
  const int64_t t = ((total + warps - 1) / warps + 31) / 32 * 32;
  return (int)std::min<int64_t>(std::max<int64_t>(t, 96), 1024);
}

ufc_status launch_direct(ufc_ctx* c, const DirectArgs& a, int blocks) {
  if (a.ntasks == 0) return UFC_OK;
  const int smem = (int)sizeof(DirectShared);
  const int grid = (int)std::min<int64_t>((int64_t)(blocks > 0 ? blocks : 2) * c->num_sms,
                                          (a.ntasks + kDWarps - 1) / kDWarps);
  UFC_CUDA(c, cudaFuncSetAttribute(k_direct<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   smem));
  {
    ProfScope ps_(c, "k_direct");
    k_direct<false><<<grid, kDT, smem, c->stream>>>(a, BoxGeom{}, 0);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

ufc_status launch_direct_images(ufc_ctx* c, DirectArgs a, const BoxGeom& g, int box) {
  const int64_t n = a.inl[0].n;
  if (n == 0) return UFC_OK;
  // eight tasks per warp of the chip (a box's images fill the shells unevenly)
  const int64_t groups = (n + 31) / 32, warps = 2ll * c->num_sms * kDWarps;
  a.nslice = (int)std::min<int64_t>(std::max<int64_t>((8 * warps + groups - 1) / groups, 1), 64);
  a.ntasks = groups * a.nslice;
  const int smem = (int)(sizeof(DirectShared) + sizeof(DirectImages));
  const int grid = (int)std::min<int64_t>(2ll * c->num_sms, (a.ntasks + kDWarps - 1) / kDWarps);
  UFC_CUDA(c, cudaFuncSetAttribute(k_direct<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   smem));
  {
    ProfScope ps_(c, "k_direct_bounds");
    k_direct_bounds<<<(int)std::min<int64_t>(4 * c->num_sms, (n + 255) / 256), 256, 0, c->stream>>>(
        a.inl[0].xyz, n, a.tab->bounds[box]);
  }
  {
    ProfScope ps_(c, "k_direct");
    k_direct<true><<<grid, kDT, smem, c->stream>>>(a, g, box);
  }
  UFC_CUDA(c, cudaGetLastError());
  return UFC_OK;
}

}  // namespace ufc
