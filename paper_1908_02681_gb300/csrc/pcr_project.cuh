// Per-point transform without a framebuffer (pcr_project_points in include/pcr.h): for every point, the pixel
// and the key the definition of Sections 1 and 2.1 gives it, or 0xFFFFFFFF and the empty key when it is culled.
// It exposes, point by point, the same decisions the raster passes take (tier 1, tier 2, FP64 arbiter), so they can be
// checked against the definition for every point and not only for the fragments that win a pixel.
#pragma once

#include "pcr_screen.cuh"

namespace pcr {

__device__ __forceinline__ void project_store(uint32_t* pix_out, unsigned long long* key_out, uint64_t i, bool visible,
                                              uint32_t pix, unsigned long long key) {
  __stcs(pix_out + i, visible ? pix : 0xFFFFFFFFu);
  __stcs(key_out + i, visible ? key : kEmptyKey);
}

// Tier 2 and the arbiter for a point that tier 1 left undecided. Out of line, as raster_deferred.
__device__ __noinline__ void project_deferred(const CertParams& P, const long long* sF, uint4 p, uint64_t i,
                                              uint32_t* pix_out, unsigned long long* key_out) {
  const CertFrag c = classify_cert(P, sF, p);
  uint32_t pix = c.pixel;
  unsigned long long q = (unsigned long long)c.q;
  bool visible = c.state == kExact;
  if (c.state != kExact && c.state != kCulled)
    visible = project_fp64(P.v, __uint_as_float(p.x), __uint_as_float(p.y), __uint_as_float(p.z), &pix, &q);
  project_store(pix_out, key_out, i, visible, pix, make_key(q, p.w));
}

// EXACT: tier 1 decides nearly every point; the others are queued by place and go through tier 2 and, if that cannot
// decide either, the FP64 definition, 32 at a time. The tiles and their loads are the screened passes'. Bound by issue
// slots and DRAM (28 bytes a point). 6M points on one GB300: 57 us with one point a thread, plain loads and tier 2 in
// line (a fifth of the warps' steps ran it for one or two lanes), 40 us now; 60M 468 and 325 (their bytes at the copy rate: 247).
template <int kPw>
__global__ void __launch_bounds__(kScreenThreads, 1) k_project_cert(const uint4* __restrict__ pts, uint64_t n,
                                                                    const __grid_constant__ CertParams P,
                                                                    uint32_t* __restrict__ pix_out,
                                                                    unsigned long long* __restrict__ key_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  long long* const sF = reinterpret_cast<long long*>(smem);
  const int tables = kPw ? P.n_pw : 1;
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t* const open = reinterpret_cast<uint32_t*>(smem + tables * kTableBytes) + (threadIdx.x >> 5) * kCand;
  const WarpTiles T = warp_tiles();
  release_next();
  build_tables(P.col, tables, sF);
  wait_previous();
  uint32_t on = 0;
  auto index = [&](uint32_t place) { return (T.g + (uint64_t)(place >> 6) * T.G) * kTile + (place & 63u); };
  auto tier2 = [&](uint32_t place) { project_deferred(P, sF, point_at(pts, T, place), index(place), pix_out, key_out); };
  auto drain = [&]() {
    __syncwarp();
    while (on >= 32u) {
      on -= 32u;
      const uint32_t place = open[on + lane];
      __syncwarp();
      tier2(place);
    }
  };
  screen_tiles<false>(
      pts, n, T, lane,
      [&](const uint4& p0, const uint4& p1, uint32_t place) {
        const uint64_t i = index(place);
        const FastFrag f0 = classify_fast<CertParams, kPw>(P, sF, p0);
        const bool o0 = f0.state >= kAmbiguous;
        if (!o0) project_store(pix_out, key_out, i, f0.state == kExact, f0.pixel, key_from_fixed(f0.a0, f0.a1, f0.a2, p0.w));
        const FastFrag f1 = classify_fast<CertParams, kPw>(P, sF, p1);
        const bool o1 = f1.state >= kAmbiguous;
        if (!o1)
          project_store(pix_out, key_out, i + 32u, f1.state == kExact, f1.pixel, key_from_fixed(f1.a0, f1.a1, f1.a2, p1.w));
        if (__any_sync(0xFFFFFFFFu, o0 | o1)) {
          push_open(o0, place, open, on, lane);
          push_open(o1, place + 32u, open, on, lane);
          drain();
        }
      },
      [&](uint32_t place, bool v0, bool v1) {
        push_open(v0, place, open, on, lane);
        push_open(v1, place + 32u, open, on, lane);
        drain();
      });
  __syncwarp();
  if (lane < on) tier2(open[lane]);
}

template <int kPw>
inline cudaError_t launch_project(const uint4* pts, uint64_t n, const CertParams& P, uint32_t* pix, unsigned long long* key,
                                  int sms, cudaStream_t s) {
  constexpr int most_tables = kPw ? kMaxRanges : 1;
  constexpr size_t queue = kCand * sizeof(uint32_t);
  static std::atomic<uint64_t> opted{0};
  const cudaError_t e = opt_in_shared(k_project_cert<kPw>, most_tables * kTableBytes + kScreenThreads / 32 * queue, opted);
  if (e != cudaSuccess) return e;
  const ScreenLaunch L = screen_launch(n, sms, kScreenThreads / 256, 1, false);
  launch_after(k_project_cert<kPw>, L.grid, L.threads, table_blocks(P) * kTableBytes + L.threads / 32 * queue, s, pts, n, P,
               pix, key);
  return cudaGetLastError();
}

// DOUBLE_FLOAT: the double-float evaluation alone, one point a thread.
__global__ void __launch_bounds__(256) k_project_df(const uint4* __restrict__ pts, uint64_t n,
                                                    const __grid_constant__ CertParams P, uint32_t* __restrict__ pix_out,
                                                    unsigned long long* __restrict__ key_out) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint4 p = pts[i];
    const CertFrag f = classify_df(P, p);
    project_store(pix_out, key_out, i, f.state == kExact, f.pixel, make_key((unsigned long long)f.q, p.w));
  }
}

// FP64 (and every view outside the single-precision preconditions, piecewise depth included): each point
// through the FP64 definition directly.
__global__ void __launch_bounds__(256) k_project_fp64(const uint4* __restrict__ pts, uint64_t n, const DevView v,
                                                      uint32_t* __restrict__ pix_out,
                                                      unsigned long long* __restrict__ key_out) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint4 p = pts[i];
    uint32_t px;
    unsigned long long q;
    const bool vis = project_fp64(v, __uint_as_float(p.x), __uint_as_float(p.y), __uint_as_float(p.z), &px, &q);
    pix_out[i] = vis ? px : 0xFFFFFFFFu;
    key_out[i] = vis ? make_key(q, p.w) : kEmptyKey;
  }
}

}  // namespace pcr
