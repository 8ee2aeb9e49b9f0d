// Screened point passes: the certified transform of pcr_certified.cuh with the depth code left out for every point
// whose float depth already settles what the pass does with it.
//
// Pass 1 (Section 2.1 of arXiv 1908.02681) only needs a point's exact 40-bit code when the point may lower its
// pixel's key, pass 2 (Section 2.2) only when it lies next to an edge of its pixel's depth band. So each pass first
// screens a point: tier 1's cull and pixel decisions, then the float depth estimate against the pixel's stored key
// with a margin that covers every rounding (see Screen). Points the screen cannot settle are gathered in a per-warp
// shared-memory queue and go through the full tiers 32 at a time, all lanes busy.
#pragma once

#include "pcr_certified.cuh"

namespace pcr {

// Constants of the screen of one view and pass. sh is the stored key's code in units of `unit` codes, as a float:
// key >> 32 (unit 2^8), or for views whose codes stay below 2^32 the code itself, saturated (unit 1).
//   Definition: code q = floor(t_d), t_d = S (w_d - off) up to 2^-11 (off = near for LINEAR, 0 for METRIC; FP64
//   roundings of a t below 2^40). The stored code qs lies in [unit sh, unit (sh + 1)).
//   |wf - w_d| <= Delta <= 4.0005u (Mw s + Mw3), |wf| <= Mw s + Mw3 (tier1_constants), u = 2^-24. An edge
//   e(sh) = RN(a sh + b), a and b >= 0 or a = 0, is within 3.1u |e| of its real value (roundings of sh, a, b, the fma).
//   With the margin m(s) = RN(k s + k3) >= (Delta + c + 3.1u |wf|)(1 + 16u), c the slack below:
//     RN(wf - e) >= m  implies  w_d >= e_real + c: wf - e >= m (1 - u), and e_real <= e + 3.1u e <= e + 3.1u wf
//     RN(wf - e) <= -m implies  w_d <= e_real - c: e_real >= e - 3.1u e, and 3.1u e = 3.1u (e - wf) + 3.1u wf
//   c S covers the width of the stored code's unit and the 2^-11 of t_d.
//   PIECEWISE (pass 1 only): codes grow with w across the ranges, so a point in range r has a larger code than qs iff it
//   lies beyond the edge lo_r + (qs + 1 - base_r) / res_r, wherever qs itself lies. Its b = lo_r + (unit - base_r) / res_r
//   may be negative: the roundings of a sh, b and the fma are then within 3.1u |e| + 3.1u |b| (e >= 0) or 4.1u |b|, and
//   k3 has 4.2u |b| more.
struct Screen {
  float k;
  float k3[kMaxRanges];                 // margin (index: PIECEWISE range, else 0)
  float a[kMaxRanges], b[kMaxRanges];   // pass 1: off + unit (sh + 1) / S; a point beyond this edge has a larger code
  float lo_a, lo_b;  // pass 2: lower band edge off + unit sh / S, or far below every w (not tested)
  float hi_a, hi_b;  // pass 2: upper band edge off + (unit sh (1 + eps) + eps Nq) / S
};

// Whether the view's codes fit 32 bits (unit 1).
inline bool screen_unit1(const DevView& v) {
  return v.depth_mode == 1 && v.far_ * v.scale < 4294967040.0;
}

// Which variant of the screened kernels a view takes.
enum ScreenMode : int { kUnit256 = 0, kUnit1 = 1, kPiecewise2 = 2, kPiecewise = 3 };  // 2: at most two ranges

inline ScreenMode screen_mode(const CertParams& P) {
  return P.n_pw > 2 ? kPiecewise : P.n_pw > 0 ? kPiecewise2 : screen_unit1(P.v) ? kUnit1 : kUnit256;
}

// The screen of a view; pass 2's edges for eps_num / eps_den (eps_den = 0: pass 1 only); lower: pass 2 also tests the
// lower edge (needed unless every point's own pass 1 has written the keys: then q >= qmin). False when the constants
// leave the float range.
inline bool make_screen(const CertParams& P, uint32_t eps_num, uint32_t eps_den, bool lower, Screen* out) {
  const DevView& v = P.v;
  const double u = 0x1p-24, up = 1.0 + 0x1p-18;
  const ScreenMode mode = screen_mode(P);
  const double unit = mode == kUnit1 ? 1.0 : 256.0, eps = eps_den ? (double)eps_num / (double)eps_den : 0.0;
  // every edge below 2^33 * 1e24 and normal: relative roundings, no overflow
  auto normal = [](float f) { return f > 1e-30f && f < 1e24f; };
  Screen s;
  std::memset(&s, 0, sizeof(s));
  s.k = host::f_up(7.2 * u * (double)P.Mw * up);
  bool ok = normal(s.k);
  int r = 0;
  auto edge = [&](double S, double off, double base) {
    const double c = (unit * (1.0 + eps) + 2.0) / S, b = off + (unit - base) / S;
    s.a[r] = (float)(unit / S);
    s.b[r] = (float)b;
    s.k3[r] = host::f_up((7.2 * u * (double)P.Mw3 + c + (b < 0.0 ? -4.2 * u * b : 0.0)) * up);
    ok = ok && normal(s.a[r]) && normal(s.k3[r]) && normal(b < 0.0 ? -s.b[r] : s.b[r]);
    ++r;
  };
  if (P.n_pw > 0) {  // the ranges that meet [near, far), in prepare_cert's order
    for (int k = 0; k < v.n_ranges; ++k)
      if (std::fmin(v.hi[k], v.far_) > std::fmax(v.lo[k], v.near_)) edge(v.res[k], v.lo[k], v.base[k]);
    *out = s;
    return ok && r == P.n_pw && eps_den == 0;
  }
  const double S = v.scale, off = P.linear ? v.near_ : 0.0;
  edge(S, off, 0.0);
  s.lo_a = lower ? s.a[0] : 0.0f;
  s.lo_b = lower ? (float)off : -3.0e38f;
  s.hi_a = (float)(unit * (1.0 + eps) / S);
  s.hi_b = (float)(off + eps * (double)v.nq / S);
  *out = s;
  return ok && normal(s.hi_a) && s.hi_b >= 0.0f && s.hi_b < 1e24f;
}

// The stored code of a pixel in the screen's units, as a float (rounded to nearest).
template <int kMode>
__device__ __forceinline__ float stored_depth(const unsigned long long* keys, uint32_t pix) {
  if constexpr (kMode == kUnit1) {
    const unsigned long long k = stored_key(keys, pix);
    const uint32_t hi = (uint32_t)(k >> 32);
    return __uint2float_rn(hi >> 24 ? 0xFFFFFFFFu : __funnelshift_r((uint32_t)k, hi, 24));
  } else {
    return __uint2float_rn(__ldca(reinterpret_cast<const uint32_t*>(keys + pix) + 1));
  }
}

// The PIECEWISE range whose window may hold w (see CertParams::pw_start).
template <int kMode>
__device__ __forceinline__ int screen_range(const CertParams& P, float w) {
  int r = 0;
  if constexpr (kMode == kPiecewise2) r = w >= P.pw_start[1] ? 1 : 0;
  if constexpr (kMode == kPiecewise)
    for (int k = 1; k < P.n_pw; ++k) r += w >= P.pw_start[k];
  return r;
}

// A range's value of a per-range constant: a select between two, or indexed.
template <int kMode>
__device__ __forceinline__ float ranged(const float* f, int r) {
  if constexpr (kMode == kPiecewise2) return r ? f[1] : f[0];
  if constexpr (kMode == kPiecewise) return f[r];
  return f[0];
}

// Tier 1 without the depth code, of one point: what the test against its stored key needs. A point that is not
// certainly visible has w = +inf, so that the ordered comparisons of both passes' tests drop it whatever its coordinates
// (their magnitude sum, hence the margin, may be infinite or NaN) and its pixel is never used.
struct ScreenPoint {
  uint32_t pixel;
  float w, m;  // depth estimate and margin
  float k;     // stored depth (screen units)
  float a, b;  // pass 1's edge
  bool open;   // undecided, and not certainly culled (tier 2 decides)
};

// Both points of a lane. One branch leads to the cull tests of the two: on scans a tile mostly has none of them (pass 2 of
// the 100M-point scan on one GB300 1.5 % faster than with a branch per point, 400M city points' pass 1 5 %; 37M shuffled
// points' pass 2 1 % slower).
struct ScreenTwo {
  ScreenPoint a, b;
};

template <int kMode>
__device__ __forceinline__ ScreenTwo screen_two(const CertParams& P, const Screen& S, const uint4& p0, const uint4& p1,
                                                const unsigned long long* keys) {
  constexpr bool kPw = kMode >= kPiecewise2;
  ScreenTwo t;
  float s[2];
  bool in[2];
  PixelEstimate e[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint4& p = h ? p1 : p0;
    ScreenPoint& o = h ? t.b : t.a;
    const float x = __uint_as_float(p.x), y = __uint_as_float(p.y), z = __uint_as_float(p.z);
    s[h] = __fadd_rn(__fadd_rn(fabsf(x), fabsf(y)), fabsf(z));
    o.w = __fmaf_rn(P.Wr[2], z, __fmaf_rn(P.Wr[1], y, __fmaf_rn(P.Wr[0], x, P.Wr[3])));
    const int r = screen_range<kMode>(P, o.w);
    const float wc = kPw ? ranged<kMode>(P.pw_wc, r) : P.wc, whk = kPw ? ranged<kMode>(P.pw_whk, r) : P.whk;
    in[h] = fabsf(__fsub_rn(o.w, wc)) < __fmaf_rn(-P.kw, s[h], whk);
    e[h] = pixel_estimate(P, x, y, z, s[h], o.w);
    o.m = __fmaf_rn(S.k, s[h], ranged<kMode>(S.k3, r));
    o.a = ranged<kMode>(S.a, r);
    o.b = ranged<kMode>(S.b, r);
    o.pixel = e[h].pixel;
    o.k = 0.0f;
    o.open = !(in[h] & e[h].ok);
    if (!o.open) o.k = stored_depth<kMode>(keys, o.pixel);
  }
  if (t.a.open | t.b.open) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      ScreenPoint& o = h ? t.b : t.a;
      if (o.open) {
        o.open = !certainly_culled(P, s[h], o.w, s[h] < P.xyz_max, in[h], e[h]);
        o.w = __int_as_float(0x7F800000);
      }
    }
  }
  return t;
}

// Whether a point certainly lies outside the clip planes.
__device__ __forceinline__ bool point_outside_depth(const CertParams& P, const uint4& p) {
  const float x = __uint_as_float(p.x), y = __uint_as_float(p.y), z = __uint_as_float(p.z);
  const float s = __fadd_rn(__fadd_rn(fabsf(x), fabsf(y)), fabsf(z));
  const float w = __fmaf_rn(P.Wr[2], z, __fmaf_rn(P.Wr[1], y, __fmaf_rn(P.Wr[0], x, P.Wr[3])));
  return (s < P.xyz_max) & certainly_outside_depth(P, s, w);
}

// Per-warp queues in shared memory: two pushes of 32 on top of at most 31 left over. Points are also known by their
// place in the warp's sequence of tiles: 64 * tile number + place in the tile (fits 32 bits: n < 2^40, and a grid over
// that many points has over 1000 warps). Open points are queued by place alone and read again for tier 2: they are
// few, and shared memory that the queues leave free is L1, which holds the stored-key reads in flight. Pass 1 keeps its
// candidates' points (reading them again cost more than their space: the 100M-point frame 1.13 against 1.06 ms), pass 2,
// with few candidates, does not (that frame 0.97 to 0.95 ms on one GB300; 37M shuffled points 0.442 to 0.452).
constexpr uint32_t kCand = 96;

struct PlaceQueues {
  uint32_t pixel[kCand];  // candidates: certainly visible points whose exact code decides, their pixels
  uint32_t place[kCand];  // and places
  uint32_t open[kCand];   // places of the points for tier 2
};
struct ScreenQueues : PlaceQueues {  // pass 1, whose candidates are many
  uint4 p[kCand];
};

// Threads of a screened pass's block at most: one block an SM (see k_raster_screen); launches over few points take
// smaller blocks, to reach every SM.
constexpr int kScreenThreads = 1024;

// A tile with at least this many points whose code decides computes it for all 64 in place instead of queueing them:
// a strip of a scan that reaches pixels first has runs of them. On the 100M-point scan pass 1 takes 0.51 ms (10, 16, 24
// or 40 points: within 1 %) against 0.58 with every candidate queued.
constexpr int kDirect = 24;

// Exact code of a certainly visible point (tier 1's depth part; PIECEWISE: with its range's table and constants);
// false when undecided between two neighbours.
template <int kMode>
__device__ __forceinline__ bool exact_code(const CertParams& P, const long long* sF, const uint4& p, FixedCode* c) {
  const float x = __uint_as_float(p.x), y = __uint_as_float(p.y), z = __uint_as_float(p.z);
  const float s = __fadd_rn(__fadd_rn(fabsf(x), fabsf(y)), fabsf(z));
  float kd = P.kd, hd0 = P.hd0;
  if constexpr (kMode >= kPiecewise2) {
    const int r = screen_range<kMode>(
        P, __fmaf_rn(P.Wr[2], z, __fmaf_rn(P.Wr[1], y, __fmaf_rn(P.Wr[0], x, P.Wr[3]))));
    *c = fixed_code(sF + r * 3 * kTableEntries, p, P.pw_BL[r], P.pw_BH[r]);
    kd = P.pw_kd[r];
    hd0 = P.pw_hd0[r];
  } else {
    *c = fixed_code(sF, p, P.BL, P.BH);
  }
  return (s < P.xyz_max) & (fabsf(__fsub_rn(c->frac, 0.5f)) < __fmaf_rn(-kd, s, hd0));
}

__device__ __forceinline__ void push_open(bool need, uint32_t place, uint32_t* q, uint32_t& qn, uint32_t lane) {
  const unsigned m = __ballot_sync(0xFFFFFFFFu, need);
  if (need) q[qn + __popc(m & ((1u << lane) - 1u))] = place;
  qn += __popc(m);
}

__device__ __forceinline__ void push_candidate(bool need, const uint4& p, uint32_t pixel, uint32_t place, ScreenQueues& q,
                                               uint32_t& qn, uint32_t lane) {
  const unsigned m = __ballot_sync(0xFFFFFFFFu, need);
  if (need) {
    const uint32_t i = qn + __popc(m & ((1u << lane) - 1u));
    q.p[i] = p;
    q.pixel[i] = pixel;
    q.place[i] = place;
  }
  qn += __popc(m);
}

// The same for pass 2, whose candidates (next to a band edge) are few and read again.
__device__ __forceinline__ void push_candidate(bool need, uint32_t pixel, uint32_t place, PlaceQueues& q, uint32_t& qn,
                                               uint32_t lane) {
  const unsigned m = __ballot_sync(0xFFFFFFFFu, need);
  if (need) {
    const uint32_t i = qn + __popc(m & ((1u << lane) - 1u));
    q.pixel[i] = pixel;
    q.place[i] = place;
  }
  qn += __popc(m);
}

// Runs tier2(place) and candidate(index, true) on batches of 32 while there are that many. Called at the end of a
// tile, where few registers are live across the out-of-line tier 2. A candidate batch leaves at most 32 open points,
// which go first. All lanes must call it.
template <typename T2, typename Cand>
__device__ __forceinline__ void drain_batches(PlaceQueues& q, uint32_t& on, uint32_t& cn, uint32_t lane, T2&& tier2,
                                              Cand&& candidate) {
  __syncwarp();
  for (;;) {
    if (on >= 32u) {
      on -= 32u;
      const uint32_t place = q.open[on + lane];
      __syncwarp();
      tier2(place);
    } else if (cn >= 32u) {
      cn -= 32u;
      candidate(cn + lane, true);
      __syncwarp();
    } else {
      break;
    }
  }
}

// The warps of the grid take the tiles of 64 points in turn.
struct WarpTiles {
  uint32_t g, G;  // this warp in the grid, warps in the grid
};

__device__ __forceinline__ WarpTiles warp_tiles() {
  const uint32_t w = blockDim.x >> 5;
  return WarpTiles{blockIdx.x * w + (threadIdx.x >> 5), gridDim.x * w};
}

__device__ __forceinline__ uint4 point_at(const uint4* pts, const WarpTiles& T, uint32_t place) {
  return ld_stream16(pts + (T.g + (uint64_t)(place >> 6) * T.G) * kTile + (place & 63u));
}

// The full tiles of a warp, both points of a lane at a time, loaded one tile ahead (as stream_direct): body(p0, p1,
// place of p0); for the partial last tile rest(place of the lane's first point, whether each of its points exists).
// kMask: the full tiles of chunks whose bit in `mask` is clear (16 tiles a chunk) are skipped; a tile's mask word is read
// two tiles ahead, so that its points are still requested one ahead.
constexpr uint32_t kTilesPerChunk = 16;

template <bool kMask, typename Body, typename Rest>
__device__ __forceinline__ void screen_tiles(const uint4* __restrict__ pts, uint64_t n, const WarpTiles& T, uint32_t lane,
                                             Body&& body, Rest&& rest, const uint32_t* __restrict__ mask = nullptr) {
  const uint64_t n_full = n / kTile;
  const uint32_t G = T.G, g = T.g;
  const uint32_t tiles = n_full > g ? (uint32_t)((n_full - g - 1u) / G) + 1u : 0u;
  const uint4* p = pts + (uint64_t)g * kTile + lane;
  const uint64_t step = (uint64_t)G * kTile;
  uint4 a0 = make_uint4(0u, 0u, 0u, 0u), a1 = a0;
  uint32_t chunk = 0, word = 0;  // kMask: the next tile's chunk and its mask word
  bool seen = true;              // kMask: whether the current tile's chunk is visible
  auto chunk_of = [&](uint32_t at) { return (uint32_t)((g + (uint64_t)(at >> 6) * G) / kTilesPerChunk); };
  auto bit = [&](uint32_t w, uint32_t c) { return ((w >> (c & 31u)) & 1u) != 0u; };
  auto mask_word = [&](uint32_t c) {  // volatile: not moved above the wait for the kernel that wrote it
    uint32_t w;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(w) : "l"(mask + (c >> 5)) : "memory");
    return w;
  };
  if (tiles) {
    if constexpr (kMask) {
      const uint32_t c = chunk_of(0);
      seen = bit(mask_word(c), c);
      chunk = chunk_of(kTile);
      if (tiles > 1u) word = mask_word(chunk);
    }
    if (!kMask || seen) {
      a0 = ld_stream16(p);
      a1 = ld_stream16(p + 32);
    }
  }
  const uint32_t end = tiles * (uint32_t)kTile + lane;
  uint32_t place = lane;
#pragma unroll 1
  while (place != end) {
    const uint4 c0 = a0, c1 = a1;
    const bool now = seen;
    p += step;
    if constexpr (kMask) {
      seen = bit(word, chunk);
      chunk = chunk_of(place + 2u * kTile);
      if (end - place > 2u * kTile) word = mask_word(chunk);
    }
    if (place + (uint32_t)kTile != end && (!kMask || seen)) {
      a0 = ld_stream16(p);
      a1 = ld_stream16(p + 32);
    }
    if (!kMask || now) body(c0, c1, place);
    place += (uint32_t)kTile;
  }
  const uint32_t rem = (uint32_t)(n - n_full * kTile);
  if (rem != 0u && n_full % G == g) rest(end, lane < rem, lane + 32u < rem);
}

// A pass over at least this many tiles a warp (2.99e7 points on 152 SMs with default tuning) samples the cloud first, a tile a
// warp spread over all of it (1.5 us: 0.6 % of a high-quality frame of 28M scanned points, 1.1 % of 15M; shuffled clouds
// below the line go without the words, which would take their frame at 22M points from 291 to 251 us and at 10M from 151 to
// 139), and its blocks take the loop that suits it:
//   far_out: a quarter of the sampled points lie outside the clip planes (scans much larger than the view): pass 1 tests
//     each tile for lying outside as a whole before the pixel work. 400M city points on one GB300: 1.32 to 1.11 ms; done
//     always, the test costs the 100M-point scan 2 % of pass 1 and piecewise depth 6 %.
//   random: fewer than one in 64 of the sampled visible points share their pixel with the next point (clouds in no
//     order): in HQ frames, from the one after that on, pass 1 leaves pass 2 words that say which points it may accept
//     (kWords). Pixels meet their nearest points early then, and pass 2 reads 38 % of 37M shuffled points: the frame 0.46 to
//     0.38 ms on one GB300. In scan order the words leave 60 to 80 % of the points and cost more than they save (100M points 0.94 to 1.00 ms).
// A block's decision depends on the cloud, the view and the launch shape alone: pass 2, of the same shape, comes to the
// same one for the same tiles.
constexpr uint32_t kSampleTiles = 96;

struct CloudSample {
  bool far_out, random;
};

template <int kMode>
__device__ __forceinline__ CloudSample sample_cloud(const CertParams& P, const uint4* pts, uint64_t n, const WarpTiles& T,
                                                    uint32_t lane) {
  CloudSample c{false, false};
  const uint64_t spread = n / kTile / T.G;
  if (spread < kSampleTiles) return c;
  // the block's samples lie all over the cloud
  const uint4* const at = pts + ((uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * spread * kTile + lane;
  const uint4 p[2] = {ld_stream16(at), ld_stream16(at + 32)};
  int outside = 0, seen = 0, same = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float x = __uint_as_float(p[h].x), y = __uint_as_float(p[h].y), z = __uint_as_float(p[h].z);
    const float s = __fadd_rn(__fadd_rn(fabsf(x), fabsf(y)), fabsf(z));
    const float w = __fmaf_rn(P.Wr[2], z, __fmaf_rn(P.Wr[1], y, __fmaf_rn(P.Wr[0], x, P.Wr[3])));
    const PixelEstimate e = pixel_estimate(P, x, y, z, s, w);
    const uint32_t pixel = w > 0.0f && e.ok ? e.pixel : 0xFFFFFFFFu - lane;
    outside += __syncthreads_count(point_outside_depth(P, p[h]));
    seen += __syncthreads_count(w > 0.0f && e.ok);
    same += __syncthreads_count(__shfl_down_sync(0xFFFFFFFFu, pixel, 1) == pixel && lane < 31u);
  }
  c.far_out = 2 * outside >= (int)blockDim.x;
  c.random = 64 * same < seen;
  return c;
}

// The points whose bit is set in `words` (two words a tile of 64), 64 at a time: body(p0, p1, their places, whether each
// exists). Places are gathered in the warp's queue from the words alone, so tiles without a set bit are not read; a
// batch's points are requested while the batch before it is processed. The words are read 32 tiles at a time, one ahead.
constexpr uint32_t kBandQueue = 128;  // at most 63 left over and 64 of a tile

// volatile: not moved above the wait for the kernel that wrote the words
__device__ __forceinline__ uint2 ld_words(const uint2* p) {
  uint2 v;
  asm volatile("ld.global.cs.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
  return v;
}

template <typename Body>
__device__ __forceinline__ void band_points(const uint4* __restrict__ pts, uint64_t n, const WarpTiles& T, uint32_t lane,
                                            const uint2* __restrict__ words, uint32_t* q, Body&& body) {
  const uint64_t n_tiles = (n + kTile - 1) / kTile;
  const uint32_t tiles = n_tiles > T.g ? (uint32_t)((n_tiles - T.g - 1u) / T.G) + 1u : 0u;
  auto block = [&](uint32_t t) {  // the words of tiles t + lane
    return t + lane < tiles ? ld_words(words + T.g + (uint64_t)(t + lane) * T.G) : make_uint2(0u, 0u);
  };
  uint2 w = make_uint2(0u, 0u), ahead = block(0);
  uint32_t t = 0, cn = 0;
  auto fill = [&]() {
    while (cn < 64u && t < tiles) {
      if ((t & 31u) == 0u) {
        w = ahead;
        ahead = block(t + 32u);
      }
      const uint32_t b0 = __shfl_sync(0xFFFFFFFFu, w.x, t & 31u), b1 = __shfl_sync(0xFFFFFFFFu, w.y, t & 31u);
      const uint32_t below = (1u << lane) - 1u, place = t * (uint32_t)kTile + lane;
      if ((b0 >> lane) & 1u) q[cn + __popc(b0 & below)] = place;
      cn += __popc(b0);
      if ((b1 >> lane) & 1u) q[cn + __popc(b1 & below)] = place + 32u;
      cn += __popc(b1);
      ++t;
    }
    __syncwarp();
  };
  uint4 a0 = make_uint4(0u, 0u, 0u, 0u), a1 = a0;
  uint32_t l0 = 0, l1 = 0, have = 0;  // the next batch: places and size
  auto take = [&]() {
    fill();
    have = cn < 64u ? cn : 64u;
    cn -= have;
    if (lane < have) {
      l0 = q[cn + lane];
      a0 = point_at(pts, T, l0);
    }
    if (lane + 32u < have) {
      l1 = q[cn + lane + 32u];
      a1 = point_at(pts, T, l1);
    }
    __syncwarp();
  };
  take();
#pragma unroll 1
  while (have) {
    const uint4 p0 = a0, p1 = a1;
    const uint32_t c0 = l0, c1 = l1;
    const bool v0 = lane < have, v1 = lane + 32u < have;
    take();
    body(p0, p1, c0, c1, v0, v1);
  }
}

// Pass 1 (Section 2.1), exact transform. Issue slots and the latency of the stored-key reads
// bound it (67 % busy and the top stall at 20M points). 32 warps an SM at 64 registers, as one block: 48 warps with one
// point a lane (40 registers) and 24 warps (80) were slower, and one block holds one table, which leaves L1 more room
// for the keys in flight than two of 512 threads (shuffled 37M points, both passes 0.44 against 0.57 ms). Against
// k_raster_cert, which computes every point's code, on one GB300: 400M city points at 4K 2.23 to 1.10 ms (the culled
// points), 37M shuffled 0.227 to 0.18, 100M in scan order 0.539 to 0.48, and frames of 0.5 to 4 points per pixel equal
// or a few per cent faster, so it runs at every size.
// kLeave (HQ frames): what else the pass leaves where `side` points. kOrder: one word, 1 where the sample finds the cloud in
// random order (an instance of its own: in the plain one the argument cost 1M points 1.6 %). kWords: per tile, two words with
// a bit for each point that pass 2 may accept, clear where the point is culled or certainly beyond the upper band edge of the
// key its pixel holds (a stored key only decreases, and the edge with it).
enum RasterLeave : int { kNothing = 0, kOrder = 1, kWords = 2 };

template <int kMode, int kLeave>
__global__ void __launch_bounds__(kScreenThreads, 1) k_raster_screen(
    const uint4* __restrict__ pts, uint64_t n, const __grid_constant__ CertParams P, const __grid_constant__ Screen S,
    unsigned long long* __restrict__ keys, uint2* __restrict__ side) {
  extern __shared__ __align__(16) unsigned char smem[];
  long long* const sF = reinterpret_cast<long long*>(smem);
  const int tables = kMode >= kPiecewise2 ? P.n_pw : 1;
  const uint32_t lane = threadIdx.x & 31u;
  ScreenQueues& q = reinterpret_cast<ScreenQueues*>(smem + tables * kTableBytes)[threadIdx.x >> 5];
  const WarpTiles T = warp_tiles();
  release_next();
  build_tables(P.col, tables, sF);
  wait_previous();
  const CloudSample sample = sample_cloud<kMode>(P, pts, n, T, lane);
  if (kLeave == kOrder && sample.random && T.g == 0u && lane == 0u) side->x = 1u;
  uint32_t cn = 0, on = 0;
  auto tier2 = [&](uint32_t place) { raster_deferred(P, sF, point_at(pts, T, place), keys); };
  auto commit = [&](bool need, const uint4& p, uint32_t pixel, uint32_t place) {
    FixedCode f;
    const bool exact = exact_code<kMode>(P, sF, p, &f);
    if (need & exact) atomicMin(keys + pixel, key_from_fixed(f.a0, f.a1, f.a2, p.w));
    if (__any_sync(0xFFFFFFFFu, need & !exact)) push_open(need & !exact, place, q.open, on, lane);
  };
  auto candidate = [&](uint32_t i, bool valid) { commit(valid, q.p[i], q.pixel[i], q.place[i]); };
  auto record = [&](bool b0, bool b1, uint32_t place) {
    const unsigned m0 = __ballot_sync(0xFFFFFFFFu, b0), m1 = __ballot_sync(0xFFFFFFFFu, b1);
    if (lane == 0) side[T.g + (uint64_t)(place >> 6) * T.G] = make_uint2(m0, m1);
  };
  auto tile = [&](const uint4& p0, const uint4& p1, uint32_t place, bool words) {
        const ScreenTwo two = screen_two<kMode>(P, S, p0, p1, keys);
        const ScreenPoint &s0 = two.a, &s1 = two.b;
        if (words)
          record(s0.open | (__fsub_rn(__fmaf_rn(s0.k, S.hi_a, S.hi_b), s0.w) > -s0.m),
                 s1.open | (__fsub_rn(__fmaf_rn(s1.k, S.hi_a, S.hi_b), s1.w) > -s1.m), place);
        if (__any_sync(0xFFFFFFFFu, s0.open | s1.open)) {
          push_open(s0.open, place, q.open, on, lane);
          push_open(s1.open, place + 32u, q.open, on, lane);
        }
        const bool n0 = __fsub_rn(s0.w, __fmaf_rn(s0.k, s0.a, s0.b)) < s0.m;
        const bool n1 = __fsub_rn(s1.w, __fmaf_rn(s1.k, s1.a, s1.b)) < s1.m;
        const int need = __popc(__ballot_sync(0xFFFFFFFFu, n0)) + __popc(__ballot_sync(0xFFFFFFFFu, n1));
        if (need >= kDirect) {
          commit(n0, p0, s0.pixel, place);
          commit(n1, p1, s1.pixel, place + 32u);
        } else if (need) {
          push_candidate(n0, p0, s0.pixel, place, q, cn, lane);
          push_candidate(n1, p1, s1.pixel, place + 32u, q, cn, lane);
        }
        if ((on | cn) >= 32u) drain_batches(q, on, cn, lane, tier2, candidate);
      };
  auto rest = [&](uint32_t place, bool v0, bool v1) {
    if (kLeave == kWords && sample.random) record(v0, v1, place);
    push_open(v0, place, q.open, on, lane);
    push_open(v1, place + 32u, q.open, on, lane);
    drain_batches(q, on, cn, lane, tier2, candidate);
  };
  auto plain = [&](const uint4& p0, const uint4& p1, uint32_t place) { tile(p0, p1, place, false); };
  if (kLeave == kWords && sample.random)
    screen_tiles<false>(
        pts, n, T, lane, [&](const uint4& p0, const uint4& p1, uint32_t place) { tile(p0, p1, place, true); }, rest);
  else if (sample.far_out)
    screen_tiles<false>(
        pts, n, T, lane,
        [&](const uint4& p0, const uint4& p1, uint32_t place) {
          if (!__all_sync(0xFFFFFFFFu, point_outside_depth(P, p0) & point_outside_depth(P, p1))) plain(p0, p1, place);
        },
        rest);
  else
    screen_tiles<false>(pts, n, T, lane, plain, rest);
  __syncwarp();
  if (cn) candidate(lane < cn ? lane : 0u, lane < cn);
  __syncwarp();
  for (uint32_t k = lane; k < on; k += 32u) tier2(q.open[k]);
}

// ------------------------------------------------------------------------------------------- HQ additions
//
// The two 64-bit additions of a fragment go to adjacent words of one 16-byte slot. Issued by one lane they are two
// requests; issued by two adjacent lanes in one instruction they are one (random slots of a 1920x1080 frame: 105 G
// fragments/s against 211 G, the rate of a single addition). So accepted fragments are gathered in a per-warp ring
// and added 64 at a time: lane pair g takes entries 4g .. 4g + 3 in order, lane 0 of the pair their {R, G} words and
// lane 1 their {B, count} words, and neighbours that fall on one pixel (runs, in scan order) are summed first.
constexpr uint32_t kAddRing = 128;

struct AddQueue {
  uint2* ring;          // kAddRing entries {pixel, rgba}
  uint32_t head, tail;  // head: a multiple of 64
};

// Adds the 64 ring entries from `head` on. kGuard: entries with pixel 0xFFFFFFFF are absent.
template <bool kGuard>
__device__ __forceinline__ void add_drain(const AddQueue& q, unsigned long long* accum, uint32_t lane) {
  const uint4* e = reinterpret_cast<const uint4*>(q.ring + (q.head & (kAddRing - 1u))) + (lane & ~1u);
  const uint4 e0 = e[0], e1 = e[1];  // entries 4g .. 4g + 3: {pixel, rgba, pixel, rgba}
  // the lane's word of each entry as two 16-bit halves: {R, G}, or {B, 1}; four of them cannot carry
  const uint32_t sel = lane & 1u ? 0x5452u : 0x5150u;
  unsigned long long* const acc = accum + (lane & 1u);
  const bool same1 = e0.z == e0.x, same2 = e1.x == e0.z, same3 = e1.z == e1.x;  // as the entry before
  const uint32_t s3 = __byte_perm(e1.w, 1u, sel), s2 = __byte_perm(e1.y, 1u, sel) + (same3 ? s3 : 0u),
                 s1 = __byte_perm(e0.w, 1u, sel) + (same2 ? s2 : 0u), s0 = __byte_perm(e0.y, 1u, sel) + (same1 ? s1 : 0u);
  auto put = [&](bool first, uint32_t pix, uint32_t sum) {  // the first entry of each run adds the run's sum
    if (first && (!kGuard || pix != 0xFFFFFFFFu))
      atomicAdd(acc + 2 * (uint64_t)pix, (unsigned long long)(sum & 0xFFFFu) | ((unsigned long long)(sum >> 16) << 32));
  };
  put(true, e0.x, s0);
  put(!same1, e0.z, s1);
  put(!same2, e1.x, s2);
  put(!same3, e1.z, s3);
}

// Queues the accepting lanes' fragments. At most two pushes between drains (63 + 64 entries fit the ring).
__device__ __forceinline__ void add_push(bool accept, uint32_t pix, uint32_t rgba, AddQueue& q, uint32_t lane) {
  const unsigned m = __ballot_sync(0xFFFFFFFFu, accept);
  if (accept) q.ring[(q.tail + __popc(m & ((1u << lane) - 1u))) & (kAddRing - 1u)] = make_uint2(pix, rgba);
  q.tail += __popc(m);
}

// Adds 64 queued fragments when there are that many. All lanes must call it.
__device__ __forceinline__ void add_drain_full(AddQueue& q, unsigned long long* accum, uint32_t lane) {
  __syncwarp();
  if (q.tail - q.head >= 64u) {
    add_drain<false>(q, accum, lane);
    q.head += 64u;
    __syncwarp();
  }
}

// Adds what is left (fewer than 64 entries).
__device__ __forceinline__ void add_finish(AddQueue& q, unsigned long long* accum, uint32_t lane) {
  const uint32_t cnt = q.tail - q.head;
  for (uint32_t i = lane; i < 64u; i += 32u)
    if (i >= cnt) q.ring[(q.head + i) & (kAddRing - 1u)] = make_uint2(0xFFFFFFFFu, 0u);
  __syncwarp();
  add_drain<true>(q, accum, lane);
}

// Pass 2 (Section 2.2), exact transform, LINEAR or METRIC depth, for bands whose u64 test does not wrap
// (band_bounds_exact): accepted means qmin <= q <= qmin + floor(eps (qmin + Nq)). Same shape and bounds as pass 1. On
// one GB300, against k_hq_cert: 100M points in scan order 0.680 to 0.44 ms, 37M shuffled 0.290 to 0.23, with the paired
// additions (see AddQueue) and the screen.
// kFrom: every tile; the tiles of the chunks whose bit is set in `mask` (k_cull; a view of a batched frame); or the points
// whose bit is set in the words that pass 1 wrote (`mask`, two words a tile; see k_raster_screen).
enum HqSource : int { kAllTiles = 0, kChunkMask = 1, kBandWords = 2 };

template <int kMode, int kFrom>
__global__ void __launch_bounds__(kScreenThreads, 1) k_hq_screen(
    const uint4* __restrict__ pts, uint64_t n, const __grid_constant__ CertParams P, const __grid_constant__ Screen S,
    const unsigned long long* __restrict__ keys, unsigned long long* __restrict__ accum, uint32_t eps_num,
    uint32_t eps_den, const uint32_t* __restrict__ mask) {
  extern __shared__ __align__(16) unsigned char smem[];
  long long* const sF = reinterpret_cast<long long*>(smem);
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  AddQueue aq{reinterpret_cast<uint2*>(smem + kTableBytes) + warp * kAddRing, 0u, 0u};
  PlaceQueues& q = reinterpret_cast<PlaceQueues*>(smem + kTableBytes + warps * kAddRing * sizeof(uint2))[warp];
  const WarpTiles T = warp_tiles();
  release_next();
  build_tables(P.col, 1, sF);
  wait_previous();
  uint32_t cn = 0, on = 0;
  auto tier2 = [&](uint32_t place) {
    hq_deferred(P, sF, point_at(pts, T, place), keys, accum, eps_num, eps_den);
  };
  auto candidate = [&](uint32_t i, bool valid) {
    const uint4 p = point_at(pts, T, q.place[i]);
    const uint32_t pixel = q.pixel[i];
    const unsigned long long qmin = stored_key(keys, pixel) >> 24;
    FixedCode f;
    const bool exact = exact_code<kMode>(P, sF, p, &f);
    add_push(valid & exact & in_band(code_from_fixed(f.a1, f.a2), qmin, P.v.nq, eps_num, eps_den), pixel, p.w, aq, lane);
    add_drain_full(aq, accum, lane);
    push_open(valid & !exact, q.place[i], q.open, on, lane);
  };
  // two points of a lane and their places
  auto two_points = [&](const uint4& p0, const uint4& p1, uint32_t place0, uint32_t place1, bool v0, bool v1) {
    ScreenTwo two = screen_two<kMode>(P, S, p0, p1, keys);
    ScreenPoint &s0 = two.a, &s1 = two.b;
    if constexpr (kFrom == kBandWords) {  // the last batch may be partial
      s0.open &= v0;
      s1.open &= v1;
      if (!v0) s0.w = __int_as_float(0x7F800000);
      if (!v1) s1.w = __int_as_float(0x7F800000);
    }
    if (__any_sync(0xFFFFFFFFu, s0.open | s1.open)) {
      push_open(s0.open, place0, q.open, on, lane);
      push_open(s1.open, place1, q.open, on, lane);
    }
    auto inside = [&](const ScreenPoint& o) {  // >= m: in the band; <= -m: outside it
      return fminf(__fsub_rn(o.w, __fmaf_rn(o.k, S.lo_a, S.lo_b)), __fsub_rn(__fmaf_rn(o.k, S.hi_a, S.hi_b), o.w));
    };
    const float d0 = inside(s0), d1 = inside(s1);
    add_push(d0 >= s0.m, s0.pixel, p0.w, aq, lane);
    add_push(d1 >= s1.m, s1.pixel, p1.w, aq, lane);
    add_drain_full(aq, accum, lane);
    const bool n0 = fabsf(d0) < s0.m, n1 = fabsf(d1) < s1.m;
    if (__any_sync(0xFFFFFFFFu, n0 | n1)) {
      push_candidate(n0, s0.pixel, place0, q, cn, lane);
      push_candidate(n1, s1.pixel, place1, q, cn, lane);
    }
    if ((on | cn) >= 32u) drain_batches(q, on, cn, lane, tier2, candidate);
  };
  const CloudSample sample = kFrom == kBandWords ? sample_cloud<kMode>(P, pts, n, T, lane) : CloudSample{false, false};
  if (kFrom == kBandWords && sample.random)
    band_points(pts, n, T, lane, reinterpret_cast<const uint2*>(mask),
                reinterpret_cast<uint32_t*>(smem + kTableBytes + warps * (kAddRing * sizeof(uint2) + sizeof(PlaceQueues))) +
                    warp * kBandQueue,
                two_points);
  else
    screen_tiles<kFrom == kChunkMask>(
        pts, n, T, lane,
        [&](const uint4& p0, const uint4& p1, uint32_t place) { two_points(p0, p1, place, place + 32u, true, true); },
        [&](uint32_t place, bool v0, bool v1) {
          push_open(v0, place, q.open, on, lane);
          push_open(v1, place + 32u, q.open, on, lane);
          drain_batches(q, on, cn, lane, tier2, candidate);
        },
        mask);
  __syncwarp();
  if (cn) candidate(lane < cn ? lane : 0u, lane < cn);
  add_finish(aq, accum, lane);
  __syncwarp();
  for (uint32_t k = lane; k < on; k += 32u) tier2(q.open[k]);
}

// ---------------------------------------------------------------------------------------------- launch

// Launch shape of a screened pass over n points: one block an SM, with as many warps as it has tiles for, at least 4
// (they build the table) and at most 8 per requested block of 256 threads; shared memory for the table and each warp's
// queues.
struct ScreenLaunch {
  unsigned grid, threads;
  size_t smem;
};

constexpr size_t screen_smem(int warps, int tables, bool hq) {
  return tables * kTableBytes + (size_t)warps * (hq ? sizeof(PlaceQueues) + kAddRing * sizeof(uint2) + kBandQueue * sizeof(uint32_t) : sizeof(ScreenQueues));
}

inline ScreenLaunch screen_launch(uint64_t n, int sms, int per_sm, int tables, bool hq) {
  const uint64_t tiles = (n + kTile - 1) / kTile, want = (tiles + sms - 1) / sms;
  const int most = per_sm * 8 < kScreenThreads / 32 ? per_sm * 8 : kScreenThreads / 32;
  const int warps = want < 4 ? 4 : want < (uint64_t)most ? (int)want : most;
  const uint64_t need = (tiles + warps - 1) / warps;
  return ScreenLaunch{(unsigned)(need < (uint64_t)sms ? need : (uint64_t)sms), (unsigned)(32 * warps),
                      screen_smem(warps, tables, hq)};
}

template <int kMode, int kLeave = kNothing>
inline void raster_screen_launch(const uint4* pts, uint64_t n, const CertParams& P, const Screen& S,
                                 unsigned long long* keys, uint2* side, int sms, int per_sm, cudaStream_t s) {
  constexpr int most = kMode == kPiecewise ? kMaxRanges : kMode == kPiecewise2 ? 2 : 1;
  static std::atomic<uint64_t> opted{0};
  opt_in_shared(k_raster_screen<kMode, kLeave>, screen_smem(kScreenThreads / 32, most, false), opted);
  const ScreenLaunch L = screen_launch(n, sms, per_sm, table_blocks(P), false);
  launch_after(k_raster_screen<kMode, kLeave>, L.grid, L.threads, L.smem, s, pts, n, P, S, keys, side);
}

// leave, side: see k_raster_screen (other than kNothing: LINEAR or METRIC views, with the screen of pass 2's eps).
inline void launch_raster_screen(const uint4* pts, uint64_t n, const CertParams& P, const Screen& S,
                                 unsigned long long* keys, RasterLeave leave, void* side, int sms, int per_sm,
                                 cudaStream_t s) {
  uint2* const to = static_cast<uint2*>(side);
  switch (screen_mode(P)) {
    case kUnit256:
      return leave == kWords   ? raster_screen_launch<kUnit256, kWords>(pts, n, P, S, keys, to, sms, per_sm, s)
             : leave == kOrder ? raster_screen_launch<kUnit256, kOrder>(pts, n, P, S, keys, to, sms, per_sm, s)
                               : raster_screen_launch<kUnit256>(pts, n, P, S, keys, nullptr, sms, per_sm, s);
    case kUnit1:
      return leave == kWords   ? raster_screen_launch<kUnit1, kWords>(pts, n, P, S, keys, to, sms, per_sm, s)
             : leave == kOrder ? raster_screen_launch<kUnit1, kOrder>(pts, n, P, S, keys, to, sms, per_sm, s)
                               : raster_screen_launch<kUnit1>(pts, n, P, S, keys, nullptr, sms, per_sm, s);
    case kPiecewise2: return raster_screen_launch<kPiecewise2>(pts, n, P, S, keys, nullptr, sms, per_sm, s);
    case kPiecewise: return raster_screen_launch<kPiecewise>(pts, n, P, S, keys, nullptr, sms, per_sm, s);
  }
}

// One launch of pass 2: the kernel, its shape and its arguments (kept together so that a captured frame's nodes can be
// given a new view's).
struct HqScreenLaunch {
  const uint4* pts;
  uint64_t n;
  CertParams P;
  Screen S;
  const unsigned long long* keys;
  unsigned long long* accum;
  uint32_t eps_num, eps_den;
  const uint32_t* mask;
  const void* kernel;
  ScreenLaunch shape;
  void* args[9];
};

template <int kMode, int kFrom>
inline const void* hq_screen_kernel() {
  static std::atomic<uint64_t> opted{0};
  opt_in_shared(k_hq_screen<kMode, kFrom>, screen_smem(kScreenThreads / 32, 1, true), opted);
  return reinterpret_cast<const void*>(k_hq_screen<kMode, kFrom>);
}

inline void make_hq_screen(const uint4* pts, uint64_t n, const CertParams& P, const Screen& S, const unsigned long long* keys,
                           unsigned long long* accum, uint32_t eps_num, uint32_t eps_den, HqSource from,
                           const uint32_t* mask, int sms, int per_sm, HqScreenLaunch* o) {
  o->pts = pts;
  o->n = n;
  o->P = P;
  o->S = S;
  o->keys = keys;
  o->accum = accum;
  o->eps_num = eps_num;
  o->eps_den = eps_den;
  o->mask = mask;
  const bool unit1 = screen_mode(P) == kUnit1;
  o->kernel = from == kBandWords   ? (unit1 ? hq_screen_kernel<kUnit1, kBandWords>() : hq_screen_kernel<kUnit256, kBandWords>())
              : from == kChunkMask ? (unit1 ? hq_screen_kernel<kUnit1, kChunkMask>() : hq_screen_kernel<kUnit256, kChunkMask>())
                                   : (unit1 ? hq_screen_kernel<kUnit1, kAllTiles>() : hq_screen_kernel<kUnit256, kAllTiles>());
  o->shape = screen_launch(n, sms, per_sm, 1, true);
  void* args[9] = {&o->pts, &o->n, &o->P, &o->S, &o->keys, &o->accum, &o->eps_num, &o->eps_den, &o->mask};
  std::memcpy(o->args, args, sizeof(args));
}

inline void launch_hq_screen(HqScreenLaunch& l, cudaStream_t s) {
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = l.shape.grid;
  c.blockDim = l.shape.threads;
  c.dynamicSmemBytes = l.shape.smem;
  c.stream = s;
  c.attrs = &a;
  c.numAttrs = 1;
  cudaLaunchKernelExC(&c, l.kernel, l.args);
}

// Pass 1 of prepared constants with default tuning: screened where the screen applies.
inline void launch_raster_default(const uint4* pts, uint64_t n, const CertParams& P, unsigned long long* keys,
                                  uint32_t* status, int sms, int per_sm, cudaStream_t s) {
  Screen S;
  if (make_screen(P, 0, 0, false, &S))
    launch_raster_screen(pts, n, P, S, keys, kNothing, nullptr, sms, per_sm, s);
  else
    raster_launch<false, false>(pts, n, P, keys, nullptr, status, sms, per_sm, s);
}

// Pass 2 of prepared constants with default tuning, by the stored keys. own_pass1: every point's pass 1 has written
// the keys (q >= qmin holds, so the lower band edge needs no test).
inline void launch_hq_default(const uint4* pts, uint64_t n, const CertParams& P, const unsigned long long* keys,
                              unsigned long long* accum, uint32_t eps_num, uint32_t eps_den, uint32_t* status, int sms,
                              int per_sm, bool own_pass1, cudaStream_t s) {
  Screen S;
  if (band_bounds_exact(P.v.nq, eps_num, eps_den) && make_screen(P, eps_num, eps_den, !own_pass1, &S))
  {
    HqScreenLaunch l;
    make_hq_screen(pts, n, P, S, keys, accum, eps_num, eps_den, kAllTiles, nullptr, sms, per_sm, &l);
    launch_hq_screen(l, s);
  }
  else
    hq_launch<false, false>(pts, n, P, keys, accum, eps_num, eps_den, status, sms, per_sm, s);
}

// Both passes of a frame over the same n points: whether pass 1 may leave pass 2 its words (enough tiles for the sample
// that decides it), and the screen of both (eps at most 1: pass 1's margin holds pass 2's edge width).
inline bool frame_screen(const CertParams& P, uint64_t n, int sms, int per_sm, uint32_t eps_num, uint32_t eps_den, Screen* S) {
  const ScreenLaunch L = screen_launch(n, sms, per_sm, 1, false);
  return n / kTile / ((uint64_t)L.grid * (L.threads / 32)) >= kSampleTiles && P.n_pw == 0 && eps_num <= eps_den && band_bounds_exact(P.v.nq, eps_num, eps_den) &&
         make_screen(P, eps_num, eps_den, false, S);
}

// Pass 1 for a view with n >= 1 points. status: the framebuffer's status word (timeout bit).
// band (mask non-null): also write the band mask for pass 2 (used only with the exact transform on LINEAR or
// METRIC views; the caller checks that before relying on it).
inline bool launch_raster_certified(const uint4* pts, uint64_t n, const DevView& v, bool approximate,
                                    unsigned long long* keys, uint32_t* status, int sms, cudaStream_t s,
                                    unsigned long long* stats = nullptr, const Tuning& t = Tuning(),
                                    BandMask band = BandMask{nullptr, 1u, 0u, 0ull}) {
  const CertParams* Pp = nullptr;
  const unsigned grid = cert_grid(n, sms, t.blocks_per_sm);
  if (!cached_cert(v, approximate, &Pp)) {
    k_raster_fp64<<<grid, 256, 0, s>>>(pts, n, v, keys);
    return true;
  }
  const int b = t.blocks_per_sm, g = t.staging;
  if (!approximate && !stats && !t.merge && !g && !band.mask) {
    launch_raster_default(pts, n, *Pp, keys, status, sms, b, s);
    return true;
  }
  if (approximate)
    t.merge ? raster_launch<true, true>(pts, n, *Pp, keys, stats, status, sms, b, s, g)
            : raster_launch<true, false>(pts, n, *Pp, keys, stats, status, sms, b, s, g);
  else
    t.merge ? raster_launch<false, true>(pts, n, *Pp, keys, stats, status, sms, b, s, g, band)
            : raster_launch<false, false>(pts, n, *Pp, keys, stats, status, sms, b, s, g, band);
  return true;
}

// Pass 2 for a view with n >= 1 points. status: the framebuffer's status word (timeout bit). band_mask: see
// hq_launch. bounds_buf: room for the accept bounds of every pixel (npx entries), or null; with the exact
// transform and band_bounds_exact they are computed (k_band_bounds) and pass 2 tests against them. Returns the
// number of kernels launched.
inline int launch_hq_certified(const uint4* pts, uint64_t n, const DevView& v, bool approximate,
                               const unsigned long long* keys, unsigned long long* accum, uint32_t eps_num,
                               uint32_t eps_den, uint32_t* status, int sms, cudaStream_t s,
                               const Tuning& t = Tuning(), const uint32_t* band_mask = nullptr, ulonglong2* bounds_buf = nullptr, bool own_pass1 = false) {
  const CertParams* Pp = nullptr;
  const unsigned grid = cert_grid(n, sms, t.blocks_per_sm);
  if (!cached_cert(v, approximate, &Pp) || Pp->n_pw > 0) {  // (HQ takes LINEAR or METRIC views only)
    k_hq_fp64<<<grid, 256, 0, s>>>(pts, n, v, keys, accum, eps_num, eps_den);
    return 1;
  }
  const int b = t.blocks_per_sm, g = t.staging;
  if (approximate) {
    t.merge ? hq_launch<true, true>(pts, n, *Pp, keys, accum, eps_num, eps_den, status, sms, b, s, g)
            : hq_launch<true, false>(pts, n, *Pp, keys, accum, eps_num, eps_den, status, sms, b, s, g);
    return 1;
  }
  if (!t.merge && !g && !band_mask && !bounds_buf) {
    launch_hq_default(pts, n, *Pp, keys, accum, eps_num, eps_den, status, sms, b, own_pass1, s);
    return 1;
  }
  const ulonglong2* bounds = nullptr;
  if (bounds_buf && band_bounds_exact(v.nq, eps_num, eps_den)) {
    const uint64_t npx = (uint64_t)v.width * v.height;
    const unsigned bgrid = (unsigned)((npx + 255) / 256 < (uint64_t)sms * 8 ? (npx + 255) / 256 : (uint64_t)sms * 8);
    k_band_bounds<<<bgrid, 256, 0, s>>>(keys, npx, v.nq, eps_num, div_magic(eps_den), bounds_buf);
    bounds = bounds_buf;
  }
  t.merge ? hq_launch<false, true>(pts, n, *Pp, keys, accum, eps_num, eps_den, status, sms, b, s, g,
                                   band_mask, bounds)
          : hq_launch<false, false>(pts, n, *Pp, keys, accum, eps_num, eps_den, status, sms, b, s, g,
                                    band_mask, bounds);
  return bounds ? 2 : 1;
}

}  // namespace pcr
