// lr_raster.cuh -- Stage 3 of the pipeline, bin rasterisation (Sec. 2, "Stage 3: bin
// rasterization"), with the exact fallback the paper sketches (Sec. 2, "Sample blending").
//
// Work decomposition. Every 32x32 bin is cut into 32 half-blocks of 8x4 pixels (the
// paper's tri-half-block granularity). A half-block is one work item and one warp: lane
// = pixel. Persistent warps take items from a device queue ordered by bin size (largest
// bins first), so high-density bins are spread over many warps instead of one CTA.
//
// Per half-block (all from the bin's reference list, already sorted front to back by
// k_bin_sort -- stage 1 of the two-stage sort, Sec. 2, Stage 3, Phase 2):
//   1. candidates: the half-block's row of the bin's transposed bitmap (written by
//      k_bin_sort: bit j set iff sorted reference j overlaps the half-block) is read with
//      one coalesced load per 1024 references, and its set bits are handed out 32 at a
//      time in sorted order, one candidate quad per lane;
//   2. coverage, lane-parallel: both triangles' 32-pixel masks (top-left rule) from the
//      quad's five edges (quad_masks_small / quad_masks_any). Triangles that cover a pixel
//      go to a small ring in shared memory; those that do not (a third of the layer frame's)
//      cost nothing further;
//   3. batches of 32 covering triangles from the ring, one per lane: the depth key's edge
//      values, steps and plane, and the colours, into shared memory. 32-bit edge values
//      where k_setup proved them exact, else 64-bit;
//   4. a 32x32 bit transpose across the warp turns "triangle -> pixels" into "pixel ->
//      triangles", one bit per covering triangle in each lane;
//   5. fragments, per lane in candidate order: the exact depth key of the fragment
//      (interpolated 1/w, identical bit for bit to the oracle's formula) is pushed into a
//      K-slot register sorter (stage 2, the paper's depth filter, Sec. 2, Stage 3,
//      Phase 3, "Sample blending"). When full,
//      the nearest element is evicted and blended front to back. If a fragment arrives
//      that is nearer than the last evicted one, the stream was not in order for this
//      pixel: the pixel is flagged (the paper's misorder detection, same passage) and
//      registered for k_overflow. While every triangle so far has a flat colour and one
//      depth (camera-facing quads), the sorted stream is the exact order of every pixel, and
//      fragments are blended as they come, without key, sorter or test.
// Sort keys are (float bits of key) << 32 | (2 * quad + triangle): distinct per pixel, so
// the per-pixel order is total and the result is unique.
//
// What bounds it and what it took (1920x1080, kernel times): at K = 1 on 1M wavy quads with vertex
// colours the shared-memory and gather wavefronts (81% of the L1 data pipe; a 16-byte load per lane
// costs four) and 70% of issue slots together; against setting up both triangles of each candidate
// with a binary search per edge and row, 349M -> 266M warp instructions and 375 -> 307 us. With
// normals 602 -> 402 us, six mixed views at K = 3 2040 -> 692, 100k
// scattered parallelograms with a few screen-filling ones 117 -> 58. Bins whose list is already in
// every pixel's order are left to k_raster_ordered.
#pragma once

#include "lr_common.cuh"

#include <type_traits>

namespace lr {

// k_raster's batches: the edge values are kept in 64 bits
constexpr uint32_t kTriWide = 256u;
constexpr unsigned long long kSent = ~0ull;
constexpr int kRasterThreads = 256;
// Resident CTAs per SM requested from the compiler: 3 caps registers at 80 per thread (24 warps
// per SM), 4 at 64; neither spills in the forward kernels up to K = 3. Four where they fit: against
// three the layer frame took 307 instead of 315 us, 200,000 parallelograms at K = 1 143 instead of 148,
// flat layers at K = 3 154 instead of 168, with the alpha threshold at K = 1, 2, 3 135, 156, 172 instead of
// 145, 174, 184, layers with it 164 instead of 172. With three the batch of mixed views at K = 3 took 833
// instead of 868, lit layers 406 instead of 422; the shared memory of the parked colours, of lit
// colours and of the backward holds three.
__host__ __device__ constexpr int raster_min_blocks(int k, bool vtx, bool bwd, bool lit) {
  return lit || bwd || k > 3 || (vtx && k > 1) ? 3 : 4;
}
constexpr int kRasterWarps = kRasterThreads / 32;
constexpr int kOvfThreads = 128;
// alpha threshold (LR_FLAG_ALPHA_THRESHOLD, the paper's opt-in early stop, Sec. 2 "Sample
// blending"): a pixel blends a fragment only while its transmittance is above this, i.e.
// until its accumulated alpha reaches 1 - 1/128
constexpr float kAlphaTMin = 1.0f / 128.0f;
// The fp32 depth key of any fragment of a quad is at most its largest vertex 1/w times
// this: the key is a convex combination of three vertex values evaluated with a handful
// of roundings of relative size 2^-24 each, far inside the 2^-16 margin.
constexpr float kKeyBoundScale = 1.0f + 1.0f / 65536.0f;

// Backward of the front-to-back composite for one pixel (flat per-quad RGBA). With
// C = sum_i T_i a_i c_i, T_i = prod_{k<i} (1 - a_k), A = 1 - prod (1 - a_k):
//   dC/dc_i = T_i a_i,   dC/da_i = T_i c_i - S_i / (1 - a_i),   dA/da_i = T_final / (1 - a_i)
// where S_i = C_final - (C accumulated through fragment i) is the colour contributed by the
// fragments behind i. C_final, T_final come from the forward image; the running sums are
// recomputed in the forward's order.
struct GradPixel {
  float gr, gg, gb, ga;      // dL/d(R, G, B, A) of the pixel
  float fr, fg, fb, fT;      // forward colour and transmittance
  float* grad;               // f32[Q][4] of the view
  __device__ __forceinline__ void load(const float* grad_out, const float* fwd, long long pidx) {
    const float4 g = reinterpret_cast<const float4*>(grad_out)[pidx];
    const float4 f = reinterpret_cast<const float4*>(fwd)[pidx];
    gr = g.x; gg = g.y; gb = g.z; ga = g.w;
    fr = f.x; fg = f.y; fb = f.z; fT = 1.0f - f.w;
  }
};

// Columns lx in [0, 8) of one half-block row where an edge is non-negative, as an 8-bit
// mask, given the edge value r at lx = 0 and its step sx per column. The edge is linear in
// lx, so the failing columns form a prefix (sx >= 0) or a suffix (sx < 0); mirroring the
// row turns the suffix into a prefix, whose length is found by a 4-step binary search on
// exact 32-bit edge values (every value evaluated is a pixel centre of the half-block).
__device__ __forceinline__ uint32_t row_cover(int r, int sx) {
  const bool neg = sx < 0;
  const uint32_t g0 = neg ? (uint32_t)r + 7u * (uint32_t)sx : (uint32_t)r;
  const uint32_t sa = neg ? 0u - (uint32_t)sx : (uint32_t)sx;
  int cnt = ((int)(g0 + 3u * sa) < 0) ? 4 : 0;
  cnt += ((int)(g0 + (uint32_t)(cnt + 1) * sa) < 0) ? 2 : 0;
  cnt += ((int)(g0 + (uint32_t)cnt * sa) < 0) ? 1 : 0;
  cnt += (cnt == 7 && (int)(g0 + 7u * sa) < 0) ? 1 : 0;
  return neg ? (0xFFu >> cnt) : ((0xFFu << cnt) & 0xFFu);
}

// ATH: the alpha-threshold variant. Once the transmittance drops to kAlphaTMin nothing
// more is blended and `last` stays at the key of the fragment that got it there, so the
// misorder test below only flags fragments that belong in front of that one.
// PARK: the held fragments' colours stay where they were put, in shared memory, and only their places
// move with the keys, where moving a colour through a slot takes eight selects (K = 3: 250k layers
// at 1024x768 148 us with colours in the sorter's registers, 139 so; six mixed views 737 and 692).
template <int K, bool VTX, bool ATH = false, bool PARK = false>
struct PixelState {
  // K = 1 with flat colours gathered at blend time: the colour of the fragment held in the
  // slot is loaded when it enters, so the gather overlaps the next fragment's work
  static constexpr bool kPrefetch = !VTX && K == 1;
  unsigned long long s[K];
  float4 c[(VTX || kPrefetch) && !PARK ? K : 1];
  uint32_t sl[PARK ? K : 1];         // place of slot i's colour
  float4* park;                      // the lane's places, 32 apart
  unsigned long long last;
  float r, g, b, T;
  bool flagged;

  // K = 1, colours carried: the empty slot holds a fully transparent colour, so
  // blending it changes nothing (T and the colour stay, last is still kSent) and the in-order
  // insert needs no test for it (layer frame rasteriser 0.409 -> 0.394 ms; the same for the
  // flat colours gathered at blend time made the particle frame's 14% slower)
  static constexpr bool kNullSlot = VTX && K == 1;

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < K; ++i) s[i] = kSent;
#pragma unroll
    for (int i = 0; i < (PARK ? K : 0); ++i) sl[i] = (uint32_t)i;
    if (kNullSlot) c[0] = make_float4(0.f, 0.f, 0.f, 0.f);
    last = kSent;
    r = g = b = 0.f;
    T = 1.f;
    flagged = false;
  }

  // the pixel still blends (always, without the threshold)
  __device__ __forceinline__ bool live() const { return !ATH || T > kAlphaTMin; }

  __device__ __forceinline__ void blend(unsigned long long key, float4 col, const ViewDev& V) {
    const uint32_t j = (uint32_t)key >> 1;
    if (!VTX && !kPrefetch) col = __ldg(reinterpret_cast<const float4*>(V.col) + j);
    const float w = T * col.w;
    r += w * col.x;
    g += w * col.y;
    b += w * col.z;
    // T (1 - a) as one fused T - T a (a rounding, not the product's two, away from it: well
    // inside the colour tolerance); the threshold variant, whose T decides which fragments
    // blend, keeps the product
    if (ATH) T *= 1.0f - col.w;
    else T = __fmaf_rn(-T, col.w, T);
  }

  // blend of a fragment known to be next in order, without the sorter
  __device__ __forceinline__ void blend_direct(float4 col) {
    const float w = T * col.w;
    r += w * col.x;
    g += w * col.y;
    b += w * col.z;
    if (ATH) T *= 1.0f - col.w;
    else T = __fmaf_rn(-T, col.w, T);
  }

  __device__ __forceinline__ void insert(unsigned long long x, float4 xc, const ViewDev& V) {
    // nearer than a fragment already blended: order not guaranteed. With carried colours this
    // only records it (the pixel's composite is discarded, so inserting the
    // fragment anyway is harmless; measured faster than the branch there, slower for the
    // colours gathered at blend time)
    if (VTX) {
      flagged |= x > last;
    } else if (x > last) {
      flagged = true;
      return;
    }
    if (VTX && K == 1 && kNullSlot && !ATH) {
      // one slot, the empty one transparent: blend the nearer of the held and the arriving
      // fragment, keep the other (selects: whichever way a lane's fragments arrive, the warp
      // runs one path; layer frame rasteriser 0.3770 -> 0.3750 ms against the branch below)
      const bool nearer = x > s[0];
      const unsigned long long bk = nearer ? x : s[0];
      const float4 bc = nearer ? xc : c[0];
      blend(bk, bc, V);
      last = bk;
      s[0] = nearer ? s[0] : x;
      c[0] = nearer ? c[0] : xc;
      return;
    }
    if (VTX && K == 1) {       // one slot (threshold): a branch
      if (x > s[0]) {          // nearer than the held fragment: blend it at once
        if (live()) {
          blend(x, xc, V);
          last = x;
        }
      } else {
        if (live()) {   // (the empty slot is transparent)
          blend(s[0], c[0], V);
          last = s[0];
        }
        s[0] = x;
        c[0] = xc;
      }
      return;
    }
    if (kPrefetch) {
      const float4* cp = reinterpret_cast<const float4*>(V.col) + ((uint32_t)x >> 1);
      if (x > s[0]) {          // nearer than the held fragment: blend it at once
        if (live()) {
          blend(x, __ldg(cp), V);
          last = x;
        }
      } else {
        if (s[0] != kSent && live()) {
          blend(s[0], c[0], V);
          last = s[0];
        }
        s[0] = x;
        c[0] = __ldg(cp);
      }
      return;
    }
    const bool xfirst = x > s[0];
    const unsigned long long ev = xfirst ? x : s[0];
    const unsigned long long y = xfirst ? s[0] : x;
    float4 evc = xc, yc = xc;
    uint32_t ys = 0;
    if (PARK) {
      // the fragment that is kept takes (or already has) the evicted one's place
      ys = sl[0];
      if (!xfirst) {
        evc = park[32 * ys];
        park[32 * ys] = xc;
      }
    } else if (VTX) {
      evc = xfirst ? xc : c[0];
      yc = xfirst ? c[0] : xc;
    }
    // new slots = {s[1..K-1], y} in decreasing order
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const bool take_next = (i + 1 < K) && (s[i + 1 < K ? i + 1 : i] > y);
      const bool take_y = (i == 0) || (s[i] > y);
      const unsigned long long nxt = s[i + 1 < K ? i + 1 : i];
      s[i] = take_next ? nxt : (take_y ? y : s[i]);
      if (PARK) {
        const uint32_t ns = sl[i + 1 < K ? i + 1 : i];
        sl[i] = take_next ? ns : (take_y ? ys : sl[i]);
      } else if (VTX) {
        const float4 nc = c[i + 1 < K ? i + 1 : i];
        c[i] = take_next ? nc : (take_y ? yc : c[i]);
      }
    }
    if (ev != kSent && live()) {
      blend(ev, evc, V);
      last = ev;
    }
  }

  __device__ __forceinline__ void flush(const ViewDev& V) {
#pragma unroll
    for (int i = 0; i < K; ++i)
      if (s[i] != kSent && live()) {
        if (PARK) blend(s[i], park[32 * sl[i]], V);
        else blend(s[i], VTX || kPrefetch ? c[i] : make_float4(0.f, 0.f, 0.f, 0.f), V);
      }
  }
};

// Backward: one pixel. The sorter's slots hold keys and the fragment's slot in the current batch
// (kOldSlot: it came with an earlier one). What a blended fragment contributes to its quad's
// gradient is, with the pixel's g = dL/d(R, G, B), two numbers times quantities of the quad or of
// the pixel alone: the transmittance T in front of it (dL/dc = a T g) and the rest
// S = g . (C_final - C through it) - ga T_final (dL/da = T g . c - S / (1 - a)). The warp's pixels
// record them per batch in shared memory, rank of the fragment in its pixel by pixel, and
// batch_gradients sums them with one lane per triangle and one vector atomic each. Only fragments
// blended after their batch (the K last of it) or beyond kGradRanks of a pixel are added one by
// one, each with a vector atomic. 25M fragments at 1024x1024, K = 1: 435 us when each blended
// fragment searched the warp for lanes with the same quad and issued four atomics per group, 291
// when only the late ones did, 258 so.
constexpr uint32_t kOldSlot = 32u;
constexpr int kGradRanks = 12;     // (eight fragments per pixel and batch are ordinary)
struct GradShared {
  float4 g[32];                    // per pixel: dL/d(R, G, B), its batch coverage (bits)
  float2 ts[kGradRanks][32];       // (T, S) by rank and pixel
};
template <int K>
struct GradState {
  unsigned long long s[K], last;
  uint32_t sl[K];
  float T, r, g, b;                // running transmittance and colour
  GradPixel gp;
  uint32_t cover, done;            // the pixel's batch mask and the slots recorded
  bool flagged;

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < K; ++i) { s[i] = kSent; sl[i] = kOldSlot; }
    last = kSent;
    T = 1.f;
    r = g = b = 0.f;
    cover = done = 0;
    flagged = false;
  }

  __device__ __forceinline__ void blend(unsigned long long key, uint32_t slot, const ViewDev& V, const float4* qc,
                                        GradShared& G) {
    const uint32_t j = (uint32_t)key >> 1;
    float4 c;
    if (slot < kOldSlot) c = qc[slot];
    else c = __ldg(reinterpret_cast<const float4*>(V.col) + j);
    const int lane = threadIdx.x & 31;
    const float w = T * c.w;
    r += w * c.x;
    g += w * c.y;
    b += w * c.z;
    const float S = gp.gr * (gp.fr - r) + gp.gg * (gp.fg - g) + gp.gb * (gp.fb - b) - gp.ga * gp.fT;
    const int rank = __popc((cover >> (slot & 31u)) >> 1);
    if (slot < kOldSlot && rank < kGradRanks) {
      G.ts[rank][lane] = make_float2(T, S);
      done |= 1u << slot;
    } else {
      const float om = 1.0f - c.w;
      const float da = T * (gp.gr * c.x + gp.gg * c.y + gp.gb * c.z) - (om > 1e-6f ? S * rcp_approx(om) : 0.f);
      atomicAdd(reinterpret_cast<float4*>(gp.grad) + j, make_float4(gp.gr * w, gp.gg * w, gp.gb * w, da));
    }
    T = __fmaf_rn(-T, c.w, T);   // as the forward, so that r, g, b are its own and S their difference
  }

  // without a gradient (gp.grad null) the order is tested, nothing is blended
  __device__ __forceinline__ void insert(unsigned long long x, uint32_t slot, const ViewDev& V, const float4* qc,
                                         GradShared& G) {
    // nearer than a fragment already blended: order not guaranteed, and the gradient is left to
    // the exact path
    if (x > last) {
      flagged = true;
      return;
    }
    const bool xfirst = x > s[0];
    const unsigned long long ev = xfirst ? x : s[0], y = xfirst ? s[0] : x;
    const uint32_t evs = xfirst ? slot : sl[0], ys = xfirst ? sl[0] : slot;
    // new slots = {s[1..K-1], y} in decreasing order
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const bool take_next = (i + 1 < K) && (s[i + 1 < K ? i + 1 : i] > y);
      const bool take_y = (i == 0) || (s[i] > y);
      const unsigned long long nxt = s[i + 1 < K ? i + 1 : i];
      const uint32_t nsl = sl[i + 1 < K ? i + 1 : i];
      sl[i] = take_next ? nsl : (take_y ? ys : sl[i]);
      s[i] = take_next ? nxt : (take_y ? y : s[i]);
    }
    if (ev != kSent) {
      if (gp.grad) blend(ev, evs, V, qc, G);
      last = ev;
    }
  }

  __device__ __forceinline__ void flush(const ViewDev& V, const float4* qc, GradShared& G) {
#pragma unroll
    for (int i = 0; i < K; ++i)
      if (s[i] != kSent) blend(s[i], sl[i], V, qc, G);
  }
};

// Adds what the warp's pixels recorded for the batch: lane = slot, the triangle of quad j.
__device__ __forceinline__ void batch_gradients(uint32_t done, uint32_t j, float* grad, const float4* qc,
                                                const GradShared& G) {
  const int lane = threadIdx.x & 31;
  uint32_t m = warp_transpose32(done, lane);   // (its shuffles precede the reads below)
  __syncwarp();
  if (!m) return;
  // (dL/da pixel by pixel: its two terms nearly cancel, so their sums would round worse)
  const float4 c = qc[lane];
  const float om = 1.0f - c.w, inv = rcp_approx(om);
  const bool thin = om > 1e-6f;   // (an opaque quad's S may be 0 times infinity)
  float r = 0.f, g = 0.f, b = 0.f, da = 0.f;
  while (m) {
    const int px = __ffs(m) - 1;
    m &= m - 1;
    const float4 p = G.g[px];
    const float2 ts = G.ts[__popc((__float_as_uint(p.w) >> lane) >> 1)][px];
    const float w = ts.x * c.w;
    r += w * p.x;
    g += w * p.y;
    b += w * p.z;
    const float front = ts.x * (p.x * c.x + p.y * c.y + p.z * c.z);
    da += thin ? front - ts.y * inv : front;
  }
  atomicAdd(reinterpret_cast<float4*>(grad) + j, make_float4(r, g, b, da));
}

__device__ __forceinline__ void write_pixel(const ViewDev& V, long long pidx, float r, float g, float b,
                                            float T) {
  const float a = 1.0f - T;
  reinterpret_cast<float4*>(V.out)[pidx] = make_float4(r, g, b, a);
  if (V.out8) {
    const uint32_t c0 = __float2uint_rn(__fmul_rn(__saturatef(r), 255.0f));
    const uint32_t c1 = __float2uint_rn(__fmul_rn(__saturatef(g), 255.0f));
    const uint32_t c2 = __float2uint_rn(__fmul_rn(__saturatef(b), 255.0f));
    const uint32_t c3 = __float2uint_rn(__fmul_rn(__saturatef(a), 255.0f));
    reinterpret_cast<uint32_t*>(V.out8)[pidx] = c0 | (c1 << 8) | (c2 << 16) | (c3 << 24);
  }
}

// ---- coverage masks ------------------------------------------------------------------------
//
// An edge u -> v at a block's first pixel centre (Px, Py). A pixel centre is covered iff
// E + bias >= 0, E = dx (Py - yu) - dy (Px - xu), bias = 0 for an owned edge, else -1. A step
// of one column adds -256 dy and one of a row 256 dx, so E + bias may be replaced by
// r = floor((E + bias) / 256) with steps -dy and dx. A row's covered columns are then
//   dy < 0: those from ceil(r / dy) on,  dy > 0: the first floor(r / dy) + 1,  dy = 0: r >= 0,
// and both counts are ceil(r / dy -+ eps) for any eps below the quotient's distance from the
// next integer, 1 / |dy| > 2^-15. The quotient is taken in fp32 as r (1 / (8 dy)), clamped to
// [0, 1] by the multiply-add's saturation: r and its row steps are exact (below 2^24), the
// approximate reciprocal and the rounding put the clamped value off by less than 2^-22, and
// eps = 2^-17 (2^-20 scaled) exceeds that, so the count is exact; the scaling back adds 2^23
// rounded up, which leaves ceil() in the low bits. Needs |E| < 2^30 and |dx|, |dy| < 2^15 on
// the block (kRecSmall). Five instructions per edge and row, against about 16 for the
// exact integer binary search (row_cover).
struct EdgeRows {
  float r, k, b, step;
  uint32_t flip;       // all ones: the count is of covered columns, else of uncovered ones
  __device__ __forceinline__ EdgeRows(int xu, int yu, int xv, int yv, int Px, int Py) {
    const int dx = xv - xu, dy = yv - yu;
    const bool owned = dy < 0 || (dy == 0 && dx > 0);
    const int e = (int)((uint32_t)dx * (uint32_t)(Py - yu) - (uint32_t)dy * (uint32_t)(Px - xu)) - (owned ? 0 : 1);
    r = __int2float_rn(e >> 8);
    step = __int2float_rn(dx);
    k = dy == 0 ? -1e20f : rcp_approx(__int2float_rn(8 * dy));
    b = dy > 0 ? 0x1p-20f : -0x1p-20f;
    flip = dy > 0 ? 0xFFFFFFFFu : 0u;
  }
  // the row's columns in the low 8 bits, before the flip (the bits above are arbitrary)
  __device__ __forceinline__ uint32_t row() const {
    const float t = __saturatef(__fmaf_rn(r, k, b));
    return __funnelshift_l(0u, 0xFFFFFFFFu, __float_as_uint(__fmaf_ru(t, 8.0f, 8388608.0f)));   // ~0 << (c mod 32)
  }
  __device__ __forceinline__ void next() { r = __fadd_rn(r, step); }
};

// Coverage masks of a quad's two triangles on a block of 8 x ROWS pixels: ROWS = 4, bit
// ly * 8 + lx of m[0]; ROWS = 8, row ly is byte ly / 2 of m[ly & 1] (even rows, odd rows).
// Under the top-left rule a pixel centre belongs to exactly one of an edge's two directions,
// so an edge traversed backwards (a triangle of negative area, or the diagonal's second
// triangle) takes the complement, and five edges serve both triangles.
template <int ROWS>
__device__ __forceinline__ void quad_masks_small(const int X[4], const int Y[4], uint32_t info, int Px, int Py,
                                                 uint32_t m0[ROWS / 4], uint32_t m1[ROWS / 4]) {
  const uint32_t s0 = (info & kInfoSwap0) ? 0xFFFFFFFFu : 0u;
  const uint32_t s1 = (info & (kInfoSwap0 << 1)) ? 0xFFFFFFFFu : 0u;
  EdgeRows d(X[2], Y[2], X[0], Y[0], Px, Py);   // the diagonal, T0's direction
  EdgeRows e1(X[0], Y[0], X[1], Y[1], Px, Py), e2(X[1], Y[1], X[2], Y[2], Px, Py);
  EdgeRows e3(X[2], Y[2], X[3], Y[3], Px, Py), e4(X[3], Y[3], X[0], Y[0], Px, Py);
  const uint32_t fd0 = d.flip ^ s0, fd1 = ~(d.flip ^ s1), f1 = e1.flip ^ s0, f2 = e2.flip ^ s0;
  const uint32_t f3 = e3.flip ^ s1, f4 = e4.flip ^ s1;
#pragma unroll
  for (int ly = 0; ly < ROWS; ++ly) {
    const uint32_t rd = d.row();
    const uint32_t a = (rd ^ fd0) & (e1.row() ^ f1) & (e2.row() ^ f2);
    const uint32_t c = (rd ^ fd1) & (e3.row() ^ f3) & (e4.row() ^ f4);
    if (ly + 1 < ROWS) { d.next(); e1.next(); e2.next(); e3.next(); e4.next(); }
    const int w = ROWS == 4 ? 0 : (ly & 1), at = ROWS == 4 ? ly : ly >> 1;
    const int sel = at == 1 ? 0x3240 : (at == 2 ? 0x3410 : 0x4210);   // byte at <- the row
    m0[w] = at == 0 ? a : __byte_perm(m0[w], a, sel);
    m1[w] = at == 0 ? c : __byte_perm(m1[w], c, sel);
  }
#pragma unroll
  for (int w = 0; w < ROWS / 4; ++w) {
    if (!(info & kInfoTri0)) m0[w] = 0u;
    if (!(info & kInfoTri1)) m1[w] = 0u;
  }
}

// The same for any quad, with 64-bit edge values. Most edges of a quad too large for the form
// above pass a block by: with all of the block's centres on one side, known from the extremes of
// E + bias (at corners), an edge covers all of it or none. Only the edges that cross the block are
// searched row by row, in 32-bit integers: then |E + bias| / 256 <= 7 |dx| + 7 |dy| < 2^27. A few
// screen-filling quads are candidates nearly everywhere: 200,000 parallelograms at 1920x1080, K = 3,
// 186 us with every row of every edge searched, 170 us so.
template <int ROWS>
__device__ __forceinline__ void quad_masks_any(const int X[4], const int Y[4], uint32_t info, int Px, int Py,
                                               uint32_t m0[ROWS / 4], uint32_t m1[ROWS / 4]) {
  const uint32_t s0 = (info & kInfoSwap0) ? 0xFFFFFFFFu : 0u;
  const uint32_t s1 = (info & (kInfoSwap0 << 1)) ? 0xFFFFFFFFu : 0u;
  uint32_t all0 = (info & kInfoTri0) ? 0xFFFFFFFFu : 0u, all1 = (info & kInfoTri1) ? 0xFFFFFFFFu : 0u, cross = 0;
  // edges v2 -> v0, v0 -> v1, v1 -> v2, v2 -> v3, v3 -> v0
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    constexpr int from[5] = {2, 0, 1, 2, 3}, to[5] = {0, 1, 2, 3, 0};
    const int dx = X[to[k]] - X[from[k]], dy = Y[to[k]] - Y[from[k]];
    const bool owned = dy < 0 || (dy == 0 && dx > 0);
    const long long e = (long long)dx * (Py - Y[from[k]]) - (long long)dy * (Px - X[from[k]]) - (owned ? 0 : 1);
    const bool in = e + 256LL * (min(0, -7 * dy) + min(0, (ROWS - 1) * dx)) >= 0;
    const bool out = e + 256LL * (max(0, -7 * dy) + max(0, (ROWS - 1) * dx)) < 0;
    if (!in && !out) {
      cross |= 1u << k;
    } else {
      const uint32_t f = in ? 0xFFFFFFFFu : 0u;
      if (k < 3) all0 &= f ^ s0;
      if (k == 0) all1 &= ~(f ^ s1);
      if (k > 2) all1 &= f ^ s1;
    }
  }
#pragma unroll
  for (int w = 0; w < ROWS / 4; ++w) { m0[w] = all0; m1[w] = all1; }
  if ((all0 | all1) == 0u) return;
#pragma unroll 1
  for (; cross; cross &= cross - 1u) {
    const int k = __ffs(cross) - 1;
    const int xu = k == 1 ? X[0] : (k == 2 ? X[1] : (k == 4 ? X[3] : X[2]));
    const int yu = k == 1 ? Y[0] : (k == 2 ? Y[1] : (k == 4 ? Y[3] : Y[2]));
    const int xv = k == 1 ? X[1] : (k == 2 ? X[2] : (k == 3 ? X[3] : X[0]));
    const int yv = k == 1 ? Y[1] : (k == 2 ? Y[2] : (k == 3 ? Y[3] : Y[0]));
    const int dx = xv - xu, dy = yv - yu;
    const bool owned = dy < 0 || (dy == 0 && dx > 0);
    const int r = (int)(((long long)dx * (Py - yu) - (long long)dy * (Px - xu) - (owned ? 0 : 1)) >> 8);
#pragma unroll
    for (int w = 0; w < ROWS / 4; ++w) {
      uint32_t f = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) f |= row_cover(r + (ROWS == 4 ? i : 2 * i + w) * dx, -dy) << (8 * i);
      if (k < 3) m0[w] &= f ^ s0;
      if (k == 0) m1[w] &= ~(f ^ s1);
      if (k > 2) m1[w] &= f ^ s1;
    }
  }
}

// Lists the set bits of the warp's words (bit 32 l + b: bit b of lane l's word) in order as
// 16-bit indices, and returns their number. One step per set bit of the fullest word, for the
// whole window of 1024 references, where finding the n-th set bit anew for every round of 32
// candidates took about 45 instructions a round.
__device__ __forceinline__ int list_bits(uint32_t word, int lane, uint16_t* list) {
  const int n = __popc(word);
  int incl = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  __syncwarp();                       // the window before has been read
  uint16_t* at = list + (incl - n);
  const int base = 32 * lane;
  while (word) {
    *at++ = (uint16_t)(base + __ffs(word) - 1);
    word &= word - 1;
  }
  __syncwarp();
  return total;
}

// Pixel-centre extent of a box-shaped quad (kRecBox) on a block of 8 x rows pixels at (ox, oy):
// columns [c0, c1) and rows [y0, y1). Under the top-left rule a centre is covered iff
// xmin <= x < xmax and ymin <= y < ymax.
struct BoxSpan {
  int c0, c1, y0, y1;
  __device__ __forceinline__ BoxSpan(const int X[4], const int Y[4], int ox, int oy, int rows) {
    // vertices 0 and 2 are opposite corners
    c0 = min(max(((min(X[0], X[2]) + 127) >> 8) - ox, 0), 8);
    c1 = min(max(((max(X[0], X[2]) + 127) >> 8) - ox, 0), 8);
    y0 = min(max(((min(Y[0], Y[2]) + 127) >> 8) - oy, 0), rows);
    y1 = min(max(((max(Y[0], Y[2]) + 127) >> 8) - oy, 0), rows);
  }
  __device__ __forceinline__ uint32_t columns() const { return (0xFFu << c0) & ~(0xFFFFFFFFu << c1); }
};

// Bytes [a, b) of a word set, 0 <= a, b <= 4.
__device__ __forceinline__ uint32_t byte_span(int a, int b) {
  // (funnel shifts by 32 clamp to zero)
  return __funnelshift_lc(0u, 0xFFFFFFFFu, 8 * a) & ~__funnelshift_lc(0u, 0xFFFFFFFFu, 8 * b);
}

// ---- k_raster's shared memory ----------------------------------------------------------------
// Per warp: the candidates of a 1024-reference window, a ring of covering triangles waiting for
// a batch, and the records of the batch the fragment loop reads, one 16-byte array per field so that a slot's fields lie at one address
// plus constants and eight neighbouring slots never share a bank.
// references per bitmap window (a word per lane; half of them in the backward and for lit views at
// K = 3, whose shared memory leaves room for three CTAs then)
__host__ __device__ constexpr int win_refs(bool half) { return half ? 512 : 1024; }
__host__ __device__ constexpr bool half_window(int k, bool bwd, bool lit) { return bwd || (lit && k == 3); }
constexpr int kPendCap = 128;      // at most 31 left over + 64 pushed per candidate round
constexpr uint32_t kPendConst = 0x80000000u;   // pending id: flat colour and constant depth
struct BatchGeo {
  int4 ea[32];                     // e1, e2 (edge values at the half-block origin; low words
                                   // of 64-bit ones), x steps sx1, sx2 (64-bit: -dy1, -dy2)
  int4 eb[32];                     // y steps sy1, sy2 (64-bit: dx1, dx2), flags, id
  float4 kq[32];                   // q0, q1 - q0, q2 - q0, 1 / area
  int2 hi[32];                     // high words of 64-bit e1, e2
};
__host__ __device__ constexpr int batch_cols(bool vtx, bool lit) { return vtx ? (lit ? 6 : 3) : 1; }
// sorters whose colours are parked in shared memory (which then still holds three CTAs). Not flat
// colours, which are gathered as they are blended (layers at K = 3: 121 us, parked 123).
__host__ __device__ constexpr bool parked(int k, bool vtx, bool bwd) { return vtx && !bwd && (k == 2 || k == 3); }
__host__ __device__ constexpr size_t batch_smem_warp(bool vtx, bool bwd, bool lit, int k) {
  return win_refs(half_window(k, bwd, lit)) * sizeof(uint16_t) + kPendCap * sizeof(uint2) + sizeof(BatchGeo) +
         (size_t)batch_cols(vtx, lit) * 32 * sizeof(float4) + (bwd ? sizeof(GradShared) : 0) +
         (parked(k, vtx, bwd) ? (size_t)k * 32 * sizeof(float4) : 0);
}
__host__ __device__ constexpr size_t raster_smem_bytes(bool vtx, bool bwd = false, bool lit = false, int k = 1) {
  return (size_t)kRasterWarps * batch_smem_warp(vtx, bwd, lit, k);
}

// q c - p with both operations rounded, as each corner's product has to be for the 8-bit values to be
// those of corners weighted before they are subtracted.
__device__ __forceinline__ float4 weighted_difference(float q, float4 c, float4 p) {
  return make_float4(__fsub_rn(__fmul_rn(q, c.x), p.x), __fsub_rn(__fmul_rn(q, c.y), p.y),
                     __fsub_rn(__fmul_rn(q, c.z), p.z), __fsub_rn(__fmul_rn(q, c.w), p.w));
}

// The record of covering triangle id (2 * quad + triangle of view V) into slot `lane` of the
// batch: the depth key's two edge values at the block's first pixel centre (Ox, Oy), their
// steps, its plane, and with colours carried (CARRY) the flat colour or the corner colours
// times 1/w as (c0, c1 - c0, c2 - c0) for the fragment's c0 + l1 (c1 - c0) + l2 (c2 - c0);
// lit: the same for the normals.
template <bool VTX, bool LIT, bool CARRY>
__device__ __forceinline__ void setup_batch(const Ws& ws, const ViewDev& V, bool flat_view, uint32_t id, int lane, int Ox,
                                            int Oy, BatchGeo& geo, float4* qc) {
  const int t = (int)(id & 1u);
  const uint32_t jl = id >> 1;
  const QuadRec R = load_rec(ws.rec, (uint32_t)(V.quad_base + jl));
  const bool sw = (R.info & (kInfoSwap0 << t)) != 0;
  // vertices a = v0 and, oriented to a positive area, b and c
  const int xa = R.X[0], ya = R.Y[0];
  const int x1 = t ? R.X[2] : R.X[1], y1 = t ? R.Y[2] : R.Y[1];
  const int x2 = t ? R.X[3] : R.X[2], y2 = t ? R.Y[3] : R.Y[2];
  const float q1 = t ? R.q[2] : R.q[1], q2 = t ? R.q[3] : R.q[2];
  const int xb = sw ? x2 : x1, yb = sw ? y2 : y1, xc = sw ? x1 : x2, yc = sw ? y1 : y2;
  const float q_a = R.q[0], q_b = sw ? q2 : q1, q_c = sw ? q1 : q2;
  geo.kq[lane] = make_float4(q_a, __fsub_rn(q_b, q_a), __fsub_rn(q_c, q_a), t ? R.inv[1] : R.inv[0]);
  // edges c -> a and a -> b, both through a
  const int dx1 = xa - xc, dy1 = ya - yc, dx2 = xb - xa, dy2 = yb - ya;
  const int ux = Ox - xa, uy = Oy - ya;
  if (R.info & (kInfoSmall0 << t)) {
    geo.ea[lane] = make_int4((int)((uint32_t)dx1 * (uint32_t)uy - (uint32_t)dy1 * (uint32_t)ux),
                             (int)((uint32_t)dx2 * (uint32_t)uy - (uint32_t)dy2 * (uint32_t)ux), -256 * dy1, -256 * dy2);
    geo.eb[lane] = make_int4(256 * dx1, 256 * dx2, 0, (int)id);
  } else {
    // 64-bit edge values: E + 256 (ly dx - lx dy)
    const long long e1 = (long long)dx1 * uy - (long long)dy1 * ux, e2 = (long long)dx2 * uy - (long long)dy2 * ux;
    geo.ea[lane] = make_int4((int)(uint32_t)e1, (int)(uint32_t)e2, -dy1, -dy2);
    geo.hi[lane] = make_int2((int)(e1 >> 32), (int)(e2 >> 32));
    geo.eb[lane] = make_int4(dx1, dx2, (int)kTriWide, (int)id);
  }
  if (VTX && !flat_view) {
    const uint4 vi = V.idx ? __ldg(reinterpret_cast<const uint4*>(V.idx) + jl)
                           : make_uint4(4 * jl, 4 * jl + 1, 4 * jl + 2, 4 * jl + 3);
    const uint32_t w1 = t ? vi.z : vi.y, w2 = t ? vi.w : vi.z;
    const uint32_t vb = sw ? w2 : w1, vc = sw ? w1 : w2;
    const float4* cv = reinterpret_cast<const float4*>(V.col);
    const bool lit = LIT && V.color_mode == LR_COLOR_LIT;
    const uint32_t cs = lit ? 2u : 1u;
    const float4 c0 = __ldg(cv + (size_t)cs * vi.x), c1 = __ldg(cv + (size_t)cs * vb), c2 = __ldg(cv + (size_t)cs * vc);
    const float4 p0 = make_float4(q_a * c0.x, q_a * c0.y, q_a * c0.z, q_a * c0.w);
    qc[lane] = p0;
    qc[32 + lane] = weighted_difference(q_b, c1, p0);
    qc[64 + lane] = weighted_difference(q_c, c2, p0);
    if (LIT && lit) {
      const float4 n0 = __ldg(cv + 2ull * vi.x + 1), n1 = __ldg(cv + 2ull * vb + 1), n2 = __ldg(cv + 2ull * vc + 1);
      const float4 o0 = make_float4(q_a * n0.x, q_a * n0.y, q_a * n0.z, 0.f);
      qc[96 + lane] = o0;
      qc[128 + lane] = weighted_difference(q_b, make_float4(n1.x, n1.y, n1.z, 0.f), o0);
      qc[160 + lane] = weighted_difference(q_c, make_float4(n2.x, n2.y, n2.z, 0.f), o0);
    }
  } else if (CARRY) {
    qc[lane] = __ldg(reinterpret_cast<const float4*>(V.col) + jl);
  }
}

// Sort key of a triangle of constant depth.
__device__ __forceinline__ unsigned long long const_key(const Ws& ws, const ViewDev& V, uint32_t id) {
  const float q0 = __ldg(reinterpret_cast<const float*>(ws.rec + 4ull * (uint32_t)(V.quad_base + (id >> 1)) + 2));
  return ((unsigned long long)__float_as_uint(q0) << 32) | id;
}

// Perspective-correct colour of a fragment: c / w interpolated with the weights l1, l2 and
// divided by the interpolated 1/w, which is the depth key (rk its reciprocal).
__device__ __forceinline__ float4 interpolate(float4 c0, float4 d1, float4 d2, float l1, float l2, float rk) {
  return make_float4((c0.x + l1 * d1.x + l2 * d2.x) * rk, (c0.y + l1 * d1.y + l2 * d2.y) * rk,
                     (c0.z + l1 * d1.z + l2 * d2.z) * rk, (c0.w + l1 * d1.w + l2 * d2.w) * rk);
}

// Lit views: RGB times the two-sided Lambert term of the interpolated normal (times the
// interpolated 1/w, which only scales it) plus ambient.
__device__ __forceinline__ void apply_light(float4& col, float4 n0, float4 n1, float4 n2, float l1, float l2, float4 light) {
  const float nx = n0.x + l1 * n1.x + l2 * n2.x;
  const float ny = n0.y + l1 * n1.y + l2 * n2.y;
  const float nz = n0.z + l1 * n1.z + l2 * n2.z;
  const float nn = nx * nx + ny * ny + nz * nz;
  const float d = fabsf(nx * light.x + ny * light.y + nz * light.z);
  const float lam = nn > 0.f ? fminf(d * rsqrtf(nn), 1.0f) : 0.f;
  const float f = light.w + (1.0f - light.w) * lam;
  col.x *= f;
  col.y *= f;
  col.z *= f;
}

// Colour of a fragment of the triangle in slot p, with barycentric weights l1, l2 and depth
// key `key`.
template <bool VTX, bool LIT>
__device__ __forceinline__ float4 shade(const float4* qc, int p, bool flat_view, bool lit, float4 light, float l1, float l2,
                                        float key) {
  float4 col = qc[p];
  if (VTX && !flat_view) {
    col = interpolate(col, qc[32 + p], qc[64 + p], l1, l2, rcp_approx(key));
    if (LIT && lit) apply_light(col, qc[96 + p], qc[128 + p], qc[160 + p], l1, l2, light);
  }
  return col;
}

// HASH: the variant that also writes the per-pixel coverage hash (a test output); the
// others carry no code or registers for it. ATH: the alpha-threshold variant (forward
// only, no hash), which also skips candidate quads that cannot reach in front of any
// pixel of the half-block still blending. LIT: the colour-carrying variant that also
// shades lit views (per-vertex normals, one directional light).
template <int K, bool VTX, bool BWD, bool HASH, bool ATH = false, bool LIT = false>
__global__ __launch_bounds__(kRasterThreads, raster_min_blocks(K, VTX, BWD, LIT)) void k_raster(Ws ws) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  // the sorter carries each fragment's colour (backward: the batch holds its triangles' colours)
  constexpr bool kCarry = VTX || K == 1 || BWD;
  constexpr int kWin = win_refs(half_window(K, BWD, LIT));
  constexpr bool kPark = parked(K, VTX, BWD);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lx = lane & (kHbW - 1), ly = lane >> 3;
  unsigned char* wbase = smem + (size_t)warp * batch_smem_warp(VTX, BWD, LIT, K);
  uint16_t* cand = reinterpret_cast<uint16_t*>(wbase);
  uint2* pend = reinterpret_cast<uint2*>(wbase + kWin * sizeof(uint16_t));
  BatchGeo& geo = *reinterpret_cast<BatchGeo*>(pend + kPendCap);
  float4* qc = reinterpret_cast<float4*>(&geo + 1);
  GradShared& gs = *reinterpret_cast<GradShared*>(qc + batch_cols(VTX, LIT) * 32);   // (backward)
  // a batch blended in stream order keeps its sort keys (alpha threshold) or ids where the
  // others keep ea
  unsigned long long* dkey = reinterpret_cast<unsigned long long*>(&geo);
  uint32_t* did = reinterpret_cast<uint32_t*>(&geo);
  // (a batch has less than 2^32 pixels)
  const uint32_t nitems = ws.ctrl->error == LR_ERR_OVERFLOW ? 0u : (uint32_t)ws.ctrl->raster_items;
  unsigned long long frag_total = 0;

  for (;;) {
    unsigned long long k = 0;
    if (lane == 0) k = atomicAdd(&ws.ctrl->raster_head, 1ull);
    const uint32_t item = __shfl_sync(0xffffffffu, (uint32_t)min(k, 0xFFFFFFF0ull), 0);
    if (item >= nitems) break;
    const int lg = ws.bin_log2, hl = bin_hb_log2(lg), cl = bin_hb_cols_log2(lg);
    const int bin_g = (int)ws.bin_order[item >> hl];
    // items 2 i and 2 i + 1 of a bin: the upper and the lower half-block of its 8x8 block i
    const int blk = (int)(item & ((1u << hl) - 1u)) >> 1;
    const int hb = ((2 * (blk >> cl) + (int)(item & 1u)) << cl) + (blk & ((1 << cl) - 1));
    const int v = view_of_bin(ws.views, ws.n_views, bin_g);
    const ViewDev& V = ws.views[v];
    const int b = bin_g - V.bin_base;
    const int bx = b % V.nbx, by = b / V.nbx;
    const int ox = (bx << lg) + (hb & ((1 << cl) - 1)) * kHbW, oy = (by << lg) + (hb >> cl) * kHbH;
    if (ox >= V.width || oy >= V.height || !tile_owned(V, ox, oy)) continue;
    const int px = ox + lx, py = oy + ly;
    const bool pix_ok = px < V.width && py < V.height;
    const uint32_t off = ws.bin_off[bin_g];
    const int n = (int)(ws.bin_off[bin_g + 1] - off);
    const bool flat_view = V.color_mode == LR_COLOR_FLAT, lit_view = LIT && V.color_mode == LR_COLOR_LIT;
    const bool hashing = HASH && V.hash != nullptr;
    const int Ox = 256 * ox + 128, Oy = 256 * oy + 128;   // first pixel centre, 1/256 px
    // lit views: unit direction toward the light and the ambient term
    const float4 light = LIT ? make_float4(V.light[0], V.light[1], V.light[2], V.light[3])
                             : make_float4(0.f, 0.f, 0.f, 0.f);

    typename std::conditional<BWD, GradState<K>, PixelState<K, kCarry, ATH, kPark>>::type st;
    if constexpr (BWD) {
      st.gp = GradPixel();
      if (pix_ok) st.gp.load(ws.grad_out, ws.fwd, (long long)py * V.width + px);
    } else {
      st.init();
      if (kPark) st.park = qc + batch_cols(VTX, LIT) * 32 + lane;
    }
    uint32_t cnt = 0;
    unsigned long long hsh = 0;

    // The backward pass streams the half-block twice: first without gradients, to learn
    // which pixels the sorter cannot order (those are left to the exact path, which
    // emits their whole gradient), then with gradients for the other pixels only.
    // With the forward's exact-path mask the detection pass is skipped.
    bool pre_flagged = false;
    int first_pass = BWD ? 0 : 1;
    if (BWD && ws.bwd_mask) {
      const uint32_t hbx = (uint32_t)ox / kHbW, hby = (uint32_t)oy / kHbH;
      const uint32_t hbw = ((uint32_t)V.width + kHbW - 1) / kHbW;
      pre_flagged = (ws.bwd_mask[hby * hbw + hbx] >> lane) & 1u;
      first_pass = 1;
    }
    for (int pass = first_pass; pass < 2; ++pass) {
    if constexpr (BWD) {
      st.init();
      st.flagged = pre_flagged;
      st.gp.grad = pass == 1 ? ws.grad_col : nullptr;
      gs.g[lane] = make_float4(st.gp.gr, st.gp.gg, st.gp.gb, 0.f);
      cnt = 0;
      hsh = 0;
    }
    // ---- 1. the half-block's candidates: set bits of its bitmap row, in sorted order ----
    const uint32_t* row = hb_row(ws, off, bin_g, n, hb);
    const int nw = (n + 31) >> 5;
    const uint32_t* ref_lo = reinterpret_cast<const uint32_t*>(ws.refs + off);   // low words
    int g = -kWin / 32, r0 = 0, total = 0;   // bitmap window, position in it, its candidates
    int head = 0, tail = 0;       // pending ring
    bool ordered = !HASH && !BWD; // everything so far was blended in stream order
    uint32_t last_id = 0xFFFFFFFFu;   // ... the last fragment's id
    for (;;) {
      // ---- 2. coverage masks of 32 candidates, one quad per lane, until a batch is full ---
      while (tail - head < 32) {
        if (r0 >= total) {
          g += kWin / 32;
          if (g >= nw) break;
          total = list_bits(lane < kWin / 32 && g + lane < nw ? __ldg(row + g + lane) : 0u, lane, cand);
          r0 = 0;
          continue;
        }
        const bool in = r0 + lane < total;
        const uint32_t rec = in ? ~ref_lo[2 * (32 * g + (int)cand[r0 + lane])] : 0u;
        r0 += 32;
        bool skip = !in;
        if constexpr (ATH) {
          // The smallest key a fragment must exceed to change any pixel of the half-block:
          // 0 while a pixel still blends; a finished pixel needs a fragment in front of the
          // one that finished it (keys are positive floats, so their bits order like them);
          // pixels outside the image and pixels left to the exact path need nothing. A
          // candidate whose largest possible key is below that is skipped: every fragment
          // of it would be dropped.
          const uint32_t need = (!pix_ok || st.flagged) ? 0xFFFFFFFFu : (st.live() ? 0u : (uint32_t)(st.last >> 32));
          const uint32_t kmin = __reduce_min_sync(0xffffffffu, need);
          if (kmin != 0u) {
            if (in) {
              const int4 qv = __ldg(ws.rec + 4ull * rec + 2);   // the record's four 1/w
              const float qm = fmaxf(fmaxf(__int_as_float(qv.x), __int_as_float(qv.y)),
                                     fmaxf(__int_as_float(qv.z), __int_as_float(qv.w)));
              skip = __float_as_uint(qm * kKeyBoundScale) < kmin;
            }
            if (__all_sync(0xffffffffu, skip)) continue;
          }
        }
        uint32_t ma = 0, mb = 0, ida = 0, idb = 0;
        if (!skip) {
          int X[4], Y[4];
          load_rec_xy(ws.rec, rec, X, Y);
          const int2 fl = __ldg(reinterpret_cast<const int2*>(ws.rec + 4ull * rec + 3) + 1);   // info, record flags
          const uint32_t info = (uint32_t)fl.x;
          const bool one = flat_view && (info & kInfoFlatDepth);
          if (!HASH && one && (fl.y & (int)kRecBox)) {
            const BoxSpan B(X, Y, ox, oy, kHbH);
            ma = (0x01010101u * B.columns()) & byte_span(B.y0, B.y1);
          } else if (fl.y & (int)kRecSmall) {
            quad_masks_small<kHbH>(X, Y, info, Ox, Oy, &ma, &mb);
          } else {
            quad_masks_any<kHbH>(X, Y, info, Ox, Oy, &ma, &mb);
          }
          ida = 2u * (uint32_t)(rec - V.quad_base);
          idb = ida + 1u;
          if (one) {
            // one colour and one depth key for the whole quad: its triangles form one entry
            // where they do not overlap, else the second goes first (it lies in front: equal
            // keys order by triangle)
            if (!HASH && (ma & mb) == 0u) {
              ma |= mb;
              mb = 0u;
            } else {
              const uint32_t t = ma; ma = mb; mb = t;
              const uint32_t u = ida; ida = idb; idb = u;
            }
            ida |= kPendConst;
            idb |= kPendConst;
          }
        }
        const unsigned ba = __ballot_sync(0xffffffffu, ma != 0u), bb = __ballot_sync(0xffffffffu, mb != 0u);
        const unsigned lt = (1u << lane) - 1u;
        int at = tail + __popc(ba & lt) + __popc(bb & lt);
        if (ma) pend[at++ & (kPendCap - 1)] = make_uint2(ida, ma);
        if (mb) pend[at & (kPendCap - 1)] = make_uint2(idb, mb);
        tail += __popc(ba) + __popc(bb);
        __syncwarp();
      }
      const int nb = min(32, tail - head);
      if (nb == 0) break;
      // ---- 3. records of the next nb covering triangles, one per lane; entry 31 - L of the
      // batch goes to lane and slot L, so that the highest set bit is the next in order ------
      const int e = 31 - lane;
      uint32_t id = 0, mk = 0;
      if (e < nb) {
        const uint2 pe = pend[(head + e) & (kPendCap - 1)];
        id = pe.x;
        mk = pe.y;
      }
      head += nb;
      const bool direct = ordered && __all_sync(0xffffffffu, e >= nb || (id & kPendConst));
      id &= ~kPendConst;
      if (direct) {
        if (e < nb) {
          qc[lane] = __ldg(reinterpret_cast<const float4*>(V.col) + (id >> 1));
          if (ATH) dkey[lane] = const_key(ws, V, id);
          else did[lane] = id;
        }
      } else if (e < nb) {
        setup_batch<VTX, LIT, kCarry>(ws, V, flat_view, id, lane, Ox, Oy, geo, qc);
      }
      // ---- 4. transpose: lane = pixel, bit L = covered by the triangle in slot L -----------
      uint32_t m = warp_transpose32(mk, lane);   // (its shuffles also order the slots' writes below)
      __syncwarp();
      if (!pix_ok) m = 0;
      cnt += __popc(m);
      if constexpr (!BWD) {
        if (direct) {
          // ---- 5a. flat colours at constant depths, everything before them likewise: the
          // stream order is the fragments' exact order (the bin sort's key is the depth key), so
          // they blend as they come, without the sorter
          const uint32_t all = m;
          uint32_t lastp = 32;
          while (m) {
            if (ATH && !st.live()) break;
            const int p = 31 - __clz(m);
            m ^= 1u << p;
            const float4 c = qc[p];
            if (ATH) lastp = (uint32_t)p;
            st.blend_direct(c);
          }
          if (!ATH) lastp = (uint32_t)(__ffs(all) - 1);
          if (ATH) { if (lastp < 32u) st.last = dkey[lastp]; }
          else if (lastp < 32u) last_id = did[lastp];
          __syncwarp();
          continue;
        }
        if (ordered) {
          if (!ATH && last_id != 0xFFFFFFFFu) st.last = const_key(ws, V, last_id);
          // the sorter starts here; with a transparent held fragment at the last key blended
          // (K = 1), so that its first eviction keeps that key
          ordered = false;
          if (PixelState<K, kCarry, ATH>::kNullSlot) st.s[0] = st.last;
        }
      } else {
        st.cover = m;
        st.done = 0u;
        gs.g[lane].w = __uint_as_float(m);
      }
      // ---- 5b. fragments in candidate order through the K-slot sorter -------------------
      auto frag_step = [&]() {
        const int p = 31 - __clz(m);
        m ^= 1u << p;
        const int4 eb = geo.eb[p];
        const uint32_t fid = (uint32_t)eb.w;
        if (hashing) hsh += splitmix64(fid);
        // (the forward discards a flagged pixel's composite, the exact path redoing it, so it
        // keeps inserting rather than testing the flag per fragment; the backward must not
        // add a flagged pixel's gradient)
        if (!BWD || !st.flagged) {
          const int4 ea = geo.ea[p];
          const float4 kq = geo.kq[p];
          float f1, f2;
          if (!((uint32_t)eb.z & kTriWide)) {
            f1 = __int2float_rn((int)((uint32_t)ea.x + (uint32_t)lx * (uint32_t)ea.z + (uint32_t)ly * (uint32_t)eb.x));
            f2 = __int2float_rn((int)((uint32_t)ea.y + (uint32_t)lx * (uint32_t)ea.w + (uint32_t)ly * (uint32_t)eb.y));
          } else {
            const int2 h = geo.hi[p];
            const long long e1 = ((long long)h.x << 32) | (uint32_t)ea.x, e2 = ((long long)h.y << 32) | (uint32_t)ea.y;
            f1 = __ll2float_rn(e1 + 256LL * (lx * ea.z + ly * eb.x));
            f2 = __ll2float_rn(e2 + 256LL * (lx * ea.w + ly * eb.y));
          }
          // exact depth key: the interpolated 1/w (Sec. 2 "Stage 3", the reading O.8)
          const float l1 = __fmul_rn(f1, kq.w), l2 = __fmul_rn(f2, kq.w);
          const float key = __fadd_rn(kq.x, __fadd_rn(__fmul_rn(l1, kq.y), __fmul_rn(l2, kq.z)));
          const unsigned long long sk = ((unsigned long long)__float_as_uint(key) << 32) | fid;
          if constexpr (BWD) {
            st.insert(sk, (uint32_t)p, V, qc, gs);
          } else {
            float4 col = make_float4(0.f, 0.f, 0.f, 0.f);
            if (kCarry) col = shade<VTX, LIT>(qc, p, flat_view, lit_view, light, l1, l2, key);
            st.insert(sk, col, V);
          }
        }
      };
      while (m) frag_step();
      __syncwarp();
      if constexpr (BWD) {
        if (st.gp.grad) batch_gradients(st.done, id >> 1, st.gp.grad, qc, gs);
#pragma unroll
        for (int i = 0; i < K; ++i) st.sl[i] = kOldSlot;
        __syncwarp();
      }
    }
    if (pass == 0) pre_flagged = st.flagged;
    }

    // ---- finish the half-block ---------------------------------------------------------
    // a pixel the given mask missed has had part of its gradient added already: report it
    if (BWD && ws.bwd_mask && st.flagged && !pre_flagged) set_error(ws.ctrl, LR_ERR_MASK_MISMATCH);
    if (!BWD && V.xmask) {
      const uint32_t fm = __ballot_sync(0xffffffffu, pix_ok && st.flagged);
      if (lane == 0) {
        const uint32_t hbw = ((uint32_t)V.width + kHbW - 1) / kHbW;
        V.xmask[((uint32_t)oy / kHbH) * hbw + (uint32_t)ox / kHbW] = fm;
      }
    }
    if (!st.flagged) {
      if constexpr (BWD) st.flush(V, qc, gs);
      else st.flush(V);
    }
    if (pix_ok) {
      const long long pidx = (long long)py * V.width + px;
      if (!BWD && V.cnt) V.cnt[pidx] = cnt;
      if (!BWD && hashing) V.hash[pidx] = hsh;
      if (!st.flagged) {
        if constexpr (!BWD) write_pixel(V, pidx, st.r, st.g, st.b, st.T);
      } else {
        const unsigned long long slot = atomicAdd(&ws.ctrl->ovf_count, 1ull);
        ws.ovf_list[slot] = (uint32_t)(V.pix_base + pidx);
      }
    }
    frag_total += cnt;
  }
  // fragments of all pixels this warp rendered
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) frag_total += __shfl_xor_sync(0xffffffffu, frag_total, o);
  if (lane == 0 && frag_total) atomicAdd(&ws.ctrl->fragments, frag_total);
}

}  // namespace lr

// Each translation unit lr_raster_k<K>.cu instantiates the rasteriser for one sorter
// capacity K (both colour layouts) through this macro, so the variants compile in
// parallel.
#define LR_DEFINE_RASTER(KK)                                                                  \
  namespace lr {                                                                              \
  template <bool VTX, bool BWD, bool HASH, bool ATH = false, bool LIT = false>                \
  static cudaError_t raster_attr_##KK() {                                                     \
    return cudaFuncSetAttribute(k_raster<KK, VTX, BWD, HASH, ATH, LIT>,                       \
                                cudaFuncAttributeMaxDynamicSharedMemorySize,                  \
                                (int)raster_smem_bytes(VTX, BWD, LIT, KK));                       \
  }                                                                                           \
  cudaError_t prepare_raster_##KK(int* blocks_flat, int* blocks_vtx, int* blocks_bwd,         \
                                  int* blocks_lit) {                                          \
    cudaError_t e = raster_attr_##KK<false, false, false>();                                  \
    if (e == cudaSuccess) e = raster_attr_##KK<true, false, false>();                         \
    if (e == cudaSuccess) e = raster_attr_##KK<false, true, false>();                         \
    if (e == cudaSuccess) e = raster_attr_##KK<false, false, true>();                         \
    if (e == cudaSuccess) e = raster_attr_##KK<true, false, true>();                          \
    if (e == cudaSuccess) e = raster_attr_##KK<false, false, false, true>();                  \
    if (e == cudaSuccess) e = raster_attr_##KK<true, false, false, true>();                   \
    if (e == cudaSuccess) e = raster_attr_##KK<true, false, false, false, true>();            \
    if (e != cudaSuccess) return e;                                                           \
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(                                        \
        blocks_lit, k_raster<KK, true, false, false, false, true>, kRasterThreads,            \
        raster_smem_bytes(true, false, true, KK));                                                \
    if (e != cudaSuccess) return e;                                                           \
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_flat, k_raster<KK, false, false, false>, \
                                                      kRasterThreads, raster_smem_bytes(false, false, false, KK)); \
    if (e != cudaSuccess) return e;                                                           \
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_bwd, k_raster<KK, false, true, false>, \
                                                      kRasterThreads, raster_smem_bytes(false, true)); \
    if (e != cudaSuccess) return e;                                                           \
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_vtx, k_raster<KK, true, false, false>, \
                                                         kRasterThreads, raster_smem_bytes(true, false, false, KK)); \
  }                                                                                           \
  /* mode: 0 flat colours, 1 colours in the sorter, 2 backward; + 4: coverage hash;        \
     + 8: alpha threshold (modes 8 and 9 only); 17: colours in the sorter with lit views */   \
  cudaError_t launch_raster_##KK(int mode, const Ws& ws, int grid, cudaStream_t st, bool pdl) { \
    const size_t sf = raster_smem_bytes(false, false, false, KK), sv = raster_smem_bytes(true, false, false, KK);                 \
    const dim3 g(grid), t(kRasterThreads);                                                    \
    switch (mode) {                                                                           \
      case 1: return launch_pdl(pdl, k_raster<KK, true, false, false>, g, t, sv, st, ws);     \
      case 2: return launch_pdl(pdl, k_raster<KK, false, true, false>, g, t, raster_smem_bytes(false, true), st, ws); \
      case 4: return launch_pdl(pdl, k_raster<KK, false, false, true>, g, t, sf, st, ws);     \
      case 5: return launch_pdl(pdl, k_raster<KK, true, false, true>, g, t, sv, st, ws);      \
      case 8: return launch_pdl(pdl, k_raster<KK, false, false, false, true>, g, t, sf, st, ws); \
      case 9: return launch_pdl(pdl, k_raster<KK, true, false, false, true>, g, t, sv, st, ws); \
      case 17:                                                                                \
        return launch_pdl(pdl, k_raster<KK, true, false, false, false, true>, g, t,           \
                          raster_smem_bytes(true, false, true, KK), st, ws);                      \
      default: return launch_pdl(pdl, k_raster<KK, false, false, false>, g, t, sf, st, ws);   \
    }                                                                                         \
  }                                                                                           \
  }
