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
// What bounds it and what it took (K = 1, 1920x1080, kernel times): on 1M wavy quads with
// vertex colours the shared-memory and gather wavefronts (80% of the L1 data pipe; a 16-byte
// load per lane costs four), 62% of issue slots; against setting up both triangles of each
// candidate with a binary search per edge and row, 349M -> 253M warp instructions and
// 375 -> 328 us. On 2M particles, 60% of issue slots and the gathers of scattered records;
// 848M -> 372M instructions, 1005 -> 506 us. With normals 602 -> 416 us, with the alpha
// threshold on the particles 389 -> 268 us, a batch of mixed views at K = 3 2040 -> 911 us,
// 100k scattered parallelograms with a few screen-filling ones 117 -> 66 us.
#pragma once

#include "lr_common.cuh"

namespace lr {

constexpr uint32_t kTriValid = 1u, kTriFast = 2u, kTriFlatCol = 4u;   // + corr bits 3..5
// all three vertices at the same 1/w: the depth key is q0 at every pixel (the
// interpolation adds l1 * 0 + l2 * 0 with l1, l2 >= 0)
constexpr uint32_t kTriConstKey = 64u;
// lit colours (LR_COLOR_LIT): the triangle's colour slots also hold its perspective-weighted
// normals, and each fragment's RGB is shaded with the view's light
constexpr uint32_t kTriLit = 128u;
// k_raster's batches: the edge values are kept in 64 bits
constexpr uint32_t kTriWide = 256u;
constexpr unsigned long long kSent = ~0ull;
constexpr int kRasterThreads = 256;
#ifndef LR_RASTER_MIN_BLOCKS
// resident CTAs per SM requested from the compiler: 3 caps registers at 80 per thread (24
// warps per SM, a few spills), measured faster than 2 (128 registers) on both the layer
// and the particle workloads; without a bound the compiler takes ~160 and one CTA fits
#define LR_RASTER_MIN_BLOCKS 3
#endif
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

// Per (triangle, half-block) record read by the fragment loop, laid out for three 16-byte
// shared-memory loads. Edges 1 (v2->v0) and 2 (v0->v1) give the barycentric numerators
// of the depth key; edge 0 is only needed for coverage, which the masks already hold.
struct __align__(16) TriSm {
  int4 ea;         // e1, e2: edge values E at the half-block's first pixel centre; sx1,
                   // sx2: change per pixel step in x
  int4 eb;         // sy1, sy2: change per pixel step in y; flags; id (2 * quad + triangle)
  float4 kq;       // q0 = 1/w at v0, d1 = q1 - q0, d2 = q2 - q0, inv = 1 / (float)area
  int X[3], Y[3];  // vertices after the orientation fix (64-bit path)
  int pad[2];
};

// exact 64-bit edge values (unbiased) of a triangle at pixel (px, py)
__device__ __forceinline__ void edges64(const TriSm& T, int px, int py, long long e[3]) {
  const long long Px = 256LL * px + 128, Py = 256LL * py + 128;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int u = k == 0 ? 1 : (k == 1 ? 2 : 0);
    const int w = k == 0 ? 2 : (k == 1 ? 0 : 1);
    e[k] = (long long)(T.X[w] - T.X[u]) * (Py - T.Y[u]) - (long long)(T.Y[w] - T.Y[u]) * (Px - T.X[u]);
  }
}

// Builds the per-half-block record of triangle t of a quad; returns false if the triangle
// has zero area or its pixel AABB misses the half-block (BH rows: 4, or 8 for the 8x8
// blocks of k_raster8).
template <int BH = kHbH>
static __device__ __noinline__ bool setup_tri(TriSm& T, const int X[4], const int Y[4], const float qv[4],
                                          uint32_t info, int t, uint32_t jl, int ox, int oy,
                                          int cor[3], int box[4], int le[3], int lsx[3], int lsy[3]) {
  if (!(info & (t ? kInfoTri1 : kInfoTri0))) return false;
  // vertices (v0, v1, v2) of T0 or (v0, v2, v3) of T1, chosen with selects (no indexing)
  int xa = X[0], ya = Y[0];
  int xb = t ? X[2] : X[1], yb = t ? Y[2] : Y[1];
  int xc = t ? X[3] : X[2], yc = t ? Y[3] : Y[2];
  float qa = qv[0], qb = t ? qv[2] : qv[1], qc = t ? qv[3] : qv[2];
  int ib = t ? 2 : 1, ic = t ? 3 : 2;
  long long A = area2(xa, ya, xb, yb, xc, yc);
  if (A < 0) {   // orientation fix: swap v1 and v2
    int ti = xb; xb = xc; xc = ti;
    ti = yb; yb = yc; yc = ti;
    const float tq = qb; qb = qc; qc = tq;
    ti = ib; ib = ic; ic = ti;
    A = -A;
  }
  const int xmin = min(xa, min(xb, xc)), xmax = max(xa, max(xb, xc));
  const int ymin = min(ya, min(yb, yc)), ymax = max(ya, max(yb, yc));
  const int bx0 = ceil_div256((long long)xmin - 128), bx1 = floor_div256((long long)xmax - 128);
  const int by0 = ceil_div256((long long)ymin - 128), by1 = floor_div256((long long)ymax - 128);
  if (bx0 > ox + kHbW - 1 || bx1 < ox || by0 > oy + BH - 1 || by1 < oy) return false;
  box[0] = max(bx0 - ox, 0);
  box[1] = min(bx1 - ox, kHbW - 1);
  box[2] = max(by0 - oy, 0);
  box[3] = min(by1 - oy, BH - 1);
  cor[0] = 0; cor[1] = ib; cor[2] = ic;
  T.X[0] = xa; T.X[1] = xb; T.X[2] = xc;
  T.Y[0] = ya; T.Y[1] = yb; T.Y[2] = yc;
  T.kq = make_float4(qa, __fsub_rn(qb, qa), __fsub_rn(qc, qa), __fdiv_rn(1.0f, __ll2float_rn(A)));
  uint32_t flags = kTriValid | ((qb == qa && qc == qa) ? kTriConstKey : 0u);
  bool fast = true;
  const long long P0x = 256LL * ox + 128, P0y = 256LL * oy + 128;
  const long long lim = 1LL << 30;
  // edges v1->v2, v2->v0, v0->v1
  const int ux[3] = {xb, xc, xa}, uy[3] = {yb, yc, ya}, wx[3] = {xc, xa, xb}, wy[3] = {yc, ya, yb};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const long long dx = (long long)wx[k] - ux[k], dy = (long long)wy[k] - uy[k];
    const bool owned = dy < 0 || (dy == 0 && dx > 0);
    const long long e0 = dx * (P0y - uy[k]) - dy * (P0x - ux[k]) + (owned ? 0 : -1);
    const long long sx = -256 * dy, sy = 256 * dx;
    const long long c1 = e0 + (kHbW - 1) * sx, c2 = e0 + (BH - 1) * sy, c3 = c1 + (BH - 1) * sy;
    fast &= (e0 > -lim && e0 < lim && c1 > -lim && c1 < lim && c2 > -lim && c2 < lim && c3 > -lim && c3 < lim);
    le[k] = (int)e0;
    lsx[k] = (int)sx;
    lsy[k] = (int)sy;
    if (!owned) flags |= 1u << (3 + k);
  }
  if (fast) flags |= kTriFast;
  // the key's edge values unbiased (the masks use the biased ones in le)
  T.ea = make_int4((int)((uint32_t)le[1] + ((flags >> 4) & 1u)), (int)((uint32_t)le[2] + ((flags >> 5) & 1u)), lsx[1],
                   lsx[2]);
  T.eb = make_int4(lsy[1], lsy[2], (int)flags, (int)(2u * jl + (uint32_t)t));
  return true;
}

// setup_tri for a triangle that k_setup marked small (kInfoSmall0 << t): the orientation
// and 1/area come precomputed, and every edge value at the pixel centres of the box's rows,
// up to 7 pixels to either side of the box, fits in 32 bits, so the whole set-up is 32-bit
// integer arithmetic (a block row outside the box is masked off, whatever its values).
template <int BH = kHbH>
__device__ __forceinline__ bool setup_tri_small(TriSm& T, const int X[4], const int Y[4], const float qv[4],
                                                float inv, uint32_t info, int t, uint32_t jl, int ox, int oy,
                                                int cor[3], int box[4], int le[3], int lsx[3], int lsy[3]) {
  if (!(info & (t ? kInfoTri1 : kInfoTri0))) return false;
  int xa = X[0], ya = Y[0];
  int xb = t ? X[2] : X[1], yb = t ? Y[2] : Y[1];
  int xc = t ? X[3] : X[2], yc = t ? Y[3] : Y[2];
  float qa = qv[0], qb = t ? qv[2] : qv[1], qc = t ? qv[3] : qv[2];
  int ib = t ? 2 : 1, ic = t ? 3 : 2;
  if (info & (kInfoSwap0 << t)) {
    int ti = xb; xb = xc; xc = ti;
    ti = yb; yb = yc; yc = ti;
    const float tq = qb; qb = qc; qc = tq;
    ti = ib; ib = ic; ic = ti;
  }
  // pixel-centre box: ceil((min - 128) / 256) .. floor((max - 128) / 256)
  const int bx0 = (min(xa, min(xb, xc)) + 127) >> 8, bx1 = (max(xa, max(xb, xc)) - 128) >> 8;
  const int by0 = (min(ya, min(yb, yc)) + 127) >> 8, by1 = (max(ya, max(yb, yc)) - 128) >> 8;
  if (bx0 > ox + kHbW - 1 || bx1 < ox || by0 > oy + BH - 1 || by1 < oy) return false;
  box[0] = max(bx0 - ox, 0);
  box[1] = min(bx1 - ox, kHbW - 1);
  box[2] = max(by0 - oy, 0);
  box[3] = min(by1 - oy, BH - 1);
  cor[0] = 0; cor[1] = ib; cor[2] = ic;
  T.kq = make_float4(qa, __fsub_rn(qb, qa), __fsub_rn(qc, qa), inv);
  uint32_t flags = kTriValid | kTriFast | ((qb == qa && qc == qa) ? kTriConstKey : 0u);
  const int P0x = 256 * ox + 128, P0y = 256 * oy + 128;
  const int ux[3] = {xb, xc, xa}, uy[3] = {yb, yc, ya}, wx[3] = {xc, xa, xb}, wy[3] = {yc, ya, yb};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int dx = wx[k] - ux[k], dy = wy[k] - uy[k];
    const bool owned = dy < 0 || (dy == 0 && dx > 0);
    le[k] = (int)((uint32_t)dx * (uint32_t)(P0y - uy[k]) - (uint32_t)dy * (uint32_t)(P0x - ux[k])) - (owned ? 0 : 1);
    lsx[k] = -256 * dy;
    lsy[k] = 256 * dx;
    if (!owned) flags |= 1u << (3 + k);
  }
  // the key's edge values unbiased (the masks use the biased ones in le)
  T.ea = make_int4((int)((uint32_t)le[1] + ((flags >> 4) & 1u)), (int)((uint32_t)le[2] + ((flags >> 5) & 1u)), lsx[1],
                   lsx[2]);
  T.eb = make_int4(lsy[1], lsy[2], (int)flags, (int)(2u * jl + (uint32_t)t));
  return true;
}

// Backward of the front-to-back composite for one pixel (flat per-quad RGBA). With
// C = sum_i T_i a_i c_i, T_i = prod_{k<i} (1 - a_k), A = 1 - prod (1 - a_k):
//   dC/dc_i = T_i a_i,   dC/da_i = T_i c_i - S_i / (1 - a_i),   dA/da_i = T_final / (1 - a_i)
// where S_i = C_final - (C accumulated through fragment i) is the colour contributed by the
// fragments behind i. C_final, T_final come from the forward image; the running sums are
// recomputed with the forward's operations in the forward's order.
struct GradPixel {
  float gr, gg, gb, ga;      // dL/d(R, G, B, A) of the pixel
  float fr, fg, fb, fT;      // forward colour and transmittance
  float* grad;               // f32[Q][4] of the view
  float4* agg;               // this warp's 32 shared-memory slots for combining lanes' gradients
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

// Coverage of the half-block's 32 pixel centres (bit ly * 8 + lx) by a "fast" triangle:
// per row the intersection of the three edges' covered columns, limited to the triangle's
// pixel bounding box.
__device__ __forceinline__ uint32_t tri_mask_fast(const int e[3], const int sx[3], const int sy[3],
                                                  const int box[4]) {
  uint32_t mask = 0;
  const uint32_t cols = ((2u << box[1]) - 1u) & ~((1u << box[0]) - 1u);
#pragma unroll
  for (int ly = 0; ly < kHbH; ++ly) {
    uint32_t row = (ly >= box[2] && ly <= box[3]) ? cols : 0u;
#pragma unroll
    for (int k = 0; k < 3; ++k)
      row &= row_cover((int)((uint32_t)e[k] + (uint32_t)ly * (uint32_t)sy[k]), sx[k]);
    mask |= row << (ly * kHbW);
  }
  return mask;
}

// The same with exact 64-bit edge values, pixel by pixel (large triangles).
static __device__ __noinline__ uint32_t tri_mask_slow(const TriSm& T, int ox, int oy, const int box[4]) {
  uint32_t mask = 0;
  for (int ly = box[2]; ly <= box[3]; ++ly)
    for (int lx = box[0]; lx <= box[1]; ++lx) {
      long long e[3];
      edges64(T, ox + lx, oy + ly, e);
      bool cov = true;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const bool owned = !((uint32_t)T.eb.z & (1u << (3 + k)));
        cov &= e[k] > 0 || (e[k] == 0 && owned);
      }
      if (cov) mask |= 1u << (ly * kHbW + lx);
    }
  return mask;
}


// Exact depth key (interpolated 1/w, Sec. 2 "Stage 3", the reading O.8 of the depth
// formula) of a triangle record at pixel (px, py) = (ox + lx, oy + ly) of its half-block;
// also returns the barycentric weights l1, l2 it used.
__device__ __forceinline__ float tri_key(const TriSm& T, int4 ea, int4 eb, float4 kq, int lx, int ly, int px,
                                         int py, float& l1, float& l2) {
  const uint32_t fl = (uint32_t)eb.z;
  float f1, f2;
  if (fl & kTriFast) {
    const int e1 = (int)((uint32_t)ea.x + (uint32_t)lx * (uint32_t)ea.z + (uint32_t)ly * (uint32_t)eb.x);
    const int e2 = (int)((uint32_t)ea.y + (uint32_t)lx * (uint32_t)ea.w + (uint32_t)ly * (uint32_t)eb.y);
    f1 = __int2float_rn(e1);
    f2 = __int2float_rn(e2);
  } else {
    long long e[3];
    edges64(T, px, py, e);
    f1 = __ll2float_rn(e[1]);
    f2 = __ll2float_rn(e[2]);
  }
  l1 = __fmul_rn(f1, kq.w);
  l2 = __fmul_rn(f2, kq.w);
  return __fadd_rn(kq.x, __fadd_rn(__fmul_rn(l1, kq.y), __fmul_rn(l2, kq.z)));
}

// ATH: the alpha-threshold variant. Once the transmittance drops to kAlphaTMin nothing
// more is blended and `last` stays at the key of the fragment that got it there, so the
// misorder test below only flags fragments that belong in front of that one.
template <int K, bool VTX, bool BWD = false, bool ATH = false>
struct PixelState {
  // K = 1 with flat colours gathered at blend time: the colour of the fragment held in the
  // slot is loaded when it enters, so the gather overlaps the next fragment's work
  static constexpr bool kPrefetch = !VTX && K == 1;
  unsigned long long s[K];
  float4 c[VTX || kPrefetch ? K : 1];
  unsigned long long last;
  float r, g, b, T;
  bool flagged;
  GradPixel gp;

  // K = 1, forward, colours carried: the empty slot holds a fully transparent colour, so
  // blending it changes nothing (T and the colour stay, last is still kSent) and the in-order
  // insert needs no test for it (layer frame rasteriser 0.409 -> 0.394 ms; the same for the
  // flat colours gathered at blend time made the particle frame's 14% slower)
  static constexpr bool kNullSlot = VTX && K == 1 && !BWD;

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < K; ++i) s[i] = kSent;
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
    if (BWD && gp.grad) {
      const float om = 1.0f - col.w;
      float da = gp.gr * T * col.x + gp.gg * T * col.y + gp.gb * T * col.z;
      if (om > 1e-6f) {
        const float inv = rcp_approx(om);   // gradients need no correctly rounded divide
        da -= (gp.gr * (gp.fr - r) + gp.gg * (gp.fg - g) + gp.gb * (gp.fb - b)) * inv;
        da += gp.ga * gp.fT * inv;
      }
      // lanes blending a fragment of the same quad at this point add their contributions
      // in shared memory first, and one of them issues the four global atomics
      const int lane = threadIdx.x & 31;
      const unsigned act = __activemask();
      const unsigned grp = __match_any_sync(act, j);
      gp.agg[lane] = make_float4(gp.gr * w, gp.gg * w, gp.gb * w, da);
      __syncwarp(act);
      if (lane == __ffs(grp) - 1) {
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        for (unsigned m = grp; m; m &= m - 1) {
          const float4 c = gp.agg[__ffs(m) - 1];
          sum.x += c.x; sum.y += c.y; sum.z += c.z; sum.w += c.w;
        }
        float* gq = gp.grad + 4ull * j;
        atomicAdd(gq + 0, sum.x);
        atomicAdd(gq + 1, sum.y);
        atomicAdd(gq + 2, sum.z);
        atomicAdd(gq + 3, sum.w);
      }
      __syncwarp(act);
    }
    // T (1 - a) as one fused T - T a (a rounding, not the product's two, away from it: well
    // inside the colour tolerance); the threshold variant, whose T decides which fragments
    // blend, and the backward keep the product
    if (ATH || BWD) T *= 1.0f - col.w;
    else T = __fmaf_rn(-T, col.w, T);
  }

  // forward blend of a fragment known to be next in order, without the sorter
  __device__ __forceinline__ void blend_direct(float4 col) {
    const float w = T * col.w;
    r += w * col.x;
    g += w * col.y;
    b += w * col.z;
    if (ATH) T *= 1.0f - col.w;
    else T = __fmaf_rn(-T, col.w, T);
  }

  __device__ __forceinline__ void insert(unsigned long long x, float4 xc, const ViewDev& V) {
    // nearer than a fragment already blended: order not guaranteed. The forward pass with
    // carried colours only records it (the pixel's composite is discarded, so inserting the
    // fragment anyway is harmless; measured faster than the branch there, slower for the
    // colours gathered at blend time)
    if (VTX && !BWD) {
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
    if (VTX && K == 1) {       // one slot (threshold, backward): a branch
      if (x > s[0]) {          // nearer than the held fragment: blend it at once
        if (live()) {
          blend(x, xc, V);
          last = x;
        }
      } else {
        if ((kNullSlot || s[0] != kSent) && live()) {
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
    if (VTX) {
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
      if (VTX) {
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
      if (s[i] != kSent && live()) blend(s[i], VTX || kPrefetch ? c[i] : make_float4(0.f, 0.f, 0.f, 0.f), V);
  }
};

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

// ---- k_raster's coverage masks -------------------------------------------------------------
//
// Forward coverage of an edge u -> v on the half-block at pixel-centre origin (Px, Py): row
// ly's columns as the low 8 bits of f[ly] (the bits above are arbitrary). Covered iff
// E + bias >= 0, E = dx (Py - yu) - dy (Px - xu), bias = 0 for an owned edge, else -1. A step
// of one column adds -256 dy and one of a row 256 dx, so E + bias may be replaced by
// r = floor((E + bias) / 256) with steps -dy and dx. The covered columns are then
//   dy < 0: those from ceil(r / dy) on,  dy > 0: the first floor(r / dy) + 1,  dy = 0: r >= 0,
// and both counts are ceil(r / dy -+ eps) for any eps below the quotient's distance from the
// next integer, 1 / |dy| > 2^-15. The quotient is taken in fp32 as r (1 / (8 dy)), clamped to
// [0, 1] by the multiply-add's saturation: r and its row steps are exact (|r| < 2^22), the
// approximate reciprocal and the rounding put the clamped value off by less than 2^-22, and
// eps = 2^-17 (2^-20 scaled) exceeds that, so the count is exact; the scaling back adds 2^23
// rounded up, which leaves ceil() in the low bits. Needs |E| < 2^30 and |dx|, |dy| < 2^15 on
// the half-block (kRecSmall). Five instructions per edge and row, against about 16 for the
// exact integer binary search (row_cover).
__device__ __forceinline__ void edge_rows(int xu, int yu, int xv, int yv, int Px, int Py, uint32_t f[kHbH]) {
  const int dx = xv - xu, dy = yv - yu;
  const bool owned = dy < 0 || (dy == 0 && dx > 0);
  const int e = (int)((uint32_t)dx * (uint32_t)(Py - yu) - (uint32_t)dy * (uint32_t)(Px - xu)) - (owned ? 0 : 1);
  float r = __int2float_rn(e >> 8);
  const float step = __int2float_rn(dx);
  const float k = dy == 0 ? -1e20f : rcp_approx(__int2float_rn(8 * dy));
  const float b = dy > 0 ? 0x1p-20f : -0x1p-20f;
  const uint32_t flip = dy > 0 ? 0xFFFFFFFFu : 0u;
#pragma unroll
  for (int ly = 0; ly < kHbH; ++ly) {
    const float t = __saturatef(__fmaf_rn(r, k, b));
    const uint32_t c = __float_as_uint(__fmaf_ru(t, 8.0f, 8388608.0f));   // count in the low 5 bits
    f[ly] = __funnelshift_l(0u, 0xFFFFFFFFu, c) ^ flip;                   // ~0 << (c mod 32)
    r = __fadd_rn(r, step);
  }
}

__device__ __forceinline__ uint32_t pack_rows(uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  return __byte_perm(__byte_perm(r0, r1, 0x0040), __byte_perm(r2, r3, 0x0040), 0x5410);
}

// Coverage masks (bit ly * 8 + lx) of a quad's two triangles on the half-block. Under the
// top-left rule a pixel centre belongs to exactly one of an edge's two directions, so an edge
// traversed backwards (a triangle of negative area, or the diagonal's second triangle) takes
// the complement, and five edges serve both triangles.
__device__ __forceinline__ void quad_masks_small(const int X[4], const int Y[4], uint32_t info, int Px, int Py,
                                                 uint32_t& m0, uint32_t& m1) {
  const uint32_t s0 = (info & kInfoSwap0) ? 0xFFFFFFFFu : 0u;
  const uint32_t s1 = (info & (kInfoSwap0 << 1)) ? 0xFFFFFFFFu : 0u;
  uint32_t d[kHbH], f[kHbH], a[kHbH], c[kHbH];
  edge_rows(X[2], Y[2], X[0], Y[0], Px, Py, d);   // the diagonal, T0's direction
  edge_rows(X[0], Y[0], X[1], Y[1], Px, Py, f);
#pragma unroll
  for (int i = 0; i < kHbH; ++i) { a[i] = (d[i] ^ s0) & (f[i] ^ s0); c[i] = ~(d[i] ^ s1); }
  edge_rows(X[1], Y[1], X[2], Y[2], Px, Py, f);
#pragma unroll
  for (int i = 0; i < kHbH; ++i) a[i] &= f[i] ^ s0;
  edge_rows(X[2], Y[2], X[3], Y[3], Px, Py, f);
#pragma unroll
  for (int i = 0; i < kHbH; ++i) c[i] &= f[i] ^ s1;
  edge_rows(X[3], Y[3], X[0], Y[0], Px, Py, f);
#pragma unroll
  for (int i = 0; i < kHbH; ++i) c[i] &= f[i] ^ s1;
  m0 = (info & kInfoTri0) ? pack_rows(a[0], a[1], a[2], a[3]) : 0u;
  m1 = (info & kInfoTri1) ? pack_rows(c[0], c[1], c[2], c[3]) : 0u;
}

// The same for any quad: the 64-bit edge value at the origin, divided by 256 as above, is
// clamped to +-2^28 (|7 dy + 3 dx| < 2^27 within the guard band, so a clamped value keeps its
// sign on the whole half-block), and the rows are searched in 32-bit integers.
__device__ __forceinline__ void quad_masks_any(const int X[4], const int Y[4], uint32_t info, int Px, int Py,
                                               uint32_t& m0, uint32_t& m1) {
  const uint32_t s0 = (info & kInfoSwap0) ? 0xFFFFFFFFu : 0u;
  const uint32_t s1 = (info & (kInfoSwap0 << 1)) ? 0xFFFFFFFFu : 0u;
  uint32_t a = 0xFFFFFFFFu, c = 0xFFFFFFFFu;
#pragma unroll 1
  for (int k = 0; k < 5; ++k) {
    // edges v2 -> v0, v0 -> v1, v1 -> v2, v2 -> v3, v3 -> v0
    const int xu = k == 1 ? X[0] : (k == 2 ? X[1] : (k == 4 ? X[3] : X[2]));
    const int yu = k == 1 ? Y[0] : (k == 2 ? Y[1] : (k == 4 ? Y[3] : Y[2]));
    const int xv = k == 1 ? X[1] : (k == 2 ? X[2] : (k == 3 ? X[3] : X[0]));
    const int yv = k == 1 ? Y[1] : (k == 2 ? Y[2] : (k == 3 ? Y[3] : Y[0]));
    const int dx = xv - xu, dy = yv - yu;
    const bool owned = dy < 0 || (dy == 0 && dx > 0);
    const long long e = ((long long)dx * (Py - yu) - (long long)dy * (Px - xu) - (owned ? 0 : 1)) >> 8;
    const int r = (int)max(min(e, 1LL << 28), -(1LL << 28));
    uint32_t f = 0;
#pragma unroll
    for (int ly = 0; ly < kHbH; ++ly) f |= row_cover(r + ly * dx, -dy) << (ly * kHbW);
    if (k < 3) a &= f ^ s0;
    if (k == 0) c = ~(f ^ s1);
    if (k > 2) c &= f ^ s1;
  }
  m0 = (info & kInfoTri0) ? a : 0u;
  m1 = (info & kInfoTri1) ? c : 0u;
}

// ---- k_raster's shared memory ----------------------------------------------------------------
// Per warp: a ring of covering triangles waiting for a batch, and the records of the batch the
// fragment loop reads, one 16-byte array per field so that a slot's fields lie at one address
// plus constants and eight neighbouring slots never share a bank.
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
__host__ __device__ constexpr size_t batch_smem_warp(bool vtx, bool bwd, bool lit) {
  return kPendCap * sizeof(uint2) + sizeof(BatchGeo) + (size_t)batch_cols(vtx, lit) * 32 * sizeof(float4) +
         (bwd ? 32 * sizeof(float4) : 0);
}
__host__ __device__ constexpr size_t raster_smem_bytes(bool vtx, bool bwd = false, bool lit = false) {
  return (size_t)kRasterWarps * batch_smem_warp(vtx, bwd, lit);
}

// HASH: the variant that also writes the per-pixel coverage hash (a test output); the
// others carry no code or registers for it. ATH: the alpha-threshold variant (forward
// only, no hash), which also skips candidate quads that cannot reach in front of any
// pixel of the half-block still blending. LIT: the colour-carrying variant that also
// shades lit views (per-vertex normals, one directional light).
template <int K, bool VTX, bool BWD, bool HASH, bool ATH = false, bool LIT = false>
__global__ __launch_bounds__(kRasterThreads, LR_RASTER_MIN_BLOCKS) void k_raster(Ws ws) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool kCarry = VTX || K == 1;   // the sorter carries each fragment's colour
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lx = lane & (kHbW - 1), ly = lane >> 3;
  unsigned char* wbase = smem + (size_t)warp * batch_smem_warp(VTX, BWD, LIT);
  uint2* pend = reinterpret_cast<uint2*>(wbase);
  BatchGeo& geo = *reinterpret_cast<BatchGeo*>(wbase + kPendCap * sizeof(uint2));
  float4* qc = reinterpret_cast<float4*>(wbase + kPendCap * sizeof(uint2) + sizeof(BatchGeo));
  float4* agg = qc + batch_cols(VTX, LIT) * 32;
  // a batch blended in stream order keeps its sort keys where the others keep ea
  unsigned long long* dkey = reinterpret_cast<unsigned long long*>(&geo);
  if (ws.ctrl->error == LR_ERR_OVERFLOW) return;
  const unsigned long long nitems = ws.ctrl->raster_items;
  unsigned long long frag_total = 0;

  for (;;) {
    unsigned long long item = 0;
    if (lane == 0) item = atomicAdd(&ws.ctrl->raster_head, 1ull);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= nitems) break;
    const int lg = ws.bin_log2, hl = bin_hb_log2(lg), cl = bin_hb_cols_log2(lg);
    const int bin_g = (int)ws.bin_order[item >> hl];
    const int hb = (int)(item & ((1u << hl) - 1u));
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
    const bool flat_view = V.color_mode == LR_COLOR_FLAT;
    const bool hashing = HASH && V.hash != nullptr;
    const int Ox = 256 * ox + 128, Oy = 256 * oy + 128;   // first pixel centre, 1/256 px
    // lit views: unit direction toward the light and the ambient term
    const float4 light = LIT ? make_float4(V.light[0], V.light[1], V.light[2], V.light[3])
                             : make_float4(0.f, 0.f, 0.f, 0.f);

    PixelState<K, kCarry, BWD, ATH> st;
    st.init();
    st.gp.grad = nullptr;
    st.gp.agg = agg;
    if (BWD && pix_ok) {
      const long long pidx = (long long)py * V.width + px;
      const float4 gq = reinterpret_cast<const float4*>(ws.grad_out)[pidx];
      const float4 fq = reinterpret_cast<const float4*>(ws.fwd)[pidx];
      st.gp.gr = gq.x; st.gp.gg = gq.y; st.gp.gb = gq.z; st.gp.ga = gq.w;
      st.gp.fr = fq.x; st.gp.fg = fq.y; st.gp.fb = fq.z; st.gp.fT = 1.0f - fq.w;
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
    if (BWD) {
      st.init();
      st.flagged = pre_flagged;
      st.gp.grad = (pass == 1 && pix_ok) ? ws.grad_col : nullptr;
      cnt = 0;
      hsh = 0;
    }
    // ---- 1. the half-block's candidates: set bits of its bitmap row, in sorted order ----
    const uint32_t* row = hb_row(ws, off, bin_g, n, hb);
    const int nw = (n + 31) >> 5;
    const uint32_t* ref_lo = reinterpret_cast<const uint32_t*>(ws.refs + off);   // low words
    int g = -32, r0 = 0;          // bitmap window and position in it
    BitRounds br;
    br.total = 0;
    int head = 0, tail = 0;       // pending ring
    bool ordered = !HASH && !BWD; // everything so far was blended in stream order
    for (;;) {
      // ---- 2. coverage masks of 32 candidates, one quad per lane, until a batch is full ---
      while (tail - head < 32) {
        if (r0 >= br.total) {
          g += 32;
          if (g >= nw) break;
          br.prepare(g + lane < nw ? __ldg(row + g + lane) : 0u, lane);
          r0 = 0;
          continue;
        }
        const int j = br.get(r0, lane);
        r0 += 32;
        const bool in = j >= 0;
        const uint32_t rec = in ? ~ref_lo[2 * (32 * g + j)] : 0u;
        bool skip = !in;
        if (ATH) {
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
          const int4* rp = ws.rec + 4ull * rec;
          const int4 r0v = __ldg(rp), r1v = __ldg(rp + 1);
          const int2 fl = __ldg(reinterpret_cast<const int2*>(rp + 3) + 1);   // info, record flags
          const int X[4] = {r0v.x, r0v.z, r1v.x, r1v.z}, Y[4] = {r0v.y, r0v.w, r1v.y, r1v.w};
          const uint32_t info = (uint32_t)fl.x;
          if (fl.y & (int)kRecSmall) quad_masks_small(X, Y, info, Ox, Oy, ma, mb);
          else quad_masks_any(X, Y, info, Ox, Oy, ma, mb);
          ida = 2u * (uint32_t)(rec - V.quad_base);
          idb = ida + 1u;
          if (flat_view && (info & kInfoFlatDepth)) {
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
          const float q0 = __ldg(reinterpret_cast<const float*>(ws.rec + 4ull * (uint32_t)(V.quad_base + (id >> 1)) + 2));
          qc[lane] = __ldg(reinterpret_cast<const float4*>(V.col) + (id >> 1));
          dkey[lane] = ((unsigned long long)__float_as_uint(q0) << 32) | id;
        }
      } else if (e < nb) {
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
        const float qb = sw ? q2 : q1, qc2 = sw ? q1 : q2;
        geo.kq[lane] = make_float4(R.q[0], __fsub_rn(qb, R.q[0]), __fsub_rn(qc2, R.q[0]), t ? R.inv[1] : R.inv[0]);
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
          // corner colours times 1/w, as (c0, c1 - c0, c2 - c0) for the fragment's
          // c0 + l1 (c1 - c0) + l2 (c2 - c0); lit: the same for the normals
          const float4 c0 = __ldg(cv + (size_t)cs * vi.x), c1 = __ldg(cv + (size_t)cs * vb), c2 = __ldg(cv + (size_t)cs * vc);
          const float qa = R.q[0];
          const float4 p0 = make_float4(qa * c0.x, qa * c0.y, qa * c0.z, qa * c0.w);
          qc[lane] = p0;
          qc[32 + lane] = make_float4(qb * c1.x - p0.x, qb * c1.y - p0.y, qb * c1.z - p0.z, qb * c1.w - p0.w);
          qc[64 + lane] = make_float4(qc2 * c2.x - p0.x, qc2 * c2.y - p0.y, qc2 * c2.z - p0.z, qc2 * c2.w - p0.w);
          if (LIT && lit) {
            const float4 n0 = __ldg(cv + 2ull * vi.x + 1), n1 = __ldg(cv + 2ull * vb + 1), n2 = __ldg(cv + 2ull * vc + 1);
            const float4 o0 = make_float4(qa * n0.x, qa * n0.y, qa * n0.z, 0.f);
            qc[96 + lane] = o0;
            qc[128 + lane] = make_float4(qb * n1.x - o0.x, qb * n1.y - o0.y, qb * n1.z - o0.z, 0.f);
            qc[160 + lane] = make_float4(qc2 * n2.x - o0.x, qc2 * n2.y - o0.y, qc2 * n2.z - o0.z, 0.f);
          }
        } else if (kCarry) {
          qc[lane] = __ldg(reinterpret_cast<const float4*>(V.col) + jl);
        }
      }
      // ---- 4. transpose: lane = pixel, bit L = covered by the triangle in slot L -----------
      uint32_t m = warp_transpose32(mk, lane);   // (its shuffles also order the slots' writes below)
      __syncwarp();
      if (!pix_ok) m = 0;
      cnt += __popc(m);
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
        if (lastp < 32u) st.last = dkey[lastp];
      } else {
        if (ordered) {
          // the sorter starts here; with a transparent held fragment at the last key blended
          // (K = 1), so that its first eviction keeps that key
          ordered = false;
          if (PixelState<K, kCarry, BWD, ATH>::kNullSlot) st.s[0] = st.last;
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
            float4 col = make_float4(0.f, 0.f, 0.f, 0.f);
            if (kCarry) col = qc[p];
            if (VTX && !flat_view) {
              // perspective-correct colour: interpolated (c / w) divided by the
              // interpolated 1/w, which is the depth key
              const float rk = rcp_approx(key);
              const float4 d1 = qc[32 + p], d2 = qc[64 + p];
              col.x = (col.x + l1 * d1.x + l2 * d2.x) * rk;
              col.y = (col.y + l1 * d1.y + l2 * d2.y) * rk;
              col.z = (col.z + l1 * d1.z + l2 * d2.z) * rk;
              col.w = (col.w + l1 * d1.w + l2 * d2.w) * rk;
              if (LIT && V.color_mode == LR_COLOR_LIT) {
                // the interpolated normal (times the interpolated 1/w, which only scales
                // it); two-sided Lambert term plus ambient on RGB
                const float4 n0 = qc[96 + p], n1 = qc[128 + p], n2 = qc[160 + p];
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
            }
            st.insert(sk, col, V);
          }
        };
        while (m) frag_step();
      }
      __syncwarp();
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
    if (!st.flagged) st.flush(V);
    if (pix_ok) {
      const long long pidx = (long long)py * V.width + px;
      if (!BWD && V.cnt) V.cnt[pidx] = cnt;
      if (!BWD && hashing) V.hash[pidx] = hsh;
      if (!st.flagged) {
        if (!BWD) write_pixel(V, pidx, st.r, st.g, st.b, st.T);
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
                                (int)raster_smem_bytes(VTX, BWD, LIT));                       \
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
        raster_smem_bytes(true, false, true));                                                \
    if (e != cudaSuccess) return e;                                                           \
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_flat, k_raster<KK, false, false, false>, \
                                                      kRasterThreads, raster_smem_bytes(false)); \
    if (e != cudaSuccess) return e;                                                           \
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_bwd, k_raster<KK, false, true, false>, \
                                                      kRasterThreads, raster_smem_bytes(false, true)); \
    if (e != cudaSuccess) return e;                                                           \
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_vtx, k_raster<KK, true, false, false>, \
                                                         kRasterThreads, raster_smem_bytes(true)); \
  }                                                                                           \
  /* mode: 0 flat colours, 1 colours in the sorter, 2 backward; + 4: coverage hash;        \
     + 8: alpha threshold (modes 8 and 9 only); 17: colours in the sorter with lit views */   \
  cudaError_t launch_raster_##KK(int mode, const Ws& ws, int grid, cudaStream_t st) {         \
    const size_t sf = raster_smem_bytes(false), sv = raster_smem_bytes(true);                 \
    /* a plain launch: with programmatic serialisation the persistent CTAs, placed early  \
       next to the bin sort's, measured slower on the particle frame */                       \
    switch (mode) {                                                                           \
      case 1: k_raster<KK, true, false, false><<<grid, kRasterThreads, sv, st>>>(ws); break;  \
      case 2: k_raster<KK, false, true, false><<<grid, kRasterThreads, raster_smem_bytes(false, true), st>>>(ws); break; \
      case 4: k_raster<KK, false, false, true><<<grid, kRasterThreads, sf, st>>>(ws); break;  \
      case 5: k_raster<KK, true, false, true><<<grid, kRasterThreads, sv, st>>>(ws); break;   \
      case 8: k_raster<KK, false, false, false, true><<<grid, kRasterThreads, sf, st>>>(ws); break; \
      case 9: k_raster<KK, true, false, false, true><<<grid, kRasterThreads, sv, st>>>(ws); break; \
      case 17:                                                                                \
        k_raster<KK, true, false, false, false, true>                                         \
            <<<grid, kRasterThreads, raster_smem_bytes(true, false, true), st>>>(ws);         \
        break;                                                                                \
      default: k_raster<KK, false, false, false><<<grid, kRasterThreads, sf, st>>>(ws); break; \
    }                                                                                         \
    return cudaGetLastError();                                                                \
  }                                                                                           \
  }
