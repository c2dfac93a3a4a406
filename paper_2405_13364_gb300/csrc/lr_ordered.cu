// lr_ordered.cu -- the rasteriser of the bins whose sorted list is every pixel's exact fragment
// order: bins that hold only flat-colour quads of one depth each (camera-facing sprites and
// particles; kBinDepths, set by the bin count). Fragments are blended as they come, without depth
// keys, sorter or exact path, in blocks of several pixels per lane. k_bin_scan puts these bins
// behind the others in bin_order; k_raster, launched next, takes the others. (As a branch of k_raster the two block
// forms cost its own loops registers: the layer frame 309 -> 317 us, mixed views at K = 3 743 ->
// 774.)
#include "lr_raster.cuh"

namespace lr {

// Bins that hold only flat-colour quads of one depth each: the bin's list, sorted by that depth with the tie
// rule, is every pixel's exact fragment order. A warp takes an 8x8 block, the half-blocks hb and
// hb_l below it, with two pixels per lane, one above the other: a record read from shared
// memory and a step of the loop serve both, and a quad that meets both half-blocks is gathered
// and masked once. (Blocks of two pixels per lane for quads of other depths measured slower than
// half-blocks, 340 against 317 us on the layer frame: the pixels' triangles differ too often for
// the second sorter's registers.) Bins of rectangles alone: box_block.
template <bool ATH>
__device__ __forceinline__ unsigned const_block(const int4* recs, const unsigned long long* refs, const ViewDev& V,
                                                const uint32_t* row_u, const uint32_t* row_l, int n, int ox, int oy, int lane,
                                                uint16_t* cand, uint2* pend, float4* qc) {
  const int px = ox + (lane & 7), py = oy + 2 * (lane >> 3);
  const bool ok_a = px < V.width && py < V.height, ok_b = px < V.width && py + 1 < V.height;
  const int Ox = 256 * ox + 128, Oy = 256 * oy + 128;
  const uint32_t* ref_lo = reinterpret_cast<const uint32_t*>(refs);   // low words
  const float4* colors = reinterpret_cast<const float4*>(V.col);
  const uint32_t quad_base = (uint32_t)V.quad_base;
  uint32_t* pend_j = reinterpret_cast<uint32_t*>(qc + 32);   // the ring's quads; pend: their masks
  PixelState<1, true, ATH> sa, sb;
  sa.init();
  sb.init();
  uint32_t cnt_a = 0, cnt_b = 0;
  const int nw = (n + 31) >> 5;
  int g = -32, r0 = 0, total = 0, head = 0, tail = 0;
  for (;;) {
    // masks of 32 candidates, one quad per lane, until a batch of covering quads is full
    while (tail - head < 32) {
      if (ATH && !__any_sync(0xffffffffu, (ok_a && sa.live()) || (ok_b && sb.live()))) break;   // all finished
      if (r0 >= total) {
        g += 32;
        if (g >= nw) break;
        total = list_bits(g + lane < nw ? (__ldg(row_u + g + lane) | __ldg(row_l + g + lane)) : 0u, lane, cand);
        r0 = 0;
        continue;
      }
      // first entry m, and for triangles that overlap (concave or crossed quads) a second one:
      // triangle 1 lies in front
      uint32_t m[2] = {0, 0}, m2[2] = {0, 0}, j = 0;
      if (r0 + lane < total) {
        const uint32_t rec = ~ref_lo[2 * (32 * g + (int)cand[r0 + lane])];
        int X[4], Y[4];
        load_rec_xy(recs, rec, X, Y);
        const int2 fl = __ldg(reinterpret_cast<const int2*>(recs + 4ull * rec + 3) + 1);   // info, record flags
        j = rec - quad_base;
        if (fl.y & (int)kRecSmall) quad_masks_small<8>(X, Y, (uint32_t)fl.x, Ox, Oy, m2, m);
        else quad_masks_any<8>(X, Y, (uint32_t)fl.x, Ox, Oy, m2, m);
        if (((m[0] & m2[0]) | (m[1] & m2[1])) == 0u) {
          m[0] |= m2[0]; m[1] |= m2[1];
          m2[0] = m2[1] = 0u;
        }
      }
      r0 += 32;
      const bool h1 = (m[0] | m[1]) != 0u, h2 = (m2[0] | m2[1]) != 0u;
      const unsigned b1 = __ballot_sync(0xffffffffu, h1), b2 = __ballot_sync(0xffffffffu, h2);
      const unsigned lt = (1u << lane) - 1u;
      int at = tail + __popc(b1 & lt) + __popc(b2 & lt);
      if (h1) {
        pend[at & (kPendCap - 1)] = make_uint2(m[0], m[1]);
        pend_j[at++ & (kPendCap - 1)] = j;
      }
      if (h2) {
        pend[at & (kPendCap - 1)] = make_uint2(m2[0], m2[1]);
        pend_j[at & (kPendCap - 1)] = j;
      }
      tail += __popc(b1) + __popc(b2);
      __syncwarp();
    }
    const int nb = min(32, tail - head);
    if (nb == 0) break;
    // entry 31 - L of the batch goes to lane and slot L: the highest set bit is the next
    uint2 k = make_uint2(0u, 0u);
    if (31 - lane < nb) {
      const int i = (head + 31 - lane) & (kPendCap - 1);
      k = pend[i];
      qc[lane] = __ldg(colors + pend_j[i]);
    }
    head += nb;
    uint32_t m_a = warp_transpose32(k.x, lane), m_b = warp_transpose32(k.y, lane);
    __syncwarp();
    if (!ok_a) m_a = 0;
    if (!ok_b) m_b = 0;
    cnt_a += __popc(m_a);
    cnt_b += __popc(m_b);
    while (m_a | m_b) {
      if (ATH) {
        if (!sa.live()) m_a = 0;
        if (!sb.live()) m_b = 0;
        if (!(m_a | m_b)) break;
      }
      const int p = 31 - __clz(m_a | m_b);
      const uint32_t bit = 1u << p;
      const float4 c = qc[p];
      if (m_a & bit) sa.blend_direct(c);
      if (m_b & bit) sb.blend_direct(c);
      m_a &= ~bit;
      m_b &= ~bit;
    }
    __syncwarp();
  }
  if (V.xmask && lane < 2 && oy + lane * kHbH < V.height) {
    const uint32_t hbw = ((uint32_t)V.width + kHbW - 1) / kHbW;
    V.xmask[((uint32_t)oy / kHbH + lane) * hbw + (uint32_t)ox / kHbW] = 0u;
  }
  const long long pa = (long long)py * V.width + px;
  if (ok_a) {
    if (V.cnt) V.cnt[pa] = cnt_a;
    write_pixel(V, pa, sa.r, sa.g, sa.b, sa.T);
  }
  if (ok_b) {
    if (V.cnt) V.cnt[pa + V.width] = cnt_b;
    write_pixel(V, pa + V.width, sb.r, sb.g, sb.b, sb.T);
  }
  return cnt_a + cnt_b;
}

// A bin of such quads that are axis-parallel rectangles too (kRecBox: particles, upright
// billboards). A warp takes 16x8 pixels, four half-blocks, with 2x2 pixels per lane. Coverage is
// separable: a candidate's columns and rows are one word, one transpose across the warp turns 32
// of them into a word per column and per row, and a pixel's candidates are the intersection of
// two. The loop runs over the candidates of a lane's four pixels together, so that its overhead and
// the colour's load serve up to four fragments. Records' corners and colours are loaded one round
// ahead, the references two. Nearly every candidate covers a pixel, so there is no ring.
// 2M particles at 1920x1080: 274 us by 8x8 blocks with a mask per candidate, 295 us so as a branch of
// k_raster.
// The four pixels of a lane, (cx, cy), (cx + 1, cy) and the two below.
template <bool ATH>
struct BoxPixels {
  PixelState<1, true, ATH> st[4];
  uint32_t cnt[4];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      st[i].init();
      cnt[i] = 0;
    }
  }
};
// Blends the references of bitmap words [w0, w1).
template <bool ATH>
__device__ __forceinline__ void box_block(BoxPixels<ATH>& P, const int4* recs, const unsigned long long* refs, const ViewDev& V,
                                          const uint32_t* row_u, const uint32_t* row_l, int nw, int w0, int w1, int ox,
                                          int oy, int lane, uint16_t* cand, float4* qc) {
  const int cx = 2 * (lane & 7), cy = 2 * (lane >> 3);
  const uint32_t* ref_lo = reinterpret_cast<const uint32_t*>(refs);   // low words
  const float4* colors = reinterpret_cast<const float4*>(V.col);
  const uint32_t quad_base = (uint32_t)V.quad_base;
  // (row_u, row_l: the left half-blocks of the upper and the lower pair)
  int g = w0 - 32, r0 = 0, total = 0;
  uint32_t words = 0;                 // the next window's bitmap words
  auto load_words = [&](int w) {
    words = w < w1 ? (__ldg(row_u + w) | __ldg(row_u + nw + w) | __ldg(row_l + w) | __ldg(row_l + nw + w)) : 0u;
  };
  load_words(g + 32 + lane);
  constexpr uint32_t kNone = 0xFFFFFFFFu;
  auto next_refs = [&](uint32_t& rec) {
    rec = kNone;
    while (r0 >= total) {
      g += 32;
      if (g >= w1) return false;
      const uint32_t cur = words;
      load_words(g + 32 + lane);
      total = list_bits(cur, lane, cand);
      r0 = 0;
    }
    // candidate 31 - L of the round in lane and slot L: the highest set bit is the next
    const int at = r0 + 31 - lane;
    if (at < total) rec = ~ref_lo[2 * (32 * g + (int)cand[at])];
    r0 += 32;
    return true;
  };
  uint32_t rec = kNone, rec_n;
  int4 xy = make_int4(0, 0, 0, 0);    // opposite corners
  float4 col = make_float4(0.f, 0.f, 0.f, 0.f);
  bool has = false, has_n = next_refs(rec_n);
  auto advance = [&]() {
    rec = rec_n;
    has = has_n;
    if (rec != kNone) {
      const int2 a = __ldg(reinterpret_cast<const int2*>(recs + 4ull * rec));
      const int2 b = __ldg(reinterpret_cast<const int2*>(recs + 4ull * rec + 1));
      xy = make_int4(a.x, a.y, b.x, b.y);
      col = __ldg(colors + (rec - quad_base));
    }
    if (has) has_n = next_refs(rec_n);
  };
  advance();
  while (has) {
    if (ATH) {   // all finished
      bool live = false;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        live |= ox + cx + (i & 1) < V.width && oy + cy + (i >> 1) < V.height && P.st[i].live();
      if (!__any_sync(0xffffffffu, live)) break;
    }
    // under the top-left rule a centre is covered iff xmin <= x < xmax and ymin <= y < ymax
    const int c0 = min(max(((min(xy.x, xy.z) + 127) >> 8) - ox, 0), 16), c1 = min(max(((max(xy.x, xy.z) + 127) >> 8) - ox, 0), 16);
    const int y0 = min(max(((min(xy.y, xy.w) + 127) >> 8) - oy, 0), 8), y1 = min(max(((max(xy.y, xy.w) + 127) >> 8) - oy, 0), 8);
    const uint32_t word = rec != kNone ? (0xFFFFu & (0xFFFFu << c0) & ~(0xFFFFFFFFu << c1)) |
                                             ((0xFFu & (0xFFu << y0) & ~(0xFFFFFFFFu << y1)) << 16)
                                       : 0u;
    qc[lane] = col;
    advance();
    // lane x < 16: the candidates covering column x; lane 16 + y: row y
    const uint32_t t = warp_transpose32(word, lane);
    const uint32_t mx0 = __shfl_sync(0xffffffffu, t, cx), mx1 = __shfl_sync(0xffffffffu, t, cx + 1);
    const uint32_t my0 = __shfl_sync(0xffffffffu, t, 16 + cy), my1 = __shfl_sync(0xffffffffu, t, 17 + cy);
    __syncwarp();
    const uint32_t m[4] = {mx0 & my0, mx1 & my0, mx0 & my1, mx1 & my1};
#pragma unroll
    for (int i = 0; i < 4; ++i) P.cnt[i] += __popc(m[i]);
    uint32_t u = (mx0 | mx1) & (my0 | my1);
    while (u) {
      const int p = 31 - __clz(u);
      const uint32_t bit = 1u << p;
      const float4 c = qc[p];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if ((m[i] & bit) && P.st[i].live()) P.st[i].blend_direct(c);
      u ^= bit;
    }
    __syncwarp();
  }
}

// Writes pixel (px, py) of the block, if it is in the image, and returns its fragments.
__device__ __forceinline__ uint32_t box_write(const ViewDev& V, int px, int py, float r, float g, float b, float T, uint32_t cnt) {
  if (px >= V.width || py >= V.height) return 0u;
  const long long pidx = (long long)py * V.width + px;
  if (V.cnt) V.cnt[pidx] = cnt;
  write_pixel(V, pidx, r, g, b, T);
  return cnt;
}
// The block's half-blocks have no pixel for the exact path.
__device__ __forceinline__ void box_xmask(const ViewDev& V, int ox, int oy, int lane) {
  const int x = ox + (lane & 1) * kHbW, y = oy + (lane >> 1) * kHbH;
  if (V.xmask && lane < 4 && x < V.width && y < V.height)
    V.xmask[((uint32_t)y / kHbH) * (((uint32_t)V.width + kHbW - 1) / kHbW) + (uint32_t)x / kHbW] = 0u;
}

constexpr size_t kOrderedSmemWarp = win_refs(false) * sizeof(uint16_t) + kPendCap * sizeof(uint2) +
                                   32 * sizeof(float4) + kPendCap * sizeof(uint32_t);
// (two CTAs per SM 266 us on the 2M particles, three 209, four 213 and 45 instead of 41 on four small
// mixed views, five 262)
#ifndef LR_ORDERED_MIN_BLOCKS
#define LR_ORDERED_MIN_BLOCKS 3
#endif

// One 16x8 block of a bin (an item of the queue).
struct OrderedBlock {
  const ViewDev* V;          // null: nothing to do
  const unsigned long long* refs;
  const uint32_t *row_u, *row_l;
  int n, ox, oy;
  bool shapes;               // the bin holds other shapes than axis-parallel rectangles
  bool bytes;                // the view wants 8-bit values
  __device__ __forceinline__ OrderedBlock(const Ws& ws, uint32_t n_general, uint32_t item) {
    const int lg = ws.bin_log2, bl = bin_hb_log2(lg) - 2, cl = bin_hb_cols_log2(lg) - 1, cols = bin_hb_cols(lg);
    const int bin_g = (int)ws.bin_order[n_general + (item >> bl)], blk = (int)(item & ((1u << bl) - 1u));
    V = ws.views + view_of_bin(ws.views, ws.n_views, bin_g);
    const int b = bin_g - V->bin_base, bx = blk & ((1 << cl) - 1), by = blk >> cl;
    ox = ((b % V->nbx) << lg) + 16 * bx;
    oy = ((b / V->nbx) << lg) + 8 * by;
    const uint32_t off = ws.bin_off[bin_g];
    n = (int)(ws.bin_off[bin_g + 1] - off);
    refs = ws.refs + off;
    const int hb = 2 * by * cols + 2 * bx;   // upper left half-block
    row_u = hb_row(ws, off, bin_g, n, hb);
    row_l = hb_row(ws, off, bin_g, n, hb + cols);
    shapes = (ws.bin_cursor[bin_g] & kBinShapes) != 0u;
    bytes = V->out8 != nullptr;
    if (ox >= V->width || oy >= V->height || !tile_owned(*V, ox, oy)) V = nullptr;
  }
};

// Persistent CTAs over the 16x8 blocks of these bins, longest lists first. Bins with long lists
// (n_ordered_long): the CTA's eight warps take an eighth of a block's list each and their composites are
// combined in order (consecutive segments combine as C1 + T1 C2, T1 T2): one warp through a dense
// bin's list took longer than all the rest of the frame (400,000 particles at 960x540: 168 us
// against 61 us, 2M at 1920x1080 295 against 207; cut from 4096 references on they took 231, since
// the longest uncut lists then start late). Then a warp per block. With the alpha
// threshold, whose stop is defined on the running product, and for views with 8-bit values, whose
// rounding would show where a list was cut, always a warp per block.
template <bool ATH>
__global__ __launch_bounds__(kRasterThreads, LR_ORDERED_MIN_BLOCKS) void k_raster_ordered(Ws ws) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint32_t s_item;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* wbase = smem + (size_t)warp * kOrderedSmemWarp;
  uint16_t* cand = reinterpret_cast<uint16_t*>(wbase);
  uint2* pend = reinterpret_cast<uint2*>(wbase + win_refs(false) * sizeof(uint16_t));
  float4* qc = reinterpret_cast<float4*>(pend + kPendCap);
  const bool run = ws.ctrl->error != LR_ERR_OVERFLOW;
  const uint32_t n_general = ws.ctrl->n_general;
  const int bl = bin_hb_log2(ws.bin_log2) - 2;
  const uint32_t nitems = run ? ((uint32_t)ws.total_bins - n_general) << bl : 0u;   // (a batch has less than 2^32 pixels)
  const uint32_t nlong = ATH || !run ? 0u : ws.ctrl->n_ordered_long << bl;
  unsigned long long frag_total = 0;
  auto draw = [&]() { return (uint32_t)min(atomicAdd(&ws.ctrl->ordered_head, 1ull), 0xFFFFFFF0ull); };
  auto whole_block = [&](const OrderedBlock& B) {   // rectangles, by one warp
    const int nw = (B.n + 31) >> 5;
    BoxPixels<ATH> P;
    P.init();
    box_block<ATH>(P, ws.rec, B.refs, *B.V, B.row_u, B.row_l, nw, 0, nw, B.ox, B.oy, lane, cand, qc);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      frag_total += box_write(*B.V, B.ox + 2 * (lane & 7) + (i & 1), B.oy + 2 * (lane >> 3) + (i >> 1), P.st[i].r, P.st[i].g, P.st[i].b,
                              P.st[i].T, P.cnt[i]);
    box_xmask(*B.V, B.ox, B.oy, lane);
  };
  uint32_t item = 0xFFFFFFFFu;         // warp 0: the first item past the CTA's
  while (nlong) {
    if (threadIdx.x == 0) s_item = draw();
    __syncthreads();
    item = s_item;
    if (item >= nlong) break;
    const OrderedBlock B(ws, n_general, item);
    const uint32_t blk = item & ((1u << bl) - 1u);
    if (!B.shapes && B.bytes) {
      // eight blocks of the bin (two of a 16-pixel bin), a warp each
      const uint32_t it = item + warp;
      if ((blk & 7u) == 0u && it >> bl == item >> bl) {
        const OrderedBlock W(ws, n_general, it);
        if (W.V) whole_block(W);
      }
    } else if (B.V && !B.shapes) {
      const int nw = (B.n + 31) >> 5, per = (nw + kRasterWarps - 1) / kRasterWarps;
      BoxPixels<ATH> P;
      P.init();
      box_block<ATH>(P, ws.rec, B.refs, *B.V, B.row_u, B.row_l, nw, warp * per, min(nw, (warp + 1) * per), B.ox, B.oy, lane, cand, qc);
      // the warp's composite in place of its candidates, its counts in place of the ring
      float4* part = reinterpret_cast<float4*>(cand);
      uint32_t* pcnt = reinterpret_cast<uint32_t*>(pend);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        part[32 * i + lane] = make_float4(P.st[i].r, P.st[i].g, P.st[i].b, P.st[i].T);
        pcnt[32 * i + lane] = P.cnt[i];
      }
      __syncthreads();
      if (threadIdx.x < 128) {
        float r = 0.f, g = 0.f, b = 0.f, T = 1.f;
        uint32_t c = 0;
#pragma unroll
        for (int w = 0; w < kRasterWarps; ++w) {
          const unsigned char* wb = smem + (size_t)w * kOrderedSmemWarp;
          const float4 p = reinterpret_cast<const float4*>(wb)[threadIdx.x];
          r += T * p.x;
          g += T * p.y;
          b += T * p.z;
          T *= p.w;
          c += reinterpret_cast<const uint32_t*>(wb + win_refs(false) * sizeof(uint16_t))[threadIdx.x];
        }
        const int px = B.ox + 2 * (lane & 7) + (warp & 1), py = B.oy + 2 * (lane >> 3) + (warp >> 1);
        frag_total += box_write(*B.V, px, py, r, g, b, T, c);
        if (warp == 0) box_xmask(*B.V, B.ox, B.oy, lane);
      }
    } else if (B.shapes && (blk & 3u) == 0u) {
      // four blocks of the bin (two of a 16-pixel bin) as eight 8x8 blocks, a warp each
      const uint32_t it = item + (warp >> 1);
      if (it >> bl == item >> bl) {
        const OrderedBlock W(ws, n_general, it);
        const int h = warp & 1, nw = (W.n + 31) >> 5;
        if (W.V && W.ox + 8 * h < W.V->width)
          frag_total += const_block<ATH>(ws.rec, W.refs, *W.V, W.row_u + h * nw, W.row_l + h * nw, W.n, W.ox + 8 * h, W.oy, lane, cand, pend, qc);
      }
    }
    __syncthreads();
  }
  for (bool drawn = nlong != 0u && warp == 0; run; drawn = false) {
    if (!drawn) {
      uint32_t k = 0;
      if (lane == 0) k = draw();
      item = __shfl_sync(0xffffffffu, k, 0);
    }
    if (item >= nitems) break;
    const OrderedBlock B(ws, n_general, item);
    if (!B.V) continue;
    const int nw = (B.n + 31) >> 5;
    if (!B.shapes) {
      whole_block(B);
    } else {
#pragma unroll 1
      for (int h = 0; h < 2 && B.ox + 8 * h < B.V->width; ++h)
        frag_total += const_block<ATH>(ws.rec, B.refs, *B.V, B.row_u + h * nw, B.row_l + h * nw, B.n, B.ox + 8 * h, B.oy, lane, cand, pend, qc);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) frag_total += __shfl_xor_sync(0xffffffffu, frag_total, o);
  if (lane == 0 && frag_total) atomicAdd(&ws.ctrl->fragments, frag_total);
}

cudaError_t prepare_ordered(int* blocks_per_sm) {
  const int smem = (int)(kRasterWarps * kOrderedSmemWarp);
  cudaError_t e = cudaFuncSetAttribute(k_raster_ordered<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_raster_ordered<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_raster_ordered<false>, kRasterThreads, smem);
}

cudaError_t launch_ordered(const Ws& ws, int grid, cudaStream_t st, bool pdl) {
  const size_t smem = kRasterWarps * kOrderedSmemWarp;
  if (ws.t_min > 0.0f) return launch_pdl(pdl, k_raster_ordered<true>, dim3(grid), dim3(kRasterThreads), smem, st, ws);
  return launch_pdl(pdl, k_raster_ordered<false>, dim3(grid), dim3(kRasterThreads), smem, st, ws);
}

}  // namespace lr
