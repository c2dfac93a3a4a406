// lr_ordered.cu -- the rasteriser of the bins whose sorted list is every pixel's exact fragment
// order: bins that hold only flat-colour quads of one depth each (camera-facing sprites and
// particles; kBinDepths, set by the bin count). Fragments are blended as they come, without depth
// keys, sorter or exact path, in blocks of one to four pixels per lane. k_bin_scan puts these bins
// behind the others in bin_order; k_raster, launched next, takes the others. (As branches of k_raster the
// block forms cost its own loops registers: the layer frame 309 -> 317 us, mixed views at K = 3 743 ->
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
// billboards). A warp takes 16x8 pixels, four half-blocks, with 2x2 pixels per lane (NP = 4), an 8x8
// block with 1x2 (NP = 2) or a half-block (NP = 1). Coverage is separable: a candidate's columns and
// rows are one word, one transpose across the warp turns 32 of them into a word per column and per
// row, and a pixel's candidates are the intersection of two. The loop runs over the candidates of a
// lane's pixels together, so that its overhead and the colour's load serve up to four fragments.
// Records' corners and colours are loaded one round ahead, the references two (further ahead measured
// no faster). Nearly every candidate covers a pixel, so there is no ring.
template <bool ATH, int NP>
struct BoxPixels {
  PixelState<1, true, ATH> st[NP];
  uint32_t cnt[NP];
  // the lane's pixel i in the block
  static __device__ __forceinline__ int px(int lane, int i) { return NP == 4 ? 2 * (lane & 7) + (i & 1) : lane & 7; }
  static __device__ __forceinline__ int py(int lane, int i) {
    return NP == 4 ? 2 * (lane >> 3) + (i >> 1) : (NP == 2 ? 2 * (lane >> 3) + i : lane >> 3);
  }
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      st[i].init();
      cnt[i] = 0;
    }
  }
};
// With this many candidates of a round on one lane, the round's 32 colours are all read in turn, by the
// whole warp from one address and ahead of their use, instead of each lane finding its own: no
// chain from bit search to load to blend. 2M particles at 1920x1080: 264 us without for NP = 1, 235 so;
// 225 and 205 for NP = 2. (Where a lane has four pixels, too few of the 32 meet any.)
__host__ __device__ constexpr int box_dense(int np) { return np == 1 ? 10 : 14; }
// Blends the bin's references that the bitmap rows list: row_u and the one behind it the upper two
// half-blocks, row_l and the one behind it the lower two; NP = 2: row_u and row_l; NP = 1: row_u.
template <bool ATH, int NP>
__device__ __forceinline__ void box_block(BoxPixels<ATH, NP>& P, const int4* recs, const unsigned long long* refs, const ViewDev& V,
                                          const uint32_t* row_u, const uint32_t* row_l, int nw, int ox, int oy, int lane,
                                          uint16_t* cand, float4* qc) {
  constexpr int BW = NP == 4 ? 16 : 8, BH = NP == 1 ? 4 : 8;
  const int cx = P.px(lane, 0), cy = P.py(lane, 0);
  const uint32_t* ref_lo = reinterpret_cast<const uint32_t*>(refs);   // low words
  const float4* colors = reinterpret_cast<const float4*>(V.col);
  const uint32_t quad_base = (uint32_t)V.quad_base;
  int g = -32, r0 = 0, total = 0;
  uint32_t words = 0;                 // the next window's bitmap words
  auto load_words = [&](int w) {
    words = 0u;
    if (w >= nw) return;
    words = __ldg(row_u + w);
    if (NP > 1) words |= __ldg(row_l + w);
    if (NP == 4) words |= __ldg(row_u + nw + w) | __ldg(row_l + nw + w);
  };
  load_words(g + 32 + lane);
  constexpr uint32_t kNone = 0xFFFFFFFFu;
  auto next_refs = [&](uint32_t& rec) {
    rec = kNone;
    while (r0 >= total) {
      g += 32;
      if (g >= nw) return false;
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
      const Int8 a = ldg32(recs + 4ull * rec);
      xy = make_int4(a.v[0], a.v[1], a.v[4], a.v[5]);
      col = __ldg(colors + (rec - quad_base));
    }
    if (has) has_n = next_refs(rec_n);
  };
  advance();
  while (has) {
    if (ATH) {   // all finished
      bool live = false;
#pragma unroll
      for (int i = 0; i < NP; ++i) live |= ox + P.px(lane, i) < V.width && oy + P.py(lane, i) < V.height && P.st[i].live();
      if (!__any_sync(0xffffffffu, live)) break;
    }
    // under the top-left rule a centre is covered iff xmin <= x < xmax and ymin <= y < ymax
    const int c0 = min(max(((min(xy.x, xy.z) + 127) >> 8) - ox, 0), BW), c1 = min(max(((max(xy.x, xy.z) + 127) >> 8) - ox, 0), BW);
    const int y0 = min(max(((min(xy.y, xy.w) + 127) >> 8) - oy, 0), BH), y1 = min(max(((max(xy.y, xy.w) + 127) >> 8) - oy, 0), BH);
    constexpr uint32_t kCols = (1u << BW) - 1u, kRows = (1u << BH) - 1u;
    const uint32_t word = rec != kNone ? (kCols & (kCols << c0) & ~(0xFFFFFFFFu << c1)) |
                                             ((kRows & (kRows << y0) & ~(0xFFFFFFFFu << y1)) << BW)
                                       : 0u;
    qc[lane] = col;
    advance();
    // lane x < BW: the candidates covering column x; lane BW + y: row y
    const uint32_t t = warp_transpose32(word, lane);
    const uint32_t mx0 = __shfl_sync(0xffffffffu, t, cx), mx1 = NP == 4 ? __shfl_sync(0xffffffffu, t, cx + 1) : mx0;
    const uint32_t my0 = __shfl_sync(0xffffffffu, t, BW + cy), my1 = NP > 1 ? __shfl_sync(0xffffffffu, t, BW + cy + 1) : my0;
    __syncwarp();
    uint32_t m[NP], u = 0u;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      m[i] = (NP == 4 && (i & 1) ? mx1 : mx0) & ((NP == 4 ? i >> 1 : i) ? my1 : my0);
      u |= m[i];
      P.cnt[i] += __popc(m[i]);
    }
    if (NP <= 2 && !ATH && __reduce_max_sync(0xffffffffu, __popc(u)) >= box_dense(NP)) {
#pragma unroll
      for (int p = 31; p >= 0; --p) {
        const float4 c = qc[p];
#pragma unroll
        for (int i = 0; i < NP; ++i)
          if (m[i] & (1u << p)) P.st[i].blend_direct(c);
      }
      u = 0u;
    }
    while (u) {
      const int p = 31 - __clz(u);
      const uint32_t bit = 1u << p;
      const float4 c = qc[p];
#pragma unroll
      for (int i = 0; i < NP; ++i)
        if ((m[i] & bit) && P.st[i].live()) P.st[i].blend_direct(c);
      u ^= bit;
    }
    __syncwarp();
  }
}

constexpr size_t kOrderedSmemWarp = win_refs(false) * sizeof(uint16_t) + kPendCap * sizeof(uint2) +
                                   32 * sizeof(float4) + kPendCap * sizeof(uint32_t);

// A bin as the queue's items see it.
struct OrderedBin {
  const ViewDev* V;
  const unsigned long long* refs;
  const uint32_t* rows;      // of its bitmap, nw words each
  int n, nw, x0, y0;
  bool shapes;               // it holds other shapes than axis-parallel rectangles
  __device__ __forceinline__ OrderedBin(const Ws& ws, int bin) {
    V = ws.views + view_of_bin(ws.views, ws.n_views, bin);
    const int b = bin - V->bin_base;
    x0 = (b % V->nbx) << ws.bin_log2;
    y0 = (b / V->nbx) << ws.bin_log2;
    const uint32_t off = ws.bin_off[bin];
    n = (int)(ws.bin_off[bin + 1] - off);
    nw = (n + 31) >> 5;
    refs = ws.refs + off;
    rows = hb_row(ws, off, bin, n, 0);
    shapes = (ws.bin_cursor[bin] & kBinShapes) != 0u;
  }
};

// Persistent warps over these bins, longest lists first, an item each: a 16x8 block, of a bin with a
// long list (n_ordered_long) an 8x8 block, of the longest (n_ordered_longest) a half-block. One warp
// through a dense bin's list for 16x8 pixels takes longer than all the rest of the frame (2M particles at
// 1920x1080: 277 us, 203 with the smaller blocks; 400,000 at 960x540 201 and 78), while smaller blocks
// everywhere repeat the candidates' work and are bound by the L1 data pipe (265 us with half-blocks
// alone). Every pixel blends its list from the front in all of them, so an image depends neither on
// the form nor on what else is in the batch or asked for. (Lists cut into segments whose composites are
// then combined take 213 and 65 us, but round differently wherever one is cut.) The alpha
// threshold, which ends most lists early, has 16x8 blocks only (70 us on the 2M, 80 with the others).
// Bins of other shapes than rectangles: 8x8 blocks always.
template <bool ATH>
__global__ __launch_bounds__(kRasterThreads, 3) void k_raster_ordered(Ws ws) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* wbase = smem + (size_t)warp * kOrderedSmemWarp;
  uint16_t* cand = reinterpret_cast<uint16_t*>(wbase);
  uint2* pend = reinterpret_cast<uint2*>(wbase + win_refs(false) * sizeof(uint16_t));
  float4* qc = reinterpret_cast<float4*>(pend + kPendCap);
  if (ws.ctrl->error == LR_ERR_OVERFLOW) return;
  const uint32_t n_general = ws.ctrl->n_general, n_longest = ATH ? 0u : ws.ctrl->n_ordered_longest, n_long = ATH ? 0u : ws.ctrl->n_ordered_long;
  const int lg = ws.bin_log2, hl = bin_hb_log2(lg), cl = bin_hb_cols_log2(lg), bl = hl - 2;
  // (a batch has less than 2^32 pixels)
  const uint32_t items1 = n_longest << hl, items2 = items1 + ((n_long - n_longest) << (hl - 1));
  const uint32_t nitems = items2 + (((uint32_t)ws.total_bins - n_general - n_long) << bl);
  unsigned long long frag_total = 0;
  // a lane's pixel, if it is in the image
  auto write = [&](const ViewDev& V, int px, int py, const PixelState<1, true, ATH>& st, uint32_t cnt) {
    if (px >= V.width || py >= V.height) return;
    const long long pidx = (long long)py * V.width + px;
    if (V.cnt) V.cnt[pidx] = cnt;
    write_pixel(V, pidx, st.r, st.g, st.b, st.T);
    frag_total += cnt;
  };
  // half-block (x, y) has no pixel for the exact path
  auto no_exact = [&](const ViewDev& V, int x, int y) {
    if (V.xmask && x < V.width && y < V.height)
      V.xmask[((uint32_t)y / kHbH) * (((uint32_t)V.width + kHbW - 1) / kHbW) + (uint32_t)x / kHbW] = 0u;
  };
  // The first items are spread so that every SM gets long and shorter lists alike: warp 0 of every CTA
  // takes the longest, warp 1 the next, and so on
  const uint32_t warps = gridDim.x * kRasterWarps;
  for (bool first = true;; first = false) {
    uint32_t item = warp * gridDim.x + blockIdx.x;
    if (!first) {
      if (lane == 0) item = warps + (uint32_t)min(atomicAdd(&ws.ctrl->ordered_head, 1ull), 0xFFF00000ull);
      item = __shfl_sync(0xffffffffu, item, 0);
    }
    if (item >= nitems) break;
    const int form = item < items1 ? 1 : (item < items2 ? 2 : 4);   // pixels per lane
    const uint32_t i = item - (form == 1 ? 0u : (form == 2 ? items1 : items2));
    const int shift = form == 1 ? hl : (form == 2 ? hl - 1 : bl);
    const OrderedBin B(ws, (int)ws.bin_order[n_general + (form == 1 ? 0u : (form == 2 ? n_longest : n_long)) + (i >> shift)]);
    const ViewDev& V = *B.V;
    if (form <= 2) {
      // of the half-blocks, 2 j and 2 j + 1 are the upper and the lower one of 8x8 block j
      const int blk = (int)(i & ((1u << shift) - 1u)) >> (form == 1), lower = form == 1 ? (int)(i & 1u) : 0;
      const int bx = blk & ((1 << cl) - 1), by = 2 * (blk >> cl) + lower;
      const int ox = B.x0 + kHbW * bx, oy = B.y0 + kHbH * by;
      if (ox >= V.width || oy >= V.height || !tile_owned(V, ox, oy)) continue;
      const uint32_t* row_u = B.rows + (size_t)((by << cl) + bx) * B.nw;
      const uint32_t* row_l = row_u + ((size_t)B.nw << cl);   // (not read for a half-block)
      if (B.shapes) {
        if (!lower) frag_total += const_block<ATH>(ws.rec, B.refs, V, row_u, row_l, B.n, ox, oy, lane, cand, pend, qc);
      } else if (form == 1) {
        BoxPixels<ATH, 1> P;
        P.init();
        box_block<ATH, 1>(P, ws.rec, B.refs, V, row_u, row_u, B.nw, ox, oy, lane, cand, qc);
        write(V, ox + (lane & 7), oy + (lane >> 3), P.st[0], P.cnt[0]);
        if (lane == 0) no_exact(V, ox, oy);
      } else {
        BoxPixels<ATH, 2> P;
        P.init();
        box_block<ATH, 2>(P, ws.rec, B.refs, V, row_u, row_l, B.nw, ox, oy, lane, cand, qc);
#pragma unroll
        for (int k = 0; k < 2; ++k) write(V, ox + (lane & 7), oy + 2 * (lane >> 3) + k, P.st[k], P.cnt[k]);
        if (lane < 2) no_exact(V, ox, oy + lane * kHbH);
      }
    } else {
      const int blk = (int)(i & ((1u << bl) - 1u)), bx = blk & ((1 << (cl - 1)) - 1), by = blk >> (cl - 1);
      const int ox = B.x0 + 2 * kHbW * bx, oy = B.y0 + 2 * kHbH * by;
      if (ox >= V.width || oy >= V.height || !tile_owned(V, ox, oy)) continue;
      const uint32_t* row_u = B.rows + (size_t)((2 * by << cl) + 2 * bx) * B.nw;   // the upper left half-block's
      const uint32_t* row_l = row_u + ((size_t)B.nw << cl);
      if (!B.shapes) {
        BoxPixels<ATH, 4> P;
        P.init();
        box_block<ATH, 4>(P, ws.rec, B.refs, V, row_u, row_l, B.nw, ox, oy, lane, cand, qc);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          write(V, ox + 2 * (lane & 7) + (k & 1), oy + 2 * (lane >> 3) + (k >> 1), P.st[k], P.cnt[k]);
        if (lane < 4) no_exact(V, ox + (lane & 1) * kHbW, oy + (lane >> 1) * kHbH);
      } else {
#pragma unroll 1
        for (int h = 0; h < 2 && ox + 8 * h < V.width; ++h)
          frag_total += const_block<ATH>(ws.rec, B.refs, V, row_u + h * B.nw, row_l + h * B.nw, B.n, ox + 8 * h, oy, lane, cand, pend, qc);
      }
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
