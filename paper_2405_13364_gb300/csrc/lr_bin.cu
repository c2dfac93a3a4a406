// lr_bin.cu -- Stage 2 of the pipeline, quad binning (Sec. 2, "Stage 2: quad binning"),
// plus the per-bin depth sort that feeds Stage 3.
//
//   k_bin_count    Phase 1: per-bin reference counts. Each CTA owns a chunk of up to 4096
//                  quads of one view and counts into shared-memory bin counters (the paper's
//                  5120-entry arrays), then adds its non-zero counters to global memory.
//                  Quads whose bin rectangle is at most 4x4 bins are counted from their
//                  AABB; larger quads are tested bin by bin with a conservative
//                  per-triangle edge test (trivial reject), the whole warp sharing one
//                  large quad's bins and the whole CTA those of one over 128 bins.
//   k_bin_scan     Phase 2: exclusive scan of the counts into list offsets, capacity
//                  check, and a categorisation of bins by size (the paper's empty / low /
//                  high) that orders the rasterisers' work queues, largest bins first.
//   k_bin_scatter  Phase 3: places the chunk's references, each (chunk, bin) in the range
//                  k_bin_count reserved for it (k_bin_count's global atomic returns the
//                  range's base, listed per chunk), slots by shared-memory atomics. A
//                  reference is a 64-bit sort key:
//                  (~representative 1/w) << 32 | ~record index.
//   k_bin_sort     Stage-1 depth sort: sorts each bin's references ascending, i.e. front
//                  to back by a representative depth, ties with the higher quad index
//                  first, and writes the half-block bitmap. Bucket sorts in shared memory,
//                  buckets spaced linearly between the list's depth extremes, ranks by
//                  comparison within a bucket: bins with fewer than 2048 references by a
//                  quarter of a 1024-thread CTA with the keys in registers, high-density bins
//                  (the paper's "high" category) of up to 20480 by the whole CTA. A list with a
//                  bucket over 64 references (many equal depths) or a longer one merge-sorts
//                  runs in shared memory (up to 2048 and 8192 references), longer ones
//                  merged through a global buffer; one below 2048 on a few planes is first
//                  bucket-sorted with the indices.
#include "lr_common.cuh"

namespace lr {

// Conservative test whether triangle t of a quad can cover a pixel centre of bin (bx, by): false
// only if one edge is negative (after the fill-rule bias) at all four corner pixel centres of the
// bin rectangle clipped to the triangle's pixel AABB and the screen. An edge value is a sum of a
// term in x and one in y, so its largest corner value takes the better x and the better y. What
// does not depend on the bin stays in registers over a quad's bins.
__device__ __forceinline__ bool tri_may_touch_bin(const int X[4], const int Y[4], uint32_t info, int t, int bx, int by, int W,
                                                  int H, int lg) {
  if (!(info & (kInfoTri0 << t))) return false;
  const bool sw = (info & (kInfoSwap0 << t)) != 0;
  const int b = sw ? 2 + t : 1 + t, c = sw ? 1 + t : 2 + t;
  const int vx[3] = {X[0], b == 1 ? X[1] : (b == 2 ? X[2] : X[3]), c == 1 ? X[1] : (c == 2 ? X[2] : X[3])};
  const int vy[3] = {Y[0], b == 1 ? Y[1] : (b == 2 ? Y[2] : Y[3]), c == 1 ? Y[1] : (c == 2 ? Y[2] : Y[3])};
  const int x0 = max(max((min(vx[0], min(vx[1], vx[2])) + 127) >> 8, 0), bx << lg);
  const int x1 = min(min((max(vx[0], max(vx[1], vx[2])) - 128) >> 8, W - 1), ((bx + 1) << lg) - 1);
  const int y0 = max(max((min(vy[0], min(vy[1], vy[2])) + 127) >> 8, 0), by << lg);
  const int y1 = min(min((max(vy[0], max(vy[1], vy[2])) - 128) >> 8, H - 1), ((by + 1) << lg) - 1);
  bool in = x0 <= x1 && y0 <= y1;
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const int u = e == 2 ? 0 : e + 1, w = e == 0 ? 2 : (e == 1 ? 0 : 1);
    const int dx = vx[w] - vx[u], dy = vy[w] - vy[u];
    const int cx = 256 * (dy < 0 ? x1 : x0) + 128, cy = 256 * (dx > 0 ? y1 : y0) + 128;
    const long long ev = (long long)dx * (cy - vy[u]) - (long long)dy * (cx - vx[u]);
    in = in && ev >= ((dy < 0 || (dy == 0 && dx > 0)) ? 0 : 1);
  }
  return in;
}

// Per-bin representative depth of a quad that spans several bins.
__device__ __forceinline__ float rep_depth(const Ws& ws, long long q, uint32_t info, int x0, int x1,
                                           int y0, int y1) {
  const int4 a = ws.rec[4 * q], b = ws.rec[4 * q + 1], c = ws.rec[4 * q + 2];
  const int X[4] = {a.x, a.z, b.x, b.z}, Y[4] = {a.y, a.w, b.y, b.w};
  const float Q[4] = {__int_as_float(c.x), __int_as_float(c.y), __int_as_float(c.z), __int_as_float(c.w)};
  return rep_depth_of(X, Y, Q, info, x0, x1, y0, y1);
}

__device__ __forceinline__ unsigned long long ref_key(float rep, long long q) {
  return ((unsigned long long)(~__float_as_uint(rep)) << 32) | (unsigned long long)(~(uint32_t)q);
}

// Shared by count and scatter: for each (visible quad, touched bin) of the CTA's chunk
// call f(q, local_bin, bx, by). Small quads enumerate their AABB bins in their own
// thread; large quads are processed by the whole warp, one bin per lane, and those whose box
// spans more than kWarpBins bins by the whole CTA afterwards: one warp walks the 2,040 bins of a
// screen-filling quad in 64 steps, which took longer than all the rest of the chunk (a frame of
// 100,000 parallelograms with a few such quads: count 15.5 us, scatter 22.4).
// PF: the next iteration's rectangle and info are loaded while this one's bins are handled
// (the count's loop is latency-bound, a dependent load per iteration otherwise: 18.4 -> 17.0
// µs on the layer frame; the scatter, with more live registers, measured no faster with it).
constexpr int kWarpBins = 128;
struct LargeList {
  uint32_t n;
  uint16_t at[kChunkQuads];   // offset in the chunk
};
template <typename F>
__device__ __forceinline__ void large_quad_bins(const Ws& ws, const ViewDev& V, long long q, uint2 rect, uint32_t info,
                                                int first, int step, F&& f) {
  const int lg = ws.bin_log2, W = V.width, H = V.height;
  const int bx0 = (int)(rect.x & 0xffff) >> lg, by0 = (int)(rect.y & 0xffff) >> lg;
  const int bw = ((int)(rect.x >> 16) >> lg) - bx0 + 1, nb = bw * (((int)(rect.y >> 16) >> lg) - by0 + 1);
  int X[4], Y[4];
  load_rec_xy(ws.rec, (uint32_t)q, X, Y);
  for (int i = first; i < nb; i += step) {
    const int by = by0 + i / bw, bx = bx0 + i - (by - by0) * bw;
    if (tri_may_touch_bin(X, Y, info, 0, bx, by, W, H, lg) || tri_may_touch_bin(X, Y, info, 1, bx, by, W, H, lg))
      f(q, by * V.nbx + bx, bx, by, rect, info);
  }
}
template <bool PF, typename F>
__device__ __forceinline__ void for_each_ref(const Ws& ws, const ViewDev& V, long long q0, long long q1,
                                             LargeList& list, F&& f) {
  const int lane = threadIdx.x & 31;
  const int lg = ws.bin_log2;
  long long base = q0 + (threadIdx.x & ~31);
  uint2 rect_n = make_uint2(kRectInvisible, kRectInvisible);
  uint32_t info_n = 0;
  if (PF && base + lane < q1) { rect_n = ws.rec_rect[base + lane]; info_n = ws.rec_info[base + lane]; }
  for (; base < q1; base += blockDim.x) {
    const long long q = base + lane;
    const bool in = q < q1;
    uint2 rect = rect_n;
    uint32_t info = info_n;
    if (PF) {
      rect_n = make_uint2(kRectInvisible, kRectInvisible);
      info_n = 0;
      if (q + blockDim.x < q1) { rect_n = ws.rec_rect[q + blockDim.x]; info_n = ws.rec_info[q + blockDim.x]; }
    } else if (in) {
      rect = ws.rec_rect[q];
      info = ws.rec_info[q];
    }
    const bool vis = in && rect.x != kRectInvisible;
    const int bx0 = (int)(rect.x & 0xffff) >> lg, bx1 = (int)(rect.x >> 16) >> lg;
    const int by0 = (int)(rect.y & 0xffff) >> lg, by1 = (int)(rect.y >> 16) >> lg;
    bool large = vis && (info & kInfoLarge);
    if (vis && !large) {
      for (int by = by0; by <= by1; ++by)
        for (int bx = bx0; bx <= bx1; ++bx) f(q, by * V.nbx + bx, bx, by, rect, info);
    }
    if (large && (bx1 - bx0 + 1) * (by1 - by0 + 1) > kWarpBins) {
      list.at[atomicAdd(&list.n, 1u)] = (uint16_t)(q - q0);
      large = false;
    }
    unsigned todo = __ballot_sync(0xffffffffu, large);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const long long lq = base + src;
      const uint2 lr = make_uint2(__shfl_sync(0xffffffffu, rect.x, src), __shfl_sync(0xffffffffu, rect.y, src));
      const uint32_t li = __shfl_sync(0xffffffffu, info, src);
      large_quad_bins(ws, V, lq, lr, li, lane, 32, f);
    }
  }
  __syncthreads();
  const int n = (int)list.n;
  for (int i = 0; i < n; ++i) {
    const long long q = q0 + list.at[i];
    large_quad_bins(ws, V, q, ws.rec_rect[q], ws.rec_info[q], threadIdx.x, blockDim.x, f);
  }
}

// count and scatter are latency-bound (gathers, atomics); chunks and threads: chunk_quads_for
__global__ __launch_bounds__(kBinThreads, kBinMinBlocks) void k_bin_count(Ws ws) {
  pdl_begin();
  __shared__ uint32_t hist[kHistSmemBins];
  __shared__ LargeList large;
  __shared__ uint32_t depths[kHistSmemBins / 32];   // bins the chunk marks kBinDepths
  const int v = view_of_chunk(ws.views, ws.n_views, blockIdx.x);
  const ViewDev& V = ws.views[v];
  const long long q0 = V.quad_base + (long long)(blockIdx.x - V.chunk_base) * ws.chunk_quads;
  const long long q1 = min(q0 + ws.chunk_quads, V.quad_base + V.num_quads);
  const int nb = V.nbx * V.nby;
  const bool smem = nb <= kHistSmemBins;
  if (threadIdx.x == 0) large.n = 0u;
  if (smem)
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
      hist[b] = 0u;
      depths[b >> 5] = 0u;
    }
  __syncthreads();
  for_each_ref<true>(ws, V, q0, q1, large, [&](long long, int b, int, int, uint2, uint32_t info) {
    if (smem) {
      atomicAdd(&hist[b], 1u);
      const uint32_t bit = 1u << (b & 31);
      uint32_t* d = &depths[b >> 5];
      if (!(info & kInfoFlatDepth) && !(*(volatile uint32_t*)d & bit)) atomicOr(d, bit);
    } else {
      atomicAdd(&ws.bin_count[V.bin_base + b], 1u);
    }
  });
  __syncthreads();
  if (!smem) return;
  // reserve the chunk's range in every bin it touches, and list (bin, base of the range)
  // for k_bin_scatter, which then places references without recounting
  __shared__ uint32_t s_n, s_start, s_pos;
  if (threadIdx.x == 0) { s_n = 0; s_pos = 0; }
  __syncthreads();
  uint32_t mine = 0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) mine += hist[b] != 0u;
  if (mine) atomicAdd(&s_n, mine);
  __syncthreads();
  if (threadIdx.x == 0) {
    s_start = (uint32_t)min(atomicAdd(&ws.ctrl->chunk_list_head, (unsigned long long)s_n), 0xFFFFFFFFull);
    ws.chunk_span[blockIdx.x] = make_uint2(s_start, s_n);
  }
  __syncthreads();
  uint2* list = reinterpret_cast<uint2*>(ws.refs_tmp);
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const uint32_t c = hist[b];
    if (!c) continue;
    if (!ws.cursors && ((depths[b >> 5] >> (b & 31)) & 1u)) atomicOr(&ws.bin_cursor[V.bin_base + b], kBinDepths);
    const uint32_t base = atomicAdd(&ws.bin_count[V.bin_base + b], c);
    const unsigned long long at = (unsigned long long)s_start + atomicAdd(&s_pos, 1u);
    // a list past the reference capacity means the references do not fit either: the scan
    // reports the overflow and the scatter does not run
    if (at < (unsigned long long)ws.refs_cap) list[at] = make_uint2((uint32_t)b, base);
  }
}

// Single CTA. Offsets (exclusive scan), capacity check, and the bin order for the rasterisers:
// k_raster's bins, then k_raster_ordered's, each by decreasing size class (class k: from 2^(k - 1)
// references, class 0: empty). Bound by latency (one CTA): each thread takes consecutive bins, four
// counts in flight, so that there is one scan however many bins there are (8160 bins: 20 us with a
// scan per 1024 of them and the two orders, 16 us so; 2040 bins 12 and 8).
__global__ __launch_bounds__(1024) void k_bin_scan(Ws ws) {
  pdl_begin();
  constexpr int kClasses = 32;       // (a view has fewer than 2^30 quads)
  __shared__ unsigned long long warp_sums[32];
  __shared__ uint32_t warp_ordered[32];   // references of k_raster_ordered's bins
  __shared__ uint32_t cls_count[2 * kClasses], cls_base[2 * kClasses];
  __shared__ uint8_t cls_of[kHistSmemBins];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int n = ws.total_bins;
  if (tid < 2 * kClasses) cls_count[tid] = 0;
  __syncthreads();
  auto class_of = [&](int bin, uint32_t c, uint32_t flags) {
    const bool ordered = ws.ordered && !(flags & kBinDepths) &&
                         ws.views[view_of_bin(ws.views, ws.n_views, bin)].color_mode == LR_COLOR_FLAT;
    return (c ? 32 - __clz(c) : 0) + (ordered ? kClasses : 0);
  };
  unsigned long long nonempty = 0, high = 0, mx = 0, sum = 0;
  uint32_t ordered_sum = 0;            // (32 bits: more references than that overflow)
  const int per = (n + 1023) >> 10, i0 = tid * per, i1 = min(n, i0 + per);
  for (int i = i0; i < i1; i += 4) {
    uint32_t c[4], f[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      c[u] = i + u < i1 ? ws.bin_count[i + u] : 0u;
      f[u] = i + u < i1 ? ws.bin_cursor[i + u] : 0u;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (i + u >= i1) break;
      sum += c[u];
      nonempty += c[u] > 0;
      high += c[u] >= (uint32_t)kSortSmemCap;
      mx = c[u] > mx ? c[u] : mx;
      const int cls = class_of(i + u, c[u], f[u]);
      if (cls >= kClasses) ordered_sum += c[u];
      if (i + u < kHistSmemBins) cls_of[i + u] = (uint8_t)cls;
      // one shared-memory atomic per warp and size class (most bins of a warp share one)
      const unsigned act = __activemask();
      const unsigned peers = __match_any_sync(act, cls);
      if (lane == __ffs(peers) - 1) atomicAdd(&cls_count[cls], (uint32_t)__popc(peers));
    }
  }
  unsigned long long x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  ordered_sum = __reduce_add_sync(0xffffffffu, ordered_sum);
  if (lane == 31) { warp_sums[wid] = x; warp_ordered[wid] = ordered_sum; }
  __syncthreads();
  if (wid == 0) {
    unsigned long long s = warp_sums[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    warp_sums[lane] = s;
  }
  __syncthreads();
  const unsigned long long total = warp_sums[31];
  unsigned long long excl = x - sum + (wid ? warp_sums[wid - 1] : 0ull);
  for (int i = i0; i < i1; ++i) {
    const uint32_t o = (uint32_t)min(excl, (unsigned long long)ws.refs_cap);
    excl += ws.bin_count[i];
    ws.bin_off[i] = o;
    if (ws.cursors) ws.bin_cursor[i] = o;
  }
  if (tid == 0) {
    ws.bin_off[n] = (uint32_t)min(total, (unsigned long long)ws.refs_cap);
    ws.ctrl->refs_total = total;
    if (total > (unsigned long long)ws.refs_cap) set_error(ws.ctrl, LR_ERR_OVERFLOW);
  }
  // statistics
  for (int o = 16; o > 0; o >>= 1) {
    nonempty += __shfl_xor_sync(0xffffffffu, nonempty, o);
    high += __shfl_xor_sync(0xffffffffu, high, o);
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = y > mx ? y : mx;
  }
  if (lane == 0) {
    atomicAdd(&ws.ctrl->bins_nonempty, nonempty);
    atomicAdd(&ws.ctrl->bins_high, high);
    atomicMax(&ws.ctrl->max_bin, mx);
  }
  // class bases, largest class first: lane l of warp 0 has class 31 - l
  if (wid == 0) {
    const int k = 31 - lane;
    const uint32_t g = cls_count[k], o = cls_count[kClasses + k];
    uint32_t gi = g, oi = o;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, gi, d), z = __shfl_up_sync(0xffffffffu, oi, d);
      if (lane >= d) { gi += y; oi += z; }
    }
    const uint32_t general = __shfl_sync(0xffffffffu, gi, 31);
    cls_base[k] = gi - g;
    cls_base[kClasses + k] = general + oi - o;
    // long lists of k_raster_ordered
    const unsigned long long blocks = (unsigned long long)__reduce_add_sync(0xffffffffu, warp_ordered[lane]) * (unsigned)(bin_hb(ws.bin_log2) / 4);
    const unsigned long long warps8 = 8ull * (unsigned)max(ws.ordered, 1), least = k > 0 ? 1ull << (k - 1) : 0ull;
    const bool is_long = least >= kOrderedLong && least * warps8 >= blocks * kOrderedLongShare8;
    const bool is_longest = is_long && least >= kOrderedLongest && least * warps8 >= blocks * kOrderedLongestShare8;
    const uint32_t n_long = __reduce_max_sync(0xffffffffu, is_long ? oi : 0u);
    const uint32_t n_longest = __reduce_max_sync(0xffffffffu, is_longest ? oi : 0u);
    if (k == 12) ws.ctrl->high_general = gi;       // from 2048 references
    if (k == 1) ws.ctrl->nonempty_general = gi;
    if (lane == 0) {
      ws.ctrl->n_general = general;
      ws.ctrl->raster_items = (unsigned long long)general * bin_hb(ws.bin_log2);
      ws.ctrl->n_ordered_long = n_long;
      ws.ctrl->n_ordered_longest = n_longest;
    }
  }
  __syncthreads();
  for (int i = tid; i < n; i += 1024) {
    const int cls = i < kHistSmemBins ? cls_of[i] : class_of(i, ws.bin_count[i], ws.bin_cursor[i]);
    // lanes of one class take consecutive positions from one atomic of their leader
    const unsigned act = __activemask();
    const unsigned peers = __match_any_sync(act, cls);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(&cls_base[cls], (uint32_t)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    ws.bin_order[base + __popc(peers & ((1u << lane) - 1u))] = (uint32_t)i;
  }
}

__global__ __launch_bounds__(kBinThreads, kBinMinBlocks) void k_bin_scatter(Ws ws) {
  pdl_begin();
  __shared__ uint32_t hist[kHistSmemBins];
  __shared__ LargeList large;
  __shared__ uint32_t shapes[kHistSmemBins / 32];   // bins the chunk has marked kBinShapes
  if (ws.ctrl->error == LR_ERR_OVERFLOW) return;
  const int v = view_of_chunk(ws.views, ws.n_views, blockIdx.x);
  const ViewDev& V = ws.views[v];
  const long long q0 = V.quad_base + (long long)(blockIdx.x - V.chunk_base) * ws.chunk_quads;
  const long long q1 = min(q0 + ws.chunk_quads, V.quad_base + V.num_quads);
  const int nb = V.nbx * V.nby;
  const bool smem = nb <= kHistSmemBins;
  if (threadIdx.x == 0) large.n = 0u;
  if (smem) {
    for (int b = threadIdx.x; b < kHistSmemBins / 32; b += blockDim.x) shapes[b] = 0u;
    // the chunk's range in each bin it touches, reserved by k_bin_count
    const uint2 sp = ws.chunk_span[blockIdx.x];
    const uint2* list = reinterpret_cast<const uint2*>(ws.refs_tmp) + sp.x;
    for (int i = threadIdx.x; i < (int)sp.y; i += blockDim.x) {
      const uint2 e = list[i];
      hist[e.x] = ws.bin_off[V.bin_base + e.x] + e.y;
    }
  }
  __syncthreads();
  for_each_ref<false>(ws, V, q0, q1, large, [&](long long q, int b, int bx, int by, uint2 rect, uint32_t info) {
    const uint32_t slot = smem ? atomicAdd(&hist[b], 1u) : atomicAdd(&ws.bin_cursor[V.bin_base + b], 1u);
    const int lg = ws.bin_log2;
    const int x0 = max((int)(rect.x & 0xffff), bx << lg);
    const int x1 = min((int)(rect.x >> 16), ((bx + 1) << lg) - 1);
    const int y0 = max((int)(rect.y & 0xffff), by << lg);
    const int y1 = min((int)(rect.y >> 16), ((by + 1) << lg) - 1);
    // a quad inside one bin, or of constant depth: its per-quad value; else the plane at its
    // box clipped to this bin
    const bool one_bin = ((rect.x & 0xffff) >> lg) == ((rect.x >> 16) >> lg) &&
                         ((rect.y & 0xffff) >> lg) == ((rect.y >> 16) >> lg);
    const bool flat = (info & kInfoFlatDepth) != 0u;
    const float rep = one_bin || flat ? ws.rec_rep[q] : rep_depth(ws, q, info, x0, x1, y0, y1);
    if (ws.ordered && flat && rep > 0.f) {   // (no rectangle; the views' bins then have shared counters)
      const uint32_t bit = 1u << (b & 31);
      uint32_t* s = &shapes[b >> 5];
      if (!(*(volatile uint32_t*)s & bit) && !(atomicOr(s, bit) & bit)) atomicOr(&ws.bin_cursor[V.bin_base + b], kBinShapes);
    }
    if (slot < (uint32_t)ws.refs_cap) ws.refs[slot] = ref_key(fabsf(rep), q);
  });
}


// Merge sorted runs a[0, na) and b[0, nb) into out, split evenly over the CTA (merge path).
__device__ void cta_merge(const unsigned long long* a, int na, const unsigned long long* b, int nb,
                          unsigned long long* out) {
  const int total = na + nb;
  const int per = (total + blockDim.x - 1) / blockDim.x;
  const int d0 = min((int)threadIdx.x * per, total), d1 = min(d0 + per, total);
  if (d0 >= d1) return;
  // find i + j = d0 with a[i-1] < b[j] and b[j-1] < a[i] (keys are unique)
  int lo = max(0, d0 - nb), hi = min(d0, na);
  while (lo < hi) {
    const int i = (lo + hi) >> 1;
    if (a[i] < b[d0 - i - 1]) lo = i + 1; else hi = i;
  }
  int i = lo, j = d0 - lo;
  for (int d = d0; d < d1; ++d) {
    if (j >= nb || (i < na && a[i] < b[j])) out[d] = a[i++];
    else out[d] = b[j++];
  }
}

// Threads that sort one bin together: the whole CTA, or one of its quarters with a named
// barrier of its own.
struct Group {
  int t, n, bar;             // thread index, threads, barrier
  __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(n) : "memory"); }
};

// Mask word m of the 8x4 half-blocks of the bin with pixel origin (x0, y0) (bit hy * cols + hx, in
// mw 32-bit words) that the pixel box rc overlaps.
__device__ __forceinline__ uint32_t hb_mask_word(uint2 rc, int x0, int y0, int lg, int m) {
  const int B = 1 << lg, cols = bin_hb_cols(lg), rpw = 32 / cols;   // half-block rows per mask word
  // bit i * cols for every row i of a word: the row pattern's replication
  const uint32_t rep = cols == 8 ? 0x01010101u : (cols == 4 ? 0x11111111u : 0x55555555u);
  const int px0 = max((int)(rc.x & 0xffff), x0) - x0, px1 = min((int)(rc.x >> 16), x0 + B - 1) - x0;
  const int py0 = max((int)(rc.y & 0xffff), y0) - y0, py1 = min((int)(rc.y >> 16), y0 + B - 1) - y0;
  if (px0 > px1 || py0 > py1) return 0u;
  const int hx0 = px0 / kHbW, hx1 = px1 / kHbW, hy0 = py0 / kHbH, hy1 = py1 / kHbH;
  // the half-block columns hx0..hx1 replicated into the rows hy0..hy1 that fall in mask
  // word m: a product, since a row's pattern never carries into the next row
  const uint32_t row = ((2u << hx1) - 1u) & ~((1u << hx0) - 1u);
  const int a = max(hy0 - m * rpw, 0), c = min(hy1 - m * rpw, rpw - 1);
  return a <= c ? row * (rep & ((2u << (c * cols)) - 1u) & ~((1u << (a * cols)) - 1u)) : 0u;
}

// The bin's transposed half-block bitmap (hb_row): for each sorted reference, the mask of
// the bin's 8x4 half-blocks that the quad's pixel AABB overlaps, computed one warp per 32
// references and transposed across the warp word by word, so that row h, word w holds the
// bits of references 32 w .. 32 w + 31 for half-block h. The rasteriser then reads a
// half-block's candidates with one coalesced load per 1024 references. When the bitmap fits
// `stage` (shared memory, stage_words 32-bit words), the transposed words are assembled there
// and copied out row by row with coalesced stores; otherwise each lane stores its word of a
// row directly. Four words' references and boxes are in flight at a time.
__device__ void write_hb_bitmap(const Ws& ws, const unsigned long long* r, int n, int bin, uint32_t* stage,
                                int stage_words, const Group& G) {
  const int v = view_of_bin(ws.views, ws.n_views, bin);
  const ViewDev& V = ws.views[v];
  const int b = bin - V.bin_base;
  const int lg = ws.bin_log2;
  const int mw = bin_mw(lg), mrows = bin_mrows(lg);
  const int x0 = (b % V.nbx) << lg, y0 = (b / V.nbx) << lg;
  const int nw = (n + 31) >> 5;
  const int lane = G.t & 31, warps = G.n >> 5;
  uint32_t* bm = ws.ref_hb + (size_t)mw * (size_t)(r - ws.refs) + (size_t)mrows * (size_t)bin;
  const bool staged = mrows * nw <= stage_words;
  uint32_t* dst = staged ? stage : bm;
  for (int w0 = G.t >> 5; w0 < nw; w0 += 4 * warps) {
    uint32_t rec[4];
    uint2 rc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = 32 * (w0 + u * warps) + lane;
      rec[u] = i < n ? ~(uint32_t)r[i] : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      rc[u] = rec[u] < (uint64_t)ws.total_quads ? ws.rec_rect[rec[u]] : make_uint2(1u, 1u);   // (an empty box)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int w = w0 + u * warps;
      if (w >= nw) break;
      for (int m = 0; m < mw; ++m)
        dst[(size_t)(32 * m + lane) * nw + w] = warp_transpose32(hb_mask_word(rc[u], x0, y0, lg, m), lane);
    }
  }
  if (staged) {
    G.sync();
    for (int i = G.t; i < mrows * nw; i += G.n) bm[i] = stage[i];
  }
}

// Bucket of a key between the depth extremes lo and hi of its list (high words of the keys): linear,
// hence monotone, so that buckets come out in order.
struct Buckets {
  uint32_t lo;
  float scale;
  int last;
  __device__ __forceinline__ Buckets(uint32_t lo_, uint32_t hi_, int nb) : lo(lo_), last(nb - 1) {
    scale = (float)nb / ((float)(hi_ - lo_) + 1.0f);
  }
  __device__ __forceinline__ int of(unsigned long long key) const {
    return min(last, (int)((float)((uint32_t)(key >> 32) - lo) * scale));
  }
};

// Reductions over the group's warps through red (one word per warp, at most 32), after a sync.
__device__ __forceinline__ uint32_t red_min(const uint32_t* red, int nw, int lane) {
  return __reduce_min_sync(0xffffffffu, lane < nw ? red[lane] : 0xFFFFFFFFu);
}
__device__ __forceinline__ uint32_t red_max(const uint32_t* red, int nw, int lane) {
  return __reduce_max_sync(0xffffffffu, lane < nw ? red[lane] : 0u);
}

// The buckets' counters are 16 bits wide, two to a word (lists are shorter than 2^16): many buckets
// keep the comparisons within a bucket few where depths cluster, and those, of a warp's fullest
// bucket, were most of the sort's instructions (2M particles: 4096 buckets for 15,000 keys 84 us,
// 16384 80 us).
__device__ __forceinline__ uint32_t count_up(uint32_t* cnt, int b) {   // the count before
  const int sh = 16 * (b & 1);
  return (atomicAdd(&cnt[b >> 1], 1u << sh) >> sh) & 0xFFFFu;
}

// Turns the counts of 2 PER * G.n buckets into exclusive prefix sums, 2 PER consecutive ones per
// thread; false when one of them exceeds kMaxBucket (the counts are then as they were unless ALWAYS).
// red: 64 words.
template <int PER, bool ALWAYS = false>
__device__ __forceinline__ bool scan_counts(uint32_t* cnt, uint32_t* red, const Group& G) {
  const int lane = G.t & 31, w = G.t >> 5, nw = G.n >> 5;
  uint32_t c[PER], sum = 0, mx = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    c[k] = cnt[PER * G.t + k];
    sum += (c[k] & 0xFFFFu) + (c[k] >> 16);
    mx = max(mx, max(c[k] & 0xFFFFu, c[k] >> 16));
  }
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += x;
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 31) { red[w] = incl; red[32 + w] = mx; }
  G.sync();
  const bool ok = red_max(red + 32, nw, lane) <= (uint32_t)kMaxBucket;
  if (!ALWAYS && !ok) return false;
  uint32_t at = incl - sum + __reduce_add_sync(0xffffffffu, lane < w ? red[lane] : 0u);
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const uint32_t odd = at + (c[k] & 0xFFFFu);
    cnt[PER * G.t + k] = at | (odd << 16);
    at = odd + (c[k] >> 16);
  }
  return ok;
}

// Position of key among the keys [s0, s1) of its bucket.
__device__ __forceinline__ int bucket_rank(const unsigned long long* keys, int s0, int s1, unsigned long long key) {
  int c = s0;
  for (int j = s0; j < s1; ++j) c += keys[j] < key;
  return c;
}

// Ascending bucket sort of the 64-bit keys r[0, n), n <= kBucketBigCap, by the whole CTA (1024
// threads), through shared memory dst[n] and cnt[kBucketsBig / 2]: counts, prefix sums, keys to their
// buckets, then each key's rank by comparison within its bucket. Returns false, with r unchanged,
// when a bucket would hold more than kMaxBucket keys (many equal or clustered depths); the caller
// then uses a comparison sort. The three passes over the list are bound by latency, so four loads
// are in flight per thread.
__device__ bool cta_bucket_sort(unsigned long long* r, int n, unsigned long long* dst, uint32_t* cnt, uint32_t* red,
                                const Group& G) {
  const int t = G.t, lane = t & 31, w = t >> 5, T = G.n;
  auto each_key = [&](auto f) {
    for (int i = t; i < n; i += 4 * T) {
      unsigned long long k[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) k[u] = i + u * T < n ? r[i + u * T] : 0ull;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i + u * T < n) f(k[u]);
    }
  };
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
  each_key([&](unsigned long long k) {
    lo = min(lo, (uint32_t)(k >> 32));
    hi = max(hi, (uint32_t)(k >> 32));
  });
  constexpr int PER = kBucketsBig / 2 / kSortThreads;
#pragma unroll
  for (int k = 0; k < PER; ++k) cnt[t + k * T] = 0u;
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) { red[w] = lo; red[32 + w] = hi; }
  G.sync();
  const Buckets bk(red_min(red, T >> 5, lane), red_max(red + 32, T >> 5, lane), kBucketsBig);
  each_key([&](unsigned long long k) { count_up(cnt, bk.of(k)); });
  G.sync();
  if (!scan_counts<PER>(cnt, red, G)) return false;
  G.sync();
  each_key([&](unsigned long long k) { dst[count_up(cnt, bk.of(k))] = k; });   // b's end afterwards
  G.sync();
  const uint16_t* end = reinterpret_cast<const uint16_t*>(cnt);
  for (int i = t; i < n; i += T) {
    const unsigned long long k = dst[i];
    const int b = bk.of(k);
    r[bucket_rank(dst, b ? (int)end[b - 1] : 0, (int)end[b], k)] = k;
  }
  G.sync();
  return true;
}

// Shared memory of a quarter CTA sorting one bin of fewer than kSortSmemCap references.
struct SmallSort {
  unsigned long long a[kSortSmemCap], b[kSortSmemCap];
  uint32_t mask[kSortSmemCap];
  uint32_t cnt[kBucketsSmall / 2 + 4];
};
constexpr int kStageWords = (int)(sizeof(SmallSort::a) / 4);   // bitmap assembled in `a`

// The same for n <= KPT * 256 keys by a quarter CTA, the keys in registers,
// each with its half-block mask (bins of up to 32 pixels: one word), loaded while the keys are
// counted; the sorted list and its bitmap are written from shared memory.
template <int KPT>
__device__ __forceinline__ bool small_bucket_sort(const Ws& ws, unsigned long long* r, int n, int bin, SmallSort& S,
                                                  uint32_t* red, const Group& G) {
  const int t = G.t, lane = t & 31, w = t >> 5;
  constexpr int T = kSortThreads / 4, NB = KPT >= 3 ? kBucketsSmall : 2 * KPT * T, PER = NB / 2 / T;
  const bool one_word = bin_mw(ws.bin_log2) == 1;
  const ViewDev& V = ws.views[view_of_bin(ws.views, ws.n_views, bin)];
  unsigned long long key[KPT];
  uint32_t at[KPT], mask[KPT], lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
  for (int k = 0; k < KPT; ++k) key[k] = t + k * T < n ? r[t + k * T] : 0ull;
#pragma unroll
  for (int k = 0; k < PER; ++k) S.cnt[t + k * T] = 0u;
#pragma unroll
  for (int k = 0; k < KPT; ++k)
    if (t + k * T < n) {
      lo = min(lo, (uint32_t)(key[k] >> 32));
      hi = max(hi, (uint32_t)(key[k] >> 32));
    }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) { red[w] = lo; red[32 + w] = hi; }
#pragma unroll
  for (int k = 0; k < KPT; ++k) mask[k] = 0u;
  if (one_word) {
    const int b = bin - V.bin_base, lg = ws.bin_log2;
    const int x0 = (b % V.nbx) << lg, y0 = (b / V.nbx) << lg;
#pragma unroll
    for (int k = 0; k < KPT; ++k) {
      const uint32_t rec = t + k * T < n ? ~(uint32_t)key[k] : 0xFFFFFFFFu;
      mask[k] = rec < (uint64_t)ws.total_quads ? hb_mask_word(ws.rec_rect[rec], x0, y0, lg, 0) : 0u;
    }
  }
  G.sync();
  lo = red_min(red, T / 32, lane);
  hi = red_max(red + 32, T / 32, lane);
  if (lo == hi && n > kMaxBucket) return false;   // one depth
  const Buckets bk(lo, hi, NB);
#pragma unroll
  for (int k = 0; k < KPT; ++k)
    if (t + k * T < n) {
      const int b = bk.of(key[k]);
      at[k] = (uint32_t)b | (count_up(S.cnt, b) << 16);
    }
  G.sync();
  if (!scan_counts<PER>(S.cnt, red, G)) return false;
  if (t == 0) S.cnt[NB / 2] = (uint32_t)n;
  const uint16_t* start = reinterpret_cast<const uint16_t*>(S.cnt);
  G.sync();
#pragma unroll
  for (int k = 0; k < KPT; ++k)
    if (t + k * T < n) S.a[start[at[k] & 0xFFFFu] + (at[k] >> 16)] = key[k];
  G.sync();
#pragma unroll
  for (int k = 0; k < KPT; ++k)
    if (t + k * T < n) {
      const int b = (int)(at[k] & 0xFFFFu);
      const int p = bucket_rank(S.a, (int)start[b], (int)start[b + 1], key[k]);
      S.b[p] = key[k];
      S.mask[p] = mask[k];
    }
  G.sync();
  for (int i = t; i < n; i += T) r[i] = S.b[i];
  uint32_t* stage = reinterpret_cast<uint32_t*>(S.a);
  if (!one_word) {
    G.sync();
    write_hb_bitmap(ws, r, n, bin, stage, kStageWords, G);
    return true;
  }
  const int nw = (n + 31) >> 5;
  uint32_t* bm = ws.ref_hb + (size_t)(r - ws.refs) + (size_t)bin_mrows(ws.bin_log2) * (size_t)bin;
  for (int i = w; i < nw; i += T / 32)
    stage[lane * nw + i] = warp_transpose32(32 * i + lane < n ? S.mask[32 * i + lane] : 0u, lane);
  G.sync();
  for (int i = t; i < 32 * nw; i += T) bm[i] = stage[i];
  return true;
}

// The same for a list of few depths (quads on a few planes), whose buckets are too full: where the keys of
// such a bucket have one depth, they are spread over as many buckets as they are by their index, and the
// list is counted anew. Returns false, with r unchanged, when a bucket is too full still or holds several
// depths. Out of line, so that the sort above stays small; its bitmap is written afterwards. Sort stage of
// 400,000 quads on one or eight planes at 1920x1080: 61 and 57 us with the merge sort, 43 so (31 at distinct
// depths); of 1M, a third of whose references are in dense lists, 129 and 123, 92 so.
__device__ __noinline__ bool small_plane_sort(unsigned long long* r, int n, SmallSort& S, uint32_t* red, const Group G) {
  const int t = G.t, lane = t & 31, w = t >> 5;
  constexpr int T = kSortThreads / 4, NB = kBucketsSmall, PER = NB / 2 / T;
  uint32_t* cnt1 = reinterpret_cast<uint32_t*>(S.b);      // counts by depth, then these buckets' starts
  uint32_t* cnt2 = S.cnt;                                 // counts with the full buckets spread
  uint32_t* depth = S.mask;                               // of a full bucket: they start more than 64 apart
  uint32_t* mixed = S.mask + kSortSmemCap / kMaxBucket;   // a full bucket holds several depths
  uint32_t lo = 0xFFFFFFFFu, hi = 0u, ilo = 0xFFFFFFFFu, ihi = 0u;
  for (int i = t; i < n; i += T) {
    const unsigned long long k = r[i];
    lo = min(lo, (uint32_t)(k >> 32));
    hi = max(hi, (uint32_t)(k >> 32));
    ilo = min(ilo, (uint32_t)k);
    ihi = max(ihi, (uint32_t)k);
  }
  for (int i = t; i < NB / 2; i += T) cnt1[i] = cnt2[i] = 0u;
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  ilo = __reduce_min_sync(0xffffffffu, ilo);
  ihi = __reduce_max_sync(0xffffffffu, ihi);
  G.sync();                                               // (red is read by the failed attempt)
  if (lane == 0) { red[w] = lo; red[8 + w] = hi; red[16 + w] = ilo; red[24 + w] = ihi; }
  if (t == 0) *mixed = 0u;
  G.sync();
  const Buckets bk(red_min(red, T / 32, lane), red_max(red + 8, T / 32, lane), NB);
  ilo = red_min(red + 16, T / 32, lane);
  const float spread = 1.0f / ((float)(red_max(red + 24, T / 32, lane) - ilo) + 1.0f);
  for (int i = t; i < n; i += T) count_up(cnt1, bk.of(r[i]));
  G.sync();
  scan_counts<PER, true>(cnt1, red, G);
  if (t == 0) cnt1[NB / 2] = (uint32_t)n;
  G.sync();
  const uint16_t* start1 = reinterpret_cast<const uint16_t*>(cnt1);
  // a key's bucket: its bucket's start, in a full one plus its share of the bucket by index (monotone)
  auto of = [&](unsigned long long k) {
    const int b = bk.of(k), s = (int)start1[b], c = (int)start1[b + 1] - s;
    return c <= kMaxBucket ? s : s + min(c - 1, (int)((float)((uint32_t)k - ilo) * spread * (float)c));
  };
  auto full = [&](unsigned long long k, int& s) {
    const int b = bk.of(k);
    s = (int)start1[b];
    return (int)start1[b + 1] - s > kMaxBucket;
  };
  int s;
  for (int i = t; i < n; i += T)
    if (full(r[i], s)) depth[s / kMaxBucket] = (uint32_t)(r[i] >> 32);   // (any of them)
  G.sync();
  for (int i = t; i < n; i += T) {
    const unsigned long long k = r[i];
    if (full(k, s) && depth[s / kMaxBucket] != (uint32_t)(k >> 32)) *mixed = 1u;
    count_up(cnt2, of(k));
  }
  G.sync();
  if (*mixed) return false;
  if (!scan_counts<PER>(cnt2, red, G)) return false;
  G.sync();
  for (int i = t; i < n; i += T) {
    const unsigned long long k = r[i];
    S.a[count_up(cnt2, of(k))] = k;                       // the bucket's end afterwards
  }
  G.sync();
  const uint16_t* end = reinterpret_cast<const uint16_t*>(cnt2);
  for (int i = t; i < n; i += T) {
    const unsigned long long k = S.a[i];
    const int b = of(k);
    r[bucket_rank(S.a, b ? (int)end[b - 1] : 0, (int)end[b], k)] = k;
  }
  G.sync();
  return true;
}

// Ascending sort of the 32 KPL keys v (KPL per lane, lane l holding elements KPL l ..
// KPL l + KPL - 1) by one warp: a bitonic network, its compare-exchanges between a lane's own
// keys (element distance below KPL) in registers and the others by shuffles with the
// partner lane.
template <int KPL>
__device__ __forceinline__ void warp_bitonic(unsigned long long v[KPL], int lane) {
#pragma unroll
  for (int k = 2; k <= 32 * KPL; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j < KPL) {
#pragma unroll
        for (int r = 0; r < KPL; ++r) {
          if (r & j) continue;   // r is the lower element of the pair (r, r + j)
          // ascending where element KPL lane + r has bit k clear
          const bool asc = k < KPL ? (r & k) == 0 : (lane & (k / KPL)) == 0;
          const unsigned long long a = v[r], b = v[r | j];
          const bool sw = asc ? (a > b) : (a < b);
          v[r] = sw ? b : a;
          v[r | j] = sw ? a : b;
        }
      } else {
        const int lj = j / KPL;
        const bool asc = (lane & (k / KPL)) == 0;
        const bool lower = (lane & lj) == 0;
#pragma unroll
        for (int r = 0; r < KPL; ++r) {
          const unsigned long long o = __shfl_xor_sync(0xffffffffu, v[r], lj);
          // the lower element of an ascending pair (or the upper of a descending one) keeps
          // the smaller key
          v[r] = (asc == lower) ? (v[r] < o ? v[r] : o) : (v[r] > o ? v[r] : o);
        }
      }
    }
  }
}

// Runs of 32 KPL keys of g[0, n), one warp each, sorted into A (padded with the largest key
// up to the end of the last run).
template <int KPL>
__device__ __forceinline__ void sort_runs(const unsigned long long* g, int n, unsigned long long* A, const Group& G) {
  constexpr int L = 32 * KPL;
  const int lane = G.t & 31, warp = G.t >> 5, nw = G.n >> 5;
  for (int r = warp; L * r < n; r += nw) {
    unsigned long long v[KPL];
    const int base = L * r + KPL * lane;
#pragma unroll
    for (int k = 0; k < KPL; ++k) v[k] = base + k < n ? g[base + k] : ~0ull;
    warp_bitonic<KPL>(v, lane);
#pragma unroll
    for (int k = 0; k < KPL; ++k) A[base + k] = v[k];
  }
}

// Ascending merge sort of g[0, n) (n <= 256 * warps of the group) in shared memory by the whole
// group: runs sorted in registers, one per warp (sort_runs), then merge levels between two
// shared buffers, each thread producing an equal slice of every level's output (merge path
// search + a sequential merge of its slice). Runs are 256 keys long when nearly every warp
// gets one, else 128 or 64 (a warp without a run would wait at the barrier). The keys are
// padded to a power of two N with the largest key, so every output position from n on
// holds padding at every level: both buffers are padded once, and the runs and output
// slices starting at n or later are skipped.
__device__ __noinline__ void merge_sort_smem(unsigned long long* g, int n, unsigned long long* A,
                                             unsigned long long* Bf, const Group G) {
  const int T = G.n, t = G.t, nw = T >> 5;
  const int run = n > (nw - 1) * 256 ? 256 : (n > (nw - 1) * 128 ? 128 : 64);
  int N = run;
  while (N < n) N <<= 1;
  if (run == 256) sort_runs<8>(g, n, A, G);
  else if (run == 128) sort_runs<4>(g, n, A, G);
  else sort_runs<2>(g, n, A, G);
  for (int i = ((n + run - 1) / run) * run + t; i < N; i += T) A[i] = ~0ull;
  for (int i = n + t; i < N; i += T) Bf[i] = ~0ull;
  G.sync();
  unsigned long long* src = A;
  unsigned long long* dst = Bf;
  for (int w = run; w < N; w <<= 1) {
    const int P = N / T > 0 ? N / T : 1;      // outputs per thread; divides 2w
    for (int d0 = t * P; d0 < n; d0 += T * P) {
      const int base = (d0 / (2 * w)) * (2 * w), loc = d0 - base;
      const unsigned long long* a = src + base;
      const unsigned long long* b = src + base + w;
      int lo = max(0, loc - w), hi = min(loc, w);
      while (lo < hi) {
        const int i = (lo + hi) >> 1;
        if (a[i] < b[loc - i - 1]) lo = i + 1; else hi = i;
      }
      int i = lo, j = loc - lo;
      for (int d = 0; d < P; ++d) {
        const bool ta = j >= w || (i < w && a[i] < b[j]);
        dst[base + loc + d] = ta ? a[i] : b[j];
        i += ta;
        j += !ta;
      }
    }
    G.sync();
    unsigned long long* tmp = src; src = dst; dst = tmp;
  }
  for (int i = t; i < n; i += T) g[i] = src[i];
}

// Whether a bin is rasterised by this render: with an owned-tile set, whether any 32x32-pixel
// tile the bin covers is owned (a bin of 16 pixels lies in one tile, one of 64 spans up to
// four).
__device__ __forceinline__ bool bin_owned(const Ws& ws, int bin) {
  const int v = view_of_bin(ws.views, ws.n_views, bin);
  const ViewDev& V = ws.views[v];
  if (!V.owned) return true;
  const int b = bin - V.bin_base, lg = ws.bin_log2;
  const int x0 = (b % V.nbx) << lg, y0 = (b / V.nbx) << lg;
  const int x1 = min(x0 + (1 << lg), V.width) - 1, y1 = min(y0 + (1 << lg), V.height) - 1;
  for (int ty = y0 >> kTileLog2; ty <= (y1 >> kTileLog2); ++ty)
    for (int tx = x0 >> kTileLog2; tx <= (x1 >> kTileLog2); ++tx)
      if (tile_owned(V, tx << kTileLog2, ty << kTileLog2)) return true;
  return false;
}

// One persistent CTA per SM. It takes the high-density bins first, one at a time with all its
// threads, then its quarters take the other non-empty bins, largest first: while a few CTAs still
// sort the largest bins, the others have gone on. Bound by latency and issue (46% of the slots). As
// two kernels one after the other, the small bins merge-sorted: 2M particles 41 + 80 us against
// 82 us, the layer frame 41 + 4 against 31, a batch of six mixed views 131 against 74.
__global__ __launch_bounds__(kSortThreads, 1) void k_bin_sort(Ws ws) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char sort_smem[];
  __shared__ int s_bin[4];
  __shared__ uint32_t s_red[4][64];
  if (ws.ctrl->error == LR_ERR_OVERFLOW) return;
  const unsigned long long n_big = ws.ctrl->bins_high, n_all = ws.ctrl->bins_nonempty;
  // bin_order holds k_raster's bins, then k_raster_ordered's: the k-th dense bin, the k-th other one
  const unsigned long long n_general = ws.ctrl->n_general, high_g = ws.ctrl->high_general, full_g = ws.ctrl->nonempty_general;
  auto dense_bin = [&](unsigned long long k) { return (int)ws.bin_order[k < high_g ? k : n_general + (k - high_g)]; };
  auto small_bin = [&](unsigned long long k) {
    return (int)ws.bin_order[high_g + k < full_g ? high_g + k : n_general + (n_big - high_g) + (high_g + k - full_g)];
  };
  const Group C{(int)threadIdx.x, kSortThreads, 0};
  unsigned long long* sbuf = reinterpret_cast<unsigned long long*>(sort_smem);
  uint32_t* stage = reinterpret_cast<uint32_t*>(sort_smem);
  while (n_big) {
    if (threadIdx.x == 0) {
      const unsigned long long k = atomicAdd(&ws.ctrl->sort_head, 1ull);
      s_bin[0] = k < n_big ? dense_bin(k) : -1;
    }
    C.sync();
    const int bin = s_bin[0];
    C.sync();
    if (bin < 0) break;
    if (!bin_owned(ws, bin)) continue;  // a tile another renderer rasterises
    const uint32_t off = ws.bin_off[bin];
    const int n = (int)(ws.bin_off[bin + 1] - off);
    unsigned long long* r = ws.refs + off;
    if (n <= kBucketBigCap && cta_bucket_sort(r, n, sbuf, reinterpret_cast<uint32_t*>(sbuf + kBucketBigCap), s_red[0], C)) {
      if (threadIdx.x == 0) atomicAdd(&ws.ctrl->sort_branch[0], 1ull);
      write_hb_bitmap(ws, r, n, bin, stage, (int)(kSortSmemBytes / 4), C);
      C.sync();
      continue;
    }
    const int run0 = n <= kSortBigCap ? n : kSortBigCap;
    if (threadIdx.x == 0) atomicAdd(&ws.ctrl->sort_branch[n <= kSortBigCap ? 1 : 2], 1ull);
    C.sync();
    // sort runs of up to kSortBigCap references in shared memory
    for (int s = 0; s < n; s += run0) {
      merge_sort_smem(r + s, min(run0, n - s), sbuf, sbuf + kSortBigCap, C);
      C.sync();
    }
    // merge the runs through the global buffer (only for more than kSortBigCap)
    unsigned long long* src = r;
    unsigned long long* dst = ws.refs_tmp + off;
    for (int run = run0; run < n; run <<= 1) {
      for (int s = 0; s < n; s += 2 * run) {
        const int na = min(run, n - s);
        const int nbb = min(run, max(0, n - s - run));
        cta_merge(src + s, na, src + s + na, nbb, dst + s);
      }
      C.sync();
      unsigned long long* t = src; src = dst; dst = t;
    }
    if (src != r) {
      for (int i = threadIdx.x; i < n; i += blockDim.x) r[i] = src[i];
    }
    C.sync();
    write_hb_bitmap(ws, r, n, bin, stage, (int)(kSortSmemBytes / 4), C);
    C.sync();
  }
  const int q = (int)(threadIdx.x / (kSortThreads / 4));
  const Group G{(int)(threadIdx.x % (kSortThreads / 4)), kSortThreads / 4, 1 + q};
  SmallSort& S = reinterpret_cast<SmallSort*>(sort_smem)[q];
  auto ticket = [&]() {
    const unsigned long long k = atomicAdd(&ws.ctrl->sort_small_head, 1ull);
    return k < n_all - n_big ? small_bin(k) : -1;
  };
  int k = 0;   // (thread 0 of the quarter; the next bin is drawn while one is sorted)
  if (G.t == 0) s_bin[q] = ticket();
  for (;;) {
    G.sync();
    const int bin = s_bin[q];
    if (bin < 0) return;
    if (G.t == 0) k = ticket();
    if (bin_owned(ws, bin)) {
      const uint32_t off = ws.bin_off[bin];
      const int n = (int)(ws.bin_off[bin + 1] - off);
      unsigned long long* r = ws.refs + off;
      const bool done = n <= kSortThreads / 4       ? small_bucket_sort<1>(ws, r, n, bin, S, s_red[q], G)
                        : n <= 2 * kSortThreads / 4 ? small_bucket_sort<2>(ws, r, n, bin, S, s_red[q], G)
                        : n <= 3 * kSortThreads / 4 ? small_bucket_sort<3>(ws, r, n, bin, S, s_red[q], G)
                        : n <= kSortThreads         ? small_bucket_sort<4>(ws, r, n, bin, S, s_red[q], G)
                                                    : small_bucket_sort<8>(ws, r, n, bin, S, s_red[q], G);
      if (!done) {
        if (!small_plane_sort(r, n, S, s_red[q], G)) {
          G.sync();
          merge_sort_smem(r, n, S.a, S.b, G);
          G.sync();
        }
        write_hb_bitmap(ws, r, n, bin, reinterpret_cast<uint32_t*>(S.a), kStageWords, G);
      }
    }
    G.sync();
    if (G.t == 0) s_bin[q] = k;
  }
}
static_assert(4 * sizeof(SmallSort) <= kSortSmemBytes, "a quarter of the CTA's shared memory each");

}  // namespace lr
