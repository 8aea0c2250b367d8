// analysis.cu -- implicit dependence analysis on the GPU.
//
// Pipeline (one graph, all launches so far):
//  1. bin count:  each rectangle -> number of tiles it overlaps
//  2. scan + expand: one (tile, packed entry) per overlap, written in
//     rectangle order with coalesced int4 loads of the rectangle arrays
//  3. stable radix sort by tile -> per tile, its candidates in program order
//  4. sweep (sweep.cu): one warp per tile walks the candidates in program
//     order, keeps per-cell run state in shared memory and emits (src, dst)
//     pairs deduplicated per task within the tile
//     (tiles whose pairs overflowed the buffer are swept again, alone, into a
//     larger one)
//  5. radix sort of the 64-bit pair keys, unique, CSR by source: row counts
//     and in-degrees by warp-aggregated atomics, row_ptr by a device scan
//  6. countdown counters (the in-degrees) and the compacted root list; the
//     executor's trigger records are packed from the CSR (exec.cu)
//
// The edge rule is the per-cell run reading of "infer the DAG from the data
// usage of tasks" (Section 2.2, Section 5): a task's rectangles combine into
// one privilege per cell, and each access gets edges from every member of the
// run preceding its own run at that cell.
#include "grt_internal.cuh"

namespace grt {

namespace {

// error bits of the device-side validation
constexpr uint32_t kErrReqOff = 1u, kErrRect = 2u, kErrPriv = 4u, kErrPred = 8u, kErrBodyArg = 16u, kErrBand = 32u;

// the last k in [0, n) with first[k] <= x (first[0] <= x, first nondecreasing)
__device__ __forceinline__ int32_t last_at_most(const int32_t* first, int32_t n, int64_t x) {
  int32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if ((int64_t)first[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Band placement of a captured batch (rt_batch_capture): rectangle r belongs
// to the task whose rectangle range holds it, which belongs to graph k; it must
// lie in graph k's own domain (kErrBand otherwise) and moves by graph k's shift
// into its band of the stacked domain. box[k] = {lo[D], hi[D], shift[D]}.
__global__ void k_band_place(const int32_t* req_off, int32_t n, const int32_t* task_first, int32_t G,
                             const int64_t* box, int D, int64_t* lo, int64_t* hi, int64_t R, uint32_t* err) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < R; r += stride) {
    const int32_t t = last_at_most(req_off, n, r);
    const int32_t k = last_at_most(task_first, G, t);
    const int64_t* b = box + (int64_t)k * 3 * D;
    bool outside = false;
    for (int d = 0; d < D; ++d) {
      const int64_t a = lo[r * D + d], c = hi[r * D + d];
      if (a < b[d] || c > b[D + d]) outside = true;
      lo[r * D + d] = a + b[2 * D + d];
      hi[r * D + d] = c + b[2 * D + d];
    }
    if (outside) atomicOr(err, kErrBand);
  }
}

// Checks one appended batch whose offsets were already shifted to graph-wide
// positions: req_off[0..n] must run from r_first to r_end without decreasing;
// pred_off likewise from p_first to p_end, every pred in [0, own id).
__global__ void k_validate_tasks(const int32_t* req_off, int32_t n, int64_t r_first, int64_t r_end,
                                 const int32_t* pred_off, const int32_t* pred, int64_t p_first,
                                 int64_t p_end, int32_t task_base, const int32_t* body_arg,
                                 int64_t body_limit, uint32_t* err) {
  int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i > n) return;
  uint32_t e = 0;
  if (i == 0 && (int64_t)req_off[0] != r_first) e |= kErrReqOff;
  if (i == n && (int64_t)req_off[n] != r_end) e |= kErrReqOff;
  if (pred_off && i == 0 && (int64_t)pred_off[0] != p_first) e |= kErrPred;
  if (pred_off && i == n && (int64_t)pred_off[n] != p_end) e |= kErrPred;
  if (i < n) {
    if (req_off[i + 1] < req_off[i]) e |= kErrReqOff;
    if (pred_off) {
      int32_t a = pred_off[i], b = pred_off[i + 1];
      if (b < a || (int64_t)a < p_first || (int64_t)b > p_end) {
        e |= kErrPred;
      } else {
        for (int32_t k = a; k < b; ++k) {
          int32_t p = pred[k];
          if (p < 0 || p >= task_base + i) {
            e |= kErrPred;
            break;
          }
        }
      }
    }
    if (body_arg && body_limit >= 0) {
      int32_t v = body_arg[i];
      if (v < 0 || (int64_t)v >= body_limit) e |= kErrBodyArg;
    }
  }
  if (e) atomicOr(err, e);
}

__global__ void k_validate_rects(const int64_t* lo, const int64_t* hi, const uint8_t* priv, int64_t R,
                                 AnalysisDims d, uint32_t* err) {
  int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= R) return;
  uint32_t e = 0;
  for (int k = 0; k < d.ndim; ++k) {
    int64_t a = lo[r * d.ndim + k], b = hi[r * d.ndim + k];
    if (a > b || a < d.dom_lo[k] || b > d.dom_lo[k] + d.ext[k] - 1) e |= kErrRect;
  }
  if (priv[r] > 2) e |= kErrPriv;
  if (e) atomicOr(err, e);
}

__global__ void k_add_offset(int32_t* a, int64_t n, int32_t add) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] += add;
}

// int32 rectangle bounds (both arrays, m values each) widened to int64 in the
// graph's own arrays
__global__ void k_widen_bounds(const int32_t* lo32, const int32_t* hi32, int64_t m, int64_t* lo, int64_t* hi) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
    lo[i] = lo32[i];
    hi[i] = hi32[i];
  }
}

// A batch's rectangles into the graph's own arrays, widened and checked in one
// pass (a copy each and a checking kernel read the bounds twice: 55 us more for
// 6.1M rectangles). priv_in may be priv. Two bounds go as one load and store
// where the caller's arrays allow it (wide).
template <class T, bool WIDE>
__global__ void __launch_bounds__(256) k_ingest_rects(const T* lo_in, const T* hi_in, const uint8_t* priv_in, int64_t R,
                                                      AnalysisDims d, int64_t* lo, int64_t* hi, uint8_t* priv,
                                                      uint32_t* err) {
  struct alignas(2 * sizeof(T)) Pair {
    T x, y;
  };
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= R) return;
  uint32_t e = 0;
  int64_t a[2] = {0, 0}, b[2] = {0, 0};
  if (WIDE) {
    const Pair p = reinterpret_cast<const Pair*>(lo_in)[r], q = reinterpret_cast<const Pair*>(hi_in)[r];
    a[0] = p.x;
    a[1] = p.y;
    b[0] = q.x;
    b[1] = q.y;
    reinterpret_cast<longlong2*>(lo)[r] = make_longlong2(a[0], a[1]);
    reinterpret_cast<longlong2*>(hi)[r] = make_longlong2(b[0], b[1]);
  } else {
    for (int k = 0; k < d.ndim; ++k) {
      lo[r * d.ndim + k] = a[k] = lo_in[r * d.ndim + k];
      hi[r * d.ndim + k] = b[k] = hi_in[r * d.ndim + k];
    }
  }
  for (int k = 0; k < d.ndim; ++k)
    if (a[k] > b[k] || a[k] < d.dom_lo[k] || b[k] > d.dom_lo[k] + d.ext[k] - 1) e |= kErrRect;
  const uint8_t p = priv_in[r];
  if (p > 2) e |= kErrPriv;
  priv[r] = p;
  if (e) atomicOr(err, e);
}

// tile range of one rectangle (coordinates relative to the domain origin)
struct TileRange {
  int64_t lx, hx, ly, hy;  // relative inclusive bounds
  int32_t tx0, ty0, ntx, nty;
};

__device__ __forceinline__ TileRange tile_range(const int64_t* lo, const int64_t* hi, int64_t r,
                                                const AnalysisDims& d) {
  TileRange t;
  if (d.ndim == 2) {
    // one 16-byte load per corner: the rectangle arrays are int64[R][2]
    longlong2 a = *reinterpret_cast<const longlong2*>(lo + 2 * r);
    longlong2 b = *reinterpret_cast<const longlong2*>(hi + 2 * r);
    t.lx = a.x - d.dom_lo[0];
    t.hx = b.x - d.dom_lo[0];
    t.ly = a.y - d.dom_lo[1];
    t.hy = b.y - d.dom_lo[1];
  } else {
    t.lx = lo[r] - d.dom_lo[0];
    t.hx = hi[r] - d.dom_lo[0];
    t.ly = 0;
    t.hy = 0;
  }
  // a 64-bit division takes about a hundred instructions, and there are four
  if (d.shx >= 0) {
    t.tx0 = (int32_t)(t.lx >> d.shx);
    t.ty0 = (int32_t)(t.ly >> d.shy);
    t.ntx = (int32_t)(t.hx >> d.shx) - t.tx0 + 1;
    t.nty = (int32_t)(t.hy >> d.shy) - t.ty0 + 1;
  } else {
    t.tx0 = (int32_t)(t.lx / d.tw);
    t.ty0 = (int32_t)(t.ly / d.th);
    t.ntx = (int32_t)(t.hx / d.tw) - t.tx0 + 1;
    t.nty = (int32_t)(t.hy / d.th) - t.ty0 + 1;
  }
  return t;
}

// Each rectangle's tiles, and its task. A warp takes the rectangles of 32
// consecutive tasks, one per lane at a time, so that the corners' loads coalesce
// (a thread per task, each walking its own rectangles: 81 us for 6.1M rectangles
// of 1M tasks). Also adds up the cells of all rectangles (area[0], zeroed by the
// caller) and their tiles (area[1], in 64 bits: the counts themselves are only
// scanned once the sum is known to fit), which together say how much of their
// tiles the entries cover; and clears zero[0..n), the pair counts per source of the CSR stage.
__global__ void __launch_bounds__(256) k_bin_count(const int32_t* __restrict__ req_off, int32_t n, int64_t R,
                                                   const int64_t* __restrict__ lo, const int64_t* __restrict__ hi,
                                                   AnalysisDims d, int32_t* __restrict__ rect_task,
                                                   uint32_t* __restrict__ cnt, unsigned long long* area,
                                                   uint32_t* __restrict__ zero) {
  __shared__ unsigned long long part[8][2];
  const int lane = threadIdx.x & 31;
  const int32_t t = blockIdx.x * blockDim.x + threadIdx.x, t0 = t - lane;
  unsigned long long sum = 0, tiles = 0;
  if (t < n) zero[t] = 0u;
  // lane l holds the first rectangle of task t0 + l
  const int32_t first = req_off[t < n ? t : n];
  int32_t end = __shfl_sync(0xffffffffu, req_off[t + 1 < n ? t + 1 : n], 31);
  if ((int64_t)end > R) end = (int32_t)R;
  const int32_t begin = __shfl_sync(0xffffffffu, first, 0);
  for (int32_t r0 = begin > 0 ? begin : 0; r0 < end; r0 += 32) {  // (offsets not yet validated)
    const int32_t r = r0 + lane;
    int own = 0;  // the last task of the 32 whose first rectangle is at most r
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1)
      if (__shfl_sync(0xffffffffu, first, own + step) <= r) own += step;
    if (r < end) {
      rect_task[r] = t0 + own;
      const TileRange tr = tile_range(lo, hi, r, d);
      cnt[r] = (uint32_t)tr.ntx * (uint32_t)tr.nty;  // at most the domain's 2^26 tiles
      tiles += (unsigned long long)tr.ntx * (unsigned long long)tr.nty;
      sum += (unsigned long long)(tr.hx - tr.lx + 1) * (unsigned long long)(tr.hy - tr.ly + 1);
    }
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    tiles += __shfl_xor_sync(0xffffffffu, tiles, o);
  }
  if (lane == 0) {
    part[threadIdx.x >> 5][0] = sum;
    part[threadIdx.x >> 5][1] = tiles;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    sum = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) sum += part[w][threadIdx.x];
    if (sum) red_add_u64(area + threadIdx.x, sum);
  }
}

// One thread per rectangle: a rectangle over a few tiles writes its own
// entries; the entries of a larger one are written by its whole warp
// (lane-strided), so that large rectangles do not serialise on one lane. Only a
// rectangle's first and last tile column (row) cut it, so an entry's box is four
// selections of 32-bit offsets.
constexpr uint32_t kOwnTiles = 4;

__global__ void __launch_bounds__(256) k_bin_expand(const int32_t* __restrict__ rect_task,
                                                    const int64_t* __restrict__ lo, const int64_t* __restrict__ hi,
                                                    const uint8_t* __restrict__ priv, int64_t R,
                                                    const uint32_t* __restrict__ off, AnalysisDims d,
                                                    uint32_t* __restrict__ keys, uint64_t* __restrict__ payload) {
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  const bool valid = r < R;
  uint32_t base = 0, cnt = 0, task = 0, pv = 0, tile0 = 0;
  int ntx = 1, nty = 1, fx = 0, lx = 0, fy = 0, ly = 0;  // first and last column (row) inside their tiles
  if (valid) {
    const TileRange tr = tile_range(lo, hi, r, d);
    base = off[r];
    cnt = off[r + 1] - base;
    task = (uint32_t)rect_task[r];
    pv = priv[r];
    ntx = tr.ntx;
    nty = tr.nty;
    fx = (int)(tr.lx - (int64_t)tr.tx0 * d.tw);
    fy = (int)(tr.ly - (int64_t)tr.ty0 * d.th);
    lx = (int)(tr.hx - (int64_t)(tr.tx0 + ntx - 1) * d.tw);
    ly = (int)(tr.hy - (int64_t)(tr.ty0 + nty - 1) * d.th);
    tile0 = (uint32_t)tr.ty0 * (uint32_t)d.ntx + (uint32_t)tr.tx0;
  }
  auto put = [&](uint32_t at, uint32_t tile, int i, int j, int nx, int ny, int x0, int x1, int y0, int y1, uint32_t tk,
                 uint32_t p) {
    keys[at] = tile + (uint32_t)j * (uint32_t)d.ntx + (uint32_t)i;
    payload[at] = pack_entry(tk, p, d.ndim, (uint32_t)(i == 0 ? x0 : 0), (uint32_t)(i == nx - 1 ? x1 : d.tw - 1),
                             (uint32_t)(j == 0 ? y0 : 0), (uint32_t)(j == ny - 1 ? y1 : d.th - 1));
  };
  // A rectangle over at most kOwnTiles tiles (the usual case: one) is written
  // by its own lane; consecutive rectangles then write consecutive entries, so
  // the stores coalesce. Larger ones are written by the whole warp below.
  const bool own = valid && cnt <= kOwnTiles;
  if (own) {
    for (uint32_t k = 0, i = 0, j = 0; k < cnt; ++k) {
      put(base + k, tile0, (int)i, (int)j, ntx, nty, fx, lx, fy, ly, task, pv);
      if (++i == (uint32_t)ntx) {
        i = 0;
        ++j;
      }
    }
  }
  unsigned shared = __ballot_sync(0xffffffffu, valid && !own);
  while (shared) {
    const int s = __ffs((int)shared) - 1;
    shared &= shared - 1;
    const uint32_t c = __shfl_sync(0xffffffffu, cnt, s), b = __shfl_sync(0xffffffffu, base, s);
    const uint32_t t0 = __shfl_sync(0xffffffffu, tile0, s);
    const int nx = __shfl_sync(0xffffffffu, ntx, s), ny = __shfl_sync(0xffffffffu, nty, s);
    const int x0 = __shfl_sync(0xffffffffu, fx, s), x1 = __shfl_sync(0xffffffffu, lx, s);
    const int y0 = __shfl_sync(0xffffffffu, fy, s), y1 = __shfl_sync(0xffffffffu, ly, s);
    const uint32_t tk = __shfl_sync(0xffffffffu, task, s), p = __shfl_sync(0xffffffffu, pv, s);
    const int dj = 32 / nx, di = 32 - dj * nx;  // 32 entries further
    int j = lane / nx, i = lane - j * nx;
    for (uint32_t k = (uint32_t)lane; k < c; k += 32) {
      put(b + k, t0, i, j, nx, ny, x0, x1, y0, y1, tk, p);
      i += di;
      j += dj;
      if (i >= nx) {
        i -= nx;
        ++j;
      }
    }
  }
}

// Where each tile's entries begin and end in the sorted keys: a binary search
// per tile. (Marking the places where the key changes read all entries: 60 us of
// 20M entries, where 32768 searches take 9.)
__global__ void k_segments(const uint32_t* keys, int64_t M, int64_t ntiles, uint32_t* seg_begin, uint32_t* seg_end) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t > ntiles) return;
  int64_t lo = 0, hi = M;  // the first entry with a key of at least t
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)__ldg(keys + mid) < t) lo = mid + 1; else hi = mid;
  }
  if (t < ntiles) seg_begin[t] = (uint32_t)lo;
  if (t > 0) seg_end[t - 1] = (uint32_t)lo;
}

__global__ void k_explicit_pairs(const int32_t* pred_off, const int32_t* pred, int32_t n, int key_bits,
                                 uint64_t* pairs) {
  int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  for (int32_t k = pred_off[t]; k < pred_off[t + 1]; ++k)
    pairs[k] = ((uint64_t)(uint32_t)pred[k] << key_bits) | (uint32_t)t;
}

__global__ void k_unique_flags(const uint64_t* keys, int64_t P, uint32_t* flags) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  uint64_t k = keys[i];
  flags[i] = (k != kEmpty64 && (i == 0 || keys[i - 1] != k)) ? 1u : 0u;
}

// warp-aggregated increment: lanes adding to the same counter elect one leader
__device__ __forceinline__ void warp_agg_inc(int32_t* base, int32_t idx, bool active) {
  int32_t key = active ? idx : -1;
  unsigned peers = __match_any_sync(0xffffffffu, key);
  if (active && (peers & lanemask_lt()) == 0) red_add_s32(base + idx, (int32_t)__popc(peers));
}

__global__ void k_emit_csr(const uint64_t* keys, const uint32_t* flags, const uint32_t* upos, int64_t P,
                           int key_bits, int32_t* col, int32_t* rowcnt, int32_t* indeg) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool act = i < P && flags[i] != 0;
  int32_t src = 0, dst = 0;
  if (act) {
    uint64_t k = keys[i];
    src = (int32_t)(k >> key_bits);
    dst = (int32_t)(k & ((1ull << key_bits) - 1ull));
    col[upos[i]] = dst;
  }
  warp_agg_inc(rowcnt, src, act);
  warp_agg_inc(indeg, dst, act);
}

constexpr uint32_t kRowStage = 2560;  // targets of 256 consecutive rows staged in shared memory

// Everything the executors need of a task, in one pass: its counter (Algorithm
// 1: one pending-edge counter per node), its place among the roots (pos: the
// roots before it) and its trigger record; over all tasks the largest
// out-degree, the longest edge and the last root (shape[0..2])
__global__ void __launch_bounds__(256) k_finish_tasks(const int32_t* __restrict__ row_ptr,
                                                      const int32_t* __restrict__ col,
                                                      const int32_t* __restrict__ indeg,
                                                      const uint32_t* __restrict__ pos, int32_t n, int32_t* count,
                                                      uint64_t* root_items, int4* adj, uint32_t* shape) {
  // a block's rows lie side by side in col: staged through shared memory, so that
  // the loads coalesce (1M rows of 5: 45 us without)
  __shared__ int32_t stage[kRowStage];
  const int32_t v0 = (int32_t)(blockIdx.x * blockDim.x), v = v0 + (int32_t)threadIdx.x;
  const int32_t v1 = v0 + 256 < n ? v0 + 256 : n;
  const int32_t base = row_ptr[v0], total = row_ptr[v1] - base;
  const bool staged = total <= (int32_t)kRowStage;
  if (staged) {
    for (int32_t i = threadIdx.x; i < total; i += 256) stage[i] = col[base + i];
    __syncthreads();
  }
  int b = 0, d = 0;
  uint32_t far = 0, last = 0;
  if (v < n) {
    b = row_ptr[v];
    d = row_ptr[v + 1] - b;
    const int32_t in = indeg[v];
    count[v] = in;
    if (in == 0) {
      root_items[pos[v]] = (uint32_t)v;
      last = (uint32_t)v;
    }
    const int32_t* const row = staged ? stage + (b - base) : col + b;
    if (d > 0) far = (uint32_t)(row[d - 1] - v);  // a row's targets ascend
    int c[kAdjInline];
#pragma unroll
    for (int j = 0; j < kAdjInline; ++j) c[j] = j < d ? row[j] : -1;
    adj[2 * (int64_t)v] = make_int4(b, d, in, c[0]);
    adj[2 * (int64_t)v + 1] = make_int4(c[1], c[2], c[3], c[4]);
  }
  const uint32_t m[3] = {__reduce_max_sync(0xffffffffu, (uint32_t)d), __reduce_max_sync(0xffffffffu, far),
                         __reduce_max_sync(0xffffffffu, last)};
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (m[k] > *(volatile uint32_t*)(shape + k)) atomicMax(shape + k, m[k]);
  }
}

// Words of device memory into pinned host memory, for the host to read after
// the stream's synchronisation: one launch in place of a small copy each.
__global__ void k_report(ReportArgs a) {
  const int i = threadIdx.x;
  if (i >= a.n) return;
  if (a.wide[i]) *(volatile uint64_t*)a.dst[i] = *(const volatile uint64_t*)a.src[i];
  else *(volatile uint32_t*)a.dst[i] = *(const volatile uint32_t*)a.src[i];
}

// ---------------------------------------------------------------------------
// CSR by buckets (graphs whose rows hold at most kBucketMaxRow candidate
// pairs): the pairs are counted per source, each pair's target is scattered
// into its source's bucket, every bucket is sorted and deduplicated in place,
// and the unique targets are compacted into the CSR. One pass over the pairs
// and a few over the targets, where an LSD radix sort of (source, target) keys
// makes five.
// ---------------------------------------------------------------------------
constexpr int kBucketSmallRow = 32;  // rows sorted by one thread
constexpr int kBucketLanes = 32;

// pairs counted per source; the pair count is read on the device (the sweep's
// cursor, capped at the buffer) so that no host sync is needed before it
__global__ void k_bucket_count(const uint64_t* pairs, const unsigned long long* cursor, unsigned long long cap,
                               int key_bits, uint32_t* cnt) {
  const unsigned long long P = *cursor < cap ? *cursor : cap;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x; i0 < (int64_t)P; i0 += stride) {
    const int64_t i = i0 + threadIdx.x;
    const uint64_t k = i < (int64_t)P ? pairs[i] : kEmpty64;
    const int src = k != kEmpty64 ? (int)(k >> key_bits) : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, src);
    if (src >= 0 && (peers & lanemask_lt()) == 0) red_add_u32(cnt + src, (uint32_t)__popc(peers));
  }
}

// the longest row (atomicMax into *out)
__global__ void k_bucket_maxrow(const uint32_t* cnt, int32_t n, uint32_t* out) {
  uint32_t m = 0;
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) m = max(m, cnt[v]);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

// each pair's target into its source's bucket: positions off[src] .. off[src]
// + cnt[src] - 1, handed out by counting cnt down (it ends at 0)
__global__ void k_bucket_scatter(const uint64_t* pairs, int64_t P, int key_bits, const uint32_t* off, uint32_t* cnt,
                                 uint32_t* bucket) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t k = i < P ? pairs[i] : kEmpty64;
  const int src = k != kEmpty64 ? (int)(k >> key_bits) : -1;
  const unsigned peers = __match_any_sync(0xffffffffu, src);
  const int leader = __ffs((int)peers) - 1;
  uint32_t old = 0;
  if (src >= 0 && (peers & lanemask_lt()) == 0) old = atomicSub(cnt + src, (uint32_t)__popc(peers));
  old = __shfl_sync(0xffffffffu, old, leader);
  if (src >= 0) {
    const uint32_t rank = (uint32_t)__popc(peers & lanemask_lt());
    bucket[off[src] + old - 1u - rank] = (uint32_t)(k & ((1ull << key_bits) - 1ull));
  }
}

// rows of at most kBucketSmallRow pairs: one thread sorts its row and keeps the
// distinct targets at its front; longer rows are listed for k_bucket_sort_large;
// the in-degrees are cleared on the way. A block's rows lie side by side: up to
// kRowStage targets they are staged in shared memory, read and written back
// coalesced (1M rows of 5: 62 us without).
__global__ void __launch_bounds__(256) k_bucket_sort_small(const uint32_t* off, int32_t n, uint32_t* bucket,
                                                           uint32_t* ucnt, uint32_t* big, uint32_t* nbig,
                                                           int32_t* indeg) {
  __shared__ uint32_t stage[kRowStage];
  const int32_t v0 = (int32_t)(blockIdx.x * blockDim.x), v = v0 + (int32_t)threadIdx.x;
  const int32_t v1 = v0 + 256 < n ? v0 + 256 : n;
  const uint32_t base = off[v0], total = off[v1] - base;
  const bool staged = total <= kRowStage;
  if (staged) {
    for (uint32_t i = threadIdx.x; i < total; i += 256) stage[i] = bucket[base + i];
    __syncthreads();
  }
  if (v < n) {
    indeg[v] = 0;  // counted by the compaction
    const uint32_t a = off[v], len = off[v + 1] - a;
    uint32_t* b = staged ? stage + (a - base) : bucket + a;
    if (len > (uint32_t)kBucketSmallRow) {
      big[atomicAdd(nbig, 1u)] = (uint32_t)v;
    } else if (len <= 8u) {
      // the usual short row in registers: 8 loads in flight and an odd-even
      // transposition network
      uint32_t x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = (uint32_t)i < len ? b[i] : 0xFFFFFFFFu;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
#pragma unroll
        for (int i = r & 1; i + 1 < 8; i += 2) {
          const uint32_t lo = min(x[i], x[i + 1]), hi = max(x[i], x[i + 1]);
          x[i] = lo;
          x[i + 1] = hi;
        }
      }
      uint32_t u = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if ((uint32_t)i < len && (i == 0 || x[i] != x[i > 0 ? i - 1 : 0])) b[u++] = x[i];
      ucnt[v] = u;
    } else {
      for (uint32_t i = 1; i < len; ++i) {
        const uint32_t x = b[i];
        int j = (int)i - 1;
        while (j >= 0 && b[j] > x) {
          b[j + 1] = b[j];
          --j;
        }
        b[j + 1] = x;
      }
      uint32_t u = 0;
      for (uint32_t i = 0; i < len; ++i)
        if (u == 0 || b[i] != b[u - 1]) b[u++] = b[i];
      ucnt[v] = u;
    }
  }
  if (staged) {
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < total; i += 256) bucket[base + i] = stage[i];
  }
}

// The same where rows are longer on average: a warp per row, its targets one per
// lane, sorted by a bitonic network of shuffles (the thread-per-row insertion
// took 61 us for 5317 rows of 25 pairs).
__global__ void __launch_bounds__(256) k_bucket_sort_warp(const uint32_t* __restrict__ off, int32_t n,
                                                          uint32_t* __restrict__ bucket, uint32_t* __restrict__ ucnt,
                                                          uint32_t* big, uint32_t* nbig, int32_t* __restrict__ indeg) {
  const int lane = threadIdx.x & 31;
  const int32_t v = (int32_t)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
  if (v >= n) return;
  const uint32_t a = off[v], len = off[v + 1] - a;
  if (lane == 0) indeg[v] = 0;  // counted by the compaction
  if (len > (uint32_t)kBucketSmallRow) {
    if (lane == 0) big[atomicAdd(nbig, 1u)] = (uint32_t)v;
    return;
  }
  uint32_t x = (uint32_t)lane < len ? bucket[a + lane] : 0xFFFFFFFFu;
#pragma unroll
  for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
      const bool low = (lane & j) == 0, up = (lane & k) == 0;
      x = low == up ? min(x, y) : max(x, y);
    }
  }
  const uint32_t before = __shfl_up_sync(0xffffffffu, x, 1);
  const bool keep = (uint32_t)lane < len && (lane == 0 || x != before);
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  if (keep) bucket[a + (uint32_t)__popc(m & lanemask_lt())] = x;
  if (lane == 0) ucnt[v] = (uint32_t)__popc(m);
}

// Row v of len targets at b, 32 < len <= 32 E, by one warp: E targets a lane
// (target 32 e + lane in x[e]), a bitonic network of shuffles and of exchanges
// between a lane's own registers; the distinct ones to the front.
template <int E>
__device__ __forceinline__ uint32_t sort_row(uint32_t* b, uint32_t len) {
  const int lane = threadIdx.x & 31;
  uint32_t x[E];
#pragma unroll
  for (int e = 0; e < E; ++e) x[e] = (uint32_t)(32 * e + lane) < len ? b[32 * e + lane] : 0xFFFFFFFFu;
#pragma unroll
  for (int k = 2; k <= 32 * E; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        if (j >= 32) {
          const int f = e ^ (j >> 5);
          if (f > e) {
            const uint32_t lo = min(x[e], x[f]), hi = max(x[e], x[f]);
            const bool up = ((32 * e) & k) == 0;
            x[e] = up ? lo : hi;
            x[f] = up ? hi : lo;
          }
        } else {
          const uint32_t y = __shfl_xor_sync(0xffffffffu, x[e], j);
          const bool low = (lane & j) == 0, up = ((32 * e + lane) & k) == 0;
          x[e] = low == up ? min(x[e], y) : max(x[e], y);
        }
      }
    }
  }
  uint32_t u = 0, last = 0xFFFFFFFFu;  // no target is ~0
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const uint32_t left = __shfl_up_sync(0xffffffffu, x[e], 1);
    const bool keep = (uint32_t)(32 * e + lane) < len && x[e] != (lane == 0 ? last : left);
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (keep) b[u + (uint32_t)__popc(m & lanemask_lt())] = x[e];
    u += (uint32_t)__popc(m);
    last = __shfl_sync(0xffffffffu, x[e], 31);
  }
  return u;
}

// the listed long rows (at most kBucketMaxRow pairs): one warp each, a bitonic
// sort in shared memory padded with ~0, then the distinct targets written back
// to the row's front. Up to 256 pairs the row stays in registers (in shared memory
// half the lanes idle in each exchange: analysis of 5317 dense launches 0.375 ->
// 0.360 ms, of the 1M-launch trace 38.2 -> 37.5).
__global__ void __launch_bounds__(128) k_bucket_sort_large(const uint32_t* off, uint32_t* bucket, uint32_t* ucnt,
                                                           const uint32_t* big, const uint32_t* nbig) {
  __shared__ uint32_t buf[4][kBucketMaxRow];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t* s = buf[warp];
  const uint32_t nb = *nbig;
  for (uint32_t r = blockIdx.x * 4 + warp; r < nb; r += gridDim.x * 4) {
    const uint32_t v = big[r];
    const uint32_t a = off[v], len = off[v + 1] - a;
    if (len <= 256u) {
      const uint32_t d = len <= 64u    ? sort_row<2>(bucket + a, len)
                         : len <= 128u ? sort_row<4>(bucket + a, len)
                                       : sort_row<8>(bucket + a, len);
      if (lane == 0) ucnt[v] = d;
      continue;
    }
    uint32_t N = 512;
    while (N < len) N <<= 1;
    for (uint32_t i = lane; i < N; i += 32) s[i] = i < len ? bucket[a + i] : 0xFFFFFFFFu;
    __syncwarp();
    for (uint32_t k = 2; k <= N; k <<= 1) {
      for (uint32_t j = k >> 1; j > 0; j >>= 1) {
        for (uint32_t i = lane; i < N; i += 32) {
          const uint32_t p = i ^ j;
          if (p > i) {
            const uint32_t x = s[i], y = s[p];
            const bool up = (i & k) == 0;
            if ((x > y) == up) {
              s[i] = y;
              s[p] = x;
            }
          }
        }
        __syncwarp();
      }
    }
    uint32_t u = 0;
    for (uint32_t i0 = 0; i0 < len; i0 += 32) {
      const uint32_t i = i0 + lane;
      const bool keep = i < len && (i == 0 || s[i] != s[i - 1]);
      const unsigned m = __ballot_sync(0xffffffffu, keep);
      if (keep) bucket[a + u + (uint32_t)__popc(m & lanemask_lt())] = s[i];
      u += (uint32_t)__popc(m);
    }
    if (lane == 0) ucnt[v] = u;
    __syncwarp();
  }
}

// the distinct targets of every row into the CSR's columns, and in-degrees (the
// columns of a block's rows, side by side, leave through shared memory)
__global__ void __launch_bounds__(256) k_bucket_compact(const uint32_t* off, const uint32_t* row_ptr, int32_t n,
                                                        const uint32_t* bucket, int32_t* col, int32_t* indeg) {
  __shared__ uint32_t stage[kRowStage];
  const int32_t v0 = (int32_t)(blockIdx.x * blockDim.x), v = v0 + (int32_t)threadIdx.x;
  const int32_t v1 = v0 + 256 < n ? v0 + 256 : n;
  const uint32_t base = row_ptr[v0], total = row_ptr[v1] - base;
  const bool staged = total <= kRowStage;
  if (v < n) {
    const uint32_t a = off[v], o = row_ptr[v], u = row_ptr[v + 1] - o;
    for (uint32_t i = 0; i < u; ++i) {
      const uint32_t t = bucket[a + i];
      if (staged) stage[o - base + i] = t; else col[o + i] = (int32_t)t;
      if (!staged) red_add_s32(indeg + t, 1);
    }
  }
  if (staged) {
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < total; i += 256) {
      const uint32_t t = stage[i];
      col[base + i] = (int32_t)t;
      red_add_s32(indeg + t, 1);
    }
  }
}

// the same with a warp per row, where rows are longer on average
__global__ void __launch_bounds__(256) k_bucket_compact_warp(const uint32_t* __restrict__ off,
                                                             const uint32_t* __restrict__ row_ptr, int32_t n,
                                                             const uint32_t* __restrict__ bucket,
                                                             int32_t* __restrict__ col, int32_t* indeg) {
  const uint32_t lane = threadIdx.x & 31u;
  const int32_t v = (int32_t)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
  if (v >= n) return;
  const uint32_t a = off[v], o = row_ptr[v], u = row_ptr[v + 1] - o;
  for (uint32_t i = lane; i < u; i += 32) {
    const uint32_t t = bucket[a + i];
    col[o + i] = (int32_t)t;
    red_add_s32(indeg + t, 1);
  }
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

void launch_validate(const int32_t* req_off, int32_t n, int64_t r_first, const int64_t* lo,
                     const int64_t* hi, const uint8_t* priv, int64_t R, bool rects_checked, const int32_t* pred_off,
                     const int32_t* pred, int64_t p_first, int64_t p_end, int32_t task_base,
                     const int32_t* body_arg, int64_t body_limit, AnalysisDims d, uint32_t* err,
                     cudaStream_t s) {
  count_launch();
  k_validate_tasks<<<nblk((int64_t)n + 1, 256), 256, 0, s>>>(req_off, n, r_first, r_first + R, pred_off,
                                                           pred, p_first, p_end, task_base, body_arg,
                                                           body_limit, err);
  if (R > 0 && !rects_checked) {
    count_launch();
    k_validate_rects<<<nblk(R, 256), 256, 0, s>>>(lo, hi, priv, R, d, err);
  }
}

void launch_band_place(const int32_t* req_off, int32_t n, const int32_t* task_first, int32_t G, const int64_t* box,
                       int D, int64_t* lo, int64_t* hi, int64_t R, uint32_t* err, cudaStream_t s) {
  if (R <= 0) return;
  unsigned blocks = nblk(R, 256);
  if (blocks > 4096) blocks = 4096;
  count_launch();
  k_band_place<<<blocks, 256, 0, s>>>(req_off, n, task_first, G, box, D, lo, hi, R, err);
}

void launch_widen_bounds(const int32_t* lo32, const int32_t* hi32, int64_t m, int64_t* lo, int64_t* hi,
                         cudaStream_t s) {
  if (m <= 0) return;
  unsigned blocks = nblk(m, 256);
  if (blocks > 8192) blocks = 8192;
  count_launch();
  k_widen_bounds<<<blocks, 256, 0, s>>>(lo32, hi32, m, lo, hi);
}

template <class T>
void launch_ingest_rects(const T* lo_in, const T* hi_in, const uint8_t* priv_in, int64_t R, AnalysisDims d, int64_t* lo,
                         int64_t* hi, uint8_t* priv, uint32_t* err, cudaStream_t s) {
  if (R <= 0) return;
  count_launch();
  const uintptr_t at = reinterpret_cast<uintptr_t>(lo_in) | reinterpret_cast<uintptr_t>(hi_in);
  const uintptr_t to = reinterpret_cast<uintptr_t>(lo) | reinterpret_cast<uintptr_t>(hi);
  if (d.ndim == 2 && at % (2 * sizeof(T)) == 0 && to % 16 == 0)
    k_ingest_rects<T, true><<<nblk(R, 256), 256, 0, s>>>(lo_in, hi_in, priv_in, R, d, lo, hi, priv, err);
  else
    k_ingest_rects<T, false><<<nblk(R, 256), 256, 0, s>>>(lo_in, hi_in, priv_in, R, d, lo, hi, priv, err);
}
template void launch_ingest_rects<int32_t>(const int32_t*, const int32_t*, const uint8_t*, int64_t, AnalysisDims,
                                           int64_t*, int64_t*, uint8_t*, uint32_t*, cudaStream_t);
template void launch_ingest_rects<int64_t>(const int64_t*, const int64_t*, const uint8_t*, int64_t, AnalysisDims,
                                           int64_t*, int64_t*, uint8_t*, uint32_t*, cudaStream_t);

void launch_add_offset(int32_t* a, int64_t n, int32_t add, cudaStream_t s) {
  if (n > 0 && add != 0) {
    count_launch();
    k_add_offset<<<nblk(n, 256), 256, 0, s>>>(a, n, add);
  }
}

void launch_bin_count(const int32_t* req_off, int32_t n, int64_t R, const int64_t* lo, const int64_t* hi,
                      AnalysisDims d, int32_t* rect_task, uint32_t* cnt, unsigned long long* area,
                      uint32_t* zero, cudaStream_t s) {
  if (n > 0) {
    count_launch();
    k_bin_count<<<nblk(n, 256), 256, 0, s>>>(req_off, n, R, lo, hi, d, rect_task, cnt, area, zero);
  }
}

void launch_bin_expand(const int32_t* rect_task, const int64_t* lo, const int64_t* hi,
                       const uint8_t* priv, int64_t R, const uint32_t* off, AnalysisDims d,
                       uint32_t* keys, uint64_t* payload, cudaStream_t s) {
  if (R > 0) {
    count_launch();
    k_bin_expand<<<nblk(R, 256), 256, 0, s>>>(rect_task, lo, hi, priv, R, off, d, keys, payload);
  }
}

void launch_segments(const uint32_t* keys, int64_t M, int64_t ntiles, uint32_t* seg_begin, uint32_t* seg_end,
                     cudaStream_t s) {
  if (M > 0) {
    count_launch();
    k_segments<<<nblk(ntiles + 1, 128), 128, 0, s>>>(keys, M, ntiles, seg_begin, seg_end);
  }
}

void launch_explicit_pairs(const int32_t* pred_off, const int32_t* pred, int32_t n, int key_bits,
                           uint64_t* pairs, cudaStream_t s) {
  if (n > 0) {
    count_launch();
    k_explicit_pairs<<<nblk(n, 256), 256, 0, s>>>(pred_off, pred, n, key_bits, pairs);
  }
}

void launch_unique_flags(const uint64_t* keys, int64_t P, uint32_t* flags, cudaStream_t s) {
  if (P > 0) {
    count_launch();
    k_unique_flags<<<nblk(P, 256), 256, 0, s>>>(keys, P, flags);
  }
}

void launch_bucket_count(const uint64_t* pairs, const unsigned long long* cursor, unsigned long long cap,
                         int key_bits, uint32_t* cnt, int32_t n, uint32_t* maxrow, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  count_launch(2);
  k_bucket_count<<<(unsigned)(sms > 0 ? sms * 8 : 1024), 256, 0, s>>>(pairs, cursor, cap, key_bits, cnt);
  unsigned mb = nblk(n, 256);
  if (mb > 1024) mb = 1024;
  if (mb < 1) mb = 1;
  k_bucket_maxrow<<<mb, 256, 0, s>>>(cnt, n, maxrow);
}

void launch_bucket_build(const uint64_t* pairs, int64_t P, int key_bits, int32_t n, uint32_t* cnt, uint32_t* off,
                         uint32_t* ucnt, uint32_t* big, uint32_t* nbig, uint32_t* bucket, uint32_t* row_ptr,
                         uint32_t* scan_ws, int32_t* col, int32_t* indeg, uint32_t maxrow, cudaStream_t s) {
  scan_exclusive<uint32_t>(cnt, off, n, scan_ws, s);
  if (P > 0) {
    count_launch();
    k_bucket_scatter<<<nblk(P, 256), 256, 0, s>>>(pairs, P, key_bits, off, cnt, bucket);
  }
  count_launch();
  // a warp per row from 6 pairs a row on
  const bool by_warp = P >= 6 * (int64_t)n;
  if (by_warp) k_bucket_sort_warp<<<nblk(n, 8), 256, 0, s>>>(off, n, bucket, ucnt, big, nbig, indeg);
  else k_bucket_sort_small<<<nblk(n, 256), 256, 0, s>>>(off, n, bucket, ucnt, big, nbig, indeg);
  if (maxrow > (uint32_t)kBucketSmallRow) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    count_launch();
    k_bucket_sort_large<<<(unsigned)(sms > 0 ? sms * 8 : 1024), 128, 0, s>>>(off, bucket, ucnt, big, nbig);
  }
  scan_exclusive<uint32_t>(ucnt, row_ptr, n, scan_ws, s);
  count_launch();
  if (by_warp) k_bucket_compact_warp<<<nblk(n, 8), 256, 0, s>>>(off, row_ptr, n, bucket, col, indeg);
  else k_bucket_compact<<<nblk(n, 256), 256, 0, s>>>(off, row_ptr, n, bucket, col, indeg);
}

void launch_emit_csr(const uint64_t* keys, const uint32_t* flags, const uint32_t* upos, int64_t P,
                     int key_bits, int32_t* col, int32_t* rowcnt, int32_t* indeg, cudaStream_t s) {
  if (P > 0) {
    count_launch();
    k_emit_csr<<<nblk(P, 256), 256, 0, s>>>(keys, flags, upos, P, key_bits, col, rowcnt, indeg);
  }
}

void launch_finish_tasks(const int32_t* row_ptr, const int32_t* col, const int32_t* indeg, const uint32_t* pos,
                         int32_t n, int32_t* count, uint64_t* root_items, int4* adj, uint32_t* shape,
                         cudaStream_t s) {
  if (n > 0) {
    count_launch();
    k_finish_tasks<<<nblk(n, 256), 256, 0, s>>>(row_ptr, col, indeg, pos, n, count, root_items, adj, shape);
  }
}

void launch_report(const ReportArgs& a, cudaStream_t s) {
  if (a.n > 0) {
    count_launch();
    k_report<<<1, 32, 0, s>>>(a);
  }
}

void preload_analysis() {
  cudaFuncAttributes a;
  cudaFuncGetAttributes(&a, k_validate_tasks);
  cudaFuncGetAttributes(&a, k_validate_rects);
  cudaFuncGetAttributes(&a, k_add_offset);
  cudaFuncGetAttributes(&a, k_bin_count);
  cudaFuncGetAttributes(&a, k_bin_expand);
  cudaFuncGetAttributes(&a, k_segments);
  cudaFuncGetAttributes(&a, k_explicit_pairs);
  cudaFuncGetAttributes(&a, k_unique_flags);
  cudaFuncGetAttributes(&a, k_emit_csr);
  cudaFuncGetAttributes(&a, k_finish_tasks);
  cudaFuncGetAttributes(&a, k_report);
  cudaFuncGetAttributes(&a, k_band_place);
  cudaFuncGetAttributes(&a, k_widen_bounds);
  cudaFuncGetAttributes(&a, k_ingest_rects<int32_t, false>);
  cudaFuncGetAttributes(&a, k_ingest_rects<int32_t, true>);
  cudaFuncGetAttributes(&a, k_ingest_rects<int64_t, false>);
  cudaFuncGetAttributes(&a, k_ingest_rects<int64_t, true>);
  cudaFuncGetAttributes(&a, k_bucket_count);
  cudaFuncGetAttributes(&a, k_bucket_maxrow);
  cudaFuncGetAttributes(&a, k_bucket_scatter);
  cudaFuncGetAttributes(&a, k_bucket_sort_small);
  cudaFuncGetAttributes(&a, k_bucket_sort_warp);
  cudaFuncGetAttributes(&a, k_bucket_sort_large);
  cudaFuncGetAttributes(&a, k_bucket_compact);
  cudaFuncGetAttributes(&a, k_bucket_compact_warp);
}

}  // namespace grt
