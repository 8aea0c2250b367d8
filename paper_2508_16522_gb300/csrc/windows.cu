// windows.cu -- interference sweep of dense 2-D inputs, window by window.
//
// sweep.cu walks a tile's candidates in program order and keeps every class
// cell's run state, so a tile is one warp's serial chain, and its state (8 KB
// at 16 x 32 tiles) keeps an SM at 18 warps. Where candidates cover much of
// their tile, a cell sees an access every step or two, and the run an access
// follows lies a few candidates back. Here a warp takes kNew new candidates of
// a tile together with the ones just before them, 32 in all, and finds every
// new candidate's predecessors from those 32 boxes alone, with no state:
//
//  * the boxes' edges split the tile into class cells; a class cell is covered
//    by one set of the 32 candidates, a 32-bit mask (a row mask AND a column
//    mask, each from one ballot per class);
//  * bit b is the candidate b steps before the newest, so "the last one before
//    me" is the lowest set bit above mine, and the run a candidate follows in a
//    cell is a dozen bit operations on the cell's mask (pred_run). Each lane is
//    one new candidate and ORs the runs of the cells into its own mask; the
//    warp's other lanes do the same candidates on other cells;
//  * the masks become (source task, target task) pairs once per window, through
//    the pair filter (pairs.cuh).
//
// A cell whose run is not decided within the 32 candidates (its coverage is
// thin, as at the domain's border) is walked further back, 32 candidates per
// step, for the rectangle of the cell on which all candidates read so far are
// uniform. A full-tile write ends every search, so candidates before the last
// one of those are left out of the window. Windows share nothing, so a tile's
// candidates spread over many warps and the last tile holds up no one.
//
// Bound by instruction issue (71% of the active cycles on 60k launches of the
// 4096 x 4096 trace; DRAM 2%), spent on class columns and rows, cells, pairs and
// walks in about that order. 32 warps an SM. The 1M-launch trace at 16 x 32 tiles
// sweeps in 29 ms where the tile sweep takes 192, 43 captured requests in 1.6 ms
// where it takes 3.4. (When the sweep stood at 33 ms, 10 candidates before a
// window made it 43, and 8 new ones with 24, 16 or 12 before them 36 to 45: more
// cells need walks.)
//
// A tile this does not suit is flagged and left to sweep.cu, which keeps state
// and so never looks back: one with a task of more than kNew candidates, with
// more class cells in a window than kMaxCells (small boxes), or with a walk
// longer than kMaxWalk or kMaxSteps (a run of hundreds of readers, which every
// window after it would walk again). Its pairs written before that
// are kept: duplicates vanish in the CSR stage.
#include "grt_internal.cuh"
#include "pairs.cuh"

namespace grt {

namespace {
constexpr unsigned kFullW = 0xffffffffu;
constexpr int kNew = 16;        // new candidates per window
constexpr int kMaxCells = 640;  // class cells of a window; more: small boxes, cheaper one by one
constexpr int kMaxSteps = 512;  // 32-candidate steps of one window's walks
constexpr int kMaxWalk = 16;    // ... of one walk

struct Sink {  // the warp's chunk of the pair buffer
  unsigned long long chunk_base;
  uint32_t chunk_left;
  int lane;
};

// a packed entry's box; a 1-D tile is one column of rows, so that the parts of
// the warp share its classes
__device__ __forceinline__ Box unpack_w(uint64_t p, int ndim) {
  Box e = unpack_entry(p, ndim);
  if (ndim == 1) {
    e.y0 = e.x0;
    e.y1 = e.x1;
    e.x0 = e.x1 = 0;
  }
  return e;
}

// the last column (row) of the class that starts at a: before the next edge
__device__ __forceinline__ int last_of(bool act, int v0, int v1, int a, int last) {
  const unsigned near = act && v0 > a ? (unsigned)v0 - 1u : 0xFFFFu;
  const unsigned far = act && v1 >= a ? (unsigned)v1 : 0xFFFFu;
  const int e = (int)__reduce_min_sync(kFullW, near < far ? near : far);
  return e < last ? e : last;
}

// The run a candidate follows in one cell. m: the cell's mask, rp / dp: which
// candidates read / reduce there (the others write), gt: the bits before this
// candidate, gts: those of them that are not of its own joinable kind. Readers
// join readers and reducers reducers, so the search skips own-kind bits down to
// the last other one (lo), and the run is lo alone if it writes, else the bits
// of lo's kind up to the next other one. open: the mask ended before the run
// was decided (kind: lo's kind, -1 when not even lo was found).
__device__ __forceinline__ unsigned pred_run(unsigned m, unsigned rp, unsigned dp, unsigned gt, unsigned gts,
                                             bool& open, unsigned& lo) {
  const unsigned o = m & gts, n = 0u - o;
  lo = o & n;
  const unsigned b = m & gt & (o | n);  // lo and everything before it (none if there is no lo)
  unsigned T = (lo & rp) ? rp : lo;
  T = (lo & dp) ? dp : T;
  const unsigned q = b & ~T;
  open = q == 0u && (lo == 0u || (lo & (rp | dp)) != 0u);
  return b & ~(q | (0u - q));  // the bits before the first other one
}

// Candidates of one task in a cell count as one access (combined privilege:
// all read, all reduce, else write), standing at the task's first candidate.
// reps: first candidates of the tasks with several; grp: in lane b, the bits of
// the task whose first candidate is b.
__device__ __forceinline__ void merge_groups(unsigned& m, unsigned& rp, unsigned& dp, unsigned reps, unsigned grp) {
  const unsigned rp0 = rp, dp0 = dp;
  for (unsigned g = reps; g; g &= g - 1u) {
    const int b = __ffs((int)g) - 1;
    const unsigned rep = 1u << b;
    const unsigned G = __shfl_sync(kFullW, grp, b);
    const unsigned c = m & G;
    if (c) {
      m = (m & ~G) | rep;
      rp = (rp & ~rep) | ((c & ~rp0) ? 0u : rep);
      dp = (dp & ~rep) | ((c & ~dp0) ? 0u : rep);
    }
  }
}

// in lane b, a task's first candidate: the bits of its candidates (itself and
// the bits just below it that start no task)
__device__ __forceinline__ unsigned group_bits(unsigned nonstart, int b) {
  const unsigned below = (1u << b) - 1u;
  const unsigned stop = ~nonstart & below;  // the highest of these is the next task's
  const unsigned keep = stop ? ~(kFullW >> __clz((int)stop)) : kFullW;
  return (1u << b) | (below & keep);
}

// the pairs (task of each bit of run, dst) of every lane; task: the candidate's
// task in the lane of its bit
__device__ void emit(Sink& x, const SweepOut& o, unsigned run, int task, int dst) {
  const unsigned lt = lanemask_lt();
  while (__any_sync(kFullW, run != 0u)) {
    // two lookups in flight
    const bool h0 = run != 0u;
    const int s0 = __shfl_sync(kFullW, task, h0 ? __ffs((int)run) - 1 : 0);
    run &= run - 1u;
    const bool h1 = run != 0u;
    const int s1 = __shfl_sync(kFullW, task, h1 ? __ffs((int)run) - 1 : 0);
    run &= run - 1u;
    bool f0 = h0, f1 = h1;
    if (o.filt) {
      uint32_t* const p0 = filt_slots(o, (uint32_t)s0, (uint32_t)dst);
      uint32_t* const p1 = filt_slots(o, (uint32_t)s1, (uint32_t)dst);
      const uint2 none = make_uint2((uint32_t)s0, (uint32_t)s1);
      const uint2 v0 = h0 ? filt_look(p0) : none, v1 = h1 ? filt_look(p1) : none;
      f0 = h0 && v0.x != (uint32_t)s0 && v0.y != (uint32_t)s0;
      f1 = h1 && v1.x != (uint32_t)s1 && v1.y != (uint32_t)s1;
      if (f0) f0 = filt_take(p0, v0, (uint32_t)s0);
      if (f1) f1 = filt_take(p1, v1, (uint32_t)s1);
    }
    const unsigned b0 = __ballot_sync(kFullW, f0), b1 = __ballot_sync(kFullW, f1);
    if (b0 | b1) {
      const uint32_t n0 = (uint32_t)__popc(b0);
      const PairDst pd = reserve_pairs(x, o, n0 + (uint32_t)__popc(b1));
      const unsigned long long p0 = pair_pos(pd, (uint32_t)__popc(b0 & lt));
      const unsigned long long p1 = pair_pos(pd, n0 + (uint32_t)__popc(b1 & lt));
      if (f0 && p0 < o.cap) o.pairs[p0] = pair_key(s0, dst, o.key_bits);
      if (f1 && p1 < o.cap) o.pairs[p1] = pair_key(s1, dst, o.key_bits);
    }
  }
}

// The 32 candidates before a window (or before another such block), oldest task
// whole: bit (lane) b is the candidate b steps before position hi.
struct Block {
  unsigned val, st, rp, dp;  // candidates of whole tasks; first ones; reads; reduces
  int lo;                    // position of the oldest: the next block ends there
};

__device__ __forceinline__ bool load_block(const uint64_t* payload, int ndim, int lane, int sb, int hi, uint64_t& p,
                                           Block& b) {
  const int idx = hi - 1 - lane;
  const bool in = idx >= sb;
  p = in ? __ldg(payload + idx) : 0ull;
  const int task = in ? (int)(uint32_t)p : -1;
  int older = __shfl_down_sync(kFullW, task, 1);
  if (lane == 31) older = idx > sb ? (int)(uint32_t)__ldg(payload + idx - 1) : -1;
  const unsigned st0 = __ballot_sync(kFullW, in && (idx == sb || older != task));
  if (!st0) return false;  // 32 candidates of one task
  const int hs = 31 - __clz((int)st0);
  b.val = __ballot_sync(kFullW, in) & ((2u << hs) - 1u);
  b.st = st0 & b.val;
  const int priv = (int)((p >> 32) & 3u);
  b.rp = __ballot_sync(kFullW, priv == kKindRead) & b.val;
  b.dp = __ballot_sync(kFullW, priv == kKindReduce) & b.val;
  b.lo = hi - 1 - hs;
  return true;
}

// Walks one class cell (tile cells [xa, xb] x [ya, yb]) back, first over the
// block before the window (kept in shared memory for all of its cells), then
// over the ones before. want: this lane's candidate (task dst) is undecided
// there; own: its kind in the cell; kind0: the kind of the run it was
// collecting (-1: none met yet). The predecessors met in the first block are
// bits of acc1. Returns false when the walk is too long.
__device__ __forceinline__ bool walk_back(Sink& x, const SweepOut& o, const uint64_t* payload, int ndim, int sb,
                                          const uint64_t* first, const Block& b1, int xa, int xb, int ya, int yb,
                                          bool want, int own, int kind0, int dst, int& steps, unsigned& acc1) {
  const int lane = x.lane;
  for (int y = ya; y <= yb;) {
    int by = yb;
    for (int cx = xa; cx <= xb;) {
      int rx = xb, ry = yb;  // the rectangle from (cx, y) on which every candidate read is uniform
      bool nd = want;
      int kind = kind0;
      Block b = b1;
      uint64_t p = first[lane];
      for (int blocks = 0;; ++blocks) {
        if (++steps > kMaxSteps || blocks > kMaxWalk) return false;
        const Box e = unpack_w(p, ndim);
        const bool act = (b.val >> lane) & 1u;
        const bool cy = e.y0 <= y && y <= e.y1, cc = e.x0 <= cx && cx <= e.x1;
        unsigned m = __ballot_sync(kFullW, act && cy && cc), rp = b.rp, dp = b.dp;
        // a covering candidate bounds the rectangle by its far edges, one that
        // starts further right (below) by its near one
        unsigned tx = 0xFFFFu, ty = 0xFFFFu;
        if (act) {
          if (cy && cc) {
            tx = (unsigned)e.x1;
            ty = (unsigned)e.y1;
          } else if (cy) {
            if (e.x0 > cx) tx = (unsigned)e.x0 - 1u;
          } else if (e.y0 > y && e.x1 >= cx) {
            ty = (unsigned)e.y0 - 1u;
          }
        }
        rx = min(rx, (int)__reduce_min_sync(kFullW, tx));
        ry = min(ry, (int)__reduce_min_sync(kFullW, ty));
        const unsigned nonst = b.val & ~b.st;
        if (nonst) merge_groups(m, rp, dp, b.st & (nonst << 1), group_bits(nonst, lane));
        unsigned run = 0u;
        if (nd) {
          if (kind < 0) {
            const unsigned S = own == kKindRead ? rp : (own == kKindReduce ? dp : 0u);
            bool open;
            unsigned lo;
            run = pred_run(m, rp, dp, kFullW, ~S, open, lo);
            nd = open;
            if (lo) kind = (lo & rp) ? kKindRead : kKindReduce;  // used while open: lo does not write
          } else {
            const unsigned q = m & ~(kind == kKindRead ? rp : dp);
            run = m & ~(q | (0u - q));
            nd = q == 0u;
          }
        }
        if (blocks == 0) acc1 |= run;
        else emit(x, o, run, (int)(uint32_t)p, dst);
        if (b.lo <= sb || !__any_sync(kFullW, nd)) break;
        if (!load_block(payload, ndim, lane, sb, b.lo, p, b)) return false;
      }
      by = min(by, ry);
      cx = rx + 1;
    }
    y = by + 1;
  }
  return true;
}

// kNew new candidates a window and the 32 - kNew before them; the warp's 32 / kNew
// parts take different cells.
// WIDE: tiles of more than 32 columns or rows (and 1-D ones), whose class
// starts are found among the boxes' own edges instead of in a word of bits.
template <bool WIDE>
__global__ void __launch_bounds__(256, 4) k_window(const uint64_t* __restrict__ payload, const uint32_t* __restrict__ keys,
                                                const uint32_t* __restrict__ seg_begin,
                                                const uint32_t* __restrict__ seg_end, int M, int span,
                                                AnalysisDims d, SweepOut o, uint8_t* __restrict__ bail,
                                                uint32_t* nbail) {
  constexpr int NEW = kNew, PARTS = 32 / NEW;
  __shared__ uint64_t before[kWindowWarps][32];  // the block before the window, where some cell asked for it
  const int lane = threadIdx.x & 31;
  uint64_t* const first = before[threadIdx.x >> 5];
  const int part = lane / NEW, k = lane % NEW;
  const unsigned me = 1u << k;
  const unsigned gt = ~((2u << k) - 1u);
  const unsigned newbits = (1u << NEW) - 1u;
  const int tw = d.ndim == 1 ? 1 : d.tw, th = d.ndim == 1 ? d.tw : d.th;
  const unsigned colbits = tw >= 32 ? kFullW : (1u << tw) - 1u;
  const unsigned rowbits = th >= 32 ? kFullW : (1u << th) - 1u;
  Sink x{0ull, 0u, lane};
  for (;;) {
    uint32_t ch = 0;
    if (lane == 0) ch = atomicAdd(o.tile_counter, 1u);
    ch = __shfl_sync(kFullW, ch, 0);
    if ((uint64_t)ch * (uint64_t)span >= (uint64_t)M) break;
    int pos = (int)ch * span;
    const int B = M - pos < span ? M : pos + span;
    int sb = 0, se = 0, fx = 0, fy = 0;
    uint32_t t = 0;
    while (pos < B) {
      if (pos >= se) {  // the next tile
        t = keys[pos];
        sb = (int)seg_begin[t];
        se = (int)seg_end[t];
        if (__ldcg(bail + t)) {
          pos = se;
          continue;
        }
        const int tx = (int)(t % (uint32_t)d.ntx), ty = (int)(t / (uint32_t)d.ntx);
        const int64_t wx = d.ext[0] - (int64_t)tx * d.tw, wy = d.ext[1] - (int64_t)ty * d.th;
        fx = (int)(wx < d.tw ? wx : d.tw) - 1;  // the tile's last column and row inside the domain
        fy = (int)(wy < d.th ? wy : d.th) - 1;
        if (d.ndim == 1) {
          fy = fx;
          fx = 0;
        }
        if (pos > sb) {  // a chunk that starts inside a task leaves it to the chunk before
          const uint32_t prev = (uint32_t)payload[pos - 1];
          for (;;) {
            const int idx = pos + lane;
            const unsigned diff = __ballot_sync(kFullW, idx >= se || (uint32_t)payload[idx] != prev);
            if (diff) {
              pos += __ffs((int)diff) - 1;
              break;
            }
            pos += 32;
          }
          continue;
        }
      }
      // ---- the window: bit (lane) b holds position pos + NEW - 1 - b ----------
      const int idx = pos + NEW - 1 - lane;
      const bool in = idx >= sb && idx < se;
      const uint64_t p = in ? payload[idx] : 0ull;
      const Box e = unpack_w(p, d.ndim);
      const int task = in ? e.task : -1;
      int older = __shfl_down_sync(kFullW, task, 1);
      if (lane == 31) older = in && idx > sb ? (int)(uint32_t)payload[idx - 1] : -1;
      const bool cut0 = lane == 0 && in && idx + 1 < se && (int)(uint32_t)payload[idx + 1] == task;
      const unsigned st0 = __ballot_sync(kFullW, in && (idx == sb || older != task));
      unsigned val = __ballot_sync(kFullW, in);
      int next = pos + NEW < se ? pos + NEW : se;
      if (__any_sync(kFullW, cut0)) {  // the newest task goes on past the window: left to the next one
        const int ls = __ffs((int)st0) - 1;
        if (ls >= NEW - 1) {  // more than NEW candidates of one task
          if (lane == 0) {
            bail[t] = 1;
            atomicAdd(nbail, 1u);
          }
          pos = se;
          continue;
        }
        val &= ~((2u << ls) - 1u);
        next = pos + NEW - 1 - ls;
      }
      if (pos + NEW > B) {  // tasks that start in the next chunk
        const unsigned sB = st0 & ((1u << (pos + NEW - B)) - 1u);
        if (sB) {
          const int top = 31 - __clz((int)sB);
          val &= ~((2u << top) - 1u);
          const int nx = pos + NEW - 1 - top;
          next = nx < next ? nx : next;
        }
      }
      // the oldest whole task, or the task of the last full-tile write before the new ones
      int hs = 31 - __clz((int)st0);
      bool more = pos + NEW - 1 - hs > sb;
      const unsigned fw = __ballot_sync(kFullW, in && e.priv == kKindWrite && e.x0 == 0 && e.y0 == 0 && e.x1 == fx &&
                                                    e.y1 == fy) &
                          ~newbits & ((2u << hs) - 1u);
      if (fw) {
        const unsigned at = st0 & ~((fw & (0u - fw)) - 1u);  // first candidates at or before that write
        hs = __ffs((int)at) - 1;
        more = false;
      }
      val &= (2u << hs) - 1u;
      const unsigned st = st0 & val;
      const bool act = (val >> lane) & 1u;
      const unsigned rp = __ballot_sync(kFullW, act && e.priv == kKindRead);
      const unsigned dp = __ballot_sync(kFullW, act && e.priv == kKindReduce);
      const unsigned nonst = val & ~st;
      const unsigned reps = st & (nonst << 1);
      const unsigned grp = nonst ? group_bits(nonst, lane) : 0u;

      // ---- class columns and rows that some new candidate covers --------------
      // (class j in lane j of colm / colx, class 32 + j in lane j of colm2 / colx2)
      unsigned colm = 0u, rowm = 0u, colm2 = 0u, rowm2 = 0u;
      int cols = 0, rows = 0, colx = 0, rowy = 0, colx2 = 0, rowy2 = 0;
      // a box left out covers nothing
      const unsigned bx0 = act ? (unsigned)e.x0 : 0x10000u, bxw = act ? (unsigned)(e.x1 - e.x0) : 0u;
      const unsigned by0 = act ? (unsigned)e.y0 : 0x10000u, byw = act ? (unsigned)(e.y1 - e.y0) : 0u;
      auto column = [&](int c) {
        const unsigned b = __ballot_sync(kFullW, (unsigned)c - bx0 <= bxw);
        if (!(b & newbits)) return;
        if (lane == (cols & 31)) {
          if (!WIDE || cols < 32) {
            colm = b;
            colx = c;
          } else {
            colm2 = b;
            colx2 = c;
          }
        }
        ++cols;
      };
      auto row = [&](int c) {
        const unsigned b = __ballot_sync(kFullW, (unsigned)c - by0 <= byw);
        if (!(b & newbits)) return;
        if (lane == (rows & 31)) {
          if (!WIDE || rows < 32) {
            rowm = b;
            rowy = c;
          } else {
            rowm2 = b;
            rowy2 = c;
          }
        }
        ++rows;
      };
      if (!WIDE) {
        const unsigned ex = act ? (1u << e.x0) | (e.x1 < 31 ? 2u << e.x1 : 0u) : 0u;
        const unsigned ey = act ? (1u << e.y0) | (e.y1 < 31 ? 2u << e.y1 : 0u) : 0u;
        for (unsigned r = __reduce_or_sync(kFullW, ex) & colbits; r; r &= r - 1u) column(__ffs((int)r) - 1);
        for (unsigned r = __reduce_or_sync(kFullW, ey) & rowbits; r; r &= r - 1u) row(__ffs((int)r) - 1);
      } else {
        // each value once: the first lane that holds it, far edges only where no
        // box starts
        auto starts = [&](int v0, int v1, bool cols_) {
          const unsigned lt = lanemask_lt();
          const unsigned p0 = __match_any_sync(kFullW, act ? v0 : -1), p1 = __match_any_sync(kFullW, act ? v1 : -1);
          for (unsigned r = __ballot_sync(kFullW, act && !(p0 & lt)); r; r &= r - 1u) {
            const int c = __shfl_sync(kFullW, v0, __ffs((int)r) - 1);
            if (cols_) column(c); else row(c);
          }
          for (unsigned r = __ballot_sync(kFullW, act && !(p1 & lt)); r; r &= r - 1u) {
            const int c = __shfl_sync(kFullW, v1, __ffs((int)r) - 1);
            if (__any_sync(kFullW, act && v0 == c)) continue;
            if (cols_) column(c); else row(c);
          }
        };
        starts(e.x0, e.x1 + 1, true);
        starts(e.y0, e.y1 + 1, false);
      }
      auto pick = [&](unsigned a, unsigned b, int i) -> unsigned {  // of class i (i per lane; i < 64)
        unsigned v = __shfl_sync(kFullW, a, i & 31);
        if (WIDE) {
          const unsigned v2 = __shfl_sync(kFullW, b, i & 31);
          v = i < 32 ? v : v2;
        }
        return v;
      };
      bool drop = rows * cols > kMaxCells;
      unsigned acc = 0u, acc1 = 0u;
      int steps = 0;
      Block b1{0u, 0u, 0u, 0u, -1};
      const int dst = __shfl_sync(kFullW, task, k);
      const unsigned S = (rp & me) ? rp : ((dp & me) ? dp : 0u);
      const unsigned gts = gt & ~S;
      // ---- every class cell, PARTS rows at a time ------------------------------
      // every run is decided here, no task has two candidates: 97% of the 1M-launch
      // trace's windows (their own loop: 35 -> 29 ms)
      const bool plain = !more && !nonst;
      for (int i = 0; plain && i < rows && !drop; i += PARTS) {
        unsigned rm = pick(rowm, rowm2, i + part);
        if (i + part >= rows) rm = 0u;
        for (int j = 0; j < cols; ++j) {
          const unsigned m = rm & pick(colm, colm2, j);
          bool open;
          unsigned lo;
          const unsigned run = pred_run(m, rp, dp, gt, gts, open, lo);
          if (m & me) acc |= run;
        }
      }
      for (int i = 0; !plain && i < rows && !drop; i += PARTS) {
        unsigned rm = pick(rowm, rowm2, i + part);
        if (i + part >= rows) rm = 0u;
        for (int j = 0; j < cols && !drop; ++j) {
          unsigned m = rm & pick(colm, colm2, j);
          const unsigned raw = m;
          unsigned lo;
          bool open, mine;
          if (!nonst) {
            const unsigned run = pred_run(m, rp, dp, gt, gts, open, lo);
            mine = (m & me) != 0u;
            if (mine) acc |= run;
          } else {
            unsigned r1 = rp, d1 = dp;
            merge_groups(m, r1, d1, reps, grp);
            const unsigned S1 = (r1 & me) ? r1 : ((d1 & me) ? d1 : 0u);
            const unsigned run = pred_run(m, r1, d1, gt, gt & ~S1, open, lo);
            mine = (m & me) != 0u;
            if (mine) acc |= run;
          }
          if (more && __any_sync(kFullW, mine && open)) {
            unsigned m1 = m, r1 = rp, d1 = dp;
            if (nonst) {  // the cell's own kinds again
              m1 = raw;
              merge_groups(m1, r1, d1, reps, grp);
            }
            if (b1.lo < 0) {
              uint64_t q;
              if (!load_block(payload, d.ndim, lane, sb, pos + NEW - 1 - hs, q, b1)) {
                drop = true;
                break;
              }
              first[lane] = q;
              __syncwarp();
            }
            const int own = (r1 & me) ? kKindRead : ((d1 & me) ? kKindReduce : kKindWrite);
            const int kind = lo == 0u ? -1 : ((lo & r1) ? kKindRead : kKindReduce);
            const int xa = (int)pick((unsigned)colx, (unsigned)colx2, j);
            int xb = last_of(act, e.x0, e.x1, xa, tw - 1);
            // the columns right of it that look the same are walked with it
            while (j + 1 < cols && (int)pick((unsigned)colx, (unsigned)colx2, j + 1) == xb + 1 &&
                   __all_sync(kFullW, (rm & pick(colm, colm2, j + 1)) == raw)) {
              ++j;
              xb = last_of(act, e.x0, e.x1, xb + 1, tw - 1);
            }
            for (int h = 0; h < PARTS && !drop; ++h) {
              const bool want = mine && open && part == h;
              if (!__any_sync(kFullW, want)) continue;
              const int ya = (int)pick((unsigned)rowy, (unsigned)rowy2, i + h);
              const int yb = last_of(act, e.y0, e.y1, ya, th - 1);
              drop = !walk_back(x, o, payload, d.ndim, sb, first, b1, xa, xb, ya, yb, want, own, kind, dst, steps, acc1);
            }
          }
        }
      }
      if (drop) {
        if (lane == 0) {
          bail[t] = 1;
          atomicAdd(nbail, 1u);
        }
        pos = se;
        continue;
      }
      // ---- the pairs: the parts share each candidate's mask --------------------
#pragma unroll
      for (int s = NEW; s < 32; s <<= 1) acc |= __shfl_xor_sync(kFullW, acc, s);
      constexpr unsigned share = 0x55555555u;  // every PARTS-th bit
      emit(x, o, acc & (share << part), task, dst);
      if (b1.lo >= 0) {
#pragma unroll
        for (int s = NEW; s < 32; s <<= 1) acc1 |= __shfl_xor_sync(kFullW, acc1, s);
        emit(x, o, acc1 & (share << part), (int)(uint32_t)first[lane], dst);
        __syncwarp();
      }
      pos = next;
    }
  }
  // the unused end of the warp's last chunk
  for (uint32_t i = lane; i < x.chunk_left; i += 32)
    if (x.chunk_base + i < o.cap) o.pairs[x.chunk_base + i] = kEmpty64;
}
}  // namespace

static bool wide_tile(const AnalysisDims& d) { return d.ndim == 1 || d.tw > 32 || d.th > 32; }

void launch_window(const uint64_t* payload, const uint32_t* keys, const uint32_t* seg_begin, const uint32_t* seg_end,
                   int64_t M, int span, AnalysisDims d, SweepOut o, uint8_t* bail, uint32_t* nbail, int blocks,
                   cudaStream_t s) {
  count_launch();
  if (wide_tile(d))
    k_window<true><<<blocks, 256, 0, s>>>(payload, keys, seg_begin, seg_end, (int)M, span, d, o, bail, nbail);
  else
    k_window<false><<<blocks, 256, 0, s>>>(payload, keys, seg_begin, seg_end, (int)M, span, d, o, bail, nbail);
}

int window_blocks_per_sm(const AnalysisDims& d) {
  int nb = 0;
  if (wide_tile(d)) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_window<true>, 256, 0);
  else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_window<false>, 256, 0);
  return nb < 1 ? 1 : nb;
}

void preload_window() {
  cudaFuncAttributes a;
  cudaFuncGetAttributes(&a, k_window<false>);
  cudaFuncGetAttributes(&a, k_window<true>);
}

}  // namespace grt
