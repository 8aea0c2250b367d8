// block_exec.cu -- Algorithm 1 for a graph inside one thread block.
//
// A small graph's run is its critical path: on the grid-wide executors
// (exec.cu) each hop costs L2 round trips (a decrement, the record, for the
// ring a reservation, a published slot and a poll): 2.7 us per hop of the 1-D
// stencil's chain of 216, whose tasks take nanoseconds. Here a block holds the
// counters in its shared memory and its warps are the workers. Two ways:
//
// k_exec_block, for any graph of up to kBlockTasks tasks: 2 bytes of countdown a
// task (two per word; an in-degree is below the task count) and a linear queue
// of ready task ids (each task enters once per run; its first kBlockQueue places
// in shared memory, the rest in global). A warp keeps up to a batch of the
// successors it makes ready and queues the rest; an idle warp takes queued ids
// by moving the head of one 64-bit word (head, tail). Trigger records stay in
// global memory; a lane touches its successors' records when it starts a task,
// so that they are in L1 when a successor becomes ready.
//
// k_exec_window, for graphs whose program order follows their dependences: see
// there.
//
// A batch's graphs take a block each, largest first, several blocks to an SM.
// Measured (before -> here): a replay of the 1-D stencil 0.58 -> 0.07 ms; a
// stencil of 32 x 1000 tasks of 256 FMAs 2.5 -> 0.84 ms (the FMAs alone take
// 0.56); 640 mixed graphs x 20 replays 34.8 -> 4.0 ms; one run of 43 captured
// requests (the largest 1923 levels deep, 22 edges a task) 9.9 -> 2.4 ms. What
// bounds them is the hop: about 0.2 us through the window's counters, 1.1 us
// through the queue.
//
// The bodies' effects need only reach the block's own warps: fences are block
// scope, and COUNTER's state may stay in L1. Every wait is bounded by
// timeout_ns without reported progress: a warp reports what it ran when it finds
// nothing kept and at the latest after kBlockReport tasks, k_exec_window's after
// four chunks of 32.
#include <mutex>
#include <set>

#include "bodies.cuh"
#include "grt_internal.cuh"

namespace grt {

namespace {
constexpr unsigned kFullB = 0xffffffffu;
constexpr int kBlockWarps = 16;
constexpr int kSmallWarps = 4;    // a batch's graphs of at most kBlockSmall tasks
constexpr int kBlockKeep = 64;  // kept ids per warp
constexpr unsigned kBlockSleep = 40;  // ns between an idle warp's polls
constexpr uint32_t kNoId = 0xFFFFu;
constexpr uint32_t kBlockReport = 1024;  // tasks a warp runs at most, and a batch, before it counts them

struct BlockCtl {
  unsigned long long ht;  // queue: head in the low 32 bits, tail in the high ones
  uint32_t done, status;
  int32_t graph;
  uint32_t pad;
  unsigned long long cnt[kCntCount];  // the block's totals: one block may run a whole graph many times
};

size_t block_smem_bytes(int32_t n, int warps) {
  const size_t q = (size_t)(n < kBlockQueue ? n : kBlockQueue);
  return sizeof(BlockCtl) + (size_t)warps * kBlockKeep * 2 + (size_t)((n + 3) / 4) * 8 + (q + 3) / 4 * 8;
}

// brings a sector into L1; nothing waits for the value
__device__ __forceinline__ void touch(const void* p) {
  int v;
  asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(p));
}

template <int WARPS, bool FENCE>
__global__ void __launch_bounds__(WARPS * 32, WARPS == kBlockWarps ? 2 : 8) k_exec_block(ExecParams p, BlockArgs a) {
  extern __shared__ __align__(16) unsigned char bsmem[];
  constexpr int T = WARPS * 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  BlockCtl* const ctl = reinterpret_cast<BlockCtl*>(bsmem);
  uint16_t* const keepq = reinterpret_cast<uint16_t*>(bsmem + sizeof(BlockCtl)) + warp * kBlockKeep;
  uint32_t* const cntw = reinterpret_cast<uint32_t*>(bsmem + sizeof(BlockCtl) + WARPS * kBlockKeep * 2);
  const unsigned lt = lanemask_lt();
  uint32_t edges = 0;  // out-edges of the tasks this lane ran in this run
  uint32_t cnt[kCntCount];
#pragma unroll
  for (int k = 0; k < kCntCount; ++k) cnt[k] = 0;
  if (tid < kCntCount) ctl->cnt[tid] = 0;
  if (tid == 0) ctl->status = 0;

  for (uint32_t turn = 0;; ++turn) {
    // the next graph: graph 0, or the batch's, largest first
    if (tid == 0) {
      const uint32_t i = a.order ? atomicAdd(a.next, 1u) : turn;
      ctl->graph = i < (uint32_t)a.n_order ? (a.order ? a.order[i] : 0) : -1;
    }
    __syncthreads();
    const int gi = ctl->graph;
    if (gi < 0 || ctl->status) break;
    const ExecGraph& G = p.graphs[gi];
    const int n = G.n_tasks, base = G.task_base, n_roots = G.n_roots, body = G.body, spin = G.spin_iters;
    int32_t* const out = G.out;
    int32_t* const state = G.state;
    const int32_t* const body_arg = G.body_arg;
    const int4* const adj = p.adj + 2 * (int64_t)base;
    const int32_t* const indeg = p.indeg + base;
    const int words = (n + 3) / 4 * 2, Q = n < kBlockQueue ? n : kBlockQueue;
    volatile uint16_t* const queue = reinterpret_cast<volatile uint16_t*>(cntw + words);
    volatile uint16_t* const spill = a.spill + base;  // place i >= Q of the queue
    uint32_t dirty = (uint32_t)n;                     // places that may hold an id

    for (int r = 0; r < p.replays; ++r) {
      // INIT: countdowns from the in-degrees, the roots queued
      for (int i = tid; i < words; i += T) {
        const int e = 2 * i, f = 2 * i + 1;
        cntw[i] = (e < n ? (uint32_t)__ldg(indeg + e) : 0u) | ((f < n ? (uint32_t)__ldg(indeg + f) : 0u) << 16);
      }
      for (int i = tid; i < (int)dirty; i += T) {
        const uint16_t v = i < n_roots ? (uint16_t)((uint32_t)p.root_items[G.root_base + i] - (uint32_t)base) : (uint16_t)kNoId;
        if (i < Q) queue[i] = v; else spill[i] = v;
      }
      if (tid == 0) {
        ctl->ht = (unsigned long long)(uint32_t)n_roots << 32;
        ctl->done = 0;
      }
      __syncthreads();
      int nl = 0;  // kept ids (warp-uniform)
      uint32_t seen = 0, pend = 0, polls = 0;
      uint64_t idle_since = 0;
      for (;;) {
        uint32_t id = kNoId;
        if (nl > 0) {
          const int m = nl < 32 ? nl : 32;
          if (lane < m) id = keepq[nl - m + lane];
          nl -= m;
          // a warp that always keeps something still reports: the others' limit
          // counts from the last finished task they know of
          if (pend >= kBlockReport) {
            cnt[kCntTasks] += pend;
            if (lane == 0) atomicAdd(&ctl->done, pend);
            pend = 0;
          }
          __syncwarp();
        } else {
          // count what ran since the last look, then up to `claim` queued ids. An
          // idle warp reads two words a poll and little else: 15 of them polling
          // with a CAS attempt, the clock and short sleeps took a third of the
          // issue slots from the one that worked
          if (pend) {
            cnt[kCntTasks] += pend;
            if (lane == 0) atomicAdd(&ctl->done, pend);
            pend = 0;
          }
          // one lane's look for the whole warp: lanes that read for themselves could
          // see different words, and part over the shuffles below
          unsigned long long v0 = 0;
          if (lane == 0) v0 = *(volatile unsigned long long*)&ctl->ht;
          v0 = __shfl_sync(kFullB, v0, 0);
          if ((uint32_t)v0 >= (uint32_t)(v0 >> 32)) {
            ++polls;
            int over = 0;
            if (lane == 0) {
              const uint32_t d = *(volatile uint32_t*)&ctl->done;
              over = d >= (uint32_t)n || *(volatile uint32_t*)&ctl->status != 0u;
              if (!over && (polls & 63u) == 0u) {
                const uint64_t now = globaltimer_ns();
                if (idle_since == 0 || d != seen) {
                  idle_since = now;
                  seen = d;
                } else if (now - idle_since > (uint64_t)p.timeout_ns) {
                  over = 1;
                  *(volatile uint32_t*)&ctl->status = (uint32_t)RT_ERR_TIMEOUT;
                }
              }
            }
            if (__shfl_sync(kFullB, over, 0)) break;
            __nanosleep(kBlockSleep);
            continue;
          }
          uint32_t h = 0, take = 0;
          if (lane == 0) {
            unsigned long long v = v0;
            for (;;) {
              const uint32_t hd = (uint32_t)v, tl = (uint32_t)(v >> 32);
              if (hd >= tl) break;
              uint32_t k = tl - hd;
              if (a.share) k = k < 2 * WARPS ? 1u : k / WARPS;
              k = k < (uint32_t)p.claim ? k : (uint32_t)p.claim;
              const unsigned long long w = atomicCAS(&ctl->ht, v, v + k);
              if (w == v) {
                h = hd;
                take = k;
                break;
              }
              v = w;
            }
          }
          take = __shfl_sync(kFullB, take, 0);
          if (take == 0) continue;
          cnt[kCntClaims] += 1;
          h = __shfl_sync(kFullB, h, 0) + (uint32_t)lane;
          if ((uint32_t)lane < take) {
            // a slot is written just after its place was taken; the clock bounds the
            // wait here too (an idle warp's may not run: all of them can be here)
            uint64_t from = 0;
            for (uint32_t tries = 1;; ++tries) {
              id = h < (uint32_t)Q ? queue[h] : spill[h];
              if (id != kNoId || *(volatile uint32_t*)&ctl->status) break;
              if ((tries & 1023u) == 0u) {
                const uint64_t now = globaltimer_ns();
                if (from == 0) from = now;
                else if (now - from > (uint64_t)p.timeout_ns) *(volatile uint32_t*)&ctl->status = (uint32_t)RT_ERR_TIMEOUT;
              }
            }
          }
          __syncwarp();
          idle_since = 0;
        }
        const bool has = id != kNoId;
        if (FENCE) __threadfence_block();  // acquire: predecessors' effects before the bodies
        int4 a0 = make_int4(0, 0, 0, -1), a1 = make_int4(-1, -1, -1, -1);
        if (has) {
          a0 = __ldg(adj + 2 * id);
          a1 = __ldg(adj + 2 * id + 1);
        }
        const int deg = a0.y;
        int s[kAdjInline] = {a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
        for (int j = 0; j < kAdjInline; ++j) {
          if (s[j] >= 0) {
            s[j] -= base;
            touch(adj + 2 * s[j]);
            if (FENCE && body == RT_BODY_COUNTER) touch(body_arg + s[j]);
          }
        }
        if (has) {
          if (body == RT_BODY_SPIN) {
            out[id] = (int32_t)spin_body(id, spin);
          } else if (body == RT_BODY_FMA) {
            out[id] = fma_body(id, spin);
          } else if (FENCE && body == RT_BODY_COUNTER) {
            int32_t* c = state + body_arg[id];
            *c = (int32_t)((uint32_t)*c + 1u);
          }
        }
        if (FENCE) __threadfence_block();  // release: bodies before the decrements
        // COMPLETED_EDGE: every lane its own task's inline successors, their
        // decrements in flight together; the edges past them shared by the warp
        const int dmax = (int)__reduce_max_sync(kFullB, (unsigned)deg);
        auto settle = [&](bool ready, int c) {
          const unsigned rm = __ballot_sync(kFullB, ready);
          if (!rm) return;
          const int rank = __popc(rm & lt), got = __popc(rm);
          const int room = p.keep - nl > 0 ? p.keep - nl : 0;
          if (ready && rank < room) keepq[nl + rank] = (uint16_t)c;
          if (got > room) {
            uint32_t at = 0;
            if (lane == 0) at = (uint32_t)(atomicAdd(&ctl->ht, (unsigned long long)(got - room) << 32) >> 32);
            at = __shfl_sync(kFullB, at, 0) + (uint32_t)(rank - room);
            if (ready && rank >= room) {
              if (at < (uint32_t)Q) queue[at] = (uint16_t)c; else spill[at] = (uint16_t)c;
            }
            cnt[kCntPushed] += (unsigned)(got - room);
          }
          const int kept = got < room ? got : room;
          cnt[kCntKept] += (unsigned)kept;
          nl += kept;
        };
        // a task that has become ready: the start of its row on its way to L1
        auto ahead = [&](bool ready, int c) {
          if (!ready) return;
          const int4 rec = __ldg(adj + 2 * c);
          if (rec.y > kAdjInline) touch(p.col + rec.x);
        };
        auto dec = [&](int c) -> bool {  // one decrement; true when it was the last
          const unsigned sh = ((unsigned)c & 1u) << 4;
          return ((atomicSub(cntw + (c >> 1), 1u << sh) >> sh) & 0xFFFFu) == 1u;
        };
        const unsigned hm = __ballot_sync(kFullB, has);
        if (dmax > kAdjInline && (hm & (hm - 1u)) == 0u) {
          // one task with many successors: a lane each, from its row
          const int L = __ffs((int)hm) - 1;
          const int row = __shfl_sync(kFullB, a0.x, L);
          for (int e0 = 0; e0 < dmax; e0 += 32) {
            const int c = e0 + lane < dmax ? __ldg(p.col + row + e0 + lane) - base : -1;
            const bool last = c >= 0 && dec(c);
            if (c >= 0) touch(adj + 2 * c);
            if (FENCE) __threadfence_block();
            settle(last, c);
            ahead(last, c);
          }
        } else {
          uint32_t old[kAdjInline];
#pragma unroll
          for (int j = 0; j < kAdjInline; ++j) {
            old[j] = 0u;
            if (s[j] >= 0) old[j] = atomicSub(cntw + (s[j] >> 1), 1u << ((s[j] & 1) << 4));
          }
          // the other predecessors' effects, seen through the counters, before the
          // successors are handed on
          if (FENCE) __threadfence_block();
          unsigned rm[kAdjInline];
          int got = 0;
#pragma unroll
          for (int j = 0; j < kAdjInline; ++j) {
            rm[j] = __ballot_sync(kFullB, s[j] >= 0 && ((old[j] >> ((s[j] & 1) << 4)) & 0xFFFFu) == 1u);
            got += __popc(rm[j]);
          }
          if (nl + got <= p.keep) {  // all kept
#pragma unroll
            for (int j = 0; j < kAdjInline; ++j) {
              if ((rm[j] >> lane) & 1u) keepq[nl + __popc(rm[j] & lt)] = (uint16_t)s[j];
              nl += __popc(rm[j]);
            }
            cnt[kCntKept] += (unsigned)got;
          } else {
#pragma unroll
            for (int j = 0; j < kAdjInline; ++j) settle((rm[j] >> lane) & 1u, s[j]);
          }
          if (dmax > kAdjInline) {
            const int extra = deg > kAdjInline ? deg - kAdjInline : 0;
            int incl = extra;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const int y = __shfl_up_sync(kFullB, incl, o);
              if (lane >= o) incl += y;
            }
            const int excl = incl - extra;
            const int D = __shfl_sync(kFullB, incl, 31);
            const int rbeg = a0.x + kAdjInline;
            constexpr int kRound = 2;  // groups of 32 edges whose columns are in flight together
            for (int e0 = 0; e0 < D; e0 += 32 * kRound) {
              int c[kRound];
              bool last[kRound];
#pragma unroll
              for (int k = 0; k < kRound; ++k) {
                const int e = e0 + 32 * k + lane;
                int owner = 0;
#pragma unroll
                for (int step = 16; step >= 1; step >>= 1) {
                  const int cand = owner + step;
                  if (__shfl_sync(kFullB, excl, cand) <= e) owner = cand;
                }
                const int oex = __shfl_sync(kFullB, excl, owner);
                const int orb = __shfl_sync(kFullB, rbeg, owner);
                c[k] = e < D ? __ldg(p.col + orb + (e - oex)) - base : -1;
              }
#pragma unroll
              for (int k = 0; k < kRound; ++k) {
                last[k] = c[k] >= 0 && dec(c[k]);
                if (c[k] >= 0) touch(adj + 2 * c[k]);
              }
              if (FENCE) __threadfence_block();
#pragma unroll
              for (int k = 0; k < kRound; ++k) settle(last[k], c[k]);
            }
          }
        }
        pend += __popc(hm);
        cnt[kCntBatches] += 1;
        edges += (uint32_t)deg;
        __syncwarp();
      }
      if (FENCE) __threadfence_block();
      const uint32_t e = __reduce_add_sync(kFullB, edges);  // one run has fewer than 2^31
      if (lane == 0) atomicAdd(&ctl->cnt[kCntEdges], (unsigned long long)e);
      edges = 0;
      __syncthreads();  // the run is over (or timed out)
      if (ctl->status) break;
      dirty = (uint32_t)(ctl->ht >> 32);
      __syncthreads();
    }
    __syncthreads();
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < kCntCount; ++k)
      if (k != kCntEdges && cnt[k]) atomicAdd(&ctl->cnt[k], (unsigned long long)cnt[k]);
  }
  __syncthreads();
  if (a.order) {
    if (tid < kCntCount && ctl->cnt[tid]) atomicAdd(&p.ctrl->counters[tid], ctl->cnt[tid]);
    if (tid == 0 && ctl->status) atomicCAS(&p.ctrl->status, 0u, ctl->status);
  } else {
    // pinned host memory: the host reads it after the stream's synchronisation
    if (tid < kCntCount) a.counters_out[tid] = ctl->cnt[tid];
    if (tid == 0) *a.status_out = ctl->status;
  }
}

// The same for a graph whose program order follows its dependences closely (no
// edge longer than BlockArgs::span, every root near the start): warp w owns the
// chunks w, w + WARPS, ... of 32 consecutive tasks, one per lane, and takes them
// in order, polling their counters in shared memory (k_exec_owned's scheme, with
// a hop of a shared-memory add and the owner's next poll: no queue, no kept
// list, no answer to wait for). A chunk's trigger records are loaded while the
// chunk before it runs.
//
// Only tasks near the front have counters: task v's is slot v mod S, which
// counts its finished predecessors up from 0 and is cleared when v runs. A
// successor of a task u lies at most `span` after u, and a warp takes no chunk
// that ends more than S - span tasks after the first one still held, so the
// slot of a successor c was last used by c - S, which has run. So the graph may
// have any number of tasks. The first unfinished task is always in a chunk its
// owner holds (or may take), with its predecessors done: no warp waits forever.
//
// WIDE: some task has successors past its trigger record (p.adjx). A graph without
// loads half the bytes a chunk, sets up 5 successor slots instead of 13 and keeps
// half the registers: 300 steps of a 600-wide stencil 285 -> 205 us, 32 wide with
// 256 FMA 1000 steps 850 -> 818. The wide kernel still tests adjx itself, although
// it is set: with those tests compiled out its schedule was worse (batch of 40
// random graphs of 60k tasks, 20 replays: 3.95 ms instead of 3.75).
template <int WARPS, bool FENCE, bool WIDE>
__global__ void __launch_bounds__(WARPS * 32, WARPS == kBlockWarps ? 2 : 4) k_exec_window(ExecParams p, BlockArgs a,
                                                                                          int S) {
  extern __shared__ __align__(16) unsigned char wsmem[];
  __shared__ uint32_t held[WARPS];  // first task of the chunk each warp holds (past the end: ~0)
  __shared__ uint32_t s_done, s_status;
  __shared__ int32_t s_graph;
  __shared__ unsigned long long s_cnt[2];
  uint32_t* const count = reinterpret_cast<uint32_t*>(wsmem);
  constexpr int T = WARPS * 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t mask = (uint32_t)S - 1u;
  constexpr int NQ = WIDE ? 4 : 2, NS = WIDE ? kAdjWide : kAdjInline;  // a record's int4s and successors
  for (int i = tid; i < S + 32; i += T) count[i] = 0u;
  if (tid == 0) {
    s_status = 0u;
    s_graph = -1;
    s_cnt[0] = s_cnt[1] = 0ull;
  }
  uint32_t edges = 0, ran = 0, batches = 0;
  __syncthreads();
  for (int turn = 0;; ++turn) {
    if (tid == 0) {
      const uint32_t i = a.order ? atomicAdd(a.next, 1u) : (uint32_t)turn;
      s_graph = i < (uint32_t)a.n_order ? (a.order ? a.order[i] : 0) : -1;
    }
    __syncthreads();
    const int gi = s_graph;
    if (gi < 0 || s_status) break;
    const ExecGraph& G = p.graphs[gi];
    const int n = G.n_tasks, base = G.task_base, body = G.body, spin = G.spin_iters;
    int32_t* const out = G.out;
    int32_t* const state = G.state;
    const int32_t* const body_arg = FENCE ? G.body_arg : nullptr;
    const int4* const adj = p.adj + 2 * (int64_t)base;
    const int4* const adjx = WIDE && p.adjx ? p.adjx + 2 * (int64_t)base : nullptr;
    const int room = S - (a.order ? a.spans[gi] : a.span);
    for (int r = 0; r < p.replays; ++r) {
      if (lane == 0) held[warp] = warp * 32 < n ? (uint32_t)(warp * 32) : 0xFFFFFFFFu;
      if (tid == 0) s_done = 0u;
      __syncthreads();
      uint32_t oldest = 0;  // no task before it is unfinished
      int4 nq[NQ];          // the next chunk's records
      int narg = 0;         // ... and counters
      auto fetch = [&](int v) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
          nq[k] = make_int4(0, 0, 0, -1);
          if (k > 0) nq[k].x = nq[k].y = nq[k].z = -1;
          if (v < n && (k < 2 || adjx)) nq[k] = __ldg(k < 2 ? adj + 2 * (int64_t)v + k : adjx + 2 * (int64_t)v + (k - 2));
        }
        if (FENCE && body == RT_BODY_COUNTER && v < n) narg = __ldg(body_arg + v);
      };
      fetch(warp * 32 + lane);
      bool stop = false;
      uint32_t turns = 0;
      for (int c0 = warp * 32; c0 < n && !stop; c0 += T) {
        const int v = c0 + lane;
        const bool has = v < n;
        unsigned pending = __ballot_sync(kFullB, has);
        const int deg = has ? nq[0].y : 0;
        const uint32_t need = (uint32_t)nq[0].z;
        const int row = nq[0].x, arg = narg;
        const int dmax = (int)__reduce_max_sync(kFullB, (unsigned)deg);
        // the successors' slots, now rather than when the chunk's tasks run; none:
        // the lane's own spare word past the window, so that the additions below
        // need no branches (a divergent one a successor took 30 cycles each)
        const uint32_t spare = (uint32_t)S + (uint32_t)lane;
        uint32_t succ[NS];
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
          auto slot = [&](int t) -> uint32_t { return t >= 0 ? (uint32_t)(t - base) & mask : spare; };
          if (k > 0) {
            succ[4 * k - 3] = slot(nq[k].x);
            succ[4 * k - 2] = slot(nq[k].y);
            succ[4 * k - 1] = slot(nq[k].z);
          }
          succ[4 * k] = slot(nq[k].w);
        }
        const uint32_t my = has ? (uint32_t)v & mask : spare;
        volatile uint32_t* const mine = count + my;
        fetch(v + T);
        uint64_t since = 0;
        uint32_t seen = 0, polls = 0;
        bool open = (uint32_t)c0 + 32u <= oldest + (uint32_t)room;  // the window reaches this chunk
        while (pending) {
          bool ready = false;
          if (open) ready = ((pending >> lane) & 1u) && *mine == need;
          const unsigned rm = __ballot_sync(kFullB, ready);
          if (!rm) {
            ++polls;
            if (!open) {
              oldest = __reduce_min_sync(kFullB, lane < WARPS ? *(volatile uint32_t*)&held[lane] : 0xFFFFFFFFu);
              __threadfence_block();  // acquire: the slots cleared before those chunks were let go
              open = (uint32_t)c0 + 32u <= oldest + (uint32_t)room;
            }
            if (polls >= 16u) __nanosleep(polls < 64u ? 20 : 100);
            if ((polls & 255u) == 0u) {
              int late = 0;
              if (lane == 0) {
                const uint32_t d = *(volatile uint32_t*)&s_done;
                const uint64_t now = globaltimer_ns();
                if (since == 0 || d != seen) {
                  since = now;
                  seen = d;
                } else if (now - since > (uint64_t)p.timeout_ns) {
                  *(volatile uint32_t*)&s_status = (uint32_t)RT_ERR_TIMEOUT;
                }
                late = *(volatile uint32_t*)&s_status != 0u;
              }
              if (__shfl_sync(kFullB, late, 0)) {
                stop = true;
                break;
              }
            }
            continue;
          }
          polls = 0;
          pending &= ~rm;
          ++batches;
          if (FENCE) __threadfence_block();  // acquire: the predecessors' effects before the bodies
          count[ready ? my : spare] = 0u;
          if (body == RT_BODY_SPIN) {
            const int32_t x = (int32_t)spin_body((uint32_t)v, spin);
            if (ready) out[v] = x;
          } else if (body == RT_BODY_FMA) {
            const int32_t x = fma_body((uint32_t)v, spin);
            if (ready) out[v] = x;
          } else if (FENCE && body == RT_BODY_COUNTER) {
            if (ready) state[arg] = (int32_t)((uint32_t)state[arg] + 1u);
          }
          if (FENCE) __threadfence_block();  // release: bodies before the counters
          // COMPLETED_EDGE
#pragma unroll
          for (int k = 0; k < NQ; ++k) {
            if (4 * k - 3 < dmax && (k < 2 || adjx)) {  // uniform
#pragma unroll
              for (int j = k > 0 ? 4 * k - 3 : 0; j <= 4 * k; ++j) atomicAdd(count + (ready ? succ[j] : spare), 1u);
            }
          }
          if (dmax > (adjx ? kAdjWide : kAdjInline) && ready)  // past the record
            for (int e = adjx ? kAdjWide : kAdjInline; e < deg; ++e)
              atomicAdd(count + ((uint32_t)(__ldg(p.col + row + e) - base) & mask), 1u);
          if (!FENCE) edges += ready ? (uint32_t)deg : 0u;
          __syncwarp();
        }
        if (stop) break;
        // (counted here the replayed 1-D stencil takes 257 us instead of 300, the narrow
        // FMA stencil 832 instead of 821: the loop above is scheduled anew)
        if (FENCE) edges += (uint32_t)deg;
        // every fourth chunk is let go (and the last): the fence, so that its
        // slots' clearing comes first, waits for the bodies' stores too
        if ((++turns & 3u) == 0u || c0 + T >= n) {
          __threadfence_block();
          __syncwarp();
          if (lane == 0) {
            *(volatile uint32_t*)&held[warp] = c0 + T < n ? (uint32_t)(c0 + T) : 0xFFFFFFFFu;
            atomicAdd(&s_done, 1u);
          }
        }
        ran += (uint32_t)(n - c0 < 32 ? n - c0 : 32);
      }
      if (FENCE) __threadfence_block();
      const uint32_t e = __reduce_add_sync(kFullB, edges);  // one run has fewer than 2^31
      if (lane == 0) atomicAdd(&s_cnt[1], (unsigned long long)e);
      edges = 0;
      __syncthreads();
      if (s_status) break;
    }
    __syncthreads();
  }
  if (lane == 0) atomicAdd(&s_cnt[0], (unsigned long long)ran);
  __syncthreads();
  if (tid == 0) {
    const unsigned long long cnt[3] = {batches, s_cnt[0], s_cnt[1]};  // batches: one warp's
    for (int k = 0; k < kCntCount; ++k) {
      const unsigned long long x = k < 3 ? cnt[k] : 0ull;
      if (!a.order) a.counters_out[k] = x;
      else if (x) atomicAdd(&p.ctrl->counters[k], x);
    }
    if (!a.order) *a.status_out = s_status;
    else if (s_status) atomicCAS(&p.ctrl->status, 0u, s_status);
  }
}

// each graph of a batch: its longest edge, last root and largest out-degree
// (shape[3g..3g+2], zeroed by the caller)
__global__ void __launch_bounds__(256) k_batch_shape(const ExecGraph* graphs, int32_t G, const int32_t* row_ptr,
                                                     const int32_t* col, const int32_t* indeg, uint32_t* shape) {
  for (int32_t g = blockIdx.x; g < G; g += gridDim.x) {
    const int32_t b = graphs[g].task_base, n = graphs[g].n_tasks;
    uint32_t span = 0, root = 0, deg = 0;
    for (int32_t i = threadIdx.x; i < n; i += blockDim.x) {
      const int32_t e0 = row_ptr[b + i], e1 = row_ptr[b + i + 1];
      if (e1 > e0) span = max(span, (uint32_t)(col[e1 - 1] - (b + i)));
      if (indeg[b + i] == 0) root = (uint32_t)i;
      deg = max(deg, (uint32_t)(e1 - e0));
    }
    span = __reduce_max_sync(kFullB, span);
    root = __reduce_max_sync(kFullB, root);
    deg = __reduce_max_sync(kFullB, deg);
    if ((threadIdx.x & 31) == 0) {
      if (span) atomicMax(shape + 3 * g, span);
      if (root) atomicMax(shape + 3 * g + 1, root);
      if (deg) atomicMax(shape + 3 * g + 2, deg);
    }
  }
}

template <int WARPS>
void launch_block(const ExecParams& p, const BlockArgs& a, int32_t max_n, int blocks, cudaStream_t s) {
  static std::mutex mu;
  static std::set<int> done;
  int dev = 0;
  cudaGetDevice(&dev);
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!done.count(dev)) {
      const int most = (int)block_smem_bytes(kBlockTasks, WARPS);
      cudaFuncSetAttribute(k_exec_block<WARPS, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
      cudaFuncSetAttribute(k_exec_block<WARPS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
      done.insert(dev);
    }
  }
  const size_t bytes = block_smem_bytes(max_n, WARPS);
  count_launch();
  if (p.need_fence) k_exec_block<WARPS, true><<<blocks, WARPS * 32, bytes, s>>>(p, a);
  else k_exec_block<WARPS, false><<<blocks, WARPS * 32, bytes, s>>>(p, a);
}

template <int WARPS, bool FENCE, bool WIDE>
void launch_window_kernel(const ExecParams& p, const BlockArgs& a, int S, int blocks, cudaStream_t s) {
  static std::mutex mu;
  static std::set<int> done;
  int dev = 0;
  cudaGetDevice(&dev);
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!done.count(dev)) {
      cudaFuncSetAttribute(k_exec_window<WARPS, FENCE, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (kWindowSlots + 32) * 4);
      done.insert(dev);
    }
  }
  count_launch();
  k_exec_window<WARPS, FENCE, WIDE><<<blocks, WARPS * 32, ((size_t)S + 32) * 4, s>>>(p, a, S);
}

template <int WARPS>
void launch_window_warps(const ExecParams& p, const BlockArgs& a, int S, int blocks, cudaStream_t s) {
  if (p.need_fence) {
    if (p.adjx) launch_window_kernel<WARPS, true, true>(p, a, S, blocks, s);
    else launch_window_kernel<WARPS, true, false>(p, a, S, blocks, s);
  } else {
    if (p.adjx) launch_window_kernel<WARPS, false, true>(p, a, S, blocks, s);
    else launch_window_kernel<WARPS, false, false>(p, a, S, blocks, s);
  }
}
}  // namespace

// how many tasks can be ready at once, on average over a run's steps: the tasks
// of the first d steps end at most d spans after the last root
static int32_t window_width(int32_t span, int32_t last_root) { return span > last_root ? span : last_root + 1; }

bool block_window_fits(int32_t span, int32_t last_root, int32_t body, int32_t spin_iters) {
  if (span > kWindowSpan || last_root > kWindowSpan) return false;
  if (body == RT_BODY_CHECK) return false;
  const int64_t iters = body == RT_BODY_SPIN || body == RT_BODY_FMA ? spin_iters : 0;
  return (int64_t)window_width(span, last_root) * (iters + 20) <= kWindowWork;
}

bool block_window_small(int32_t span, int32_t last_root) { return window_width(span, last_root) <= kSmallSpan; }

void launch_exec_window(const ExecParams& p, const BlockArgs& a, int blocks, bool small, cudaStream_t s) {
  if (small) launch_window_warps<kSmallWarps>(p, a, kSmallSlots, blocks, s);
  else launch_window_warps<kBlockWarps>(p, a, kWindowSlots, blocks, s);
}

void launch_batch_shape(const ExecGraph* graphs, int32_t G, const int32_t* row_ptr, const int32_t* col,
                        const int32_t* indeg, uint32_t* shape, cudaStream_t s) {
  if (G <= 0) return;
  count_launch();
  k_batch_shape<<<(unsigned)(G < 4096 ? G : 4096), 256, 0, s>>>(graphs, G, row_ptr, col, indeg, shape);
}

bool block_exec_fits(int32_t n, int64_t n_roots, int32_t body, int32_t spin_iters) {
  if (n > kBlockTasks || n_roots > kBlockRoots) return false;
  if (body == RT_BODY_CHECK) return false;  // its time depends on its rectangles' cells
  const int64_t iters = body == RT_BODY_SPIN || body == RT_BODY_FMA ? spin_iters : 0;
  return iters * n <= kBlockWork && iters * n_roots <= kBlockStep;
}

bool block_exec_small(int32_t n, int32_t body, int32_t spin_iters) {
  const int64_t iters = body == RT_BODY_SPIN || body == RT_BODY_FMA ? spin_iters : 0;
  return n <= kBlockSmall && iters * n <= kBlockSmallWork;
}

bool block_exec_alone(int32_t n, int64_t n_roots, int64_t n_edges, int32_t body, int32_t spin_iters, bool owned) {
  if (n <= 0 || !block_exec_fits(n, n_roots, body, spin_iters)) return false;
  const int64_t iters = body == RT_BODY_SPIN || body == RT_BODY_FMA ? spin_iters : 0;
  if (owned) return n <= kBlockTiny && iters * n <= kBlockTinyWork;
  return n_roots <= (n_edges / n >= 6 ? kBlockAloneRootsDense : kBlockAloneRoots);
}

int block_exec_warps() { return kBlockWarps; }
int block_small_warps() { return kSmallWarps; }

void launch_exec_block(ExecParams p, const BlockArgs& a, int32_t max_n, int blocks, bool small, cudaStream_t s) {
  if (p.keep > kBlockKeep) p.keep = kBlockKeep;
  if (p.claim > 32) p.claim = 32;
  if (p.claim < 1) p.claim = 1;
  if (small) launch_block<kSmallWarps>(p, a, max_n, blocks, s);
  else launch_block<kBlockWarps>(p, a, max_n, blocks, s);
}

void preload_block_exec() {
  cudaFuncAttributes a;
  cudaFuncGetAttributes(&a, k_batch_shape);
  cudaFuncGetAttributes(&a, k_exec_window<kBlockWarps, false, false>);
  cudaFuncGetAttributes(&a, k_exec_window<kBlockWarps, false, true>);
  cudaFuncGetAttributes(&a, k_exec_window<kBlockWarps, true, false>);
  cudaFuncGetAttributes(&a, k_exec_window<kBlockWarps, true, true>);
  cudaFuncGetAttributes(&a, k_exec_window<kSmallWarps, false, false>);
  cudaFuncGetAttributes(&a, k_exec_window<kSmallWarps, false, true>);
  cudaFuncGetAttributes(&a, k_exec_window<kSmallWarps, true, false>);
  cudaFuncGetAttributes(&a, k_exec_window<kSmallWarps, true, true>);
  cudaFuncGetAttributes(&a, k_exec_block<kBlockWarps, false>);
  cudaFuncGetAttributes(&a, k_exec_block<kBlockWarps, true>);
  cudaFuncGetAttributes(&a, k_exec_block<kSmallWarps, false>);
  cudaFuncGetAttributes(&a, k_exec_block<kSmallWarps, true>);
}

}  // namespace grt
