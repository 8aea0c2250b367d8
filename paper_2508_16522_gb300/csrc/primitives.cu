// primitives.cu -- device exclusive scan and stable LSD radix sort.
//
// Scan: reduce-then-scan over blocks of 2048 items (256 threads x 8), the
// block totals scanned recursively. out[n] receives the total, so arrays are
// sized n+1; in == out is allowed.
//
// Up to kScanOne items one block does it all.
//
// Radix sort: 8-bit digits, least significant first. Per pass: a per-block
// digit histogram, an exclusive scan of the digit-major histogram matrix, and
// a scatter whose in-block ranks are computed warp by warp with match_any (so
// the sort is stable: keys keep their input order within a digit); the block
// reorders its keys by digit in shared memory before writing them, so each
// digit's run goes out in coalesced writes.

#include <mutex>
#include <set>
#include <type_traits>

#include "grt_internal.cuh"

namespace grt {

std::atomic<long long> g_kernel_launches{0};

namespace {
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

template <typename T>
__device__ T block_exclusive_sum(T v, T* warp_tot, T* block_total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    T w = lane < (kScanThreads / 32) ? warp_tot[lane] : T(0);
    T wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < (kScanThreads / 32)) warp_tot[lane] = wi - w;
    if (lane == (kScanThreads / 32) - 1) *block_total = wi;
  }
  __syncthreads();
  return incl - v + warp_tot[warp];
}

// what a scan adds up: the array's values, or (ZERO) one per zero
template <bool ZERO, typename T>
__device__ __forceinline__ T scan_value(T v) {
  return ZERO ? T(v == T(0)) : v;
}

template <typename T, bool ZERO>
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const T* in, int64_t n, T* partial) {
  __shared__ T warp_tot[32];
  __shared__ T tot;
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  T s = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    int64_t k = base + j * kScanThreads + threadIdx.x;  // coalesced
    if (k < n) s += scan_value<ZERO>(in[k]);
  }
  (void)block_exclusive_sum<T>(s, warp_tot, &tot);
  if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

template <typename T, bool ZERO>
__global__ void __launch_bounds__(kScanThreads) k_scan_down(const T* in, T* out, int64_t n,
                                                           const T* block_base) {
  __shared__ T stage[kScanTile];
  __shared__ T warp_tot[32];
  __shared__ T tot;
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  // coalesced load into shared memory, then each thread owns 8 consecutive items
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    int64_t k = base + j * kScanThreads + threadIdx.x;
    stage[j * kScanThreads + threadIdx.x] = k < n ? scan_value<ZERO>(in[k]) : T(0);
  }
  __syncthreads();
  T v[kScanItems];
  T s = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    v[j] = stage[threadIdx.x * kScanItems + j];
    s += v[j];
  }
  T run = block_exclusive_sum<T>(s, warp_tot, &tot);
  if (block_base) run += block_base[blockIdx.x];
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    stage[threadIdx.x * kScanItems + j] = run;
    run += v[j];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    int64_t k = base + j * kScanThreads + threadIdx.x;
    if (k < n) out[k] = stage[j * kScanThreads + threadIdx.x];
  }
  if (base + kScanTile >= n && threadIdx.x == 0) {
    // the last block writes the grand total
    T total = tot + (block_base ? block_base[blockIdx.x] : T(0));
    out[n] = total;
  }
}
// A short scan in one block: kOneTile items a step, staged in shared memory so
// that loads and stores coalesce, the next step's loads in flight meanwhile and
// the running total carried along. Up to kScanOne items it beats the three
// launches of reduce, scan of the totals and down-sweep (about 3 us each on the
// device and as much on the host). 512 threads: a block of 1024 at 52 registers
// would not fit an SM beside a resident serving kernel, and never start.
constexpr int kOneThreads = 512;
constexpr int kOneItems = 8;
constexpr int kOneTile = kOneThreads * kOneItems;
constexpr int kScanOne = 6 * kOneTile;

template <typename T, bool ZERO>
__global__ void __launch_bounds__(kOneThreads) k_scan_one(const T* in, T* out, int32_t n) {
  constexpr int kWarps = kOneThreads / 32;
  __shared__ T stage[kOneTile];
  __shared__ T wtot[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T next[kOneItems];
#pragma unroll
  for (int j = 0; j < kOneItems; ++j) {
    const int32_t k = j * kOneThreads + tid;
    next[j] = k < n ? scan_value<ZERO>(in[k]) : T(0);
  }
  T carry = 0;
  for (int32_t base = 0; base < n; base += kOneTile) {
#pragma unroll
    for (int j = 0; j < kOneItems; ++j) stage[j * kOneThreads + tid] = next[j];
    __syncthreads();
    // in place is allowed: this step's items have been read, none written yet
    if (base + kOneTile < n) {
#pragma unroll
      for (int j = 0; j < kOneItems; ++j) {
        const int32_t k = base + kOneTile + j * kOneThreads + tid;
        next[j] = k < n ? scan_value<ZERO>(in[k]) : T(0);
      }
    }
    T v[kOneItems];
    T sum = 0;
#pragma unroll
    for (int j = 0; j < kOneItems; ++j) {
      v[j] = stage[tid * kOneItems + j];
      sum += v[j];
    }
    T incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wtot[warp] = incl;
    __syncthreads();
    T wi = lane < kWarps ? wtot[lane] : T(0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    const T before = __shfl_sync(0xffffffffu, wi, warp > 0 ? warp - 1 : 0);
    T run = carry + (warp > 0 ? before : T(0)) + incl - sum;
    carry += __shfl_sync(0xffffffffu, wi, 31);
#pragma unroll
    for (int j = 0; j < kOneItems; ++j) {
      stage[tid * kOneItems + j] = run;
      run += v[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kOneItems; ++j) {
      const int32_t k = base + j * kOneThreads + tid;
      if (k < n) out[k] = stage[j * kOneThreads + tid];
    }
    __syncthreads();
  }
  if (tid == 0) out[n] = carry;
}
}  // namespace

template <typename T>
size_t scan_ws_elems(int64_t n) {
  size_t total = 0;
  while (n > kScanTile) {
    int64_t nb = (n + kScanTile - 1) / kScanTile;
    total += 2 * nb + 1;
    n = nb;
  }
  return total + 1;
}

namespace {
template <typename T, bool ZERO>
void scan_any(const T* in, T* out, int64_t n, T* ws, cudaStream_t s) {
  if (n <= 0) {
    cudaMemsetAsync(out, 0, sizeof(T), s);
    return;
  }
  count_launch();
  if (n <= kScanTile) {
    k_scan_down<T, ZERO><<<1, kScanThreads, 0, s>>>(in, out, n, nullptr);
    return;
  }
  if (n <= kScanOne) {
    k_scan_one<T, ZERO><<<1, kOneThreads, 0, s>>>(in, out, (int32_t)n);
    return;
  }
  const int64_t nb = (n + kScanTile - 1) / kScanTile;
  T* part = ws;
  T* part_scan = ws + nb;
  k_scan_reduce<T, ZERO><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, part);
  scan_any<T, false>(part, part_scan, nb, ws + 2 * nb + 1, s);
  count_launch();
  k_scan_down<T, ZERO><<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, part_scan);
}
}  // namespace

template <typename T>
void scan_exclusive(const T* in, T* out, int64_t n, T* ws, cudaStream_t s) {
  scan_any<T, false>(in, out, n, ws, s);
}

void scan_zeros(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* ws, cudaStream_t s) {
  scan_any<uint32_t, true>(in, out, n, ws, s);
}

template size_t scan_ws_elems<uint32_t>(int64_t);
template void scan_exclusive<uint32_t>(const uint32_t*, uint32_t*, int64_t, uint32_t*, cudaStream_t);

// ---------------------------------------------------------------------------
// radix sort
// ---------------------------------------------------------------------------
namespace {
constexpr int kRadixThreads = 256;
constexpr int kRadixWarps = kRadixThreads / 32;
// Keys per thread: 12 (3072 a block: 53 KB of shared memory, four blocks an SM;
// with 16 three, 6.6 ms for the two passes over 343M entries instead of 6.0, and
// with 8 five but more digit counts, 6.2), or 4 for small sorts, whose few blocks
// are a chain of ranking rounds each (6200 keys: 13.9 us a pass with 16).
constexpr int kRadixIpt = 12, kRadixIptSmall = 4;
constexpr int64_t kRadixSmall = 96 * kRadixThreads * kRadixIptSmall;  // its digit counts still fit one scan block
inline int64_t radix_blocks(int64_t n) {
  const int64_t tile = kRadixThreads * (n <= kRadixSmall ? kRadixIptSmall : kRadixIpt);
  return (n + tile - 1) / tile;
}

template <typename K, int IPT>
__global__ void __launch_bounds__(kRadixThreads) k_radix_hist(const K* keys, int64_t n, int shift,
                                                             uint32_t mask, uint32_t* hist,
                                                             int64_t nblocks) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * (kRadixThreads * IPT);
  K kv[IPT];
#pragma unroll
  for (int j = 0; j < IPT; ++j) {
    const int64_t k = base + j * kRadixThreads + threadIdx.x;
    kv[j] = k < n ? keys[k] : K(0);
  }
#pragma unroll
  for (int j = 0; j < IPT; ++j)
    if (base + j * kRadixThreads + threadIdx.x < n) atomicAdd(&h[(uint32_t)(kv[j] >> shift) & mask], 1u);
  __syncthreads();
  hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// dynamic shared memory of one scatter block: its keys (and values) in
// block-sorted order
template <typename K, bool HAS_V, int IPT>
constexpr size_t scatter_smem_bytes() {
  return (size_t)(kRadixThreads * IPT) * (sizeof(K) + (HAS_V ? sizeof(uint64_t) + sizeof(uint16_t) : 0));
}

__device__ __forceinline__ void copy8_async(void* to, const void* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from)
               : "memory");
}

// One pass of the LSD radix sort over a block of (kRadixThreads * IPT) keys: every key is
// ranked within its warp and digit (match_any), the ranks become positions in
// the block's digit-sorted order, the keys are reordered in shared memory, and
// consecutive threads then write consecutive keys of each digit run to the
// run's global offset, so the global writes are coalesced. Stable. The values go
// to shared memory as they lie, by asynchronous copies under the ranking, and
// are picked by a 16-bit index when they are written: held in registers over the
// ranking they cost a third of the resident warps and their own load latency
// (two passes over 343M entries of 12 bytes: 7.06 -> 6.0 ms, with the write
// loop unrolled and 12 keys a thread; copy rate allows 2.9).
template <typename K, bool HAS_V, int IPT>
__global__ void __launch_bounds__(kRadixThreads, 3) k_radix_scatter(
    const K* __restrict__ keys, const uint64_t* __restrict__ vals, K* __restrict__ keys_out,
    uint64_t* __restrict__ vals_out, int64_t n, int shift, uint32_t mask,
    const uint32_t* __restrict__ offs, int64_t nblocks) {
  __shared__ uint32_t wcnt[kRadixWarps][256];
  __shared__ uint32_t boff[256];    // the digit's first position in the output
  __shared__ uint32_t bstart[257];  // the digit's first position in the block's sorted order
  __shared__ uint32_t wsum[kRadixWarps];
  extern __shared__ __align__(16) unsigned char rsmem[];
  K* sk = reinterpret_cast<K*>(rsmem);
  uint64_t* sv = reinterpret_cast<uint64_t*>(rsmem + (size_t)(kRadixThreads * IPT) * sizeof(K));
  uint16_t* from = reinterpret_cast<uint16_t*>(sv + kRadixThreads * IPT);  // the value of a sorted position
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int w = 0; w < kRadixWarps; ++w) wcnt[w][threadIdx.x] = 0;
  boff[threadIdx.x] = offs[(int64_t)threadIdx.x * nblocks + blockIdx.x];
  __syncthreads();
  const int64_t wbase = (int64_t)blockIdx.x * (kRadixThreads * IPT) + (int64_t)warp * (32 * IPT);
  K kv[IPT];
  uint32_t rk[IPT];
  const unsigned lt = lanemask_lt();
  // every key's load in flight before the ranking, whose warp barriers would hold
  // each round's loads back until the round before it is done (two passes over the
  // 343M entries of the 1M-launch trace: 9.9 -> 7.1 ms)
#pragma unroll
  for (int r = 0; r < IPT; ++r) {
    const int64_t idx = wbase + r * 32 + lane;
    kv[r] = idx < n ? keys[idx] : K(0);
  }
  // the values go to shared memory as they lie, while the keys are ranked
  if (HAS_V) {
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
      const int64_t idx = wbase + r * 32 + lane;
      if (idx < n) copy8_async(sv + (warp * (32 * IPT) + r * 32 + lane), vals + idx);
    }
  }
#pragma unroll
  for (int r = 0; r < IPT; ++r) {
    int64_t idx = wbase + r * 32 + lane;
    bool valid = idx < n;
    const K k = kv[r];
    uint32_t d = valid ? ((uint32_t)(k >> shift) & mask) : 256u;
    unsigned peers = __match_any_sync(0xffffffffu, d);
    uint32_t before = __popc(peers & lt);
    uint32_t base = valid ? wcnt[warp][d] : 0u;
    __syncwarp();
    if (valid && before == 0) wcnt[warp][d] = base + __popc(peers);
    __syncwarp();
    rk[r] = base + before;
  }
  __syncthreads();
  // per digit (thread d): warp prefixes, and the digit's block total
  uint32_t tot = 0;
#pragma unroll
  for (int w = 0; w < kRadixWarps; ++w) {
    uint32_t t = wcnt[w][threadIdx.x];
    wcnt[w][threadIdx.x] = tot;
    tot += t;
  }
  // exclusive scan of the totals over the 256 digits (warp scans, then warps)
  uint32_t incl = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  uint32_t wpre = 0;
#pragma unroll
  for (int w = 0; w < kRadixWarps; ++w) wpre += w < warp ? wsum[w] : 0u;
  bstart[threadIdx.x] = wpre + incl - tot;
  boff[threadIdx.x] -= wpre + incl - tot;  // read back after the next barriers: where position 0 would go
  if (threadIdx.x == kRadixThreads - 1) bstart[256] = wpre + incl;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < IPT; ++r) {
    int64_t idx = wbase + r * 32 + lane;
    if (idx < n) {
      const uint32_t d = (uint32_t)(kv[r] >> shift) & mask;
      const uint32_t lp = bstart[d] + wcnt[warp][d] + rk[r];
      sk[lp] = kv[r];
      if (HAS_V) from[lp] = (uint16_t)(warp * (32 * IPT) + r * 32 + lane);
    }
  }
  if (HAS_V) asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const uint32_t nvalid = bstart[256];
#pragma unroll
  for (int r = 0; r < IPT; ++r) {
    const uint32_t i = r * kRadixThreads + threadIdx.x;
    if (i < nvalid) {
      const K k = sk[i];
      const uint32_t dst = boff[(uint32_t)(k >> shift) & mask] + i;
      keys_out[dst] = k;
      if (HAS_V) vals_out[dst] = sv[from[i]];
    }
  }
}

template <typename K, bool HAS_V, int IPT>
void launch_scatter(const K* kin, const uint64_t* vin, K* kout, uint64_t* vout, int64_t n, int shift, uint32_t mask,
                    const uint32_t* offs, int64_t nb, cudaStream_t s) {
  // above the default 48 KB of dynamic shared memory for some instantiations:
  // one fixed size per instantiation, set once per device
  static std::mutex mu;
  static std::set<int> done;
  int dev = 0;
  cudaGetDevice(&dev);
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!done.count(dev)) {
      cudaFuncSetAttribute(k_radix_scatter<K, HAS_V, IPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)scatter_smem_bytes<K, HAS_V, IPT>());
      done.insert(dev);
    }
  }
  count_launch();
  k_radix_scatter<K, HAS_V, IPT><<<(unsigned)nb, kRadixThreads, scatter_smem_bytes<K, HAS_V, IPT>(), s>>>(
      kin, vin, kout, vout, n, shift, mask, offs, nb);
}
}  // namespace

size_t radix_ws_bytes(int64_t n) {
  const int64_t nb = radix_blocks(n);
  int64_t h = 256 * (nb > 0 ? nb : 1);
  return (size_t)(2 * h + 1 + scan_ws_elems<uint32_t>(h)) * sizeof(uint32_t) + 256;
}

template <typename K>
int radix_sort(K* keys, K* keys_alt, uint64_t* vals, uint64_t* vals_alt, int64_t n, int nbits,
               void* ws, cudaStream_t s) {
  if (n <= 1 || nbits <= 0) return 0;
  const int64_t nb = radix_blocks(n);
  const bool small = n <= kRadixSmall;
  int64_t h = 256 * nb;
  uint32_t* hist = (uint32_t*)ws;
  uint32_t* offs = hist + h;
  uint32_t* sws = offs + h + 1;
  K* kin = keys;
  K* kout = keys_alt;
  uint64_t* vin = vals;
  uint64_t* vout = vals_alt;
  int flips = 0;
  for (int shift = 0; shift < nbits; shift += 8) {
    int bits = nbits - shift < 8 ? nbits - shift : 8;
    uint32_t mask = (1u << bits) - 1u;
    auto pass = [&](auto ipt) {
      constexpr int IPT = decltype(ipt)::value;
      count_launch();
      k_radix_hist<K, IPT><<<(unsigned)nb, kRadixThreads, 0, s>>>(kin, n, shift, mask, hist, nb);
      scan_exclusive<uint32_t>(hist, offs, h, sws, s);
      if (vals) launch_scatter<K, true, IPT>(kin, vin, kout, vout, n, shift, mask, offs, nb, s);
      else launch_scatter<K, false, IPT>(kin, nullptr, kout, nullptr, n, shift, mask, offs, nb, s);
    };
    if (small) pass(std::integral_constant<int, kRadixIptSmall>());
    else pass(std::integral_constant<int, kRadixIpt>());
    K* t = kin;
    kin = kout;
    kout = t;
    uint64_t* tv = vin;
    vin = vout;
    vout = tv;
    flips ^= 1;
  }
  return flips;
}

template int radix_sort<uint32_t>(uint32_t*, uint32_t*, uint64_t*, uint64_t*, int64_t, int, void*,
                                  cudaStream_t);
template int radix_sort<uint64_t>(uint64_t*, uint64_t*, uint64_t*, uint64_t*, int64_t, int, void*,
                                  cudaStream_t);

// Loads every kernel of this file now (lazy module loading would otherwise
// load a kernel at its first launch, which can wait on a running persistent
// kernel, e.g. the serving kernel).
void preload_primitives() {
  cudaFuncAttributes a;
  cudaFuncGetAttributes(&a, k_scan_reduce<uint32_t, false>);
  cudaFuncGetAttributes(&a, k_scan_reduce<uint32_t, true>);
  cudaFuncGetAttributes(&a, k_scan_down<uint32_t, false>);
  cudaFuncGetAttributes(&a, k_scan_down<uint32_t, true>);
  cudaFuncGetAttributes(&a, k_scan_one<uint32_t, false>);
  cudaFuncGetAttributes(&a, k_scan_one<uint32_t, true>);
  cudaFuncGetAttributes(&a, k_radix_hist<uint32_t, kRadixIpt>);
  cudaFuncGetAttributes(&a, k_radix_hist<uint64_t, kRadixIpt>);
  cudaFuncGetAttributes(&a, k_radix_hist<uint32_t, kRadixIptSmall>);
  cudaFuncGetAttributes(&a, k_radix_hist<uint64_t, kRadixIptSmall>);
  cudaFuncGetAttributes(&a, k_radix_scatter<uint32_t, true, kRadixIpt>);
  cudaFuncGetAttributes(&a, k_radix_scatter<uint32_t, false, kRadixIpt>);
  cudaFuncGetAttributes(&a, k_radix_scatter<uint64_t, true, kRadixIpt>);
  cudaFuncGetAttributes(&a, k_radix_scatter<uint64_t, false, kRadixIpt>);
  cudaFuncGetAttributes(&a, k_radix_scatter<uint32_t, true, kRadixIptSmall>);
  cudaFuncGetAttributes(&a, k_radix_scatter<uint32_t, false, kRadixIptSmall>);
  cudaFuncGetAttributes(&a, k_radix_scatter<uint64_t, true, kRadixIptSmall>);
  cudaFuncGetAttributes(&a, k_radix_scatter<uint64_t, false, kRadixIptSmall>);
}

void preload_all() {
  preload_primitives();
  preload_analysis();
  preload_sweep();
  preload_window();
  preload_exec();
  preload_block_exec();
  preload_serve();
  preload_events();
  preload_task_kernel();
  preload_stitch();
  preload_static();
  preload_microbench();
}

}  // namespace grt
