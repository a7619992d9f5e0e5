// Device-wide primitives of libgwcp: exclusive scan of u32 and a stable LSD radix sort
// of (u64 key, u32 value) pairs restricted to the key bits that vary.
#include <algorithm>
#include <atomic>

#include "gwcp_internal.cuh"

namespace gwcp {

static std::atomic<unsigned long long> g_launches{0};
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
unsigned long long launch_count() { return g_launches.load(std::memory_order_relaxed); }

namespace {

// ---- exclusive scan --------------------------------------------------------------------
// Up to SC_ONE elements: one block, one launch (the pipeline's many small scans are launch
// latency and nothing else). Up to SC_TILE * SC_SUMS: each block's sum, then each block adds
// the sums before it itself and scans its tile (two launches, no block waits for another).
// Beyond: the sums are scanned by a kernel of their own in between.
constexpr int SC_THREADS = 256, SC_ITEMS = 16, SC_TILE = SC_THREADS * SC_ITEMS;
constexpr int SC_ONE_THREADS = 1024, SC_ONE_ITEMS = 16, SC_ONE = SC_ONE_THREADS * SC_ONE_ITEMS;
constexpr uint32_t SC_SUMS = 4096;

// exclusive scan of one value per thread (THREADS a multiple of 32); *total: the sum
template <int THREADS>
__device__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t warp_tot[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t inc = warp_inclusive_scan(v);
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = lane < THREADS / 32 ? warp_tot[lane] : 0;
    const uint32_t wi = warp_inclusive_scan(w);
    warp_tot[lane] = wi - w;
    if (lane == 31) *total = wi;
  }
  __syncthreads();
  const uint32_t r = warp_tot[warp] + inc - v;
  __syncthreads();
  return r;
}

// ITEMS values of the thread from base (16 consecutive words: four 128-bit loads where the
// array allows them)
template <int ITEMS>
__device__ __forceinline__ void load_items(const uint32_t* in, size_t base, size_t n, uint32_t (&v)[ITEMS]) {
  if (base + ITEMS <= n && (reinterpret_cast<uintptr_t>(in) & 15) == 0) {
#pragma unroll
    for (int j = 0; j < ITEMS; j += 4) {
      const uint4 q = *reinterpret_cast<const uint4*>(in + base + j);
      v[j] = q.x;
      v[j + 1] = q.y;
      v[j + 2] = q.z;
      v[j + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) v[j] = base + j < n ? in[base + j] : 0;
  }
}
template <int ITEMS>
__device__ __forceinline__ void store_items(uint32_t* out, size_t base, size_t n, const uint32_t (&v)[ITEMS]) {
  if (base + ITEMS <= n && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
#pragma unroll
    for (int j = 0; j < ITEMS; j += 4)
      *reinterpret_cast<uint4*>(out + base + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
  } else {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
      if (base + j < n) out[base + j] = v[j];
  }
}

__global__ void __launch_bounds__(SC_ONE_THREADS) k_scan_one(ScanBatch b) {
  grid_begin();
  const ScanJob job = b.job[blockIdx.x];
  const size_t base = size_t(threadIdx.x) * SC_ONE_ITEMS;
  uint32_t v[SC_ONE_ITEMS], s = 0;
  load_items<SC_ONE_ITEMS>(job.in, base, job.n, v);
#pragma unroll
  for (int j = 0; j < SC_ONE_ITEMS; ++j) s += v[j];
  __shared__ uint32_t tot;
  uint32_t ex = block_exclusive_scan<SC_ONE_THREADS>(s, &tot);
#pragma unroll
  for (int j = 0; j < SC_ONE_ITEMS; ++j) {
    const uint32_t t = v[j];
    v[j] = ex;
    ex += t;
  }
  store_items<SC_ONE_ITEMS>(job.out, base, job.n, v);
  if (threadIdx.x == 0 && job.total) *job.total = tot;
}

__global__ void __launch_bounds__(SC_THREADS) k_scan_reduce(const uint32_t* in, size_t n, uint32_t* sums) {
  grid_begin();
  const size_t base = size_t(blockIdx.x) * SC_TILE + size_t(threadIdx.x) * SC_ITEMS;
  uint32_t v[SC_ITEMS], s = 0;
  load_items<SC_ITEMS>(in, base, n, v);
#pragma unroll
  for (int j = 0; j < SC_ITEMS; ++j) s += v[j];
  __shared__ uint32_t tot;
  block_exclusive_scan<SC_THREADS>(s, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(SC_ONE_THREADS) k_scan_sums(uint32_t* sums, uint32_t nb, uint32_t* total) {
  grid_begin();
  __shared__ uint32_t tot;
  uint32_t carry = 0;
  for (uint32_t base = 0; base < nb; base += SC_ONE_THREADS) {
    const uint32_t i = base + threadIdx.x;
    const uint32_t v = i < nb ? sums[i] : 0;
    const uint32_t ex = block_exclusive_scan<SC_ONE_THREADS>(v, &tot);
    if (i < nb) sums[i] = carry + ex;
    carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

// scanned: sums holds the blocks' exclusive prefixes already; else their sums, and the last
// block writes the total
__global__ void __launch_bounds__(SC_THREADS) k_scan_apply(const uint32_t* in, uint32_t* out, size_t n,
                                                           const uint32_t* sums, bool scanned, uint32_t* total) {
  grid_begin();
  __shared__ uint32_t tot, before;
  uint32_t prefix;
  if (scanned) {
    prefix = sums[blockIdx.x];
  } else {
    uint32_t s = 0;
    for (uint32_t i = threadIdx.x; i < blockIdx.x; i += SC_THREADS) s += sums[i];
    block_exclusive_scan<SC_THREADS>(s, &before);
    prefix = before;
  }
  const size_t base = size_t(blockIdx.x) * SC_TILE + size_t(threadIdx.x) * SC_ITEMS;
  uint32_t v[SC_ITEMS], s = 0;
  load_items<SC_ITEMS>(in, base, n, v);
#pragma unroll
  for (int j = 0; j < SC_ITEMS; ++j) s += v[j];
  uint32_t ex = block_exclusive_scan<SC_THREADS>(s, &tot) + prefix;
#pragma unroll
  for (int j = 0; j < SC_ITEMS; ++j) {
    const uint32_t t = v[j];
    v[j] = ex;
    ex += t;
  }
  store_items<SC_ITEMS>(out, base, n, v);
  if (!scanned && total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = prefix + tot;
}

// ---- radix sort ------------------------------------------------------------------------
// One histogram pass over the keys counts the digits of every pass; then one kernel per
// digit: a tile ranks its pairs, publishes its digit counts, finds how many pairs of each
// digit the tiles before it hold by looking back over their published counts, and scatters
// the tile. Against a histogram, a scan and a scatter kernel per digit this reads the keys
// once per pass instead of twice and takes two launches plus one per digit instead of five
// per digit. A tile reads the counts of LOOK tiles at a time: when all tiles start together,
// tile i finds a complete prefix after about i / (2 LOOK) rounds of memory latency. The wait is
// bounded, and a tile that gives up counts its digits in the pairs before it itself: the sort
// has one result, whatever the waits do, so it has no status and no caller reads one.
// A digit takes the next eight varying bits of the key, in up to four separate runs, so the
// number of passes is that of the varying bits alone (with runs of eight adjacent bits, the
// composite keys of 64 agents took 6 passes instead of 5).
// Measured, 50M pairs, per pass: 0.46 ms (2.6 TB/s of the 24 bytes a pass moves), bound by
// the latency of a tile's phases at four blocks per SM; the three-kernel passes took 0.9 ms.
// Tiles of 256 x 12 pairs; 256 x 8 0.53 ms, 512 x 8 0.60, 256 x 16 0.65 (too many registers
// for four blocks). Ranks by eight ballots; match.any measured 9% slower.
constexpr int LOOK = 8;
constexpr int kMaxPasses = 9;

// a pair the filter of the first pass keeps
__device__ __forceinline__ bool radix_kept(uint64_t key, const RadixKeep& kp) {
  if (!kp.bits) return true;
  const uint32_t h = wl_bit(key >> kp.shift, kp.log2);
  return (__ldg(kp.bits + (h >> 5)) >> (h & 31)) & 1u;
}

// a digit: up to four runs of key bits, each shifted to its place
struct Digit {
  uint8_t sh[4], mask[4];
  __host__ __device__ __forceinline__ uint32_t of(uint64_t k) const {
    return (uint32_t(k >> sh[0]) & mask[0]) | (uint32_t(k >> sh[1]) & mask[1]) | (uint32_t(k >> sh[2]) & mask[2]) |
           (uint32_t(k >> sh[3]) & mask[3]);
  }
};
struct SweepPlan {
  int passes;
  Digit dig[kMaxPasses];
};

// digit counts of all passes (kept keys only); also clears the tiles' published counts
constexpr int HI_THREADS = 512;
__global__ void __launch_bounds__(HI_THREADS) k_sweep_hist(const uint64_t* keys, size_t n, const uint32_t* n_dev,
                                                           const __grid_constant__ SweepPlan pl, uint32_t* hist, uint4* status,
                                                           size_t status_quads, RadixKeep kp) {
  grid_begin();
  __shared__ uint32_t h[kMaxPasses * 256];
  for (int i = threadIdx.x; i < pl.passes * 256; i += HI_THREADS) h[i] = 0;
  const size_t first = size_t(blockIdx.x) * HI_THREADS + threadIdx.x, step = size_t(gridDim.x) * HI_THREADS;
  for (size_t i = first; i < status_quads; i += step) status[i] = make_uint4(0, 0, 0, 0);
  if (n_dev && *n_dev < n) n = *n_dev;
  __syncthreads();
  constexpr int U = 4;  // keys in flight per thread
  for (size_t i0 = first; i0 < n; i0 += U * step) {
    uint64_t k[U];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const size_t i = i0 + u * step;
      k[u] = i < n ? keys[i] : 0;
      ok[u] = i < n;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!ok[u] || !radix_kept(k[u], kp)) continue;
      for (int p = 0; p < pl.passes; ++p) atomicAdd(&h[p * 256 + pl.dig[p].of(k[u])], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < pl.passes * 256; i += HI_THREADS)
    if (h[i]) atomicAdd(hist + i, h[i]);
}

// the lanes with the same digit among those with a pair
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, bool valid) {
  uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const bool one = (d >> q) & 1u;
    const uint32_t b = __ballot_sync(0xffffffffu, one);
    peers &= one ? b : ~b;
  }
  return peers;
}

struct SweepArgs {
  const uint64_t* kin;
  const uint32_t* vin;
  uint64_t* kout;
  uint32_t* vout;
  size_t n;
  const uint32_t* n_dev;
  Digit dig;
  const uint32_t* hist;        // [256] digit counts of this pass
  unsigned long long* status;  // [tiles][256] (tag << 32 | count): the tile's own, or up to and with it
  uint32_t* counter;           // tiles handed out, in order
  uint32_t tag;                // this pass's tag of an own count; tag + 1: of a prefix
  RadixKeep kp;
  uint32_t polls;  // looks without news before a tile gives up
};

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

template <int THREADS, int ITEMS>
constexpr size_t sweep_smem() {
  return size_t(THREADS) * ITEMS * 12 + size_t(THREADS / 32) * 256 * 4;
}

// What a tile that has given up does in the place of the rest of its wait: it counts the kept
// pairs of each digit in front of it (cnt: 256 words), publishes its prefixes and sets glob,
// by the whole block. Out of line, with all it needs computed again: no other tile pays for it.
template <int THREADS>
__device__ __noinline__ void count_before(const SweepArgs& a, size_t tile, size_t before, uint32_t* cnt,
                                          const uint32_t* tile_off, uint32_t nvalid, uint32_t* glob) {
  __shared__ uint32_t all;
  const uint32_t tid = threadIdx.x;
  if (tid < 256) cnt[tid] = 0;
  __syncthreads();
  for (size_t i = tid; i < before; i += THREADS) {
    const uint64_t k = a.kin[i];
    if (radix_kept(k, a.kp)) atomicAdd(&cnt[a.dig.of(k)], 1u);
  }
  __syncthreads();
  const uint32_t dig_base = block_exclusive_scan<THREADS>(tid < 256 ? a.hist[tid] : 0u, &all);
  if (tid < 256) {
    const uint32_t own = (tid < 255 ? tile_off[tid + 1] : nvalid) - tile_off[tid];
    st_relaxed(a.status + tile * 256 + tid, (static_cast<unsigned long long>(a.tag + 1) << 32) | (cnt[tid] + own));
    glob[tid] = dig_base + cnt[tid];
  }
  __syncthreads();
}

// Warp w of a tile owns items [w * 32 * ITEMS, ..) of it, visited in rounds of 32 consecutive
// items; ranks within a round follow lane order, so the sort is stable. The tile is first put
// in digit order in shared memory, so that consecutive threads write consecutive positions
// of one digit's run.
template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS, ITEMS <= 4 ? 6 : 4) k_sweep(const __grid_constant__ SweepArgs a) {
  grid_begin();
  constexpr int WARPS = THREADS / 32, TILE = THREADS * ITEMS;
  static_assert(THREADS >= 256, "a thread per digit");
  extern __shared__ __align__(16) unsigned char dyn[];
  uint64_t* const sk = reinterpret_cast<uint64_t*>(dyn);
  uint32_t* const sv = reinterpret_cast<uint32_t*>(sk + TILE);
  uint32_t* const cnt = sv + TILE;  // [WARPS][256]
  __shared__ uint32_t tile_off[256], glob[256], s_tile, tot, tot2;
  __shared__ int s_gone;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  size_t n = a.n;
  if (a.n_dev && *a.n_dev < n) n = *a.n_dev;
  if (tid == 0) {
    s_tile = atomicAdd(a.counter, 1u);  // tiles start in order: those before this one run or have run
    s_gone = 0;
  }
  for (int i = tid; i < WARPS * 256; i += THREADS) cnt[i] = 0;
  __syncthreads();
  const uint32_t tile = s_tile;
  if (size_t(tile) * TILE >= n) return;
  const size_t base = size_t(tile) * TILE + size_t(warp) * (ITEMS * 32) + lane;
  uint64_t k[ITEMS];
  uint32_t rank[ITEMS];
  bool valid[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const size_t i = base + size_t(r) * 32;
    k[r] = i < n ? a.kin[i] : 0;
  }
  if (a.vin) {  // the values are read after the ranks; their lines are fetched meanwhile
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
      if (base + size_t(r) * 32 < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.vin + base + size_t(r) * 32));
  }
  uint32_t* const wcnt = cnt + warp * 256;
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    valid[r] = base + size_t(r) * 32 < n && radix_kept(k[r], a.kp);
    const uint32_t d = a.dig.of(k[r]);
    const uint32_t peers = digit_peers(d, valid[r]);
    const uint32_t before = __popc(peers & lt);
    uint32_t b0 = 0;
    if (valid[r] && before == 0) b0 = atomicAdd(&wcnt[d], __popc(peers));
    rank[r] = __shfl_sync(0xffffffffu, b0, (__ffs(peers) - 1) & 31) + before;
  }
  __syncthreads();
  uint32_t own = 0;
  unsigned long long* const status = a.status + size_t(tile) * 256;
  if (tid < 256) {  // a digit per thread: the warps' offsets, the tile's count
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
      const uint32_t t = cnt[w * 256 + tid];
      cnt[w * 256 + tid] = own;
      own += t;
    }
    st_relaxed(status + tid, (static_cast<unsigned long long>(tile ? a.tag : a.tag + 1) << 32) | own);
  }
  const uint32_t dig_base = block_exclusive_scan<THREADS>(tid < 256 ? a.hist[tid] : 0u, &tot2);
  const uint32_t off = block_exclusive_scan<THREADS>(own, &tot);
  if (tid < 256) tile_off[tid] = off;
  if (a.kp.bits && tile == 0 && tid == 0) *a.kp.n_out = tot2;  // all kept pairs
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    if (valid[r]) {
      const uint32_t d = a.dig.of(k[r]);
      const uint32_t lp = tile_off[d] + wcnt[d] + rank[r];
      sk[lp] = k[r];
      if (a.vin) sv[lp] = a.vin[base + size_t(r) * 32];
    }
  }
  if (tid < 256) {
    // pairs of this digit in the tiles before
    uint32_t excl = 0, spins = 0;
    bool gone = false;
    for (int64_t t = int64_t(tile) - 1; t >= 0;) {
      unsigned long long w[LOOK];
#pragma unroll
      for (int j = 0; j < LOOK; ++j)
        w[j] = t >= j ? ld_relaxed(a.status + size_t(t - j) * 256 + tid)
                      : static_cast<unsigned long long>(a.tag + 1) << 32;
      bool stop = false;
      int used = 0;
#pragma unroll
      for (int j = 0; j < LOOK; ++j) {
        if (stop) continue;
        const uint32_t tg = uint32_t(w[j] >> 32);
        if (tg == a.tag + 1) {  // a complete prefix
          excl += uint32_t(w[j]);
          used = -1;
          stop = true;
        } else if (tg == a.tag) {
          excl += uint32_t(w[j]);
          used = j + 1;
        } else {
          stop = true;  // not published yet: look again from here
        }
      }
      if (used < 0) break;
      t -= used;
      if (used == 0 && ++spins > a.polls) {
        gone = true;
        break;
      }
    }
    if (gone)
      s_gone = 1;
    else if (tile)
      st_relaxed(status + tid, (static_cast<unsigned long long>(a.tag + 1) << 32) | (excl + own));
    glob[tid] = dig_base + excl;
  }
  __syncthreads();
  const uint32_t nvalid = tot;
  // (the input stays as it is until every tile of this pass is done)
  if (s_gone) count_before<THREADS>(a, tile, size_t(tile) * TILE, cnt, tile_off, nvalid, glob);
  for (uint32_t i = tid; i < nvalid; i += THREADS) {
    const uint64_t key = sk[i];
    const uint32_t d = a.dig.of(key);
    const uint32_t pos = glob[d] + (i - tile_off[d]);
    a.kout[pos] = key;
    if (a.vout) a.vout[pos] = sv[i];
  }
}

// The whole sort of up to ONE_MAX pairs in one block (the tile passes of k_sweep on one
// tile, every pass in shared memory).
constexpr int ONE_THREADS = 1024, ONE_ITEMS = 4, ONE_MAX = ONE_THREADS * ONE_ITEMS;
__global__ void __launch_bounds__(ONE_THREADS) k_sort_one(const uint64_t* kin, const uint32_t* vin, uint64_t* kout,
                                                          uint32_t* vout, uint32_t n, const uint32_t* n_dev,
                                                          const __grid_constant__ SweepPlan pl, RadixKeep kp) {
  grid_begin();
  constexpr int WARPS = ONE_THREADS / 32;
  extern __shared__ __align__(16) unsigned char dyn[];
  uint64_t* const sk = reinterpret_cast<uint64_t*>(dyn);
  uint32_t* const sv = reinterpret_cast<uint32_t*>(sk + ONE_MAX);
  uint32_t* const cnt = sv + ONE_MAX;  // [WARPS][256]
  __shared__ uint32_t tile_off[256], tot;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (n_dev && *n_dev < n) n = *n_dev;
  const uint32_t base = warp * (ONE_ITEMS * 32) + lane;
  const uint32_t lt = lanemask_lt();
  uint64_t k[ONE_ITEMS];
  uint32_t v[ONE_ITEMS], rank[ONE_ITEMS];
  bool valid[ONE_ITEMS];
#pragma unroll
  for (int r = 0; r < ONE_ITEMS; ++r) {
    const uint32_t i = base + r * 32;
    k[r] = i < n ? kin[i] : 0;
    v[r] = i < n && vin ? vin[i] : 0;
    valid[r] = i < n && radix_kept(k[r], kp);
  }
  uint32_t* const wcnt = cnt + warp * 256;
  for (int p = 0; p < pl.passes; ++p) {
    for (int i = tid; i < WARPS * 256; i += ONE_THREADS) cnt[i] = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ONE_ITEMS; ++r) {
      const uint32_t d = pl.dig[p].of(k[r]);
      const uint32_t peers = digit_peers(d, valid[r]);
      const uint32_t before = __popc(peers & lt);
      uint32_t b0 = 0;
      if (valid[r] && before == 0) b0 = atomicAdd(&wcnt[d], __popc(peers));
      rank[r] = __shfl_sync(0xffffffffu, b0, (__ffs(peers) - 1) & 31) + before;
    }
    __syncthreads();
    uint32_t own = 0;
    if (tid < 256) {
#pragma unroll 8
      for (int w = 0; w < WARPS; ++w) {
        const uint32_t t = cnt[w * 256 + tid];
        cnt[w * 256 + tid] = own;
        own += t;
      }
    }
    const uint32_t off = block_exclusive_scan<ONE_THREADS>(own, &tot);
    if (tid < 256) tile_off[tid] = off;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ONE_ITEMS; ++r) {
      if (valid[r]) {
        const uint32_t d = pl.dig[p].of(k[r]);
        const uint32_t lp = tile_off[d] + wcnt[d] + rank[r];
        sk[lp] = k[r];
        sv[lp] = v[r];
      }
    }
    __syncthreads();
    n = tot;  // the kept pairs
#pragma unroll
    for (int r = 0; r < ONE_ITEMS; ++r) {
      const uint32_t i = base + r * 32;
      valid[r] = i < n;
      k[r] = valid[r] ? sk[i] : 0;
      v[r] = valid[r] ? sv[i] : 0;
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < ONE_ITEMS; ++r) {
    const uint32_t i = base + r * 32;
    if (valid[r]) {
      kout[i] = k[r];
      if (vout) vout[i] = v[r];
    }
  }
  if (kp.bits && tid == 0) *kp.n_out = n;
}

// tiles of 1,024 pairs up to this count (more blocks for small sorts), of 3,072 beyond
constexpr size_t kSmallSort = size_t(1) << 18;
constexpr size_t kSmallTile = 1024, kLargeTile = 256 * 12;
size_t sweep_tile(size_t n) { return n <= kSmallSort ? kSmallTile : kLargeTile; }
constexpr size_t kSweepHead = kMaxPasses * 256 + 16;  // words before the tiles' counts: histograms, counters

template <int THREADS, int ITEMS>
void launch_sweep(const SweepArgs& a, uint32_t tiles, cudaStream_t s) {
  constexpr size_t smem = sweep_smem<THREADS, ITEMS>();
  if (smem > 48 * 1024)
    cudaFuncSetAttribute(k_sweep<THREADS, ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  launch(k_sweep<THREADS, ITEMS>, tiles, THREADS, smem, s)(a);
  count_launch();
}

}  // namespace

size_t scan_tmp_need(size_t n) { return (n + SC_TILE - 1) / SC_TILE + 1; }

void scan_small(const ScanBatch& b, int jobs, cudaStream_t s) {
  launch(k_scan_one, jobs, SC_ONE_THREADS, 0, s)(b);
  count_launch();
}

namespace {
__global__ void __launch_bounds__(256) k_fill(const __grid_constant__ FillBatch b) {
  grid_begin();
  const size_t t = size_t(blockIdx.x) * blockDim.x + threadIdx.x, all = size_t(gridDim.x) * blockDim.x;
  for (int j = 0; j < b.n; ++j) {
    const uint32_t v = b.job[j].value;
    const size_t n = b.job[j].words;
    uint4* const q = static_cast<uint4*>(b.job[j].ptr);
    for (size_t i = t; i < n / 4; i += all) q[i] = make_uint4(v, v, v, v);
    if (t < n % 4) static_cast<uint32_t*>(b.job[j].ptr)[n / 4 * 4 + t] = v;
  }
}
__global__ void k_read_back(const DevStatus* st, const __grid_constant__ ReadBack r, DevStatus* st_out, uint32_t* val_out) {
  grid_begin();
  const int t = threadIdx.x;
  constexpr int words = sizeof(DevStatus) / 4;
  static_assert(sizeof(DevStatus) % 4 == 0 && words + 8 <= 64);
  if (t < words) reinterpret_cast<uint32_t*>(st_out)[t] = reinterpret_cast<const uint32_t*>(st)[t];
  if (t < r.n) val_out[t] = *r.word[t];
}
__global__ void k_status_init(DevStatus* st, const __grid_constant__ DevStatus v) { grid_begin(); *st = v; }
}  // namespace

void fill_all(const FillBatch& b, cudaStream_t s) {
  size_t most = 0;
  for (int j = 0; j < b.n; ++j) most = std::max(most, b.job[j].words);
  if (!b.n) return;
  launch(k_fill, unsigned(std::min<size_t>((most + 1023) / 1024, kSms * 8)), 256, 0, s)(b);
  count_launch();
}
void read_back_to(const DevStatus* st, const ReadBack& r, DevStatus* st_out, uint32_t* val_out, cudaStream_t s) {
  launch(k_read_back, 1, 64, 0, s)(st, r, st_out, val_out);
  count_launch();
}
void status_init(DevStatus* st, const DevStatus& v, cudaStream_t s) {
  launch(k_status_init, 1, 1, 0, s)(st, v);
  count_launch();
}

bool scan_is_small(size_t n) { return n <= size_t(SC_ONE); }

void scan_exclusive(const uint32_t* in, uint32_t* out, size_t n, uint32_t* total_dev, uint32_t* tmp,
                    cudaStream_t s) {
  if (n == 0) {
    if (total_dev) cudaMemsetAsync(total_dev, 0, sizeof(uint32_t), s);
    return;
  }
  if (scan_is_small(n)) {
    ScanBatch b{};
    b.job[0] = ScanJob{in, out, total_dev, uint32_t(n)};
    scan_small(b, 1, s);
    return;
  }
  const uint32_t nb = uint32_t((n + SC_TILE - 1) / SC_TILE);
  launch(k_scan_reduce, nb, SC_THREADS, 0, s)(in, n, tmp);
  count_launch();
  const bool own_sums = nb <= SC_SUMS;
  if (!own_sums) {
    launch(k_scan_sums, 1, SC_ONE_THREADS, 0, s)(tmp, nb, total_dev);
    count_launch();
  }
  launch(k_scan_apply, nb, SC_THREADS, 0, s)(in, out, n, tmp, !own_sums, total_dev);
  count_launch();
}

void scan_all(const ScanBatch& b, int jobs, uint32_t* tmp, cudaStream_t s) {
  bool small = true;
  for (int j = 0; j < jobs; ++j) small = small && scan_is_small(b.job[j].n);
  if (small) {
    scan_small(b, jobs, s);
    return;
  }
  for (int j = 0; j < jobs; ++j) {
    const ScanJob& q = b.job[j];
    scan_exclusive(q.in, q.out, q.n, q.total, tmp, s);
  }
}

namespace {
SweepPlan sweep_plan(uint64_t mask) {
  SweepPlan pl{};
  int bit = 0;
  while (bit < 64 && (mask >> bit)) {
    Digit& d = pl.dig[pl.passes++];
    int have = 0;  // bits of the digit so far
    for (int q = 0; q < 4 && have < 8; ++q) {
      while (bit < 64 && !((mask >> bit) & 1)) ++bit;
      int len = 0;
      while (bit + len < 64 && ((mask >> (bit + len)) & 1) && have + len < 8) ++len;
      if (!len) break;
      d.sh[q] = uint8_t(bit - have);  // have <= bit: every bit of the digit has its own key bit
      d.mask[q] = uint8_t(((1u << len) - 1u) << have);
      have += len;
      bit += len;
    }
    while (bit < 64 && !((mask >> bit) & 1)) ++bit;
  }
  return pl;
}
}  // namespace

int radix_passes(uint64_t mask) { return sweep_plan(mask).passes; }

size_t radix_tmp_need(size_t n) {
  if (n <= size_t(ONE_MAX)) return 1;
  const size_t tiles = std::max((n + kLargeTile - 1) / kLargeTile, (std::min(n, kSmallSort) + kSmallTile - 1) / kSmallTile);
  return kSweepHead + 2 + 512 * tiles;
}

bool radix_sort_pairs(uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, size_t n, uint64_t mask,
                      uint32_t* tmp, cudaStream_t s, const uint32_t* n_dev, RadixKeep keep, uint32_t polls) {
  if (keep.bits) {
    if (n == 0) {
      cudaMemsetAsync(keep.n_out, 0, 4, s);
      return false;
    }
    if (mask == 0) mask = 1;  // the filter needs one pass
  } else if (n <= 1) {
    return false;
  }
  const SweepPlan pl = sweep_plan(mask);
  if (!pl.passes) return false;
  if (n <= size_t(ONE_MAX)) {
    constexpr size_t smem = size_t(ONE_MAX) * 12 + size_t(ONE_THREADS / 32) * 256 * 4;
    cudaFuncSetAttribute(k_sort_one, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    launch(k_sort_one, 1, ONE_THREADS, smem, s)(k0, v0, k1, v1, uint32_t(n), n_dev, pl, keep);
    count_launch();
    return true;
  }
  const size_t tile = sweep_tile(n);
  const uint32_t tiles = uint32_t((n + tile - 1) / tile);
  uint32_t* hist = tmp;
  uint32_t* counters = tmp + kMaxPasses * 256;
  auto* status = reinterpret_cast<unsigned long long*>((reinterpret_cast<uintptr_t>(tmp + kSweepHead) + 15) & ~uintptr_t(15));
  cudaMemsetAsync(tmp, 0, kSweepHead * 4, s);
  const uint32_t hist_blocks = uint32_t(std::min<size_t>((n + 2047) / 2048, kSms * 4));
  launch(k_sweep_hist, hist_blocks, HI_THREADS, 0, s)(k0, n, n_dev, pl, hist, reinterpret_cast<uint4*>(status),
                                                 size_t(tiles) * 128, keep);
  count_launch();
  bool in_second = false;
  for (int p = 0; p < pl.passes; ++p) {
    SweepArgs a{};
    a.kin = in_second ? k1 : k0;
    a.vin = in_second ? v1 : v0;
    a.kout = in_second ? k0 : k1;
    a.vout = in_second ? v0 : v1;
    a.n = n;
    a.n_dev = n_dev;
    a.dig = pl.dig[p];
    a.hist = hist + p * 256;
    a.status = status;
    a.counter = counters + p;
    a.tag = uint32_t(2 * p + 1);
    if (p == 0) a.kp = keep;
    a.polls = polls;
    if (tile == kSmallTile)
      launch_sweep<256, 4>(a, tiles, s);
    else
      launch_sweep<256, 12>(a, tiles, s);
    if (p == 0 && keep.bits) n_dev = keep.n_out;  // later passes sort the kept pairs
    in_second = !in_second;
  }
  return in_second;
}

int debug_sort(uint64_t* key, uint32_t* val, uint64_t n, uint64_t mask, uint32_t polls) {
  unsigned char* mem = nullptr;
  const size_t kb = n * 8, vb = val ? (n * 4 + 15) & ~size_t(15) : 0;
  if (cudaMalloc(&mem, 2 * (kb + vb) + 512 + radix_tmp_need(n) * 4) != cudaSuccess) {
    cudaGetLastError();
    return GWCP_ERR_OOM;
  }
  // scratch first (256-byte aligned), then keys, then values
  auto* tmp = reinterpret_cast<uint32_t*>(mem);
  unsigned char* at = mem + ((radix_tmp_need(n) * 4 + 255) & ~size_t(255));
  auto *k0 = reinterpret_cast<uint64_t*>(at), *k1 = reinterpret_cast<uint64_t*>(at + kb);
  uint32_t *v0 = nullptr, *v1 = nullptr;
  if (val) {
    v0 = reinterpret_cast<uint32_t*>(at + 2 * kb);
    v1 = reinterpret_cast<uint32_t*>(at + 2 * kb + vb);
  }
  cudaMemcpy(k0, key, kb, cudaMemcpyHostToDevice);
  if (val) cudaMemcpy(v0, val, n * 4, cudaMemcpyHostToDevice);
  const bool second = radix_sort_pairs(k0, v0, k1, v1, n, mask, tmp, nullptr, nullptr, {}, polls);
  cudaMemcpy(key, second ? k1 : k0, kb, cudaMemcpyDeviceToHost);
  if (val) cudaMemcpy(val, second ? v1 : v0, n * 4, cudaMemcpyDeviceToHost);
  const int rc = cudaDeviceSynchronize() == cudaSuccess && cudaGetLastError() == cudaSuccess ? GWCP_OK : GWCP_ERR_CUDA;
  cudaFree(mem);
  return rc;
}

}  // namespace gwcp
