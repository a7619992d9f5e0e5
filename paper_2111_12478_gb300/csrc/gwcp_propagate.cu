// Clock propagation of libgwcp (Algorithms 1 and 2 of the paper).
//
// One warp per agent walks the agent's clock-changing entries in trace order:
// acquires, releases, barrier participations and accesses made while holding a lock.
// The agent's P_t and H_t live in registers, blocked so that lane l holds entries
// [l*K, l*K+K) (K = Wp/32); every join is a 32-lane vector max over the whole clock
// width (64-, 128- or 256-bit loads). After each entry the warp stores P_t as the
// agent's next clock version; the race check reads those rows.
//
// A third clock, JN_t, is the join of every H snapshot that entered P_t: joined from the
// lock's published JN at an acquire, over the members at a barrier, and with every H
// snapshot joined in the release loop or at an in-section access. H moves only by joins of
// whole H clocks, so JN_t[v] >= e means that P_t already holds the H snapshot of v's release
// at local time e, and a join of that release (release loop, L^w / L^r) changes nothing and
// is skipped.
//
// Cross-agent values are snapshots written once: a release stores P_t, H_t and JN_t (the
// paper's P_<l,s>, H_<l,s> and its Rel-queue entry) over rows filled with a sentinel word; a
// row without a sentinel word is complete. An acquire waits (bounded) for the releases it
// joins - the latest release on every overlapping scope of the lock, precomputed per
// acquire. Because every dependence points backwards in trace order and each walker
// processes its own entries in trace order, the earliest unprocessed event can always
// proceed, so all waits end on a well-formed trace. All walkers are co-resident
// (cooperative launch). A barrier whose block fits in one CTA is a shared-memory join: two
// buffers in turn hold the block's joined rows, and since clocks only grow a member adds its
// rows with max reductions only if they changed since the last barrier, else its own entry
// alone. Other barriers use a per-barrier global join with atomics and a bounded wait. A wait
// that gives up sets GWCP_ERR_TIMEOUT and the walker continues without waiting, so no CTA
// barrier is left short of arrivals.
//
// What bounds it: the chain of barrier periods and lock hand-offs, each as long as its
// slowest walker's steps (two walkers per scheduler issue an instruction every five to eight
// cycles), so everything a step does not need is kept off that path. Plan entries are read
// from shared memory, loaded 16 at a time a batch ahead; the records of the next release and
// the snapshot rows of coming acquires are fetched by walkers that reach a barrier without
// another step since the last one (they are early), or after a release when no barrier is
// near. Propagation, ms, against register-held plan entries decoded by shuffles, staging at
// every step and joins without JN_t: 64 warps, 10M events 16.4 -> 11.2; 256 warps, 5M
// 6.1 -> 1.87; 512 warps (8 per block), 3M 2.9 (tile tables) and 1.0; two blocks of 128
// threads, 250k 6.2 -> 0.48; 64 threads, 10k 0.28 -> 0.07; compressed versions, 64 warps, 3M
// 7.1 -> 5.2. An mbarrier polled between pieces of that work measured 11.6 on the first.
#include "gwcp_internal.cuh"

namespace gwcp {

namespace {

constexpr uint32_t kSpinLimit = 1u << 23;

struct PropArgs {
  Geo g;
  const Event* ev;
  DevStatus* st;
  const uint32_t *sy_start, *sy_idx, *sy_kind, *sy_N, *sy_ver, *sy_aux, *sy_agent;
  const uint32_t *incs_off, *incs_ver, *incs_k, *sy_inner, *cs_parent, *cs_exp, *cs_r0, *ex_dep_off, *ex_dep_cnt;
  const uint32_t* rowbase;
  const uint32_t *cs_of_sync, *cs_agent, *cs_sid, *cs_epoch, *cs_rel_idx, *cs_lock, *lock_cs_lo, *cs_rel_epoch;
  const uint32_t *acq_dep_off, *acq_dep_cnt, *pool;
  const uint32_t* flat;
  uint4* plan;   // two per step
  uint4* plan2;  // two per step, in-section accesses only: (agent, release epoch) per joined release
  uint4* recmeta;
  uint32_t hb_only;  // publish H_t instead of P_t as the clock versions the check reads
  uint32_t* rows;
  uint32_t *psnap, *hsnap, *jsnap, *cursor;
  uint32_t *bar_j, *bar_jj, *bar_cnt;
  uint32_t n_locks;
  int cta_barriers;
  // shared memory of a CTA, in words: the barrier joins' rows, then per warp its plan entries,
  // a row, the H rows of the last acquire (keep_h) and `slots` staged acquires of up to `deps`
  // releases each
  uint32_t acc_words, warp_words, slots, deps, keep_h;
  uint32_t forced;  // forced compression at barriers: local times come from the plan
  // compressed clock versions: rows holds B header words per version
  uint32_t compress;
  uint32_t* cv_pool;
  unsigned long long cv_cap;
  unsigned long long *cv_used, *cv_words;  // pool words handed out; words written
};

// Clock rows another walker may still be writing: every word goes once from SENTINEL to
// its value, and a reader takes a row only when no word is SENTINEL, so relaxed gpu-scope
// accesses (each word single-copy atomic, no order between words needed) make the
// exchange race-free under the PTX memory model; they cost what .cg accesses cost.
template <int K>
__device__ __forceinline__ void load_row(const uint32_t* row, uint32_t (&x)[K]) {
  const int lane = threadIdx.x & 31;
  const uint32_t* p = row + lane * K;
  if constexpr (K == 1) {
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(x[0]) : "l"(p) : "memory");
  } else if constexpr (K == 2) {
    asm volatile("ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(x[0]), "=r"(x[1]) : "l"(p) : "memory");
  } else {
#pragma unroll
    for (int j = 0; j < K; j += 4)
      asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(x[j]), "=r"(x[j + 1]), "=r"(x[j + 2]), "=r"(x[j + 3])
                   : "l"(p + j)
                   : "memory");
  }
}

template <int K>
__device__ __forceinline__ void store_row(uint32_t* row, const uint32_t (&x)[K]) {
  const int lane = threadIdx.x & 31;
  uint32_t* p = row + lane * K;
  if constexpr (K == 1) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(x[0]) : "memory");
  } else if constexpr (K == 2) {
    asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(x[0]), "r"(x[1]) : "memory");
  } else {
#pragma unroll
    for (int j = 0; j < K; j += 4)
      asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p + j), "r"(x[j]), "r"(x[j + 1]),
                   "r"(x[j + 2]), "r"(x[j + 3])
                   : "memory");
  }
}

// the same blocked layout in shared memory (plain stores: __stcg is for global memory)
template <int K>
__device__ __forceinline__ void store_row_shared(uint32_t* row, const uint32_t (&x)[K]) {
  uint32_t* p = row + (threadIdx.x & 31) * K;
#pragma unroll
  for (int j = 0; j < K; ++j) p[j] = x[j];
}

// Walker state of the compressed-version pool: the chunk being filled, words written.
struct CvState {
  unsigned long long cur, end, words;
};

// Stores the clock the warp left in `scratch` (its Wc shared words, entry e at e) as the
// compressed version `row` (the blockVC / warpVC form): B header words at rows + row * B;
// the words of expanded blocks go to the pool, from a chunk of kCvChunk words the walker
// takes at a time. A version that does not fit the pool gets zero headers, and the host
// runs again with a larger pool (cv_used keeps counting). Only the compressing walker
// instantiations contain it, out of line (the register path below is the common one).
__device__ __noinline__ CvState put_row_c(const PropArgs& a, uint32_t row, const uint32_t* scratch, CvState cs) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t apb = a.g.apb, nb = a.g.B, gs = cv_group(a.g.gran), nw = (apb + gs - 1) / gs;
  // pass 1: which of the lane's blocks (b = lane + 32 i) are uniform, and the words the
  // others need: nw warp words, plus 32 lane values per warp that is not uniform
  uint32_t need = 0, umask = 0;
  for (uint32_t b = lane, i = 0; b < nb; b += 32, ++i) {
    const uint32_t* q = scratch + b * apb;
    bool uni = true;
    uint32_t ew = 0;
    for (uint32_t w = 0; w < nw; ++w) {
      const uint32_t lo = w * gs, hi = min(lo + gs, apb), v = q[lo];
      bool wu = true;
      for (uint32_t e = lo; e < hi; ++e) wu &= q[e] == v;
      uni &= wu && v == q[0];
      ew += wu ? 0u : 1u;
    }
    if (uni)
      umask |= 1u << i;
    else
      need += nw + 32 * ew;
  }
  const uint32_t incl = warp_inclusive_scan(need);
  const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
  if (total && cs.cur + total > cs.end) {
    unsigned long long base = 0;
    const unsigned long long take = max(total, kCvChunk);
    if (lane == 0) base = atomicAdd(a.cv_used, take);
    base = __shfl_sync(0xffffffffu, base, 0);
    cs.cur = base;
    cs.end = base + take;
  }
  unsigned long long o = cs.cur + (incl - need);
  cs.cur += total;
  cs.words += nb + total;
  const bool fits = cs.cur <= a.cv_cap;  // the whole version lies inside the pool
  uint32_t* hdr = a.rows + size_t(row) * nb;
  // pass 2: headers, warp words and lane values
  for (uint32_t b = lane, i = 0; b < nb; b += 32, ++i) {
    const uint32_t* q = scratch + b * apb;
    if ((umask >> i) & 1u) {
      __stcg(hdr + b, q[0]);
      continue;
    }
    if (!fits) {
      __stcg(hdr + b, 0u);
      continue;
    }
    __stcg(hdr + b, kCvExpanded | uint32_t(o));
    unsigned long long o2 = o + nw;
    for (uint32_t w = 0; w < nw; ++w) {
      const uint32_t lo = w * gs, hi = min(lo + gs, apb), v = q[lo];
      bool wu = true;
      for (uint32_t e = lo; e < hi; ++e) wu &= q[e] == v;
      if (wu) {
        __stcg(a.cv_pool + o + w, v);
      } else {
        __stcg(a.cv_pool + o + w, kCvExpanded | uint32_t(o2));
        for (uint32_t e = 0; e < 32; ++e) __stcg(a.cv_pool + o2 + e, lo + e < apb ? q[lo + e] : 0u);
        o2 += 32;
      }
    }
    o = o2;
  }
  __syncwarp();
  return cs;
}

// The same store from registers, for warp granularity with K dividing agents_per_block:
// a block is L = apb / K consecutive lanes, so its uniformity is one ballot and its
// expanded words are the lanes' own entries (one per agent, in agent order).
template <int K>
__device__ __forceinline__ CvState put_row_lanes(const PropArgs& a, uint32_t row, const uint32_t (&x)[K], CvState cs) {
  const uint32_t lane = threadIdx.x & 31, apb = a.g.apb, nb = a.g.B, L = apb / K;
  const uint32_t grp = lane / L, first = grp * L;
  const bool live = grp < nb;  // lanes past the last block hold padding
  bool same = true;
#pragma unroll
  for (int j = 0; j < K; ++j) same &= x[j] == x[0];
  const uint32_t head_v = __shfl_sync(0xffffffffu, x[0], live ? first : lane);
  const uint32_t ok = __ballot_sync(0xffffffffu, live && same && x[0] == head_v);
  const uint32_t gmask = live ? ((L == 32 ? 0xffffffffu : (1u << L) - 1u) << first) : 0u;
  const bool uni = live && (ok & gmask) == gmask;
  const bool head = live && lane == first;
  const uint32_t expm = __ballot_sync(0xffffffffu, head && !uni);  // bit at each expanded block's first lane
  const uint32_t total = __popc(expm) * apb;
  if (total && cs.cur + total > cs.end) {
    unsigned long long base = 0;
    const unsigned long long take = max(total, kCvChunk);
    if (lane == 0) base = atomicAdd(a.cv_used, take);
    base = __shfl_sync(0xffffffffu, base, 0);
    cs.cur = base;
    cs.end = base + take;
  }
  const unsigned long long o = cs.cur + (unsigned long long)apb * __popc(expm & ((1u << first) - 1u));
  cs.cur += total;
  cs.words += nb + total;
  const bool fits = cs.cur <= a.cv_cap;
  if (head) __stcg(a.rows + size_t(row) * nb + grp, uni ? x[0] : fits ? kCvExpanded | uint32_t(o) : 0u);
  if (live && !uni && fits) {
#pragma unroll
    for (int j = 0; j < K; ++j) __stcg(a.cv_pool + o + (lane - first) * K + j, x[j]);
  }
  return cs;
}

// entry v of a blocked clock (owner lane v / K, register v % K), broadcast to the warp. The
// registers are selected by bit tests of v, so that the array is never indexed (indexed, it
// lives in local memory).
template <int K>
__device__ __forceinline__ uint32_t get_entry(const uint32_t (&x)[K], uint32_t v) {
  uint32_t t[K];
#pragma unroll
  for (int j = 0; j < K; ++j) t[j] = x[j];
#pragma unroll
  for (int h = K / 2; h >= 1; h /= 2)
#pragma unroll
    for (int j = 0; j < h; ++j) t[j] = (v & h) ? t[j + h] : t[j];
  return __shfl_sync(0xffffffffu, t[0], int(v / K));
}

template <int K>
__device__ __forceinline__ void set_entry(uint32_t (&x)[K], uint32_t v, uint32_t val) {
  const uint32_t first = (threadIdx.x & 31) * K;
#pragma unroll
  for (int j = 0; j < K; ++j) x[j] = first + j == v ? val : x[j];
}

constexpr uint32_t SENTINEL = 0xFFFFFFFFu;  // no clock entry ever takes this value
enum : uint32_t { P_ACQ = 0, P_REL = 1, P_BAR = 2, P_INCS = 3 };
enum : uint32_t { BAR_SINGLE = 0, BAR_CTA = 1, BAR_GLOBAL = 2 };

// Snapshot rows are written once by another walker. They start filled with SENTINEL;
// each 32-bit word is written exactly once, so a row with no SENTINEL word is complete.
// Rows are always read through L2 (ld.cg, cp.async.cg), never cached in L1. No flag or
// fence is involved.
template <int K>
__device__ __forceinline__ bool row_complete(const uint32_t (&y)[K]) {
  bool ok = true;
#pragma unroll
  for (int j = 0; j < K; ++j) ok &= y[j] != SENTINEL;
  return __all_sync(0xffffffffu, ok);
}

template <int K>
__device__ __forceinline__ bool rows_complete(const uint32_t (&x)[K], const uint32_t (&y)[K], const uint32_t (&z)[K]) {
  bool ok = true;
#pragma unroll
  for (int j = 0; j < K; ++j) ok &= x[j] != SENTINEL && y[j] != SENTINEL && z[j] != SENTINEL;
  return __all_sync(0xffffffffu, ok);
}

// re-read from L2 until complete (bounded: after `limit` polls the wait gives up, sets
// GWCP_ERR_TIMEOUT and the walker carries on)
template <int K>
__device__ __forceinline__ void wait_row(const uint32_t* row, uint32_t (&y)[K], bool& abort, DevStatus* st,
                                         uint32_t limit = kSpinLimit) {
  for (uint32_t it = 0;;) {
    load_row<K>(row, y);
    if (row_complete<K>(y) || abort) return;
    if (++it > limit) {
      if ((threadIdx.x & 31) == 0) atomicCAS(&st->code, 0, GWCP_ERR_TIMEOUT);
      abort = true;
      return;
    }
    if (it > 16) __nanosleep(32);
  }
}

// x |= row, y |= row for the n rows at base + ids[q] * Wp, all loads issued before any is used
template <int K, int M>
__device__ __forceinline__ void join_rows(uint32_t (&x)[K], uint32_t (&y)[K], const uint32_t* base,
                                          const uint32_t (&ids)[M], int n, bool& abort, DevStatus* st) {
  uint32_t r[M][K];
#pragma unroll
  for (int q = 0; q < M; ++q)
    if (q < n) load_row<K>(base + size_t(ids[q]) * 32 * K, r[q]);
#pragma unroll
  for (int q = 0; q < M; ++q) {
    if (q < n) {
      if (!row_complete<K>(r[q])) wait_row<K>(base + size_t(ids[q]) * 32 * K, r[q], abort, st);
#pragma unroll
      for (int j = 0; j < K; ++j) {
        x[j] = max(x[j], r[q][j]);
        y[j] = max(y[j], r[q][j]);
      }
    }
  }
}

// entry v of x for a lane-varying v: by K shuffles, or with many entries per lane through
// the warp's shared row
template <int K>
__device__ __forceinline__ uint32_t lookup_entry(const uint32_t (&x)[K], uint32_t v, uint32_t* scratch) {
  if constexpr (K <= 4) {
    uint32_t r = 0;
    const int src = int(min(v, 32u * K - 1) / K);
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const uint32_t t = __shfl_sync(0xffffffffu, x[j], src);
      if (j == int(v % K)) r = t;
    }
    return r;
  } else {
    __syncwarp();
    store_row_shared<K>(scratch, x);
    __syncwarp();
    return v < 32u * K ? scratch[v] : 0u;
  }
}

// cp.async (LDGSTS): 16-byte copy global -> shared through L2 only (no L1 line that
// could hold a row before its release wrote it)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// until at most n (< 4) of the youngest groups are in flight
__device__ __forceinline__ void cp_async_wait(uint32_t n) {
  if (n == 0)
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  else if (n == 1)
    asm volatile("cp.async.wait_group 1;" ::: "memory");
  else if (n == 2)
    asm volatile("cp.async.wait_group 2;" ::: "memory");
  else
    asm volatile("cp.async.wait_group 3;" ::: "memory");
}

template <int K>
__device__ __forceinline__ void read_row_shared(const uint32_t* row, uint32_t (&y)[K]) {
  const uint32_t* p = row + (threadIdx.x & 31) * K;
#pragma unroll
  for (int j = 0; j < K; ++j) y[j] = p[j];
}

// Shared memory by 32-bit address (the walkers' inner loop counts instructions).
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t lds(uint32_t at) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ uint4 lds4(uint32_t at) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ void red_max(uint32_t at, uint32_t v) {
  asm volatile("red.shared.max.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}
// A row of a barrier buffer: the lane's K entries at lane * K (two or fewer: one load), else
// entry j of all lanes together (no bank conflicts).
template <int K>
__device__ __forceinline__ constexpr uint32_t brow(int j) {
  return K <= 2 ? 4 * j : 128 * j;
}
template <int K>
__device__ __forceinline__ void lds_row(uint32_t at, uint32_t (&x)[K]) {
  if constexpr (K == 2) {
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(x[0]), "=r"(x[1]) : "r"(at) : "memory");
  } else {
#pragma unroll
    for (int j = 0; j < K; ++j) x[j] = lds(at + brow<K>(j));
  }
}

// plan entries per batch (64 bytes each in shared memory, two batches per warp)
template <int K>
__host__ __device__ constexpr int plan_batch() {
  return K >= 32 ? 8 : 16;
}

// One warp per agent walks the agent's plan (its clock-changing steps in trace order).
// CV: clock versions stored compressed (a separate instantiation, so that the plain
// walkers' register allocation does not carry it).
template <int K, int MAXT, bool CV>
__global__ void __launch_bounds__(MAXT, 1) k_propagate(const __grid_constant__ PropArgs a) {
  constexpr int Wc = 32 * K;
  constexpr int PB = plan_batch<K>();
  constexpr uint32_t EW = 16;  // words of a plan entry in shared memory
  extern __shared__ __align__(16) uint32_t sm[];
  const Geo& g = a.g;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const uint32_t u = a.cta_barriers ? blockIdx.x * g.apb + warp : blockIdx.x * nwarps + warp;
  uint32_t* const acc = sm;  // barrier joins: two buffers of (C, H, JN) rows (brow)
  uint32_t* const plan_s = sm + a.acc_words + size_t(warp) * a.warp_words;  // [2][PB][EW]
  uint32_t* const scratch = plan_s + 2 * PB * EW;                                // [Wc]
  uint32_t* const last_h = scratch + Wc;                                         // [2][Wc] with keep_h
  uint32_t* const slots = last_h + (a.keep_h ? 2 * Wc : 0);                      // [slots][deps][P, H, JN][Wc]
  const uint32_t slot_words = a.deps * 3 * Wc;
  // one read of the status per CTA, so all warps of a CTA agree on whether to run
  __shared__ int start_code;
  if (threadIdx.x == 0) start_code = *(volatile int*)&a.st->code;
  for (uint32_t i = threadIdx.x; i < a.acc_words; i += blockDim.x) acc[i] = 0;
  __syncthreads();
  if (start_code) return;
  if (u >= g.W) return;  // (only without CTA barriers)

  uint32_t P[K], H[K], J[K];
#pragma unroll
  for (int j = 0; j < K; ++j) P[j] = H[j] = J[j] = 0;
  // H_t = bottom{t := 1}. H_t[t] = N_t is kept in N alone and put into the row where it is
  // published (the row's own entry may lag).
  uint32_t N = 1;  // N_t
  bool abort = false;
  uint32_t joins = 0, visits = 0, nbar = 0;
  bool busy = false;     // a step other than a barrier since the block's last barrier
  bool changed = false;  // P_t, H_t or JN_t took in more than its own entry since the block's last barrier
  uint32_t last0 = NONE, last1 = NONE;  // the releases whose H rows last_h holds
  CvState cvs{0, 0, 0};  // compressed versions
  const bool cv_lanes = g.gran == GWCP_GRAN_WARP && g.apb % K == 0;
  auto put_version = [&](uint32_t r) {
    if (a.hb_only) set_entry<K>(H, u, N);
    if constexpr (CV) {
      if (cv_lanes) {
        cvs = a.hb_only ? put_row_lanes<K>(a, r, H, cvs) : put_row_lanes<K>(a, r, P, cvs);
        return;
      }
      __syncwarp();
      if (a.hb_only)
        store_row_shared<K>(scratch, H);
      else
        store_row_shared<K>(scratch, P);
      __syncwarp();
      cvs = put_row_c(a, r, scratch, cvs);
    } else if (a.hb_only) {
      store_row<K>(a.rows + size_t(r) * Wc, H);
    } else {
      store_row<K>(a.rows + size_t(r) * Wc, P);
    }
  };
  put_version(a.rowbase[u]);
  const uint32_t k0 = a.sy_start[u], k1 = a.sy_start[u + 1];
  const uint32_t pb = k0 + a.incs_off[k0], pe = k1 + a.incs_off[k1];
  uint32_t* const cursor_row = a.cursor + size_t(u) * a.n_locks;

  // Batches of PB plan entries: the current one (first step `base`, in half `half` of the
  // plan buffer) and the next, whose entries are loaded into registers when the current batch
  // begins and put into shared memory later, with the loads of its releases' cursors. This,
  // the rows of coming acquires and the records of the next release are fetched while the
  // walker waits at a barrier or after it has published a release (`ahead` below).
  constexpr int LD = PB * 4 / 32;
  uint4 nx[LD];
  auto load_entries = [&](uint32_t b0) {
#pragma unroll
    for (int q = 0; q < LD; ++q) {
      const uint32_t c = q * 32 + lane, e = b0 + c / 4;
      nx[q] = make_uint4(0, 0, 0, 0);
      if (e < pe) nx[q] = (c & 2) ? __ldcg(a.plan2 + 2 * size_t(e) + (c & 1)) : __ldcg(a.plan + 2 * size_t(e) + (c & 1));
    }
  };
  // lane l < PB: the lock and the cursor of entry l when it is a release, else NONE
  uint32_t lock_a = NONE, cur_a = 0, lock_b = NONE, cur_b = 0;
  uint32_t acq_a = 0, acq_b = 0;  // the batch's acquires (bit per entry)
  uint32_t rel_a = 0, rel_b = 0;  // releases
  uint32_t bar_a = 0, bar_b = 0;  // and block barriers
  bool put = false;               // the next batch is in shared memory
  auto put_entries = [&](uint32_t b0, uint32_t h) {
    uint4* d = reinterpret_cast<uint4*>(plan_s + h * PB * EW);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < LD; ++q) d[q * 32 + lane] = nx[q];
    __syncwarp();
    const bool mine = lane < PB && b0 + lane < pe;
    const uint32_t* e = plan_s + (h * PB + (lane & (PB - 1))) * EW;
    const uint32_t t = mine ? e[0] & 0xFF : 0xFFu;
    acq_b = __ballot_sync(0xffffffffu, t == P_ACQ);
    rel_b = __ballot_sync(0xffffffffu, t == P_REL);
    bar_b = __ballot_sync(0xffffffffu, t == P_BAR && e[4] == BAR_CTA);
    put = true;
    lock_b = NONE;
    if (t == P_REL) {
      lock_b = e[3];
      cur_b = __ldcg(cursor_row + lock_b);
    }
  };
  uint32_t base = pb, half = 0;
  if (pb < pe) {
    load_entries(pb);
    put_entries(pb, 0);
    lock_a = lock_b;
    cur_a = cur_b;
    acq_a = acq_b;
    rel_a = rel_b;
    bar_a = bar_b;
    lock_b = NONE;
    acq_b = rel_b = bar_b = 0;
    put = false;
    load_entries(pb + PB);
  }
  auto entry = [&](uint32_t i) {  // entry i of the current batch, or i - PB of the next
    return plan_s + (((i >= uint32_t(PB)) ? half ^ 1u : half) * PB + (i & (PB - 1))) * EW;
  };

  // Staged acquires, in trace order: the rows of steps q0, q1, .. (NONE: none) are in slots
  // first, first + 1, ..; the search for the next one starts at step sq.
  uint32_t q0 = NONE, q1 = NONE, q2 = NONE, q3 = NONE, staged = 0, first = 0, sq = pb;
  // Records of the next release (step rec_p), a lane each from its lock's cursor on: the agent
  // (NONE past the lock's last record), the acquire's local time (0 for an own record) and
  // the release's (0 unless the release may join it).
  uint32_t rec_ag = NONE, rec_acq = 0, rec_rel = 0;
  uint32_t rec_p = NONE;
  auto load_records = [&](uint32_t rec, uint32_t hi, uint32_t s, uint32_t my_idx) {
    uint4 m = make_uint4(NONE, 0, NONE, 0);
    if (rec < hi) m = __ldg(a.recmeta + rec);
    rec_ag = m.x == NONE ? NONE : (m.x & 0xFFFF);
    const bool mine = rec_ag == u;
    rec_acq = mine ? 0u : m.y;
    rec_rel = !mine && m.z != NONE && m.z < my_idx && scopes_overlap(m.x >> 16, s) ? m.w : 0u;
  };
  // One piece of work for later steps, at step p; false when there is none.
  auto ahead = [&](uint32_t p) -> bool {
    if (int(sq - p) <= 0) sq = p + 1;
    const uint32_t m_acq =
        staged < a.slots && sq - base < 2 * PB ? (acq_a | (acq_b << PB)) & (0xFFFFFFFFu << (sq - base)) : 0u;
    if (!m_acq) {
      // the records of the next release; then the next batch's entries. Neither is touched
      // before its loads (the batch's cursors, the entries) have had a few steps to arrive.
      const uint32_t m = (rel_a | (p - base >= 3 * PB / 4 ? rel_b << PB : 0u)) & (0xFFFFFFFEu << (p - base));
      const uint32_t i = m ? uint32_t(__ffs(m) - 1) : 0u;
      if (m && rec_p != base + i) {
        rec_p = base + i;
        const uint32_t* e = entry(i);
        const uint32_t c = __shfl_sync(0xffffffffu, i < uint32_t(PB) ? cur_a : cur_b, i & (PB - 1));
        load_records(e[4] + c + lane, e[5], e[6], e[7]);
        return true;
      }
      if (!put && p - base >= PB / 4 && base + PB < pe) {
        put_entries(base + PB, half ^ 1u);
        return true;
      }
      return false;
    }
    const uint32_t i = uint32_t(__ffs(m_acq) - 1);
    const uint32_t* e = entry(i);
    sq = base + i + 1;
    const uint32_t cnt = e[3];
    if (cnt == 0 || cnt > a.deps) return true;
    uint32_t* slot = slots + ((first + staged) & (a.slots - 1)) * slot_words;
    for (uint32_t d = 0; d < cnt; ++d) {
      const size_t at = size_t(e[4 + d]) * Wc;
      uint32_t* dst = slot + d * 3 * Wc;
#pragma unroll
      for (int c = lane; c < 3 * Wc / 4; c += 32) {
        const int r = c / (Wc / 4);
        const uint32_t* src = (r == 0 ? a.psnap : r == 1 ? a.hsnap : a.jsnap) + at;
        cp_async16(dst + 4 * c, src + 4 * (c % (Wc / 4)));
      }
    }
    cp_async_commit();
    q0 = staged == 0 ? base + i : q0;
    q1 = staged == 1 ? base + i : q1;
    q2 = staged == 2 ? base + i : q2;
    q3 = staged == 3 ? base + i : q3;
    ++staged;
    return true;
  };

  // the barrier buffer in turn (bufs: the sum of both addresses), and the agent's own entries
  // in it: lane 0 the C row's, lane 1 the H row's
  uint32_t buf = smem_addr(acc);
  const uint32_t bufs = 2 * buf + 12 * Wc;
  const uint32_t own = (lane & 1) * Wc * 4 + u / K * (K <= 2 ? 4 * K : 4) +
                       (u % K) * (K <= 2 ? 4 : 128);
  uint32_t e_at = smem_addr(plan_s);  // the entry of step p
  for (uint32_t p = pb; p < pe; ++p) {
    const uint4 ea = lds4(e_at), eb = lds4(e_at + 16);
    const uint32_t t = ea.x, z = ea.z, w = ea.w;
    if (t == P_BAR) {
      // sync (Algorithm 1): join C_t and H_t over the barrier's scope. The plan holds N_t
      // entering the join (under forced compression at barriers the highest N among the
      // members)
      const uint32_t mode = eb.x;
      N = eb.y;
      if (mode == BAR_CTA) {
        // Two buffers in turn hold the block's joined rows, which only grow: a member whose
        // rows are still the last join's adds its own entries alone.
        if (changed) {
          const uint32_t at = buf + (K <= 2 ? lane * K : lane) * 4;
#pragma unroll
          for (int j = 0; j < K; ++j) {
            red_max(at + brow<K>(j), P[j]);
            red_max(at + Wc * 4 + brow<K>(j), H[j]);
            red_max(at + Wc * 8 + brow<K>(j), J[j]);
          }
        }
        // (no other member holds a larger value, but other members' reductions of this word may
        // be under way, so it is a reduction as well: a plain store could be lost to one)
        if (lane < 2) red_max(buf + own, N);
        // a member with no other step since the last barrier is early: it works ahead
        if (!busy) ahead(p);
        changed = busy = false;
        __syncthreads();
        {
          const uint32_t at = buf + (K <= 2 ? lane * K : lane) * 4;
          lds_row<K>(at, P);
          lds_row<K>(at + Wc * 4, H);
          lds_row<K>(at + Wc * 8, J);
        }
        // the other buffer, which every member has read after the barrier before, takes this
        // join in (members that are ahead may already add to it)
        const uint32_t other = bufs - buf;
        for (uint32_t q = threadIdx.x * 4; q < 12 * Wc; q += blockDim.x * 4) {
          const uint32_t v = lds(buf + q);
          if (v > lds(other + q)) red_max(other + q, v);
        }
        buf = other;
        ++nbar;
      } else {
        set_entry<K>(P, u, N);  // C_t
        if (mode == BAR_GLOBAL) {
          const uint32_t bid = z, count = w;
          uint32_t* JP = a.bar_j + size_t(bid) * 2 * Wc;
          uint32_t* JJ = a.bar_jj + size_t(bid) * Wc;
          set_entry<K>(H, u, N);
#pragma unroll
          for (int j = 0; j < K; ++j) {
            atomicMax(JP + lane * K + j, P[j]);
            atomicMax(JP + Wc + lane * K + j, H[j]);
            atomicMax(JJ + lane * K + j, J[j]);
          }
          __threadfence();
          __syncwarp();
          if (lane == 0) atomicAdd(a.bar_cnt + bid, 1u);
          if (!abort) {
            bool ok = true;
            if (lane == 0) {
              uint32_t it = 0;
              while (ld_acquire(a.bar_cnt + bid) < count) {
                if (++it > kSpinLimit) {
                  ok = false;
                  break;
                }
                if (it > 16) __nanosleep(64);
              }
              if (!ok) atomicCAS(&a.st->code, 0, GWCP_ERR_TIMEOUT);
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            __syncwarp();
            if (!ok) abort = true;
          }
          load_row<K>(JP, P);
          load_row<K>(JP + Wc, H);
          load_row<K>(JJ, J);
          changed = true;
          joins += 2;
        }
      }
      ++N;
    } else if (t == P_INCS) {
      busy = true;
      // in-section access (Algorithm 2): P_t |= L^w (| L^r), each the H snapshot of an earlier
      // section's release, unless JN_t already covers it
      for (uint32_t q = 0; q < w; ++q) {
        uint32_t x, ag, ep;
        if (w <= 4) {
          x = q == 0 ? eb.x : q == 1 ? eb.y : q == 2 ? eb.z : eb.w;
          ag = lds(e_at + 32 + 8 * q);
          ep = lds(e_at + 36 + 8 * q);
        } else {
          x = __ldcg(a.flat + z + q);
          const uint4 mx = __ldg(a.recmeta + x);
          ag = mx.x & 0xFFFF;
          ep = mx.w;
        }
        if (get_entry<K>(J, ag) >= ep) continue;
        uint32_t y[K];
        if (x == last0 || x == last1)
          read_row_shared<K>(last_h + (x == last0 ? 0 : Wc), y);
        else
          wait_row<K>(a.hsnap + size_t(x) * Wc, y, abort, a.st);
#pragma unroll
        for (int j = 0; j < K; ++j) {
          P[j] = max(P[j], y[j]);
          J[j] = max(J[j], y[j]);
        }
        changed = true;
        ++joins;
      }
    } else if (t == P_ACQ) {
      busy = true;
      // acquire (Algorithm 1): P_t |= P_<l,s'>, H_t |= H_<l,s'> over the overlapping
      // scopes' latest releases
      const bool here = q0 == p;  // its rows are in slot `first`
      const uint32_t* slot = slots + (first & (a.slots - 1)) * slot_words;
      if (here) {
        --staged;
        cp_async_wait(staged);
        ++first;
        q0 = q1;
        q1 = q2;
        q2 = q3;
        q3 = NONE;
        __syncwarp();  // every lane's copies
      }
      for (uint32_t q = 0; q < w; ++q) {
        const uint32_t x = w > 4 ? __ldcg(a.pool + z + q) : q == 0 ? eb.x : q == 1 ? eb.y : q == 2 ? eb.z : eb.w;
        const size_t at = size_t(x) * Wc;
        if constexpr (K <= 8) {
          uint32_t yp[K], yh[K], yj[K];
          bool ok = false;
          if (here) {
            const uint32_t* rows = slot + q * 3 * Wc;
            read_row_shared<K>(rows, yp);
            read_row_shared<K>(rows + Wc, yh);
            read_row_shared<K>(rows + 2 * Wc, yj);
            ok = rows_complete<K>(yp, yh, yj);
          }
          for (uint32_t it = 0; !ok; ++it) {  // the three rows polled together
            load_row<K>(a.psnap + at, yp);
            load_row<K>(a.hsnap + at, yh);
            load_row<K>(a.jsnap + at, yj);
            ok = rows_complete<K>(yp, yh, yj);
            if (ok || abort) break;
            if (it >= kSpinLimit) {
              if (lane == 0) atomicCAS(&a.st->code, 0, GWCP_ERR_TIMEOUT);
              abort = true;
              break;
            }
            if (it > 16) __nanosleep(32);
          }
#pragma unroll
          for (int j = 0; j < K; ++j) {
            P[j] = max(P[j], yp[j]);
            H[j] = max(H[j], yh[j]);
            J[j] = max(J[j], yj[j]);
          }
          if (a.keep_h && q < 2) store_row_shared<K>(last_h + q * Wc, yh);
        } else {
          uint32_t y[K];
          wait_row<K>(a.psnap + at, y, abort, a.st);
#pragma unroll
          for (int j = 0; j < K; ++j) P[j] = max(P[j], y[j]);
          wait_row<K>(a.jsnap + at, y, abort, a.st);
#pragma unroll
          for (int j = 0; j < K; ++j) J[j] = max(J[j], y[j]);
          wait_row<K>(a.hsnap + at, y, abort, a.st);
#pragma unroll
          for (int j = 0; j < K; ++j) H[j] = max(H[j], y[j]);
          if (a.keep_h && q < 2) store_row_shared<K>(last_h + q * Wc, y);
        }
      }
      joins += 2 * w;
      changed |= w != 0;
      last0 = w > 0 && w <= 4 && a.keep_h ? eb.x : NONE;
      last1 = w > 1 && w <= 4 && a.keep_h ? eb.y : NONE;
    } else {
      // release (Algorithm 1): pop other agents' records on this lock while their
      // acquire is ordered before C_t; join the released ones whose scope overlaps.
      // Waves: every record before the first one failing the test against the current
      // P passes (P only grows), so their snapshots are joined together; the failing
      // record is tested again only if the wave changed P.
      busy = true;
      const uint32_t i = p - base, c = z, L = w;
      const uint32_t lo = eb.x, hi = eb.y;
      uint32_t cur = __shfl_sync(0xffffffffu, cur_a, i);
      bool fetched = rec_p == p;
      while (lo + cur < hi) {
        if (!fetched) load_records(lo + cur + lane, hi, eb.z, eb.w);
        fetched = false;
        const uint32_t nbr = min(32u, hi - (lo + cur));
        const uint32_t others = __ballot_sync(0xffffffffu, rec_ag != u);  // (lanes past the last record too)
        uint32_t start = 0;
        bool stop = false;
        for (;;) {
          const uint32_t pv = lookup_entry<K>(P, rec_ag, scratch);
          const uint32_t jv = lookup_entry<K>(J, rec_ag, scratch);
          const uint32_t from = 0xFFFFFFFFu << start;  // start < 32
          const uint32_t fail = __ballot_sync(0xffffffffu, rec_acq > pv) & from;
          const uint32_t f = fail ? uint32_t(__ffs(fail) - 1) : nbr;  // first failing record
          const uint32_t below = f < 32 ? (1u << f) - 1u : 0xFFFFFFFFu;
          visits += __popc(others & from & (fail ? below | (1u << f) : below));
          // of the popped releases, join only those not dominated, and per agent only
          // the latest (records of one agent are in acquire order)
          uint32_t wave = __ballot_sync(0xffffffffu, rec_rel > jv) & from & below;
          if (wave) {
            changed = true;
            if (wave & (wave - 1)) {
              const bool cand = (wave >> lane) & 1u;
              const uint32_t same = __match_any_sync(0xffffffffu, cand ? rec_ag : 0xFFFFFFFFu);
              wave = __ballot_sync(0xffffffffu, cand && (same >> lane) <= 1u);
            }
            constexpr int M = K <= 4 ? 4 : K <= 8 ? 2 : 1;
            for (uint32_t wm = wave; wm;) {
              uint32_t ids[M];
              int n = 0;
#pragma unroll
              for (int q = 0; q < M; ++q) {
                ids[q] = 0;
                if (wm) {
                  ids[q] = lo + cur + (__ffs(wm) - 1);
                  wm &= wm - 1;
                  ++n;
                }
              }
              join_rows<K, M>(P, J, a.hsnap, ids, n, abort, a.st);
              joins += n;
            }
          }
          start = f;
          if (!fail) break;
          if (!wave) {
            stop = true;  // P unchanged: the record stays unordered
            break;
          }
          // P grew: test the failing record again
        }
        cur += start;
        if (stop) break;
      }
      set_entry<K>(H, u, N);  // H_t[t] = N_t
      const size_t at = size_t(c) * Wc;
      store_row<K>(a.psnap + at, P);
      store_row<K>(a.hsnap + at, H);
      store_row<K>(a.jsnap + at, J);
      if (lane == 0) __stcg(cursor_row + L, cur);
      // later releases of L, in this batch and the next, start from the new cursor
      if (lane > int(i) && lock_a == L) cur_a = cur;
      if (lock_b == L) cur_b = cur;
      ++N;  // H_t[t]++
      // a barrier later in the batch has time for the work ahead; otherwise a piece is done here
      if (!(bar_a >> i)) ahead(p);
    }
    put_version(ea.y);
    e_at += EW * 4;
    if (p + 1 - base == PB) {  // next batch
      if (!put) put_entries(base + PB, half ^ 1u);
      base += PB;
      half ^= 1u;
      e_at = smem_addr(plan_s) + half * PB * EW * 4;
      lock_a = lock_b;
      cur_a = cur_b;
      acq_a = acq_b;
      rel_a = rel_b;
      bar_a = bar_b;
      lock_b = NONE;
      acq_b = rel_b = bar_b = 0;
      put = false;
      load_entries(base + PB);
    }
  }
  joins += 2 * nbar;  // at a block barrier each member's C_t and H_t enter the block's
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (lane == 0) {
    atomicAdd(&a.st->joins, (unsigned long long)joins);
    atomicAdd(&a.st->loop_visits, (unsigned long long)visits);
    if constexpr (CV) atomicAdd(a.cv_words, cvs.words);
  }
}

// ---- plan construction -------------------------------------------------------------


// Per section, its record as the release loop reads it: (agent | scope id << 16, acquire
// epoch, release index, release epoch). Per in-section access, the number of releases it
// joins, over the sections that it is held in.
__global__ void k_plan_counts(PropArgs a, uint32_t n_cs, const uint32_t* cs_epoch, const uint32_t* cs_rel_epoch,
                              uint32_t n_incs, uint32_t* cnt) {
  grid_begin();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_cs) a.recmeta[i] = make_uint4(a.cs_agent[i] | (a.cs_sid[i] << 16), cs_epoch[i], a.cs_rel_idx[i], cs_rel_epoch[i]);
  if (i >= n_incs) return;
  uint32_t t = 0;
  if (!a.st->code)  // (after an error the lists are incomplete)
    for (uint32_t c = a.cs_of_sync[a.sy_inner[a.incs_k[i]]]; c != NONE; c = a.cs_parent[c])
      t += a.ex_dep_cnt[a.cs_exp[c] + (i - a.cs_r0[c])];
  cnt[i] = t;
}

// the entry of synchronisation entry k
__device__ __forceinline__ void plan_sync(const PropArgs& a, const uint32_t* sy_kind_, const uint32_t* sy_ver, uint32_t k) {
  const Geo& g = a.g;
  const uint32_t u = a.sy_agent[k];
  const uint32_t row = a.rowbase[u] + sy_ver[k];
  const uint32_t kind = sy_kind_[k];
  uint4 ea, eb = make_uint4(0, 0, 0, 0);
  if (kind == K_ACQ) {
    const uint32_t c = a.cs_of_sync[k];
    const uint32_t off = a.acq_dep_off[c], cnt = a.acq_dep_cnt[c];
    ea = make_uint4(P_ACQ, row, off, cnt);
    if (cnt <= 4)  // up to four dependency ids ride in the entry itself
      eb = make_uint4(cnt > 0 ? a.pool[off] : 0, cnt > 1 ? a.pool[off + 1] : 0, cnt > 2 ? a.pool[off + 2] : 0,
                      cnt > 3 ? a.pool[off + 3] : 0);
  } else if (kind == K_REL) {
    const uint32_t c = a.cs_of_sync[k];
    const uint32_t L = a.cs_lock[c];
    ea = make_uint4(P_REL, row, c, L);
    eb = make_uint4(a.lock_cs_lo[L], a.lock_cs_lo[L + 1], a.cs_sid[c], a.sy_idx[k]);
  } else {
    const Event e = a.ev[a.sy_idx[k]];
    const BarMembers bm = barrier_members(e, g);
    const uint32_t mode = bm.count == 1 ? BAR_SINGLE
                          : (a.cta_barriers && e.scope == GWCP_SCOPE_CTA) ? BAR_CTA
                                                                          : BAR_GLOBAL;
    ea = make_uint4(P_BAR, row, a.sy_aux[k], bm.count);
    eb.x = mode;
    eb.y = a.sy_N[k] - 1;  // N_t entering the join (after the barrier, N_t = eb.y + 1)
  }
  const size_t p = size_t(k) + a.incs_off[k];
  a.plan[2 * p] = ea;
  a.plan[2 * p + 1] = eb;
}

// The plan's entries: per synchronisation entry, and per in-section access with its flattened
// list (its sections from the inside out).
__global__ void k_plan(const __grid_constant__ PropArgs a, const uint32_t* sy_kind_, const uint32_t* sy_ver, uint32_t n_sync,
                       const uint32_t* flat_off, uint32_t* flat, uint32_t n_incs) {
  grid_begin();
  const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
  if (a.st->code) return;  // (the lists are incomplete, the walkers stand down)
  if (r < n_sync) plan_sync(a, sy_kind_, sy_ver, r);
  if (r >= n_incs) return;
  const uint32_t k = a.incs_k[r];
  const uint32_t u = a.sy_agent[k];
  const size_t p = size_t(k) + 1 + r;
  const uint32_t off = flat_off[r], cnt = flat_off[r + 1] - off;
  uint32_t o = off;
  if (cnt)
    for (uint32_t c = a.cs_of_sync[a.sy_inner[k]]; c != NONE; c = a.cs_parent[c]) {
      const uint32_t e = a.cs_exp[c] + (r - a.cs_r0[c]);
      const uint32_t* list = a.pool + a.ex_dep_off[e];
      for (uint32_t q = 0; q < a.ex_dep_cnt[e]; ++q) flat[o++] = list[q];
    }
  a.plan[2 * p] = make_uint4(P_INCS, a.rowbase[u] + a.incs_ver[r], off, cnt);
  uint32_t id[4] = {0, 0, 0, 0}, meta[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  if (cnt <= 4) {
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
      if (q >= cnt) break;
      id[q] = flat[off + q];
      const uint4 m = a.recmeta[id[q]];
      meta[2 * q] = m.x & 0xFFFF;  // the releasing agent and its local time at the release
      meta[2 * q + 1] = m.w;
    }
  }
  a.plan[2 * p + 1] = make_uint4(id[0], id[1], id[2], id[3]);
  a.plan2[2 * p] = make_uint4(meta[0], meta[1], meta[2], meta[3]);
  a.plan2[2 * p + 1] = make_uint4(meta[4], meta[5], meta[6], meta[7]);
}

// Launches the walkers with the most staging that fits a CTA's shared memory and keeps all
// CTAs co-resident.
template <int K, int MAXT, bool CV>
int launch(const PropArgs& args, uint32_t grid, uint32_t threads, cudaStream_t s) {
  auto kern = k_propagate<K, MAXT, CV>;
  constexpr uint32_t Wc = 32 * K;
  const uint32_t warps = threads / 32;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // (one limit for every launch: other threads may be launching with another size)
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kMaxDynamicSmem)) != cudaSuccess)
    return GWCP_ERR_CUDA;
  // (slots, releases per staged acquire, keep the acquired H rows)
  constexpr uint32_t kShapes[6][3] = {{4, 2, 1}, {2, 2, 1}, {2, 1, 1}, {1, 1, 1}, {0, 0, 1}, {0, 0, 0}};
  for (const auto& sh : kShapes) {
    if (sh[0] && K > 8) continue;  // three rows at a time do not fit the registers
    PropArgs a = args;
    a.slots = sh[0];
    a.deps = sh[1];
    a.keep_h = sh[2];
    a.acc_words = a.cta_barriers && a.g.apb > 1 ? 6 * Wc : 0;
    a.warp_words = 2 * plan_batch<K>() * 16 + Wc + (a.keep_h ? 2 * Wc : 0) + a.slots * a.deps * 3 * Wc;
    const size_t smem = (size_t(a.acc_words) + size_t(warps) * a.warp_words) * 4;
    if (smem > kMaxDynamicSmem) continue;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, int(threads), smem) != cudaSuccess)
      return GWCP_ERR_CUDA;
    if (uint64_t(per_sm) * sms < grid) continue;  // walkers must be co-resident
    void* kargs[] = {&a};
    if (cudaLaunchCooperativeKernel(reinterpret_cast<void*>(kern), dim3(grid), dim3(threads), kargs, smem, s) !=
        cudaSuccess)
      return GWCP_ERR_CUDA;
    count_launch();
    return GWCP_OK;
  }
  return GWCP_ERR_UNSUPPORTED;
}

// CTAs of up to eight and sixteen walkers have the registers of 256 and 512 threads
template <int K>
int launch_k(const PropArgs& a, uint32_t grid, uint32_t threads, cudaStream_t s) {
  if (threads <= 256)
    return a.compress ? launch<K, 256, true>(a, grid, threads, s) : launch<K, 256, false>(a, grid, threads, s);
  if (threads <= 512)
    return a.compress ? launch<K, 512, true>(a, grid, threads, s) : launch<K, 512, false>(a, grid, threads, s);
  return a.compress ? launch<K, 1024, true>(a, grid, threads, s) : launch<K, 1024, false>(a, grid, threads, s);
}

// failure-detection test: one warp waits, with the walkers' bounded wait, on a clock row
// that nothing completes
__global__ void k_wait_probe(const uint32_t* row, DevStatus* st, uint32_t limit) {
  uint32_t y[1];
  bool abort = false;
  wait_row<1>(row, y, abort, st, limit);
}

}  // namespace

int wait_probe(uint32_t limit, int* code) {
  // a 32-word row of SENTINEL words (never completed) and a status record
  void* mem = nullptr;
  if (cudaMalloc(&mem, 256 + sizeof(DevStatus)) != cudaSuccess) {
    cudaGetLastError();
    return GWCP_ERR_OOM;
  }
  auto* row = static_cast<uint32_t*>(mem);
  auto* st = reinterpret_cast<DevStatus*>(static_cast<char*>(mem) + 256);
  cudaMemset(row, 0xFF, 256);
  cudaMemset(st, 0, sizeof(DevStatus));
  k_wait_probe<<<1, 32>>>(row, st, limit);
  count_launch();
  int rc = cudaDeviceSynchronize() == cudaSuccess ? GWCP_OK : GWCP_ERR_CUDA;
  if (!rc && cudaMemcpy(code, &st->code, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) rc = GWCP_ERR_CUDA;
  cudaFree(mem);
  return rc;
}

int phaseG_propagate(const Bufs& b, const Geo& g, const Sizes& z, cudaStream_t s, Prof& p) {
  PropArgs a{};
  a.g = g;
  a.ev = b.ev;
  a.st = b.st;
  a.sy_start = b.sy_start;
  a.sy_idx = b.sy_idx;
  a.sy_kind = b.sy_kind;
  a.sy_N = b.sy_N;
  a.sy_ver = b.sy_ver;
  a.sy_aux = b.sy_aux;
  a.sy_agent = b.sy_agent;
  a.incs_off = b.incs_cnt;
  a.incs_ver = b.incs_ver;
  a.incs_k = b.incs_k;
  a.sy_inner = b.sy_inner;
  a.cs_parent = b.cs_parent;
  a.cs_exp = b.cs_exp;
  a.cs_r0 = b.cs_r0;
  a.ex_dep_off = b.ex_dep_off;
  a.ex_dep_cnt = b.ex_dep_cnt;
  a.rowbase = b.vcount;
  a.cs_of_sync = b.cs_of_sync;
  a.cs_agent = b.cs_agent;
  a.cs_sid = b.cs_sid;
  a.cs_epoch = b.cs_epoch;
  a.cs_rel_idx = b.cs_rel_idx;
  a.cs_lock = b.cs_lock;
  a.cs_rel_epoch = b.cs_rel_epoch;
  a.lock_cs_lo = b.lock_cs_lo;
  a.acq_dep_off = b.acq_dep_off;
  a.acq_dep_cnt = b.acq_dep_cnt;
  a.pool = b.dep_pool;
  a.rows = b.rows;
  a.psnap = b.psnap;
  a.hsnap = b.hsnap;
  a.jsnap = b.jsnap;
  a.cursor = b.cursor;
  a.bar_j = b.bar_j;
  a.bar_jj = b.bar_jj;
  a.bar_cnt = b.bar_cnt;
  a.n_locks = z.n_locks;
  a.cta_barriers = z.cta_barriers;
  a.flat = b.flat;
  a.plan = b.plan;
  a.plan2 = b.plan2;
  a.recmeta = b.recmeta;
  a.hb_only = z.hb_only;
  a.forced = z.forced_barrier;
  a.compress = z.compress;
  a.cv_pool = b.cv_pool;
  a.cv_cap = z.cv_cap;
  a.cv_used = reinterpret_cast<unsigned long long*>(&b.st->spare[3]);
  a.cv_words = reinterpret_cast<unsigned long long*>(&b.st->spare[4]);
  // plan: per-agent stream of clock-changing steps with their static data resolved
  p.begin("g_plan", double(z.n_sync + z.n_incs) * 64 + double(z.n_cs) * 2 * g.RW * 4);
  if (z.n_cs) {
    const uint32_t most = std::max(z.n_cs, z.n_incs);
    launch(k_plan_counts, (most + 255) / 256, 256, 0, s)(a, z.n_cs, b.cs_epoch, b.cs_rel_epoch, z.n_incs, b.flat_off);
    count_launch();
  }
  FillBatch f;
  // snapshot rows start as SENTINEL: a reader accepts a row once none is left
  for (uint32_t* snap : {b.psnap, b.hsnap, b.jsnap}) f.add(snap, size_t(z.n_cs) * g.RW, 0xFFFFFFFFu);
  f.add(b.cursor, size_t(g.W) * (z.n_locks + 1), 0);
  if ((!z.cta_barriers || g.gran == GWCP_GRAN_THREAD) && z.n_bar) {  // barriers joined in global memory
    f.add(b.bar_j, size_t(z.n_bar) * 2 * g.Wp, 0);
    f.add(b.bar_jj, size_t(z.n_bar) * g.Wp, 0);
    f.add(b.bar_cnt, z.n_bar, 0);
  }
  if (g.nT) f.add(b.tiles, kTileW, 0);  // tile 0 is the zero tile; ids are handed out from 1
  fill_all(f, s);
  if (z.n_incs) {
    scan_exclusive(b.flat_off, b.flat_off, size_t(z.n_incs) + 1, nullptr, b.scan_tmp, s);
  }
  if (z.n_sync) {  // (no in-section access without a synchronisation entry)
    const uint32_t most = std::max(z.n_sync, z.n_incs);
    launch(k_plan, (most + 255) / 256, 256, 0, s)(a, b.sy_kind, b.sy_ver, z.n_sync, b.flat_off, b.flat, z.n_incs);
    count_launch();
  }
  p.end();
  if (z.before_walk) cudaEventRecord(z.before_walk, s);
  if (g.nT) {
    // tile tables: each clock version and snapshot is a table (new tiles counted apart)
    p.begin("g_propagate", double(z.n_rows) * g.RW * 4 + double(z.n_cs) * 2 * g.RW * 4);
    const int rc = phaseG_wide(b, g, z, s);
    p.end();
    return rc;
  }
  // a CTA per block of the traced program; without CTA barriers the walkers are spread eight
  // to a CTA over the SMs
  const uint32_t threads = z.cta_barriers ? g.apb * 32 : 256;
  const uint32_t grid = z.cta_barriers ? g.B : (g.W + 7) / 8;
  // algorithmic bytes: each clock version written once, each join reads a row
  p.begin("g_propagate", double(z.n_rows) * g.Wp * 4 + double(z.n_cs) * 2 * g.Wp * 4);
  int rc;
  switch (g.K) {
    case 1: rc = launch_k<1>(a, grid, threads, s); break;
    case 2: rc = launch_k<2>(a, grid, threads, s); break;
    case 4: rc = launch_k<4>(a, grid, threads, s); break;
    case 8: rc = launch_k<8>(a, grid, threads, s); break;
    case 16: rc = launch_k<16>(a, grid, threads, s); break;
    case 32: rc = launch_k<32>(a, grid, threads, s); break;
    default: rc = GWCP_ERR_UNSUPPORTED;
  }
  p.end();
  return rc;
}

}  // namespace gwcp
