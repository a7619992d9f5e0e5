// Wide clocks (many agents, up to 8192): clock propagation and race check over
// copy-on-write clock tiles.
//
// A clock of width W is cut into nT = ceil(W / 256) tiles of 256 u32 entries. Tiles live
// in one pool and are immutable once written; a clock is a table of nT tile ids (id 0 is
// the all-zero tile). A warp walks one agent as in the register-resident walker, but
// lane T holds the ids of tile T of P_t and H_t instead of the entries themselves. A join
// P_t |= X (Algorithms 1-2) compares ids tile by tile: an equal or zero tile costs
// nothing, a differing one is merged by the whole warp (8 entries per lane) and the
// result keeps an input's id when it equals that input, else it is written as a new
// tile. Clocks shared after a barrier or an acquire therefore share their tiles, and a
// clock version (the row the check reads) is a 128-byte table. A release snapshot is
// two tables. H_t[t] = N_t is kept implicit: the walker holds N_t in a register and the
// table's own entry may lag, so an increment copies no tile; the release snapshot of H_t
// writes the entry out (one tile copy), and a barrier raises every member's own entry to
// its local time while it joins the members' tables, as it does for C_t.
//
// Publication: a writer fences after writing new tiles and before storing a table that
// refers to them; tables are written once over SENTINEL words, so a reader accepts a
// table once none of its nT words is SENTINEL. All waits are bounded (GWCP_ERR_TIMEOUT).
// Pool exhaustion sets GWCP_ERR_OOM; the walker then keeps its old tile (the host grows
// the pool and runs the analysis again).
//
// The partner check enumerates partners per access instead of holding a W-wide table:
// accesses sorted by location are re-sorted stably by (location, class, agent);
// for access b every (class, agent) group of its location whose class conflicts with b
// is searched for its latest access before b, and an agent is tested once, against its
// latest conflicting non-exempt access a*: race iff N(a*) > C_b[v] (the paper's check).
#include <algorithm>

#include "gwcp_internal.cuh"
#include "gwcp_post.cuh"

namespace gwcp {

namespace {

constexpr uint32_t kSpinLimitW = 1u << 23;
constexpr uint32_t kPlanBatch = 16;
constexpr unsigned long long kBarrierLimitNs = 60ull * 1000 * 1000 * 1000;
constexpr uint32_t SENT = 0xFFFFFFFFu;
enum : uint32_t { P_ACQ = 0, P_REL = 1, P_BAR = 2, P_INCS = 3 };
enum : uint32_t { BAR_SINGLE = 0, BAR_CTA = 1, BAR_GLOBAL = 2 };

struct WideArgs {
  Geo g;
  DevStatus* st;
  const uint32_t *sy_start, *incs_off, *rowbase;
  const uint4* plan;
  const uint4* recmeta;
  const uint32_t *pool, *flat;
  uint32_t *rows, *psnap, *hsnap, *jsnap, *cursor;
  uint32_t* tiles;
  unsigned long long* tile_ctr;
  unsigned long long tile_cap;
  uint32_t n_locks;
  uint32_t hb_only;  // publish H_t instead of P_t as the clock versions
};

__device__ __forceinline__ uint4 max4(uint4 x, uint4 y) {
  return make_uint4(max(x.x, y.x), max(x.y, y.y), max(x.z, y.z), max(x.w, y.w));
}
__device__ __forceinline__ bool eq4(uint4 x, uint4 y) { return x.x == y.x && x.y == y.y && x.z == y.z && x.w == y.w; }

// Tiles are immutable once written and a tile id becomes known to a walker only through a
// table published after the tile (or through its own CTA after a barrier), so no L1 line
// can hold a tile's address before the tile is written (L1 starts clean each launch):
// tile reads may go through L1, and a merge first prefetches every tile it will read.
__device__ __forceinline__ void prefetch_tile(const WideArgs& a, uint32_t id) {
  const char* p = reinterpret_cast<const char*>(a.tiles + size_t(id) * kTileW);
#pragma unroll
  for (int q = 0; q < 8; ++q) asm volatile("prefetch.global.L1 [%0];" ::"l"(p + q * 128));
}
__device__ __forceinline__ const uint4* tile_src(const WideArgs& a, uint32_t id) {
  return reinterpret_cast<const uint4*>(a.tiles + size_t(id) * kTileW) + (threadIdx.x & 31) * 2;
}
__device__ __forceinline__ uint4* tile_dst(const WideArgs& a, uint32_t id) {
  return reinterpret_cast<uint4*>(a.tiles + size_t(id) * kTileW) + (threadIdx.x & 31) * 2;
}

// A lane holds 8 consecutive entries of a tile as (x0, x1). These update entry c (0..7)
// with register selects only, so the pair is never addressed through memory.
__device__ __forceinline__ void set8(uint4& x0, uint4& x1, uint32_t c, uint32_t val) {
  x0.x = c == 0 ? val : x0.x;
  x0.y = c == 1 ? val : x0.y;
  x0.z = c == 2 ? val : x0.z;
  x0.w = c == 3 ? val : x0.w;
  x1.x = c == 4 ? val : x1.x;
  x1.y = c == 5 ? val : x1.y;
  x1.z = c == 6 ? val : x1.z;
  x1.w = c == 7 ? val : x1.w;
}

// Tile ids are handed to each warp kTileChunk at a time (one atomic per chunk instead of
// one per tile on a single counter); the warp-uniform state lives in the walker. The next
// chunk is asked for when the current one is begun, so that its atomic's latency is over
// when it is needed.
constexpr uint32_t kTileChunk = 4;
struct TileAlloc {
  uint32_t next = 0, end = 0;  // ids [next, end) are the warp's; both clamped to the pool size
  unsigned long long ahead = 0;  // lane 0: the next chunk's first id
  uint32_t* cnt = nullptr;     // shared words: tiles read, tiles written (lane 0 adds)
  __device__ __forceinline__ void count(uint32_t rd, uint32_t wr) const {
    if ((threadIdx.x & 31) == 0) {
      cnt[0] += rd;
      cnt[1] += wr;
    }
  }
};
__device__ __forceinline__ void ask_chunk(const WideArgs& a, TileAlloc& ta) {
  if ((threadIdx.x & 31) == 0) ta.ahead = atomicAdd(a.tile_ctr, (unsigned long long)kTileChunk);
}

// a fresh tile id (warp-uniform); 0 when the pool is exhausted (GWCP_ERR_OOM set)
__device__ __forceinline__ uint32_t alloc_tile(const WideArgs& a, TileAlloc& ta) {
  if (ta.next == ta.end) {
    const unsigned long long base = __shfl_sync(0xffffffffu, ta.ahead, 0);
    ask_chunk(a, ta);
    ta.next = uint32_t(min(base, a.tile_cap));
    ta.end = uint32_t(min(base + kTileChunk, a.tile_cap));
    if (ta.next == ta.end) {
      if ((threadIdx.x & 31) == 0) atomicCAS(&a.st->code, 0, GWCP_ERR_OOM);
      return 0;
    }
  }
  return ta.next++;
}

// max of tiles ia and ib by the whole warp: an input's id when the result equals it, else that
// of a new tile (ia when the pool is exhausted)
__device__ __forceinline__ uint32_t merge_one(const WideArgs& a, uint32_t ia, uint32_t ib, bool& fresh,
                                              TileAlloc& ta) {
  const uint4* pa = tile_src(a, ia);
  const uint4* pb = tile_src(a, ib);
  const uint4 x0 = __ldca(pa), x1 = __ldca(pa + 1), y0 = __ldca(pb), y1 = __ldca(pb + 1);
  const uint4 r0 = max4(x0, y0), r1 = max4(x1, y1);
  fresh = false;
  if (__all_sync(0xffffffffu, eq4(r0, x0) && eq4(r1, x1))) return ia;
  if (__all_sync(0xffffffffu, eq4(r0, y0) && eq4(r1, y1))) return ib;
  const uint32_t nid = alloc_tile(a, ta);
  if (!nid) return ia;
  uint4* d = tile_dst(a, nid);
  d[0] = r0;
  d[1] = r1;
  fresh = true;
  return nid;
}

// A merge of whole tables is up to 32 merges of tiles per table, each a chain of loads, votes,
// an id and stores: 1,400 cycles, and 65 us for the three tables of an acquire with 8192 warps
// when one warp walks them, while the other walkers of its CTA mostly wait at the block's
// barrier. So a walker posts its merges in shared memory, and walkers that wait (at a barrier,
// or for a release) take them one by one, as does the walker itself. Propagation, with the
// plan ring and the members' own entries raised from shared memory (the barrier join 35,000
// -> 17,000 cycles): 8192 warps, 50M events 16.7 -> 9.5 ms; 4096 warps, 4M 4.2 -> 1.86; 512
// warps, 2.3M 2.2 -> 1.3. (The pairs of eight merges copied to shared memory ahead of the
// one walker: 13.5 and 3.0 ms; four tiles per warp at a time: slower than one.)
// A post is reused only after all its merges are done, and opened by the store to `word`
// after everything else is written. A walker that draws a merge thereby knows that the post
// stays as it is until the merge is done; one that comes late draws nothing, or a merge of the
// new post together with that post's own limit.
struct Post {
  uint32_t word, done, pad[2];  // merges and merges handed out (gwcp_post.cuh); merges done
  uint32_t ida[96], idb[96];    // the merges: my tile (then the result), the source's
};
constexpr uint32_t kPosts = 4;  // per CTA; a walker that finds none free walks its merges alone

struct __align__(16) Shared {  // a CTA's posts
  uint32_t open;     // posts with merges left (bit each)
  uint32_t arrived;  // walkers that have reached a block barrier, all barriers together
  uint32_t used;     // posts taken (bit each)
  uint32_t pad;
  Post post[kPosts];
};

// takes one merge of post b, if one is left
__device__ __forceinline__ bool take_merge(const WideArgs& a, Shared& sh, int b, TileAlloc& ta) {
  const int lane = threadIdx.x & 31;
  Post& q = sh.post[b];
  uint32_t w = kPostClosed;
  if (lane == 0) {
    w = *(volatile uint32_t*)&q.word;
    if (post_left(w)) w = atomicAdd(&q.word, 1u);
    __threadfence_block();
  }
  w = __shfl_sync(0xffffffffu, w, 0);
  __syncwarp();
  if (!post_left(w)) return false;
  const uint32_t j = post_merge(w);
  if (j + 1 == post_merges(w) && lane == 0) atomicAnd(&sh.open, ~(1u << b));
  bool fresh;
  const uint32_t id = merge_one(a, *(volatile uint32_t*)&q.ida[j], *(volatile uint32_t*)&q.idb[j], fresh, ta);
  ta.count(2, fresh ? 1u : 0u);
  // (the tile is ordered before `done`, and the poster fences before it publishes a table)
  __syncwarp();
  if (lane == 0) {
    *(volatile uint32_t*)&q.ida[j] = id;
    __threadfence_block();
    atomicAdd(&q.done, 1u);
  }
  return true;
}

// (posts with merges left, arrivals at block barriers): one load, the same for all lanes. The
// waiting walkers poll it, up to 62 on an SM beside the ones that work, so a poll is few
// instructions and polls are kWaitNs apart.
constexpr uint32_t kWaitNs = 300;
__device__ __forceinline__ uint2 look(const Shared& sh) {
  uint2 v;
  asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];"
               : "=r"(v.x), "=r"(v.y)
               : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(&sh.open)))
               : "memory");
  return make_uint2(__shfl_sync(0xffffffffu, v.x, 0), __shfl_sync(0xffffffffu, v.y, 0));
}
__device__ __noinline__ void help(const WideArgs& a, Shared& sh, uint32_t open, TileAlloc& ta) {
  take_merge(a, sh, __ffs(open) - 1, ta);
}

// my[q] |= src[q] tile by tile for the tables q < NT (lane T < nT holds the ids of tile T)
template <int NT>
__device__ __noinline__ void merge_tables(const WideArgs& a, uint32_t (&my)[NT], const uint32_t (&src)[NT], bool& dirty,
                                          TileAlloc& ta, Shared& sh) {
  const int lane = threadIdx.x & 31;
  uint32_t total = 0, at[NT];
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int q = 0; q < NT; ++q) {
    bool need = lane < int(a.g.nT) && src[q] != 0 && src[q] != my[q];
    if (need && my[q] == 0) {
      my[q] = src[q];
      need = false;
    }
    const uint32_t m = __ballot_sync(0xffffffffu, need);
    at[q] = need ? total + __popc(m & lt) : NONE;  // the merge's place in the post
    total += __popc(m);
  }
  if (!total) return;
  int b = -1;
  if (total > 1 && blockDim.x > 32) {
    if (lane == 0) {
      const uint32_t left = ~*(volatile uint32_t*)&sh.used & ((1u << kPosts) - 1u);
      if (left) {
        const int q = __ffs(left) - 1;
        if (!(atomicOr(&sh.used, 1u << q) & (1u << q))) b = q;
      }
    }
    b = __shfl_sync(0xffffffffu, b, 0);
  }
  if (b < 0) {  // alone
#pragma unroll
    for (int q = 0; q < NT; ++q) {
      if (at[q] != NONE) {
        prefetch_tile(a, my[q]);
        prefetch_tile(a, src[q]);
      }
      for (uint32_t m = __ballot_sync(0xffffffffu, at[q] != NONE); m; m &= m - 1) {
        const int T = __ffs(m) - 1;
        bool fresh;
        const uint32_t id = merge_one(a, __shfl_sync(0xffffffffu, my[q], T), __shfl_sync(0xffffffffu, src[q], T),
                                      fresh, ta);
        if (lane == T) my[q] = id;
        ta.count(2, fresh ? 1u : 0u);
        dirty |= fresh;
      }
    }
    return;
  }
  Post& post = sh.post[b];
#pragma unroll
  for (int q = 0; q < NT; ++q) {
    if (at[q] != NONE) {
      post.ida[at[q]] = my[q];
      post.idb[at[q]] = src[q];
    }
  }
  if (lane == 0) post.done = 0;
  __threadfence_block();
  __syncwarp();
  if (lane == 0) {
    atomicOr(&sh.open, 1u << b);  // (before the first merge can be taken: the last one taken clears it)
    __threadfence_block();
    atomicExch(&post.word, post_open(total));
  }
  while (take_merge(a, sh, b, ta)) {
  }
  // helpers finish what they took (they wait for nothing meanwhile); bounded all the same
  for (uint32_t it = 0; it < kSpinLimitW; ++it) {
    if (__all_sync(0xffffffffu, *(volatile uint32_t*)&post.done >= total)) break;
    if (it + 1 == kSpinLimitW && lane == 0) atomicCAS(&a.st->code, 0, GWCP_ERR_TIMEOUT);
  }
  __threadfence_block();
#pragma unroll
  for (int q = 0; q < NT; ++q)
    if (at[q] != NONE) my[q] = *(volatile uint32_t*)&post.ida[at[q]];
  __syncwarp();
  if (lane == 0) {
    atomicExch(&post.word, kPostClosed);
    atomicAnd(&sh.used, ~(1u << b));
  }
  dirty = true;
}

// copy of tile `id` with entry e set to val; returns the new id (warp-uniform)
__device__ __forceinline__ uint32_t cow_set(const WideArgs& a, uint32_t id, uint32_t e, uint32_t val, bool& dirty, TileAlloc& ta) {
  const int lane = threadIdx.x & 31;
  const uint4* p = tile_src(a, id);
  uint4 x0 = __ldca(p), x1 = __ldca(p + 1);
  if (lane == int(e >> 3)) set8(x0, x1, e & 7, val);
  const uint32_t nid = alloc_tile(a, ta);
  ta.count(1, 1);
  if (!nid) return id;
  uint4* d = tile_dst(a, nid);
  d[0] = x0;
  d[1] = x1;
  dirty = true;
  return nid;
}

// entry t of the table held by the warp := val (copy of the tile holding t)
__device__ __forceinline__ void set_entry_w(const WideArgs& a, uint32_t& my, uint32_t t, uint32_t val, bool& dirty,
                                            TileAlloc& ta) {
  const uint32_t T = t / kTileW;
  const uint32_t id = __shfl_sync(0xffffffffu, my, T);
  const uint32_t nid = cow_set(a, id, t % kTileW, val, dirty, ta);
  if ((threadIdx.x & 31) == int(T)) my = nid;
}

// a published table: wait (bounded) until none of its nT words is SENTINEL
__device__ __forceinline__ uint32_t read_table(const WideArgs& a, const uint32_t* tab, bool& abort, Shared& sh,
                                               TileAlloc& ta) {
  const int lane = threadIdx.x & 31;
  const bool act = lane < int(a.g.nT);
  uint32_t v = act ? __ldcg(tab + lane) : 0;
  if (__all_sync(0xffffffffu, v != SENT)) return v;
  uint32_t it = 0;
  while (!abort) {
    const uint32_t open = look(sh).x;
    if (open)
      help(a, sh, open, ta);
    else
      __nanosleep(64);
    v = act ? __ldcg(tab + lane) : 0;
    if (__all_sync(0xffffffffu, v != SENT)) return v;
    if (++it > kSpinLimitW) {
      if (lane == 0) atomicCAS(&a.st->code, 0, GWCP_ERR_TIMEOUT);
      abort = true;
    }
  }
  return v == SENT ? 0u : v;
}

__device__ __forceinline__ void publish(const WideArgs& a, uint32_t* tab, uint32_t id, bool& dirty) {
  if (dirty) __threadfence();  // the tiles this warp wrote are visible before the table is
  dirty = false;
  if ((threadIdx.x & 31) < int(a.g.nT)) __stcg(tab + (threadIdx.x & 31), id);
}

__device__ __forceinline__ uint32_t entry_of(const WideArgs& a, uint32_t my, uint32_t t) {
  // entry t of the warp's table, 0 for t >= W; every lane may ask for a different t.
  // All lanes take part in the shuffle.
  const bool ok = t < a.g.W;
  const uint32_t id = __shfl_sync(0xffffffffu, my, ok ? int(t / kTileW) : 0);
  return ok ? __ldcg(a.tiles + size_t(id) * kTileW + t % kTileW) : 0u;
}

// Join of one tile over a CTA's members (lane m holds member m's id for the tile), with
// the members' own entries raised to their local times nbuf[m] (C_m[u_m] = N_m; H_m[u_m] =
// N_m, which the walker keeps implicit). One pass over the distinct input tiles keeps the
// running maximum and which input equals it so far (an input equals the final maximum
// iff it is >= every other input); the result keeps that input's id when the own
// entries raise nothing, else it is written as a new tile.
__device__ __noinline__ uint32_t join_members(const WideArgs& a, uint32_t idm, const uint32_t* nbuf, uint32_t apb,
                                              uint32_t first, uint32_t T, bool own, bool& dirty, TileAlloc& ta) {
  const int lane = threadIdx.x & 31;
  const bool act = uint32_t(lane) < apb && idm != 0;
  const uint32_t any = __ballot_sync(0xffffffffu, act);
  // members whose own entry lies in tile T
  const uint32_t lo = T * kTileW;
  const bool own_here = own && first < lo + kTileW && first + apb > lo;
  // the usual case: one tile, shared since the last barrier, and no own entries
  const uint32_t id0 = __shfl_sync(0xffffffffu, idm, any ? __ffs(any) - 1 : 0);
  uint32_t leaders = any & (0u - any);
  if (!__all_sync(0xffffffffu, !act || idm == id0)) {
    const uint32_t same = __match_any_sync(0xffffffffu, act ? idm : 0xFFFFFFFFu);
    leaders = __ballot_sync(0xffffffffu, act && (__ffs(same) - 1) == lane);
  }
  if (!own_here && !(leaders & (leaders - 1))) return any ? id0 : 0u;
  uint4 r0 = make_uint4(0, 0, 0, 0), r1 = r0;
  bool have = leaders == 0;  // no input: the zero tile (id 0) equals the maximum so far
  uint32_t cid = 0;          // id of an input equal to the maximum so far (when have)
  auto take = [&](uint32_t id, const uint4& x0, const uint4& x1) {
    const uint4 m0 = max4(r0, x0), m1 = max4(r1, x1);
    const bool le = __all_sync(0xffffffffu, eq4(m0, r0) && eq4(m1, r1));  // x <= r
    const bool ge = __all_sync(0xffffffffu, eq4(m0, x0) && eq4(m1, x1));  // x >= r
    r0 = m0;
    r1 = m1;
    if (!(le && have)) cid = id;
    have = (le && have) || ge;
  };
  for (uint32_t m = leaders; m;) {  // two inputs' loads at a time
    const uint32_t ia = __shfl_sync(0xffffffffu, idm, __ffs(m) - 1);
    m &= m - 1;
    const uint32_t ib = __shfl_sync(0xffffffffu, idm, m ? __ffs(m) - 1 : 0);
    const uint4* p = tile_src(a, ia);
    const uint4* q = tile_src(a, m ? ib : ia);
    const uint4 x0 = __ldca(p), x1 = __ldca(p + 1), y0 = __ldca(q), y1 = __ldca(q + 1);
    take(ia, x0, x1);
    if (m) take(ib, y0, y1);
    m &= m - 1;
  }
  bool raised = false;
  if (own_here) {  // the lane's entries lo + 8 lane + c are those of members lo + 8 lane + c - first
    const int m0 = int(lo + 8 * lane) - int(first);
    if (m0 > -8 && m0 < int(apb)) {
      auto raise = [&](uint32_t x, int c) {
        const int m = m0 + c;
        const uint32_t v = m >= 0 && m < int(apb) ? nbuf[m] : 0u;
        raised |= v > x;
        return max(x, v);
      };
      r0 = make_uint4(raise(r0.x, 0), raise(r0.y, 1), raise(r0.z, 2), raise(r0.w, 3));
      r1 = make_uint4(raise(r1.x, 4), raise(r1.y, 5), raise(r1.z, 6), raise(r1.w, 7));
    }
  }
  const bool keep = have && !__any_sync(0xffffffffu, raised);
  ta.count(__popc(leaders), keep ? 0u : 1u);
  if (keep) return cid;
  const uint32_t nid = alloc_tile(a, ta);
  if (!nid) return any ? id0 : 0u;
  uint4* d = tile_dst(a, nid);
  d[0] = r0;
  d[1] = r1;
  dirty = true;
  return nid;
}

// One warp per agent, one CTA per block of the traced program (agents_per_block <= 32).
// MINB = CTAs of 1024 threads that must share an SM for all blocks to be co-resident.
template <int MINB>
__global__ void __launch_bounds__(1024, MINB) k_prop_wide(const __grid_constant__ WideArgs a) {
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ Shared sh;
  const Geo& g = a.g;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t apb = g.apb;
  const uint32_t first = blockIdx.x * apb;
  const uint32_t u = first + warp;
  uint32_t* const ring = sm + warp * 2 * kPlanBatch * 8;  // [apb][2][kPlanBatch] plan entries
  uint32_t* tabs = sm + apb * 2 * kPlanBatch * 8;         // [apb][3][32] member tables (P, H, JN)
  uint32_t* nbuf = tabs + apb * 96;     // [apb] member epochs
  uint32_t* J = nbuf + 32;              // [3][32] joined tables
  uint32_t* tcnt = J + 96 + warp * 2;   // [apb][2] tiles this warp read and wrote (lane 0 counts)
  __shared__ int start_code;
  if (threadIdx.x == 0) {
    start_code = *(volatile int*)&a.st->code;
    sh.used = sh.open = sh.arrived = 0;
    for (uint32_t q = 0; q < kPosts; ++q) sh.post[q].word = kPostClosed;
  }
  // a walker whose wait gave up goes on without waiting for its block: what it then reads of
  // members that have not arrived is the zero tile and the local time 0
  for (uint32_t i = threadIdx.x; i < apb * 96 + 32 + 96; i += blockDim.x) tabs[i] = 0;  // and nbuf, J
  __syncthreads();
  if (start_code) return;
  const bool act = lane < int(g.nT);
  bool dirty = false, abort = false;
  TileAlloc ta;
  ta.cnt = tcnt;
  if (lane == 0) tcnt[0] = tcnt[1] = 0;
  ask_chunk(a, ta);
  // H_t = bottom{t := 1}: the table starts at bottom and H_t[t] = N_t is kept implicit (in
  // N), so no tile is copied when it increments; a release snapshot writes it out
  // JN_t (jid): the join of every H snapshot joined into P_t, carried along with P_t (joined
  // at acquires from the lock's published JN, at barriers over the members). H moves only by
  // whole-clock joins, so JN_t[v] >= e means P_t already holds the H snapshot of v's release
  // at epoch e: such a join (release loop, in-section access) changes nothing and is skipped.
  uint32_t pid = 0, hid = 0, jid = 0;
  uint32_t N = 1;
  uint32_t arrivals = 0;  // arrivals that complete the block barrier at hand
  unsigned long long joins = 0, visits = 0;
  if (act) a.rows[size_t(a.rowbase[u]) * kTabW + lane] = a.hb_only ? hid : 0u;
  const uint32_t k0 = a.sy_start[u], k1 = a.sy_start[u + 1];
  const uint32_t pb = k0 + a.incs_off[k0], pe = k1 + a.incs_off[k1];
  uint32_t* const cursor_row = a.cursor + size_t(u) * a.n_locks;
  // plan entries, 16 at a time in two halves of the warp's ring: the next ones are copied in
  // while these are walked (read one step ahead they were 1,900 cycles of memory latency each)
  auto fetch = [&](uint32_t b0, uint32_t half) {
    const uint32_t e = b0 + lane / 2;
    if (e < pe)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(
                       __cvta_generic_to_shared(ring + half * kPlanBatch * 8 + lane * 4))),
                   "l"(a.plan + 2 * size_t(b0) + lane)
                   : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(pb, 0);
  for (uint32_t p = pb; p < pe; ++p) {
    const uint32_t i = (p - pb) % kPlanBatch, half = ((p - pb) / kPlanBatch) & 1u;
    if (i == 0) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncwarp();
      fetch(p + kPlanBatch, half ^ 1u);
    }
    const uint4 ea = *reinterpret_cast<const uint4*>(ring + (half * kPlanBatch + i) * 8),
                eb = *reinterpret_cast<const uint4*>(ring + (half * kPlanBatch + i) * 8 + 4);
    const uint32_t t = ea.x & 0xFF, row = ea.y;
    if (t == P_ACQ || t == P_INCS) {
      // acquire: P_t |= P_<l,s'>, H_t |= H_<l,s'>; in-section access: P_t |= L^w (| L^r)
      const uint32_t off = ea.z, w = ea.w;
      const uint32_t* list = t == P_ACQ ? a.pool : a.flat;
      for (uint32_t q = 0; q < w; ++q) {
        uint32_t x;
        if (w <= 4)
          x = q == 0 ? eb.x : q == 1 ? eb.y : q == 2 ? eb.z : eb.w;
        else
          x = __ldcg(list + off + q);
        if (t == P_ACQ) {
          // the three published tables are loaded together (a table still being written is
          // then waited for)
          uint32_t sp = lane < int(g.nT) ? __ldcg(a.psnap + size_t(x) * kTabW + lane) : 0;
          uint32_t sq = lane < int(g.nT) ? __ldcg(a.hsnap + size_t(x) * kTabW + lane) : 0;
          uint32_t sj = lane < int(g.nT) ? __ldcg(a.jsnap + size_t(x) * kTabW + lane) : 0;
          if (!__all_sync(0xffffffffu, sp != SENT && sq != SENT && sj != SENT)) {
            sp = read_table(a, a.psnap + size_t(x) * kTabW, abort, sh, ta);
            sq = read_table(a, a.hsnap + size_t(x) * kTabW, abort, sh, ta);
            sj = read_table(a, a.jsnap + size_t(x) * kTabW, abort, sh, ta);
          }
          uint32_t mine[3] = {pid, hid, jid};
          const uint32_t theirs[3] = {sp, sq, sj};
          merge_tables<3>(a, mine, theirs, dirty, ta, sh);
          pid = mine[0];
          hid = mine[1];
          jid = mine[2];
          joins += 2;
        } else {
          // L^w / L^r: the H snapshot of section x's release, unless JN_t already covers it
          const uint4 mx = __ldg(a.recmeta + x);
          if (entry_of(a, jid, mx.x & 0xFFFF) < mx.w) {
            const uint32_t sx = read_table(a, a.hsnap + size_t(x) * kTabW, abort, sh, ta);
            uint32_t mine[2] = {pid, jid};
            const uint32_t theirs[2] = {sx, sx};
            merge_tables<2>(a, mine, theirs, dirty, ta, sh);
            pid = mine[0];
            jid = mine[1];
            joins += 1;
          }
        }
      }
    } else if (t == P_REL) {
      // release: pop other agents' records on this lock while their acquire is ordered
      // before C_t, joining the released ones whose scope overlaps; then publish
      const uint32_t c = ea.z, L = ea.w;
      const uint32_t lo = eb.x, hi = eb.y, s = eb.z, my_idx = eb.w;
      uint32_t cur = __ldcg(cursor_row + L);
      bool stop = false;
      while (!stop && lo + cur < hi) {
        const uint32_t rec = lo + cur + lane;
        const uint32_t nbr = min(32u, hi - (lo + cur));
        uint4 m = make_uint4(NONE, 0, NONE, 0);
        if (rec < hi) m = __ldg(a.recmeta + rec);
        const uint32_t mag = m.x == NONE ? NONE : (m.x & 0xFFFF);
        const uint32_t msid = m.x >> 16;
        const bool mine = mag == u;
        const bool joinable = !mine && m.z != NONE && m.z < my_idx && scopes_overlap(msid, s);
        uint32_t start = 0;
        uint32_t pv = entry_of(a, pid, mag), jv = entry_of(a, jid, mag);
        while (start < nbr) {
          const bool in = uint32_t(lane) >= start && uint32_t(lane) < nbr;
          const uint32_t fail = __ballot_sync(0xffffffffu, in && !mine && m.y > pv);
          const uint32_t f = fail ? uint32_t(__ffs(fail) - 1) : nbr;
          const uint32_t popped = __ballot_sync(0xffffffffu, in && uint32_t(lane) < f && joinable);
          // join only releases not already in P, and of one agent's popped records only the
          // latest (records of one agent are in acquire order, so its H dominates)
          const bool cand = ((popped >> lane) & 1u) && m.w > jv;
          const uint32_t same = __match_any_sync(0xffffffffu, cand ? mag : 0xFFFFFFFFu);
          const uint32_t wave = __ballot_sync(0xffffffffu, cand && (same >> lane) <= 1u);
          visits += __popc(__ballot_sync(0xffffffffu, in && uint32_t(lane) <= f && !mine));
          for (uint32_t wm = wave; wm; wm &= wm - 1) {
            const uint32_t r = lo + cur + (__ffs(wm) - 1);
            const uint32_t sx = read_table(a, a.hsnap + size_t(r) * kTabW, abort, sh, ta);
            uint32_t mine[2] = {pid, jid};
            const uint32_t theirs[2] = {sx, sx};
            merge_tables<2>(a, mine, theirs, dirty, ta, sh);
            pid = mine[0];
            jid = mine[1];
            ++joins;
          }
          if (f == nbr) {
            start = nbr;
          } else if (wave) {
            start = f;  // P grew: test the failing record again
            pv = entry_of(a, pid, mag);
            jv = entry_of(a, jid, mag);
          } else {
            stop = true;  // P unchanged: the record stays unordered
            start = f;
            break;
          }
        }
        cur += start;
      }
      if (lane == 0) __stcg(cursor_row + L, cur);
      uint32_t hp = hid;  // the snapshot of H_t carries its own entry N_t
      set_entry_w(a, hp, u, N, dirty, ta);
      publish(a, a.psnap + size_t(c) * kTabW, pid, dirty);
      publish(a, a.hsnap + size_t(c) * kTabW, hp, dirty);
      publish(a, a.jsnap + size_t(c) * kTabW, jid, dirty);
      ++N;  // H_t[t] = N_t, implicit
    } else {
      // barrier: C and H joined over the members
      const uint32_t mode = eb.x;
      if (eb.y != N) N = eb.y;  // forced compression at barriers: enter with the members' highest N
      if (mode == BAR_SINGLE) {
        set_entry_w(a, pid, u, N, dirty, ta);  // P_t = C_t
      } else {
        if (act) {
          tabs[(warp * 3) * 32 + lane] = pid;
          tabs[(warp * 3 + 1) * 32 + lane] = hid;
          tabs[(warp * 3 + 2) * 32 + lane] = jid;
        }
        if (lane == 0) nbuf[warp] = N;
        // all members have arrived when the count says so; until then merges of others are
        // taken. The members' own waits are bounded and always end in an arrival; the time
        // limit here only backs them up.
        const uint32_t nw = blockDim.x >> 5;
        arrivals += nw;
        __threadfence_block();
        __syncwarp();
        if (lane == 0) atomicAdd(&sh.arrived, 1u);
        unsigned long long t0 = 0;
        for (uint32_t it = 1; !abort; ++it) {
          const uint2 seen = look(sh);
          if (int(seen.y - arrivals) >= 0) break;
          if (seen.x)
            help(a, sh, seen.x, ta);
          else
            __nanosleep(kWaitNs);
          if ((it & 0xFFFFu) == 0) {
            const unsigned long long now = global_ns();
            if (!t0) t0 = now;
            if (__any_sync(0xffffffffu, now - t0 > kBarrierLimitNs)) {
              if (lane == 0) atomicCAS(&a.st->code, 0, GWCP_ERR_TIMEOUT);
              abort = true;
            }
          }
        }
        __threadfence_block();
        bool wrote = false;  // (members fence before they publish the joined tiles)
        // (table, tile) pairs over the warps (asking for their inputs with L1 prefetches first
        // measured 8% slower)
        for (uint32_t job = warp; job < 3 * g.nT; job += nw) {
          const uint32_t tab = job / g.nT, T = job - tab * g.nT;
          const uint32_t id = uint32_t(lane) < apb ? tabs[(lane * 3 + tab) * 32 + T] : 0;
          const uint32_t j = join_members(a, id, nbuf, apb, first, T, tab < 2, wrote, ta);
          if (lane == 0) J[tab * 32 + T] = j;
        }
        __syncthreads();
        dirty = true;
        pid = act ? J[lane] : 0;
        hid = act ? J[32 + lane] : 0;
        jid = act ? J[64 + lane] : 0;
        joins += 2;  // this member's C_t and H_t joined into the block's
        // J is rewritten only after every member has arrived at the next barrier, after reading
        // it here (or by a walker that has given up, with ids of this launch: the analysis has
        // failed then, and every id that can be read is of a tile in the pool)
      }
      ++N;  // H_t[t] = N_t, implicit
    }
    if (act) a.rows[size_t(row) * kTabW + lane] = a.hb_only ? hid : pid;
  }
  if (dirty) __threadfence();
  if (lane == 0) {
    atomicAdd(&a.st->joins, joins);
    atomicAdd(&a.st->loop_visits, visits);
    atomicAdd(&a.st->tiles_read, (unsigned long long)tcnt[0]);
    atomicAdd(&a.st->tiles_written, (unsigned long long)tcnt[1]);
  }
}

// ---- check ---------------------------------------------------------------------------

__global__ void k_wc_runflags(const uint64_t* key, uint32_t n, uint32_t* flag) {
  grid_begin();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) flag[p] = (p == 0 || key[p] != key[p - 1]) ? 1u : 0u;
}

// composite key (run, class, agent) for the stable regrouping; value = key-order position
// composite keys (run, class, agent) of the key-ordered accesses; also the fields of each
// access record the check needs, copied into key order (a sequential read for the check
// instead of a gather by trace index)
__global__ void k_wc_compose(const uint32_t* run_excl, const uint32_t* flag, const uint32_t* idx,
                             const AccInfo* info, uint32_t n, uint64_t* ck, uint32_t* cv, uint32_t* s_who,
                             uint32_t* s_row, uint32_t* s_ep) {
  grid_begin();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const uint32_t run = run_excl[p] + flag[p] - 1;
  const AccInfo in = info[idx[p]];
  ck[p] = (uint64_t(run) << 15) | (uint64_t(who_class(in.who)) << 13) | who_agent(in.who);
  cv[p] = p;
  s_who[p] = in.who;
  s_row[p] = in.row;
  s_ep[p] = in.epoch;
}

// A location that no write-class access touches has no races (two reads never conflict):
// its accesses are left out of the regrouping, so the check finds no partner groups there.
__global__ void k_wc_runwrite(const uint64_t* ck, uint32_t n, uint32_t* run_w) {
  grid_begin();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n && ((ck[p] >> 13) & 3u) != C_READ) run_w[ck[p] >> 15] = 1u;
}
__global__ void k_wc_keep(const uint64_t* ck, uint32_t n, const uint32_t* run_w, uint32_t* keep) {
  grid_begin();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) keep[p] = run_w[ck[p] >> 15];
}
__global__ void k_wc_compact(const uint64_t* ck, const uint32_t* cv, const uint32_t* keep, const uint32_t* kpos,
                             uint32_t n, uint64_t* ck2, uint32_t* cv2) {
  grid_begin();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n && keep[p]) {
    ck2[kpos[p]] = ck[p];
    cv2[kpos[p]] = cv[p];
  }
}

// group starts over the sorted composite keys (the first *n_dev of n), and per (run, class)
// group counts
__global__ void k_wc_groupflags(const uint64_t* ck, uint32_t n, const uint32_t* n_dev, uint32_t* gflag) {
  grid_begin();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) gflag[i] = (i < *n_dev && (i == 0 || ck[i] != ck[i - 1])) ? 1u : 0u;
}

__global__ void k_wc_groups(const uint64_t* ck, const uint32_t* gflag, const uint32_t* gexcl, uint32_t n,
                            uint32_t* grp_lo, uint32_t* grp_agent, uint32_t* rc_cnt) {
  grid_begin();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || !gflag[i]) return;
  const uint32_t gi = gexcl[i];
  grp_lo[gi] = i;
  grp_agent[gi] = uint32_t(ck[i] & 0x1FFF);
  atomicAdd(rc_cnt + (ck[i] >> 13), 1u);  // (run << 2 | class)
}

struct WideCheckArgs {
  Geo g;
  uint32_t n;
  const uint32_t* n_dev;     // the count on the device (at most n), or null
  const uint32_t* idx;       // key order -> trace index
  const uint32_t* flag;      // run starts
  const uint32_t* run_excl;  // exclusive scan of flag
  const uint32_t* gs;        // grouped order -> key-order position (grouped: the trace index itself)
  uint32_t grouped;          // the primary order is the grouped order (compare trace indices)
  const uint32_t* grp_lo;    // [n_groups + 1]
  const uint32_t* grp_agent;
  const uint32_t* rc_off;    // [(run << 2 | class) + 1]
  const AccInfo* info;
  const uint32_t *s_who, *s_row, *s_ep;  // record fields in key order
  const uint32_t* rows;
  const uint32_t* tiles;
  unsigned long long tile_cap;  // ids at or above it (rows a failed walk left stale) read as zero
  uint64_t* races;
  unsigned long long race_cap;
  DevStatus* st;
  uint32_t dense_wp;             // 0: clocks are tile tables; else dense rows of this many words
  const uint32_t* cv_pool;       // non-null: compressed versions (rows holds B headers each)
  unsigned long long cv_cap;
  uint32_t row_words;            // words per entry of rows
  unsigned long long* chunk_ns;  // optional timeline: globaltimer at each block's end
  uint32_t* chunk_races;         // and the races it found
  uint2* big;         // (position, piece | pieces << 16) items of k_wc_big
  uint32_t big_cap;   // items it holds
};

// position j in group gi of the latest member with gs[j] < x (gs ascends within a group:
// key-order positions, or trace indices in the grouped order), or NONE
__device__ __forceinline__ uint32_t pred_in_group(const WideCheckArgs& a, uint32_t gi, uint32_t x) {
  uint32_t lo = a.grp_lo[gi], hi = a.grp_lo[gi + 1];
  if (lo == hi || a.gs[lo] >= x) return NONE;
  while (hi - lo > 1) {  // invariant: gs[lo] < x, and gs[hi] >= x or hi is the end
    const uint32_t mid = (lo + hi) >> 1;
    if (a.gs[mid] < x)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// classes a later access of class cb conflicts with and is not exempt from (bit q = class
// q), given whether the partner shares b's block
__device__ __forceinline__ uint32_t conflict_classes(uint32_t cb, bool same_block) {
  switch (cb) {
    case C_READ: return 0b1110;
    case C_WRITE: return 0b1111;
    case C_ATOM_CTA: return same_block ? 0b0011 : 0b0111;
    default: return 0b0011;
  }
}

// Races found by a warp are staged in shared memory and appended with one global atomic
// per warp; a warp that finds more than kRaceStage spills the rest with one atomic each.
// Per warp, not per block: the threads of an access at a hot location search many more
// partner groups than the rest, and a block-wide append would hold every warp of the
// block until its slowest thread is done.
constexpr uint32_t kRaceStage = 256;
constexpr uint32_t kCheckThreads = 256;

__device__ __forceinline__ void emit_race(const WideCheckArgs& a, uint64_t v, uint32_t* s_cnt, uint64_t* s_buf) {
  const uint32_t slot = atomicAdd(s_cnt, 1u);
  if (slot == 0) atomicCAS(&a.st->first_race_ns, 0ull, global_ns());  // the warp's first race: the earliest
                                                                       // stamp wins
  if (slot < kRaceStage) {
    s_buf[slot] = v;
    return;
  }
  const unsigned long long at = atomicAdd(&a.st->n_races, 1ull);
  if (at < a.race_cap) a.races[at] = v;
}

// REP: how the clock versions are held (one instantiation each, so that the common
// representations keep their registers and occupancy)
enum : int { REP_TILES = 0, REP_DENSE = 1, REP_COMPRESSED = 2 };

// One access to check, and the groups of its location by class.
struct CheckAcc {
  uint32_t b, who, run;    // trace index, agent / class / block, location run
  uint32_t x;              // "earlier than b" in the order gs holds
  const uint32_t* rowtab;  // b's clock version
};
__device__ __forceinline__ CheckAcc check_acc(const WideCheckArgs& a, uint32_t p) {
  CheckAcc c;
  c.b = a.idx[p];
  c.who = a.s_who[p];
  c.run = a.run_excl[p] + a.flag[p] - 1;
  c.x = a.grouped ? c.b : p;
  c.rowtab = a.rows + size_t(a.s_row[p]) * a.row_words;
  return c;
}
// the groups [cur[q], end[q]) of the classes the access may conflict with
__device__ __forceinline__ void check_lists(const WideCheckArgs& a, const CheckAcc& c, uint32_t (&cur)[4],
                                            uint32_t (&end)[4]) {
  const uint32_t cb = who_class(c.who);
  const uint32_t any_mask = conflict_classes(cb, false) | conflict_classes(cb, true);
#pragma unroll
  for (uint32_t q = 0; q < 4; ++q) {
    const bool on = (any_mask >> q) & 1u;
    cur[q] = on ? a.rc_off[(c.run << 2) | q] : 0u;
    end[q] = on ? a.rc_off[((c.run << 2) | q) + 1] : 0u;
  }
}

// Partner tests of access c against the groups [cur[q], end[q]); returns how many were made.
// The location's groups of each class are sorted by agent: walk the classes' lists
// together (a merge by agent), so that each agent is handled once, from the class
// holding its latest conflicting access before b (ties: the lower class).
template <int REP>
__device__ __forceinline__ uint32_t check_merge(const WideCheckArgs& a, const CheckAcc& c, uint32_t (&cur)[4],
                                                const uint32_t (&end)[4], uint32_t* s_cnt, uint64_t* s_buf) {
  const uint32_t u = who_agent(c.who), cb = who_class(c.who), bu = who_block(c.who);
  uint32_t tests = 0;
  for (;;) {
    uint32_t v = NONE;
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q)
      if (cur[q] < end[q]) v = min(v, a.grp_agent[cur[q]]);
    if (v == NONE) break;
    const uint32_t cm = conflict_classes(cb, v / a.g.apb == bu);
    uint32_t j = NONE, pos = NONE;
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
      if (cur[q] >= end[q] || a.grp_agent[cur[q]] != v) continue;
      const uint32_t gi = cur[q]++;
      if (v == u || !((cm >> q) & 1u)) continue;
      const uint32_t jq = pred_in_group(a, gi, c.x);
      if (jq == NONE) continue;
      const uint32_t pq = a.gs[jq];
      if (pos == NONE || pq > pos) {
        pos = pq;
        j = jq;
      }
    }
    if (pos == NONE) continue;
    {
      ++tests;
      const uint32_t qa = a.grouped ? j : pos;  // a*'s position in the primary order
      const uint32_t ai = a.idx[qa];
      const uint32_t na = a.s_ep[qa];
      uint32_t cv;
      if constexpr (REP == REP_COMPRESSED) {
        cv = cv_entry(c.rowtab, a.cv_pool, a.cv_cap, v, a.g.apb, cv_group(a.g.gran));
      } else if constexpr (REP == REP_DENSE) {
        cv = __ldg(c.rowtab + v);
      } else {
        const uint32_t tid = __ldg(c.rowtab + v / kTileW);
        cv = tid < a.tile_cap ? __ldg(a.tiles + size_t(tid) * kTileW + v % kTileW) : 0u;
      }
      if (na > cv) emit_race(a, (uint64_t(c.b) << 32) | ai, s_cnt, s_buf);  // N(a*) > C_b[v]
    }
  }
  return tests;
}

// An access at a location that many agents touched walks up to a group per agent and class,
// a chain of dependent loads of 1 to 2 us per group: one thread for each such access left a
// tail of 10 ms after everything else (4M events, 4096 warps: writes to a location that all
// warps read). Such accesses are cut by agent into parts, one per lane, each walking its own
// agents' groups: 9.8 -> 0.51 ms there (1.67 -> 0.23 at 512 warps and 2.3M events).
//   part `part` of `parts`: the longest class list is cut evenly, the other lists at the
//   same agents (binary searches).
__device__ __forceinline__ uint32_t group_lower_bound(const WideCheckArgs& a, uint32_t lo, uint32_t hi,
                                                      uint32_t agent) {
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (a.grp_agent[mid] < agent)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}
__device__ __forceinline__ void cut_lists(const WideCheckArgs& a, uint32_t part, uint32_t parts, uint32_t (&cur)[4],
                                          uint32_t (&end)[4]) {
  uint32_t lo = cur[0], len = end[0] - cur[0];
#pragma unroll
  for (uint32_t q = 1; q < 4; ++q) {
    if (end[q] - cur[q] > len) {
      len = end[q] - cur[q];
      lo = cur[q];
    }
  }
  // agents [a0, a1): the part's share of the longest list (the first part also takes the
  // agents below it, the last part those above). A part with an empty share has a0 == a1.
  const uint32_t s0 = uint32_t(uint64_t(len) * part / parts), s1 = uint32_t(uint64_t(len) * (part + 1) / parts);
  const bool first = part == 0, last = part + 1 == parts;
  const uint32_t a0 = first ? 0u : a.grp_agent[lo + s0], a1 = last ? NONE : a.grp_agent[lo + s1];
#pragma unroll
  for (uint32_t q = 0; q < 4; ++q) {
    const uint32_t c0 = cur[q], c1 = end[q];
    cur[q] = first ? c0 : group_lower_bound(a, c0, c1, a0);
    end[q] = last ? c1 : group_lower_bound(a, cur[q], c1, a1);
  }
}

// Part `part` of `parts` of the access at position p (out of line: k_wc_check's registers
// are those of the common walk).
template <int REP>
__device__ __noinline__ uint32_t check_part(const WideCheckArgs& a, uint32_t p, uint32_t part, uint32_t parts,
                                            uint32_t* s_cnt, uint64_t* s_buf) {
  const CheckAcc c = check_acc(a, p);
  uint32_t cur[4], end[4];
  check_lists(a, c, cur, end);
  cut_lists(a, part, parts, cur, end);
  return check_merge<REP>(a, c, cur, end, s_cnt, s_buf);
}

// A lane walks its access's groups itself up to a limit; an access with more is put aside. The
// longest walk left to a lane is a tail of about 1 us per group after everything else, so the
// limit is low where it can be: but an access that is put aside costs the searches that place
// its parts, and at the locations that most agents use nearly every access is as long as the
// longest. So the limit is the lowest step that at most kAsideMost accesses of this trace are
// above: about one for each warp of k_wc_big that the GPU holds. k_wc_fields (in the ranked order
// k_wc_lists) counts them, beside the walkers. The check (ms) by limit, with the accesses above it:
//   events, agents     32              48              64              96             192
//   1M, 64        0.056  218      0.066  188      0.103  119      0.178    0     0.180    0
//   2M, 128       0.334  83k      0.096  1717     0.106  424      0.125  377     0.480    0
//   3M, 256       0.696  179k     0.524  122k     0.533  122k     0.170  603     0.244  507
//   5M, 64        0.993  294k     0.766  200k     0.290  649      0.379  175     0.414    0
//   8M, 128       2.286  674k     1.979  554k     1.319  317k     0.414  6629    0.795  188
//   1M, 4096      0.215  42k      0.082  228      0.088  210      0.123  198     0.158  176
//   3M, 512 thr.  0.205  57k      0.201  48k      0.201  42k      0.196  24k     0.226  3
constexpr uint32_t kAsideMost = 8192;
__host__ __device__ constexpr uint32_t list_step(int j) {
  constexpr uint32_t step[kListSteps] = {32, 48, 64, 80, 96, 128, 192, 384};
  return step[j];
}
__device__ __forceinline__ uint32_t list_limit(const DevStatus* st) {
  uint32_t limit = list_step(kListSteps - 1);
#pragma unroll
  for (int j = kListSteps - 2; j >= 0; --j)
    if (st->long_lists[j] <= kAsideMost) limit = list_step(j);  // (the counts fall from step to step)
  return limit;
}

// The partner groups of an access of class cb in a run.
__device__ __forceinline__ uint32_t list_length(const uint32_t* rc_off, uint32_t run, uint32_t cb) {
  const uint32_t any_mask = conflict_classes(cb, false) | conflict_classes(cb, true);
  uint32_t groups = 0, at = rc_off[run << 2];
#pragma unroll
  for (uint32_t q = 0; q < 4; ++q) {
    const uint32_t next = rc_off[((run << 2) | q) + 1];
    groups += (any_mask >> q) & 1u ? next - at : 0u;
    at = next;
  }
  return groups;
}
// Counts the block's accesses above each step (every thread of it calls this).
__device__ __forceinline__ void count_lists(uint32_t groups, DevStatus* st) {
  __shared__ uint32_t s_over[kListSteps];
  if (threadIdx.x < kListSteps) s_over[threadIdx.x] = 0;
  if (!__syncthreads_or(groups > list_step(0))) return;
#pragma unroll
  for (int j = 0; j < kListSteps; ++j) {
    const uint32_t over = __popc(__ballot_sync(0xffffffffu, groups > list_step(j)));
    if ((threadIdx.x & 31) == 0 && over) atomicAdd(&s_over[j], over);
  }
  __syncthreads();
  if (threadIdx.x < kListSteps && s_over[threadIdx.x]) atomicAdd(&st->long_lists[threadIdx.x], s_over[threadIdx.x]);
}
__global__ void __launch_bounds__(kCheckThreads) k_wc_lists(const uint32_t* flag, const uint32_t* run_excl,
                                                            const uint32_t* s_who, const uint32_t* rc_off, uint32_t n,
                                                            DevStatus* st) {
  grid_begin();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  count_lists(p < n ? list_length(rc_off, run_excl[p] + flag[p] - 1, who_class(s_who[p])) : 0u, st);
}

constexpr uint32_t kPieceGroups = 128;  // groups per item of k_wc_big: four per lane

// appends the warp's staged races (one global atomic) and its test count; returns the races found
__device__ __forceinline__ uint32_t flush_warp(const WideCheckArgs& a, uint32_t tests, uint32_t* s_cnt,
                                               const uint64_t* s_buf) {
  const uint32_t lane = threadIdx.x & 31;
  tests = __reduce_add_sync(0xffffffffu, tests);
  __syncwarp();
  const uint32_t found = *s_cnt;
  const uint32_t n = min(found, kRaceStage);
  unsigned long long base = 0;
  if (lane == 0) {
    if (tests) atomicAdd(&a.st->partner_tests, (unsigned long long)tests);
    if (n) base = atomicAdd(&a.st->n_races, (unsigned long long)n);
  }
  base = __shfl_sync(0xffffffffu, base, 0);
  for (uint32_t i = lane; i < n; i += 32)
    if (base + i < a.race_cap) a.races[base + i] = s_buf[i];
  return found;
}

// ASIDE: accesses with many groups become items of k_wc_big (those that find no room are
// walked here); otherwise the lanes of their warp share them (a ranked check keeps its order).
template <int REP, bool ASIDE>
__global__ void __launch_bounds__(kCheckThreads, 8) k_wc_check(const __grid_constant__ WideCheckArgs a) {
  grid_begin();
  const uint32_t limit = list_limit(a.st);
  if (a.st->code) return;  // (the access records or clocks are incomplete)
  constexpr uint32_t kWarps = kCheckThreads / 32;
  __shared__ uint32_t s_cnt[kWarps];
  __shared__ uint64_t s_buf[kWarps][kRaceStage];
  __shared__ uint32_t s_done, s_found;  // timeline: warps finished, races found by the block
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) s_cnt[warp] = 0;
  if (threadIdx.x == 0) s_done = s_found = 0;
  __syncthreads();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t n_eff = a.n_dev ? min(a.n, *a.n_dev) : a.n;
  uint32_t tests = 0;
  bool big = false;
  {
    CheckAcc c{};
    uint32_t cur[4] = {0, 0, 0, 0}, end[4] = {0, 0, 0, 0};
    if (p < n_eff) {
      c = check_acc(a, p);
      check_lists(a, c, cur, end);
    }
    uint32_t groups = 0;
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) groups += end[q] - cur[q];
    big = groups > limit;
    if constexpr (ASIDE) {
      if (big) {
        const uint32_t pieces = (groups + kPieceGroups - 1) / kPieceGroups;
        const unsigned long long at = atomicAdd(&a.st->big_items, (unsigned long long)pieces);
        const bool fits = at + pieces <= a.big_cap;
        for (unsigned long long i = 0; i < pieces && at + i < a.big_cap; ++i)
          a.big[at + i] = fits ? make_uint2(p, uint32_t(i) | (pieces << 16)) : make_uint2(NONE, 0);
        big = fits;
      }
    }
    if (!big) tests = check_merge<REP>(a, c, cur, end, &s_cnt[warp], s_buf[warp]);
  }
  if constexpr (!ASIDE) {
    for (uint32_t m = __ballot_sync(0xffffffffu, big); m; m &= m - 1) {
      const uint32_t first = blockIdx.x * blockDim.x + warp * 32;
      tests += check_part<REP>(a, first + (__ffs(m) - 1), lane, 32, &s_cnt[warp], s_buf[warp]);
      __syncwarp();
    }
  }
  const uint32_t found = flush_warp(a, tests, &s_cnt[warp], s_buf[warp]);
  if (a.chunk_ns && lane == 0) {  // the block's last warp stamps the block's end
    atomicAdd(&s_found, found);
    __threadfence_block();
    if (atomicAdd(&s_done, 1u) == kWarps - 1) {
      a.chunk_ns[blockIdx.x] = global_ns();
      a.chunk_races[blockIdx.x] = atomicAdd(&s_found, 0u);
    }
  }
}

// The items that k_wc_check put aside, a warp each: piece i of an access's lists, cut into
// 32 parts per piece. Runs after k_wc_check; the grid strides over the items, so accesses
// at one hot location (neighbours in the order) spread over all SMs.
template <int REP>
__global__ void __launch_bounds__(kCheckThreads, 6) k_wc_big(const __grid_constant__ WideCheckArgs a) {
  grid_begin();
  if (a.st->code) return;  // (the access records or clocks are incomplete)
  constexpr uint32_t kWarps = kCheckThreads / 32;
  __shared__ uint32_t s_cnt[kWarps];
  __shared__ uint64_t s_buf[kWarps][kRaceStage];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned long long items = min(a.st->big_items, (unsigned long long)a.big_cap);
  for (unsigned long long t = blockIdx.x * kWarps + warp; t < items; t += gridDim.x * kWarps) {
    const uint2 it = a.big[t];
    if (it.x == NONE) continue;
    if (lane == 0) s_cnt[warp] = 0;
    __syncwarp();
    const uint32_t tests =
        check_part<REP>(a, it.x, (it.y & 0xFFFFu) * 32 + lane, (it.y >> 16) * 32, &s_cnt[warp], s_buf[warp]);
    __syncwarp();
    const uint32_t found = flush_warp(a, tests, &s_cnt[warp], s_buf[warp]);
    if (a.chunk_ns && lane == 0) {  // the item belongs to its access's chunk of the timeline
      atomicAdd(a.chunk_races + it.x / kCheckThreads, found);
      atomicMax(a.chunk_ns + it.x / kCheckThreads, global_ns());
    }
    __syncwarp();
  }
}

// ---- grouped order: the accesses sorted once by (location, class, agent, trace index) ----
// Before the sort, the accesses of locations without a write-class access are left out
// (two reads never race): the sort's first pass keeps only those whose location's bit is
// set in the hashed bitmap that the decoding pass filled from the write-class accesses. A
// bit shared with a written location keeps a few read-only locations; they have no partners.

// location runs and (class, agent) groups of the composite keys (the first *n_dev keys)
__global__ void k_gr_flags(const uint64_t* ck, uint32_t n, const uint32_t* n_dev, uint32_t* run_flag,
                           uint32_t* grp_flag) {
  grid_begin();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  if (p >= *n_dev) {
    run_flag[p] = 0;
    grp_flag[p] = 0;
    return;
  }
  run_flag[p] = (p == 0 || (ck[p] >> 15) != (ck[p - 1] >> 15)) ? 1u : 0u;
  grp_flag[p] = (p == 0 || ck[p] != ck[p - 1]) ? 1u : 0u;
}

// The groups ascend by (run, class, agent); rc_off[(run << 2) | q] is the first group whose
// (run, class) slot is >= (run, q). The first group of a slot writes it and the empty slots
// before it; the last access writes the slots after the last group (up to 4 * runs).
__global__ void k_gr_groups(const uint64_t* ck, const uint32_t* run_flag, const uint32_t* run_excl,
                            const uint32_t* gflag, const uint32_t* gexcl, const uint32_t* n_dev, uint32_t* grp_lo,
                            uint32_t* grp_agent, uint32_t* rc_off) {
  grid_begin();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t n = *n_dev;
  if (i >= n) return;
  const uint32_t run = run_excl[i] + run_flag[i] - 1;
  const uint32_t slot = (run << 2) | uint32_t((ck[i] >> 13) & 3u);
  if (i == n - 1) {
    const uint32_t n_groups = gexcl[i] + gflag[i];
    grp_lo[n_groups] = n;
    for (uint32_t t = slot + 1; t <= (run << 2) + 4; ++t) rc_off[t] = n_groups;
  }
  if (!gflag[i]) return;
  const uint32_t gi = gexcl[i];
  grp_lo[gi] = i;
  grp_agent[gi] = uint32_t(ck[i] & 0x1FFF);
  // slot of the previous group (-1 before the first)
  const int64_t prev = i == 0 ? -1 : int64_t(((run - run_flag[i]) << 2) | uint32_t((ck[i - 1] >> 13) & 3u));
  for (int64_t t = prev + 1; t <= int64_t(slot); ++t) rc_off[t] = gi;
}

// the fields of each access record the check needs, copied into the primary order; and the
// counts of long lists
__global__ void __launch_bounds__(kCheckThreads) k_wc_fields(const uint32_t* idx, const AccInfo* info, const uint32_t* n_dev,
                                                             uint32_t* s_who, uint32_t* s_row, uint32_t* s_ep,
                                                             const uint32_t* flag, const uint32_t* run_excl,
                                                             const uint32_t* rc_off, DevStatus* st) {
  grid_begin();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t groups = 0;
  if (p < *n_dev) {
    const AccInfo in = info[idx[p]];
    s_who[p] = in.who;
    s_row[p] = in.row;
    s_ep[p] = in.epoch;
    groups = list_length(rc_off, run_excl[p] + flag[p] - 1, who_class(in.who));
  }
  count_lists(groups, st);
}

__global__ void k_wc_grp_end(const uint32_t* n_groups, const uint32_t* n_dev, uint32_t* grp_lo) {
  grid_begin();
  grp_lo[*n_groups] = *n_dev;
}

inline uint32_t nblk(uint64_t n, uint32_t t) { return uint32_t((n + t - 1) / t); }

}  // namespace

// Launch of the wide walker (the plan stream is already built on s).
int phaseG_wide(const Bufs& b, const Geo& g, const Sizes& z, cudaStream_t s) {
  WideArgs a{};
  a.g = g;
  a.st = b.st;
  a.sy_start = b.sy_start;
  a.incs_off = b.incs_cnt;
  a.rowbase = b.vcount;
  a.plan = b.plan;
  a.recmeta = b.recmeta;
  a.pool = b.dep_pool;
  a.flat = b.flat;
  a.rows = b.rows;
  a.psnap = b.psnap;
  a.hsnap = b.hsnap;
  a.cursor = b.cursor;
  a.jsnap = b.jsnap;
  a.tiles = b.tiles;
  a.tile_ctr = reinterpret_cast<unsigned long long*>(&b.st->spare[2]);
  a.tile_cap = z.tile_cap;
  a.n_locks = z.n_locks;
  a.hb_only = z.hb_only;
  const uint32_t threads = g.apb * 32;
  // member tables, epochs, joined tables, tile counts, plan rings
  const size_t smem = (size_t(g.apb) * 96 + 32 + 96 + 2 * size_t(g.apb) + size_t(g.apb) * 2 * kPlanBatch * 8) * 4;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // the variant with the most registers whose CTAs are all co-resident; packed: two CTAs
  // per SM first, which leaves SMs to other streams' kernels
  void* kern = nullptr;
  void* order[2] = {reinterpret_cast<void*>(k_prop_wide<1>), reinterpret_cast<void*>(k_prop_wide<2>)};
  if (z.pack_walkers) std::swap(order[0], order[1]);
  for (void* k : order) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kMaxDynamicSmem)) != cudaSuccess)
      return GWCP_ERR_CUDA;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, int(threads), smem) != cudaSuccess)
      return GWCP_ERR_CUDA;
    if (uint64_t(per_sm) * sms >= g.B) {
      kern = k;
      break;
    }
  }
  if (!kern) return GWCP_ERR_UNSUPPORTED;  // walkers must be co-resident
  void* args[] = {&a};
  if (cudaLaunchCooperativeKernel(kern, dim3(g.B), dim3(threads), args, smem, s) != cudaSuccess) return GWCP_ERR_CUDA;
  count_launch();
  return GWCP_OK;
}

// Regrouping of the key-sorted accesses by (location, class, agent); runs beside the
// propagation (it needs AccInfo and the key order, not the clocks).
void phaseI_wide_group(Bufs& b, const Geo& g, Sizes& z, uint32_t* tmp, cudaStream_t s, Prof& p) {
  const uint32_t n = z.n_acc;
  if (!n) return;
  p.begin("i_wide_group", double(n) * (8 + 4 + 16 + 12 * 3 * 5 + 16), s);
  launch(k_wc_runflags, nblk(n, 256), 256, 0, s)(b.acc_key, n, b.wc_flag);
  count_launch();
  scan_exclusive(b.wc_flag, b.wc_run, n, b.wc_run + n, tmp, s);
  launch(k_wc_compose, nblk(n, 256), 256, 0, s)(b.wc_run, b.wc_flag, b.acc_idx, b.acc_info, n, b.wc_key, b.wc_val,
                                            b.wc_who, b.wc_row, b.wc_ep);
  count_launch();
  // accesses of locations with a write-class access, compacted (count on the device, at
  // wc_gexcl[n]); wc_grp_lo, wc_gflag and wc_gexcl serve as scratch until the groups are built
  uint32_t* run_w = b.wc_grp_lo;
  uint32_t* keep = b.wc_gflag;
  uint32_t* kpos = b.wc_gexcl;
  uint32_t* n_keep = b.wc_gexcl + n;
  cudaMemsetAsync(run_w, 0, (size_t(n) + 1) * 4, s);
  launch(k_wc_runwrite, nblk(n, 256), 256, 0, s)(b.wc_key, n, run_w);
  count_launch();
  launch(k_wc_keep, nblk(n, 256), 256, 0, s)(b.wc_key, n, run_w, keep);
  count_launch();
  scan_exclusive(keep, kpos, n, n_keep, tmp, s);
  launch(k_wc_compact, nblk(n, 256), 256, 0, s)(b.wc_key, b.wc_val, keep, kpos, n, b.wc_key2, b.wc_val2);
  count_launch();
  std::swap(b.wc_key, b.wc_key2);
  std::swap(b.wc_val, b.wc_val2);
  uint32_t* const n_kept = b.wc_run + n + 1;  // the count, copied out of the scratch
  cudaMemcpyAsync(n_kept, n_keep, 4, cudaMemcpyDeviceToDevice, s);
  // runs < n <= 2^30: key bits 15 .. 15 + ceil(log2 n); class bits 13-14; agent bits below
  // 13, of which only ceil(log2 W) vary
  uint32_t rb = 1, ab = 0;
  while ((1ull << rb) < n) ++rb;
  while ((1u << ab) < g.W) ++ab;
  const uint64_t mask = (((1ull << rb) - 1) << 15) | (3ull << 13) | ((1ull << ab) - 1);
  if (radix_sort_pairs(b.wc_key, b.wc_val, b.wc_key2, b.wc_val2, n, mask, tmp, s, n_kept)) {
    std::swap(b.wc_key, b.wc_key2);
    std::swap(b.wc_val, b.wc_val2);
  }
  launch(k_wc_groupflags, nblk(n, 256), 256, 0, s)(b.wc_key, n, n_kept, b.wc_gflag);
  count_launch();
  scan_exclusive(b.wc_gflag, b.wc_gexcl, n, b.wc_gexcl + n, tmp, s);
  cudaMemsetAsync(b.wc_rc, 0, (size_t(n) * 4 + 2) * 4, s);
  launch(k_wc_groups, nblk(n, 256), 256, 0, s)(b.wc_key, b.wc_gflag, b.wc_gexcl, n, b.wc_grp_lo, b.wc_grp_agent,
                                          b.wc_rc);
  count_launch();
  launch(k_wc_grp_end, 1, 1, 0, s)(b.wc_gexcl + n, n_kept, b.wc_grp_lo);  // grp_lo[n_groups] = kept count
  count_launch();
  scan_exclusive(b.wc_rc, b.wc_rc, size_t(n) * 4 + 1, nullptr, tmp, s);
  launch(k_wc_lists, nblk(n, kCheckThreads), kCheckThreads, 0, s)(b.wc_flag, b.wc_run, b.wc_who, b.wc_rc, n, b.st);
  count_launch();
  p.end();
}

// Groups of the grouped order (the accesses already sorted by (location, class, agent),
// trace order within): location runs, (class, agent) groups, the first group of each
// (run, class), and the record fields in that order. One sort instead of a location sort
// followed by a regrouping sort.
void phaseI_grouped(Bufs& b, const Geo& g, Sizes& z, uint32_t* tmp, cudaStream_t s, Prof& p) {
  (void)g;
  const uint32_t n = z.n_kept;  // the accesses the written-location filter kept
  if (!n) return;
  p.begin("i_wide_group", double(n) * (8 + 4 * 4 + 16 + 12 + 16), s);  // ~ per access
  launch(k_gr_flags, nblk(n, 256), 256, 0, s)(b.acc_key, n, b.n_kept, b.wc_flag, b.wc_gflag);
  count_launch();
  ScanBatch sb{};
  sb.job[0] = ScanJob{b.wc_flag, b.wc_run, b.wc_run + n, n};
  sb.job[1] = ScanJob{b.wc_gflag, b.wc_gexcl, b.wc_gexcl + n, n};
  scan_all(sb, 2, tmp, s);
  launch(k_gr_groups, nblk(n, 256), 256, 0, s)(b.acc_key, b.wc_flag, b.wc_run, b.wc_gflag, b.wc_gexcl, b.n_kept,
                                          b.wc_grp_lo, b.wc_grp_agent, b.wc_rc);
  count_launch();
  launch(k_wc_fields, nblk(n, kCheckThreads), kCheckThreads, 0, s)(b.acc_idx, b.acc_info, b.n_kept, b.wc_who, b.wc_row,
                                                              b.wc_ep, b.wc_flag, b.wc_run, b.wc_rc, b.st);
  count_launch();
  p.end();
}


uint32_t sparse_check_blocks(uint32_t n_acc) { return nblk(n_acc, kCheckThreads); }

void phaseI_wide_check(const Bufs& b, const Geo& g, const Sizes& z, cudaStream_t s, Prof& p) {
  const uint32_t n = z.grouped ? z.n_kept : z.n_acc;
  if (!n) return;
  WideCheckArgs a{};
  a.g = g;
  a.n = n;
  a.n_dev = z.grouped ? b.n_kept : nullptr;
  a.idx = b.acc_idx;
  a.flag = b.wc_flag;
  a.run_excl = b.wc_run;
  a.gs = z.grouped ? b.acc_idx : b.wc_val;
  a.grouped = z.grouped ? 1u : 0u;
  a.grp_lo = b.wc_grp_lo;
  a.grp_agent = b.wc_grp_agent;
  a.rc_off = b.wc_rc;
  a.info = b.acc_info;
  a.s_who = b.wc_who;
  a.s_row = b.wc_row;
  a.s_ep = b.wc_ep;
  a.rows = b.rows;
  a.tiles = b.tiles;
  a.tile_cap = z.tile_cap;
  a.races = b.races;
  a.race_cap = z.race_cap;
  a.st = b.st;
  a.dense_wp = g.nT ? 0u : g.Wp;
  a.cv_pool = z.compress ? b.cv_pool : nullptr;
  a.cv_cap = z.cv_cap;
  a.row_words = z.compress ? g.B : g.RW;
  a.chunk_ns = b.chunk_ns;
  a.chunk_races = b.chunk_races;
  a.big = reinterpret_cast<uint2*>(b.wc_big);
  a.big_cap = z.grouped ? z.big_cap : 0;
  p.begin("i_check", double(n) * (4 + 16 + 4 + 4 + 4 + 8));
  int rep = g.nT ? REP_TILES : REP_DENSE;
  if (z.compress) rep = REP_COMPRESSED;
  auto check = rep == REP_TILES ? k_wc_check<REP_TILES, true>
               : rep == REP_DENSE ? k_wc_check<REP_DENSE, true> : k_wc_check<REP_COMPRESSED, true>;
  if (!z.grouped)
    check = rep == REP_TILES ? k_wc_check<REP_TILES, false>
            : rep == REP_DENSE ? k_wc_check<REP_DENSE, false> : k_wc_check<REP_COMPRESSED, false>;
  launch(check, nblk(n, kCheckThreads), kCheckThreads, 0, s)(a);
  count_launch();
  if (z.grouped && 4 * g.W > list_step(0)) {  // fewer agents have no such access
    auto big = rep == REP_TILES ? k_wc_big<REP_TILES>
               : rep == REP_DENSE ? k_wc_big<REP_DENSE> : k_wc_big<REP_COMPRESSED>;
    launch(big, std::min<uint32_t>(nblk(n, 32), kSms * 6), kCheckThreads, 0, s)(a);
    count_launch();
  }
  p.end();
}

}  // namespace gwcp
