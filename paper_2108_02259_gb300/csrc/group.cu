// Grouping of the particles into work items (sm_103a): from each particle's
// key -- ((global page of its grid block) * max_bodies + body) << 6 | cell in
// the block -- to the sorted order, the items (pieces of the runs of one body
// in one grid block), the active grid blocks and the page table.
//
// Two ways there.  By sorting (sort.cu), then k_runs: any keys, stable, so the
// order is the same in every run (the deterministic mode, the first step of a
// context, boxes much larger than their particles).  By counting, once the
// page-table boxes and the number of (block, body) pairs are known from the
// step before:
//
//   k_cells    (kernels.cu) flags each particle's (block, body) pair
//   k_pairs    numbers the flagged pairs
//   k_rank     a particle's rank in its cell: one atomic on the cell's count
//   k_offsets  16 pairs a CTA: first positions of their cells (a scan over
//              1,024 cells, one atomic for the CTA's share of the order), their
//              items, and the blocks their stencils reach
//   k_place    the particle's position: first position of its cell + rank
//
// A pair's cells are consecutive and in order, as the transfer kernel needs;
// the order of the particles in a cell is left to the atomics (node sums are
// atomics as well).  Pairs come in the order of their pages from kOrderedGroup
// particles on, where CTAs that number them look back at the CTAs before;
// below, one atomic per CTA gives it the next free place.  Four short launches in
// the place of a histogram, three radix passes, two scans of three launches and
// three item kernels: every one of those waits for the one before and reads or
// writes all keys.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "apic_internal.h"

namespace apic {

#ifdef APIC_DEBUG_BOUNDS
__device__ unsigned g_dbg_group;  // bounds-check bits of this translation unit
namespace {
__device__ __forceinline__ void dbg_record(unsigned bit) { atomicOr(&g_dbg_group, bit); }
}  // namespace
#endif

unsigned group_debug_flags(int clear) {
#ifdef APIC_DEBUG_BOUNDS
  unsigned v = 0;
  if (cudaMemcpyFromSymbol(&v, g_dbg_group, sizeof(v)) != cudaSuccess) return ~0u;
  if (clear) {
    const unsigned z = 0;
    if (cudaMemcpyToSymbol(g_dbg_group, &z, sizeof(z)) != cudaSuccess) return ~0u;
  }
  return v;
#else
  (void)clear;
  return 0;
#endif
}

namespace {

constexpr int kGroupThreads = 256;
constexpr int kGroupWarps = kGroupThreads / 32;

// Exclusive sum of one value per thread over the CTA; *total the CTA's sum.
// warp_tot holds kGroupWarps ints; ends with a barrier.
__device__ __forceinline__ int cta_exclusive(int x, int* warp_tot, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[w] = incl;
  __syncthreads();
  int before = 0, sum = 0;
#pragma unroll
  for (int q = 0; q < kGroupWarps; ++q) {
    const int t = warp_tot[q];
    if (q < w) before += t;
    sum += t;
  }
  __syncthreads();
  *total = sum;
  return before + incl - x;
}

// The sum of the totals of the CTAs before this one (tile: its number in the
// order of starting), by decoupled look-back over 64-bit status words: a CTA
// publishes its own total, adds up the totals before it 32 at a time back to
// the nearest full prefix, and publishes its prefix.  Called by one whole
// warp.  A word carries its two flag bits with its value, so relaxed accesses
// are enough.  A CTA waits only for CTAs that started before it, each wait is
// bounded, and a CTA that gives up sets `gave_up` in the error word (the host
// fails the call) and publishes all the same, so that no later CTA waits for
// it.  What it returns, and so every later prefix, is then too small: places
// drawn from it overlap but stay inside the tables.  Pairs numbered from it
// leave numbers without an owner, whose entries and counts nothing has
// written, so the kernels after k_pairs do nothing (kErrWaits).
constexpr unsigned long long kOwnTotal = 1ull << 62, kFullPrefix = 2ull << 62, kStatusValue = kOwnTotal - 1ull;
constexpr int kLookbackSpins = 1 << 20;
#ifdef APIC_DEBUG_BOUNDS
__device__ int g_dbg_wait[2] = {kLookbackSpins, kLookbackSpins};  // (apic_debug_wait_limit)
__device__ __forceinline__ int wait_limit(int gave_up) { return g_dbg_wait[gave_up == kErrPairWait ? 0 : 1]; }
#else
__device__ __forceinline__ int wait_limit(int) { return kLookbackSpins; }
#endif
__device__ __forceinline__ void st_word(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long look_back(unsigned long long* status, int tile, unsigned long long total,
                                                        int* err, int gave_up) {
  const int lane = threadIdx.x & 31;
  const int limit = wait_limit(gave_up);
  if (lane == 0) st_word(status + tile, (tile == 0 ? kFullPrefix : kOwnTotal) | total);
  unsigned long long before = 0;
  for (int t0 = tile - 1; t0 >= 0; t0 -= 32) {
    unsigned long long v = kFullPrefix;  // (lanes before the first tile)
    if (t0 - lane >= 0) {
      v = ld_word(status + t0 - lane);
      for (int spins = 0; limit < 0 || (v & ~kStatusValue) == 0ull; ++spins) {
        if (spins > limit) {
          atomicOr(err, gave_up);
          v = kFullPrefix;
          break;
        }
        __nanosleep(32);
        v = ld_word(status + t0 - lane);
      }
    }
    const unsigned full = __ballot_sync(0xffffffffu, (v & kFullPrefix) != 0ull);
    const int stop = full ? __ffs(full) - 1 : 31;  // nearest full prefix
    unsigned long long x = lane <= stop ? v & kStatusValue : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    before += x;
    if (full) break;
  }
  if (lane == 0 && tile > 0) st_word(status + tile, kFullPrefix | ((before + total) & kStatusValue));
  return before;
}

// The blocks that a particle's stencil reaches.  Along an axis, from cell l of
// its block B (bits 0, 1, 2: B-1, B, B+1): B-1 when l = 0, B+1 when l >= 2.  Of
// the 3x3x3 blocks around B, one bit each, every combination of the axes' (so
// the OR over cells is exact however the particles are divided between threads,
// and a step has as many active blocks by sorting as by counting).
__device__ __forceinline__ unsigned axis_reach(unsigned l) { return 2u | (l == 0 ? 1u : 0u) | (l >= 2 ? 4u : 0u); }
__device__ __forceinline__ unsigned reach(unsigned x, unsigned y, unsigned z) {
  const unsigned xy = x * ((y & 1u) | (y & 2u) << 2 | (y & 4u) << 4);
  return xy * ((z & 1u) | (z & 2u) << 8 | (z & 4u) << 16);
}

// Flag neighbour q (of the 3x3x3 blocks around the block at page gpage) if its
// particles reach it.  Every particle block keeps a one-block margin inside its
// scene's box, so the page stays in the box.
__device__ __forceinline__ void mark_neighbour(int q, unsigned reached, long long gpage, const Box& box, int* flags,
                                               int64_t n_pages) {
  const int dx = q % 3 - 1, dy = (q / 3) % 3 - 1, dz = q / 9 - 1;
  const long long page = gpage + ((long long)dz * box.ny + dy) * box.nx + dx;
  if (((reached >> q) & 1u) && APIC_DBG_CHECK(page >= 0 && page < n_pages, kDbgPage)) flags[page] = 1;
}

// Item j of the k = ceil(len / chunk) items of a run of len particles from
// sorted position s: items are cut at whole warps.  Of the run's W = ceil(len
// / 32) warps, item j takes [floor(j W / k), floor((j + 1) W / k)), so sizes
// differ by at most one warp and only a run's last warp is partly filled (a
// cut into equal particle counts left the last warp of every item partly
// filled, and phases 1 and 2 of the transfer cost the same for a partial warp
// as for a full one: 4.086 -> 4.041 ms a step at 4,000,000 nodes).  chunk is a
// multiple of 32, so W <= k chunk / 32 and no item exceeds chunk.
__device__ __forceinline__ void write_item(int j, int k, int s, int len, int o, int4 info, int* item_start,
                                           int4* item_info, int64_t n) {
  const long long W = (len + 31) >> 5;
  const int a = (int)(j * W / k) * 32, b = min((int)((j + 1) * W / k) * 32, len);
  // (there are at most as many items as particles)
  if (!APIC_DBG_CHECK(o + j >= 0 && o + j < n && s >= 0 && s + b <= n && a < b, kDbgItem)) return;
  item_start[o + j] = s + a;
  info.w = b - a;
  item_info[o + j] = info;
}

// Work items and active blocks from the sorted keys.  A run is a maximal
// range of equal (grid block, body).  A CTA takes 1,024 keys, a warp four
// groups of 32: a group's run heads come from a ballot, a run's end is the
// next head of the group or, for the group's last run, a 32-way search over
// the keys that follow; one atomic per CTA draws its items' places, so items
// come out in nearly sorted order.  Each group also flags the blocks that its
// particles' stencils reach.
constexpr int kRunGroups = 4;
template <class K>
__global__ void __launch_bounds__(kGroupThreads)
    k_runs(int64_t n, const K* __restrict__ keys, int chunk, int max_bodies, const SceneDev* __restrict__ sc, int ns,
           int* item_start, int4* item_info, DevScalars* ds, int* flags, int64_t n_pages) {
  __shared__ int warp_tot[kGroupWarps];
  __shared__ int s_items;
  if (ds->err & kErrWaits) return;  // the keys may not be sorted, nor keys of this call
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t base = ((int64_t)blockIdx.x * kGroupWarps + w) * (32 * kRunGroups);
  int end[kRunGroups], my = 0, runs = 0;
#pragma unroll
  for (int r = 0; r < kRunGroups; ++r) end[r] = 0;
#pragma unroll
  for (int r = 0; r < kRunGroups; ++r) {
    const int64_t s = base + 32 * r + lane;
    const bool in = s < n;
    const K key = in ? keys[s] : K(0);
    const K q = key >> 6;
    K before = __shfl_up_sync(0xffffffffu, q, 1);
    if (lane == 0 && in && s > 0) before = keys[s - 1] >> 6;
    const bool head = in && (s == 0 || before != q);
    const unsigned valid = __ballot_sync(0xffffffffu, in);
    const unsigned heads = __ballot_sync(0xffffffffu, head);
    if (valid == 0) break;  // (uniform over the warp)
    // blocks reached, segment by segment (a segment: lanes of one run)
    const unsigned loc = (unsigned)(key & 63);
    const unsigned mine = in ? reach(axis_reach(loc & 3), axis_reach((loc >> 2) & 3), axis_reach(loc >> 4)) : 0u;
    for (unsigned starts = heads | 1u; starts != 0u; starts &= starts - 1u) {
      const int a = __ffs(starts) - 1;
      const unsigned above = heads & ~((2u << a) - 1u);
      const int b = above ? __ffs(above) - 1 : 32;
      const unsigned seg = __reduce_or_sync(0xffffffffu, lane >= a && lane < b ? mine : 0u);
      const K qa = __shfl_sync(0xffffffffu, q, a);
      const long long gpage = (long long)(qa / (K)max_bodies);
      const SceneDev& S = sc[scene_of_page(sc, ns, gpage)];
      if (lane < 27) mark_neighbour(lane, seg, gpage, S.box, flags, n_pages);
    }
    if (heads == 0) continue;
    const unsigned above = heads & ~((2u << lane) - 1u);
    if (head && above) end[r] = (int)(base + 32 * r + __ffs(above) - 1);
    // the group's last run: 32 probes a round, widening while all are equal
    const int last = 31 - __clz(heads);
    const K ql = __shfl_sync(0xffffffffu, q, last);
    int64_t lo = base + 32 * r + (32 - __clz(__ballot_sync(0xffffffffu, in && q == ql)));
    if (lo == base + 32 * r + 32) {
      int64_t step = 1;
      while (true) {
        const int64_t probe = lo + step * (lane + 1) - 1;
        const int eq = __popc(__ballot_sync(0xffffffffu, probe < n && (keys[probe < n ? probe : 0] >> 6) == ql));
        lo += step * eq;
        if (eq == 32) {
          if (step < (int64_t(1) << 20)) step *= 32;
        } else if (step == 1) {
          break;
        } else {
          step /= 32;
        }
      }
    }
    if (lane == last) end[r] = (int)lo;
    if (head) {
      my += (end[r] - (int)s + chunk - 1) / chunk;
      ++runs;
    }
  }
  int total;
  const int o0 = cta_exclusive(my, warp_tot, &total);
  if (threadIdx.x == 0) s_items = total > 0 ? atomicAdd(&ds->n_items, total) : 0;
  const int wr = __reduce_add_sync(0xffffffffu, runs);
  if (lane == 0 && wr > 0) atomicAdd(&ds->n_runs, wr);
  __syncthreads();
  int o = s_items + o0;
#pragma unroll
  for (int r = 0; r < kRunGroups; ++r) {
    // the warp writes its runs' items together, run by run
    for (unsigned todo = __ballot_sync(0xffffffffu, end[r] > 0); todo != 0u; todo &= todo - 1u) {
      const int a = __ffs(todo) - 1;
      const int s = (int)(base + 32 * r + a);
      const int len = __shfl_sync(0xffffffffu, end[r], a) - s;
      const int k = (len + chunk - 1) / chunk;
      const int oa = __shfl_sync(0xffffffffu, o, a);
      const K q = keys[s] >> 6;
      const long long gpage = (long long)(q / (K)max_bodies);
      const int4 info = make_int4((int)gpage, (int)(q % (K)max_bodies), scene_of_page(sc, ns, gpage), 0);
      for (int j = lane; j < k; j += 32) write_item(j, k, s, len, oa, info, item_start, item_info, n);
      if (lane == a) o += k;
    }
  }
}

// Number the flagged (block, body) pairs: pairs[e] = the pair's number (in
// place of its flag), and its cell counts cleared.  A pair beyond `cap` (more
// pairs than the step before left room for) is counted, and its particles go
// to pair 0: the host sizes afresh (kErrPairs).
__global__ void __launch_bounds__(kGroupThreads)
    k_pairs(int64_t n_entries, int* pairs, int cap, int* pair_entry, int* cnt, DevScalars* ds,
            unsigned long long* status) {
  __shared__ int warp_tot[kGroupWarps];
  __shared__ int s_base, s_tile;
  int tile = blockIdx.x;
  if (status) {
    if (threadIdx.x == 0) s_tile = atomicAdd(&ds->ticket_pairs, 1);
    __syncthreads();
    tile = s_tile;
  }
  const int64_t e0 = ((int64_t)tile * kGroupThreads + threadIdx.x) * 4;
  int4 f = make_int4(0, 0, 0, 0);
  if (e0 < n_entries) f = *reinterpret_cast<const int4*>(pairs + e0);  // (the array is padded to whole int4)
  const int fl[4] = {f.x, f.y, f.z, f.w};
  int mine = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) mine += fl[j] != 0;
  int total;
  int id = cta_exclusive(mine, warp_tot, &total);
  if (status) {
    if (threadIdx.x < 32) {
      const int before = (int)look_back(status, tile, (unsigned long long)total, &ds->err, kErrPairWait);
      if (threadIdx.x == 0) s_base = before;
      if (threadIdx.x == 0 && total > 0) atomicAdd(&ds->n_runs, total);
    }
  } else if (threadIdx.x == 0) {
    s_base = total > 0 ? atomicAdd(&ds->n_runs, total) : 0;
  }
  if (total == 0) return;  // (uniform over the CTA)
  __syncthreads();
  if (threadIdx.x == 0 && s_base + total > cap) atomicOr(&ds->err, kErrPairs);
  const int base = s_base;
  id += base;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (fl[j]) {
      if (id < cap && APIC_DBG_CHECK(id >= 0 && e0 + j < n_entries, kDbgPair)) pair_entry[id] = (int)(e0 + j);
      pairs[e0 + j] = id < cap ? id : 0;
      ++id;
    }
  const int lim = min(base + total, cap) - base;
  int4* c4 = reinterpret_cast<int4*>(cnt + (int64_t)base * 64);
  for (int i = threadIdx.x; i < lim * 16; i += kGroupThreads) c4[i] = make_int4(0, 0, 0, 0);
}

// Each particle's cell (pair * 64 + cell in block) and its rank in it.
template <class K>
__global__ void __launch_bounds__(kGroupThreads)
    k_rank(int64_t n, const K* __restrict__ keys, const int* __restrict__ pairs, int64_t n_entries, int cap,
           int* __restrict__ cnt, int* __restrict__ slot, int* __restrict__ rank, const int* __restrict__ err) {
  const int64_t i = (int64_t)blockIdx.x * kGroupThreads + threadIdx.x;
  if (i >= n) return;
  const int e = err ? *err : 0;  // (both loads in flight: these launches are short)
  const K key = keys[i];
  if (e & kErrWaits) return;
  if (!APIC_DBG_CHECK((int64_t)(key >> 6) < n_entries, kDbgPair)) return;
  const int pair = pairs[key >> 6];
  if (!APIC_DBG_CHECK(pair >= 0 && pair < cap, kDbgPair)) return;
  const int c = pair * 64 + (int)(key & 63);
  slot[i] = c;
  rank[i] = atomicAdd(&cnt[c], 1);
}

// 16 pairs a CTA, 16 threads a pair, 4 cells a thread: counts to first
// positions (in place), items, and the blocks the pair's cells reach; the
// pair's flag is cleared.
__global__ void __launch_bounds__(kGroupThreads)
    k_offsets(int64_t n, int64_t n_entries, int cap, const int* __restrict__ pair_entry, int* __restrict__ pairs,
              int* __restrict__ cnt, int chunk, int max_bodies, const SceneDev* __restrict__ sc, int ns,
              int* item_start, int4* item_info, DevScalars* ds, int* flags, int64_t n_pages,
              unsigned long long* status) {
  constexpr int kPairs = kGroupThreads / 16;
  __shared__ int warp_tot[kGroupWarps];
  __shared__ int s_k[kPairs], s_o[kPairs];
  __shared__ int s_base, s_items, s_total, s_tile;
  const int e = status ? ds->err : 0, n_pairs = min(ds->n_runs, cap);
  if (e & kErrPairWait) return;  // (set by an earlier launch only, so the whole grid leaves)
  int tile = blockIdx.x;
  if (status) {
    if (threadIdx.x == 0) s_tile = atomicAdd(&ds->ticket_offsets, 1);
    __syncthreads();
    tile = s_tile;
  }
  const int pl = threadIdx.x >> 4, l = threadIdx.x & 15;  // pair in the CTA, thread of the pair
  const int pair = tile * kPairs + pl;
  if (tile * kPairs >= n_pairs) return;  // (uniform over the CTA; no later tile has pairs)
  const bool live = pair < n_pairs;
  int4* c4 = reinterpret_cast<int4*>(cnt + (int64_t)pair * 64) + l;
  const int4 c = live ? *c4 : make_int4(0, 0, 0, 0);
  const int sum = c.x + c.y + c.z + c.w;
  int total;
  const int excl = cta_exclusive(sum, warp_tot, &total);
  // over the pair's 16 threads: its particles and the blocks they reach
  int len = sum;
  const unsigned x = (c.x ? axis_reach(0) : 0u) | (c.y ? axis_reach(1) : 0u) | (c.z ? axis_reach(2) : 0u) |
                     (c.w ? axis_reach(3) : 0u);
  unsigned reached = reach(x, axis_reach(l & 3), axis_reach(l >> 2));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    len += __shfl_xor_sync(0xffffffffu, len, o);
    reached |= __shfl_xor_sync(0xffffffffu, reached, o);
  }
  const int k = (len + chunk - 1) / chunk;
  if (l == 0) s_k[pl] = k;
  __syncthreads();
  if (threadIdx.x == 0) {
    int items = 0;
#pragma unroll
    for (int q = 0; q < kPairs; ++q) {
      s_o[q] = items;
      items += s_k[q];
    }
    s_total = items;
    const int at = atomicAdd(&ds->n_items, items);
    if (!status) {
      s_items = at;
      s_base = atomicAdd(&ds->n_placed, total);
    }
  }
  if (status && threadIdx.x < 32) {
    // items and particles together: at most 2^29 of each
    __syncwarp();
    const unsigned long long before =
        look_back(status, tile, ((unsigned long long)s_total << 31) | (unsigned long long)total, &ds->err,
                  kErrItemWait);
    if (threadIdx.x == 0) {
      s_items = (int)(before >> 31);
      s_base = (int)(before & 0x7fffffffull);
    }
  }
  __syncthreads();
  const int first = s_base + excl;
  if (live) *c4 = make_int4(first, first + c.x, first + c.x + c.y, first + c.x + c.y + c.z);
  if (!live || len == 0) return;
  // the pair's first position (its 16 threads are half a warp)
  const int s = __shfl_sync(0xffffu << (threadIdx.x & 16), first, threadIdx.x & 16);
  const unsigned entry = (unsigned)pair_entry[pair];
  if (!APIC_DBG_CHECK((int64_t)entry < n_entries, kDbgPair)) return;
  if (l == 0) pairs[entry] = 0;  // for the next step
  const unsigned gpage = entry / (unsigned)max_bodies;
  const int scene = scene_of_page(sc, ns, gpage);
  const int4 info = make_int4((int)gpage, (int)(entry % (unsigned)max_bodies), scene, 0);
  for (int j = l; j < k; j += 16) write_item(j, k, s, len, s_items + s_o[pl], info, item_start, item_info, n);
  const Box box = sc[scene].box;
  for (int q = l; q < 27; q += 16) mark_neighbour(q, reached, gpage, box, flags, n_pages);
}

// The particles' positions: (particle, cell in its block) in sorted order, one
// 8-byte record so that a particle costs one scattered store.
__global__ void __launch_bounds__(kGroupThreads)
    k_place(int64_t n, const int* __restrict__ slot, const int* __restrict__ rank, const int* __restrict__ first,
            int2* __restrict__ placed, const int* __restrict__ err) {
  const int64_t i = (int64_t)blockIdx.x * kGroupThreads + threadIdx.x;
  if (i >= n) return;
  const int e = err ? *err : 0, c = slot[i], r = rank[i];
  if (e & kErrWaits) return;
  const int at = first[c] + r;
  if (APIC_DBG_CHECK(at >= 0 && at < n, kDbgSortPos)) placed[at] = make_int2((int)i, c & 63);
}

// Compact ids of the flagged blocks: the list of their pages, each page's id
// (or -1) and their number.  One launch: a CTA's 1,024 pages are numbered in
// order from a place that one atomic draws.  Flags and status words are left
// clear for the next step, and the last CTA to finish writes the counters to
// the host's page-locked copy: a memset and a copy in the launch sequence cost
// 4-5 us each.
__global__ void __launch_bounds__(kGroupThreads)
    k_compact(int64_t n, int* __restrict__ flags, int* __restrict__ list, int* __restrict__ page, DevScalars* ds,
              unsigned long long* status, int64_t n_status, DevScalars* host) {
  __shared__ int warp_tot[kGroupWarps];
  __shared__ int s_base;
  for (int64_t i = (int64_t)blockIdx.x * kGroupThreads + threadIdx.x; i < n_status;
       i += (int64_t)gridDim.x * kGroupThreads)
    status[i] = 0ull;
  const int64_t i0 = ((int64_t)blockIdx.x * kGroupThreads + threadIdx.x) * 4;
  int fl[4], mine = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    fl[j] = i0 + j < n ? flags[i0 + j] : 0;
    mine += fl[j] != 0;
  }
  int total;
  int o = cta_exclusive(mine, warp_tot, &total);
  if (threadIdx.x == 0) s_base = total > 0 ? atomicAdd(&ds->n_blocks, total) : 0;
  __syncthreads();
  o += s_base;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (i0 + j >= n) break;
    page[i0 + j] = fl[j] ? o : -1;
    if (fl[j]) {
      flags[i0 + j] = 0;
      if (APIC_DBG_CHECK(o >= 0 && o < n, kDbgPage)) list[o] = (int)(i0 + j);
      ++o;
    }
  }
  if (host != nullptr && threadIdx.x == 0) {
    __threadfence();  // this CTA's share of n_blocks before its ticket
    if (atomicAdd(&ds->ticket_compact, 1) == (int)gridDim.x - 1) {
      __threadfence();
      const int4 a = __ldcg(reinterpret_cast<const int4*>(ds)), b = __ldcg(reinterpret_cast<const int4*>(ds) + 1);
      reinterpret_cast<int4*>(host)[0] = a;
      reinterpret_cast<int4*>(host)[1] = b;
    }
  }
}

inline unsigned blocks_for(int64_t n, int64_t per) { return (unsigned)((n + per - 1) / per); }

}  // namespace

template <class K>
cudaError_t launch_runs(int64_t n, const K* keys, int chunk, int max_bodies, const SceneDev* sc, int ns,
                        int* item_start, int4* item_info, DevScalars* ds, int* flags, int64_t n_pages,
                        cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (chunk < 32 || chunk > kChunk || chunk % 32 != 0) return cudaErrorInvalidValue;
  k_runs<K><<<blocks_for(n, (int64_t)kGroupThreads * kRunGroups), kGroupThreads, 0, s>>>(
      n, keys, chunk, max_bodies, sc, ns, item_start, item_info, ds, flags, n_pages);
  return cudaGetLastError();
}

cudaError_t launch_pairs(int64_t n_entries, int* pairs, int cap, int* pair_entry, int* cnt, DevScalars* ds,
                         unsigned long long* status, cudaStream_t s) {
  if (n_entries <= 0) return cudaSuccess;
  k_pairs<<<blocks_for(n_entries, kGroupThreads * 4), kGroupThreads, 0, s>>>(n_entries, pairs, cap, pair_entry, cnt,
                                                                              ds, status);
  return cudaGetLastError();
}

template <class K>
cudaError_t launch_rank(int64_t n, const K* keys, const int* pairs, int64_t n_entries, int cap, int* cnt, int* slot,
                        int* rank, const int* err, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_rank<K><<<blocks_for(n, kGroupThreads), kGroupThreads, 0, s>>>(n, keys, pairs, n_entries, cap, cnt, slot, rank,
                                                                    err);
  return cudaGetLastError();
}

cudaError_t launch_offsets(int64_t n, int64_t n_entries, int cap, const int* pair_entry, int* pairs, int* cnt,
                           int chunk, int max_bodies, const SceneDev* sc, int ns, int* item_start, int4* item_info,
                           DevScalars* ds, int* flags, int64_t n_pages, unsigned long long* status, cudaStream_t s) {
  if (cap <= 0) return cudaSuccess;
  if (chunk < 32 || chunk > kChunk || chunk % 32 != 0) return cudaErrorInvalidValue;
  k_offsets<<<blocks_for(cap, kGroupThreads / 16), kGroupThreads, 0, s>>>(
      n, n_entries, cap, pair_entry, pairs, cnt, chunk, max_bodies, sc, ns, item_start, item_info, ds, flags, n_pages,
      status);
  return cudaGetLastError();
}

cudaError_t group_debug_wait_limit(int pairs, int items) {
#ifdef APIC_DEBUG_BOUNDS
  const int v[2] = {pairs, items};
  return cudaMemcpyToSymbol(g_dbg_wait, v, sizeof(v));
#else
  (void)pairs;
  (void)items;
  return cudaErrorNotSupported;
#endif
}

int64_t group_status_words(int64_t n, int64_t n_entries, int cap) {
  return n < kOrderedGroup ? 0 : blocks_for(n_entries, kGroupThreads * 4) + blocks_for(cap, kGroupThreads / 16);
}
int64_t group_status_split(int64_t n_entries) { return blocks_for(n_entries, kGroupThreads * 4); }

cudaError_t launch_place(int64_t n, const int* slot, const int* rank, const int* first, int2* placed, const int* err,
                         cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_place<<<blocks_for(n, kGroupThreads), kGroupThreads, 0, s>>>(n, slot, rank, first, placed, err);
  return cudaGetLastError();
}

cudaError_t launch_compact(int64_t n, int* flags, int* list, int* page, DevScalars* ds, unsigned long long* status,
                           int64_t n_status, DevScalars* host, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_compact<<<blocks_for(n, kGroupThreads * 4), kGroupThreads, 0, s>>>(n, flags, list, page, ds, status, n_status,
                                                                        host);
  return cudaGetLastError();
}

template cudaError_t launch_runs<uint32_t>(int64_t, const uint32_t*, int, int, const SceneDev*, int, int*, int4*,
                                           DevScalars*, int*, int64_t, cudaStream_t);
template cudaError_t launch_runs<uint64_t>(int64_t, const uint64_t*, int, int, const SceneDev*, int, int*, int4*,
                                           DevScalars*, int*, int64_t, cudaStream_t);
template cudaError_t launch_rank<uint32_t>(int64_t, const uint32_t*, const int*, int64_t, int, int*, int*, int*,
                                           const int*, cudaStream_t);
template cudaError_t launch_rank<uint64_t>(int64_t, const uint64_t*, const int*, int64_t, int, int*, int*, int*,
                                           const int*, cudaStream_t);

}  // namespace apic
