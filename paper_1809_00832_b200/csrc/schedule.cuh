// On-device ready-set construction for a forest given as child-index arrays.
//
// Paper, Section 4.1.1: an operation with no unresolved input is ready; when an operation
// completes, the operations that waited on it and have all inputs resolved become ready.  For a
// tree node this gives wavefront ("level") 0 for leaves and 1 + max(level of children) for
// internal nodes.  Section 4.1.2: every invocation keeps a pointer to its caller -> parent[].
// The ready order reported to the caller is canonical: ascending (level, node id).
//
// The schedulers of one CTA and of one cluster, as device functions: they are kernels of their own (schedule.cu), and the
// first cluster of the launch whose other clusters evaluate trees meanwhile (trees_tc.cu).
#pragma once

#include <stddef.h>

#include "common.cuh"

namespace tl {
namespace {

constexpr int kSingleThreads = 1024;
constexpr int kSingleWarps = kSingleThreads / 32;
// the dependency words share their shared memory with what comes after them: the radix histogram
// (256 x 32 ints) or the per-thread level counts of the few-levels placement (32 x 1024 uint16)
constexpr size_t kSingleScratch = 65536;
constexpr unsigned kWarpMask = 0xffffffffu;

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Node check shared by both paths.  Returns 0, or the error code.  is_leaf is set for valid nodes.
__device__ __forceinline__ int check_node(int n, int k, int l, int r, const int* token, int vocab,
                                          bool* is_leaf) {
  if (l < 0 && r < 0) {
    *is_leaf = true;
    if (l != -1 || r != -1) return TREELSTM_ERR_INVALID_FOREST;
    int t = token[k];
    if (t < 0 || t >= vocab) return TREELSTM_ERR_TOKEN_OUT_OF_RANGE;
    return 0;
  }
  *is_leaf = false;
  if (l < 0 || r < 0 || l >= n || r >= n || l == r || l == k || r == k)
    return TREELSTM_ERR_INVALID_FOREST;
  return 0;
}

// ------------------------------------------------------------------------------------------ //
// Stable counting pass executed by one CTA of 32 warps over `n` items.
// Item r of the source sequence is src ? src[r] : r.  key(item) in [0, 256).  Items are written
// to dst ordered by key, ties in source order.  hist is shared memory [256][32] ints.
// After the scan step, bin_starts[b] (b < n_bin_starts) receives the position of the first item
// with key b.
// ------------------------------------------------------------------------------------------ //
struct NoPlace {
  __device__ void operator()(int, int) const {}
};

template <class KeyFn, class PlaceFn = NoPlace>
__device__ void block_counting_pass(int n, const int* src, int* dst, KeyFn key, int* hist,
                                    int* scan_tmp, int* bin_starts, int n_bin_starts,
                                    PlaceFn place = NoPlace()) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < kRadixBins * kSingleWarps; i += kSingleThreads) hist[i] = 0;
  __syncthreads();
  int per_warp = (n + kSingleWarps - 1) / kSingleWarps;
  per_warp = (per_warp + 31) & ~31;
  const int begin = min(n, warp * per_warp), end = min(n, begin + per_warp);
  for (int r0 = begin; r0 < end; r0 += 32) {   // one add per distinct key of the 32 items
    const int r = r0 + lane;
    const bool valid = r < end;
    const unsigned act = __ballot_sync(kWarpMask, valid);
    if (valid) {
      const int k = key(src ? src[r] : r);
      const unsigned peers = __match_any_sync(act, k);
      if (lane == __ffs(peers) - 1) hist[k * kSingleWarps + warp] += __popc(peers);
    }
    __syncwarp();
  }
  __syncthreads();
  // exclusive scan of hist in (bin-major, warp-minor) order: 8 consecutive entries per thread
  {
    constexpr int kPer = kRadixBins * kSingleWarps / kSingleThreads;  // 8
    int v[kPer], sum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) { v[j] = hist[tid * kPer + j]; sum += v[j]; }
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      int t = __shfl_up_sync(kWarpMask, incl, d);
      if (lane >= d) incl += t;
    }
    if (lane == 31) scan_tmp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      int w = scan_tmp[lane], wi = w;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        int t = __shfl_up_sync(kWarpMask, wi, d);
        if (lane >= d) wi += t;
      }
      scan_tmp[lane] = wi - w;
    }
    __syncthreads();
    int run = scan_tmp[warp] + incl - sum;
#pragma unroll
    for (int j = 0; j < kPer; ++j) { hist[tid * kPer + j] = run; run += v[j]; }
  }
  __syncthreads();
  for (int b = tid; b < n_bin_starts; b += kSingleThreads) bin_starts[b] = hist[b * kSingleWarps];
  __syncthreads();
  for (int r0 = begin; r0 < end; r0 += 32) {
    const int r = r0 + lane;
    const bool valid = r < end;
    const unsigned act = __ballot_sync(kWarpMask, valid);
    int item = 0, k = 0, base = 0;
    unsigned peers = 0;
    if (valid) {
      item = src ? src[r] : r;
      k = key(item);
      peers = __match_any_sync(act, k);
      base = hist[k * kSingleWarps + warp];
    }
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) hist[k * kSingleWarps + warp] = base + __popc(peers);
    __syncwarp();
    if (valid) {
      const int pos = base + __popc(peers & lanemask_lt());
      dst[pos] = item;
      place(pos, item);
    }
  }
  __syncthreads();
}

// Ids of the items with flag(item) set, in ascending order, to dst; returns their number to every
// thread.  One CTA of 32 warps; warp w owns a contiguous range of ids.
template <class FlagFn, class PlaceFn = NoPlace>
__device__ int block_compact(int n, int* dst, FlagFn flag, int* scan_tmp, PlaceFn place = NoPlace()) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int per_warp = (n + kSingleWarps - 1) / kSingleWarps;
  per_warp = (per_warp + 31) & ~31;
  const int begin = min(n, warp * per_warp), end = min(n, begin + per_warp);
  int count = 0;
  for (int r0 = begin; r0 < end; r0 += 32) {
    const int r = r0 + lane;
    count += __popc(__ballot_sync(kWarpMask, r < end && flag(r)));
  }
  __syncthreads();
  if (lane == 0) scan_tmp[warp] = count;
  __syncthreads();
  int total = 0, base = 0;
  for (int w2 = 0; w2 < kSingleWarps; ++w2) {
    const int c = scan_tmp[w2];
    if (w2 < warp) base += c;
    total += c;
  }
  for (int r0 = begin; r0 < end; r0 += 32) {
    const int r = r0 + lane;
    const bool f = r < end && flag(r);
    const unsigned m = __ballot_sync(kWarpMask, f);
    if (f) {
      const int idx = base + __popc(m & lanemask_lt());
      dst[idx] = r;
      place(idx, r);
    }
    base += __popc(m);
  }
  __syncthreads();
  return total;
}

// Ready order, wavefront boundaries and roots in one go for forests of at most 32 wavefronts (the
// usual case: depth grows with the logarithm of the sentence length).  One CTA of 1024 threads;
// thread t owns the contiguous ids [t * npt, (t + 1) * npt).  tab[L][t] (uint16, n_levels x 1024: 2 KB of
// shared memory per wavefront) first counts the thread's nodes of level L, then warp L turns row L into its
// exclusive prefix over the threads, and finally thread t hands out positions level_start[L] +
// tab[L][t]++ to its nodes in ascending id - ascending (level, id) overall, with no key matching at
// all.  The positions are scattered into a shared-memory copy of the order (uint16 ids, `staged`) and
// go out to global memory as whole lines afterwards: one SM cannot afford 4-byte stores to n
// different sectors.  Output as the general path: order[], level_offset[0 .. n_levels), roots[] by
// ascending id; returns the number of roots to every thread.  scan_tmp: shared int[32].
__device__ int place_few_levels(int n, int n_levels, const unsigned short* lv16, int* order, int* level_offset,
                                int* roots, unsigned short* tab, unsigned short* staged, int* scan_tmp,
                                int* stamps) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#ifdef TREELSTM_TRACE
  const long long t_in = clock64();
#define TL_PLACE_STAMP(i) do { if (tid == 0 && stamps) stamps[i] = (int)(clock64() - t_in); } while (0)
#else
  (void)stamps;
#define TL_PLACE_STAMP(i) do { } while (0)
#endif
  __shared__ int s_level_start[32];
  __shared__ int s_root_total;
  const int npt = ((n + kSingleThreads - 1) / kSingleThreads) | 1;   // odd: the threads' ranges start in different banks
  const int k0 = min(n, tid * npt), k1 = min(n, k0 + npt);
  {
    uint4* z = reinterpret_cast<uint4*>(tab);                   // 2 KB = 128 pieces of 16 bytes per wavefront
    for (int i = tid; i < n_levels * kSingleThreads * 2 / 16; i += kSingleThreads) z[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  __syncthreads();
  TL_PLACE_STAMP(0);
  int my_roots = 0;
  for (int k = k0; k < k1; ++k) {
    const unsigned short v = lv16[k];
    tab[(v & 0x7FFF) * kSingleThreads + tid] += 1;
    my_roots += v >> 15;
  }
  __syncthreads();
  TL_PLACE_STAMP(1);
  // row L -> exclusive prefix over the threads (warp L; lane j takes the 32 threads 32 j .. 32 j + 31)
  if (warp < n_levels) {
    unsigned short* row = tab + warp * kSingleThreads + lane * 32;
    unsigned short v[32];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 x = reinterpret_cast<const uint4*>(row)[q];
      const unsigned int w4[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) { v[q * 8 + 2 * j] = (unsigned short)(w4[j] & 0xFFFFu); v[q * 8 + 2 * j + 1] = (unsigned short)(w4[j] >> 16); }
    }
    int sum = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) { const int c = v[j]; v[j] = (unsigned short)sum; sum += c; }
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(kWarpMask, incl, d);
      if (lane >= d) incl += t;
    }
    const int base = incl - sum;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      unsigned int w4[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        w4[j] = (unsigned int)(unsigned short)(v[q * 8 + 2 * j] + base) | ((unsigned int)(unsigned short)(v[q * 8 + 2 * j + 1] + base) << 16);
      reinterpret_cast<uint4*>(row)[q] = make_uint4(w4[0], w4[1], w4[2], w4[3]);
    }
    if (lane == 31) scan_tmp[warp] = incl;                      // nodes of level `warp`
  }
  __syncthreads();
  TL_PLACE_STAMP(2);
  // level starts (warp 0) and the roots' prefix over the threads (all warps, one value per thread)
  if (warp == 0) {
    const int c = lane < n_levels ? scan_tmp[lane] : 0;
    int incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(kWarpMask, incl, d);
      if (lane >= d) incl += t;
    }
    s_level_start[lane] = incl - c;
    if (lane < n_levels) level_offset[lane] = incl - c;
  }
  __syncthreads();
  int rincl = my_roots;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(kWarpMask, rincl, d);
    if (lane >= d) rincl += t;
  }
  if (lane == 31) scan_tmp[warp] = rincl;
  __syncthreads();
  if (warp == 0) {
    const int c = scan_tmp[lane];
    int incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(kWarpMask, incl, d);
      if (lane >= d) incl += t;
    }
    scan_tmp[lane] = incl - c;
    if (lane == 31) s_root_total = incl;
  }
  __syncthreads();
  TL_PLACE_STAMP(3);
  int rpos = scan_tmp[warp] + rincl - my_roots;
  for (int k = k0; k < k1; ++k) {
    const unsigned short v = lv16[k];
    const int lv = v & 0x7FFF;
    unsigned short* cell = tab + lv * kSingleThreads + tid;
    const int pos = s_level_start[lv] + *cell;
    *cell += 1;
    staged[pos] = (unsigned short)k;
    if (v >> 15) roots[rpos++] = k;
  }
  __syncthreads();
  TL_PLACE_STAMP(4);
  for (int i = tid; i < n; i += kSingleThreads) order[i] = staged[i];
  return s_root_total;
}

// A scheduler is a programmatic dependent of whatever is ahead of it on the stream (behind_last): it comes up while that ends, and reads, writes
// and lets go nothing before.  (The pointers pass through, so that no load moves ahead of the wait; and the arrays, which the kernel ahead may still write when
// this one has started, are not read as constant data.)
__device__ __forceinline__ void wait_for_last(const int*& left, const int*& right, const int*& token) {
  asm volatile("griddepcontrol.wait;" : "+l"(left), "+l"(right), "+l"(token) :: "memory");
}

__device__ __forceinline__ void clear_status(DevStatus* st, bool keep_choice) {
  const int word = (int)threadIdx.x;
  if (word < (int)(sizeof(DevStatus) / sizeof(int)) && !(keep_choice && word == (int)(offsetof(DevStatus, trees_fwd) / sizeof(int))))
    reinterpret_cast<int*>(st)[word] = 0;
}

// One CTA schedules the whole forest in shared memory (forests up to 32768 nodes).
//
// Dependency counters, as in Section 4.1.1: every internal node waits for two inputs.  A finished
// child swaps (its level + 1) into its caller's word; the child that finds the word empty was first
// and stops, the one that finds its sibling's entry knows both inputs are resolved, gives the caller
// level 1 + max and goes on upwards.  No global atomics, no grid-wide rounds.
//
// Dynamic shared memory: uint32 w[n] (dependency words; later the sort's scratch, at least 64 KB),
// uint16 par[n] (caller of each node, the return location of Section 4.1.2; later level | root
// flag), uint16 queue[n / 2] (start nodes of the climb), and with n_parts > 0 uint16 lab[n].
//
// n_parts > 0 additionally deals the trees out to n_parts sub-forests (trees are independent,
// Section 2.2): every node learns the root of its tree by pointer jumping over the caller links,
// the t-th root (ascending node id) goes to sub-forest t mod n_parts, and part_order receives the
// node ids by ascending (sub-forest, level, node id) with part_offset[0 .. n_parts] marking where
// each sub-forest starts.  slot[] (if given) is set to -1 for every node.
//
// Called by all kSingleThreads threads of one CTA.  keep_choice: the control block's word trees_fwd is another CTA's to write.
__device__ __forceinline__ void
schedule_single(unsigned char* smem, bool keep_choice, int n, const int* left, const int* right, const int* token,
                  int vocab, int* parent, int* level, int* order,
                  int* order_tmp, int* level_offset, int* roots, int* n_levels_out, DevStatus* st,
                  int n_parts, int* part_order, int* part_offset, int* slot, int cache_children) {
  const size_t w_bytes = (size_t)n * 4 > kSingleScratch ? (((size_t)n * 4 + 15) & ~(size_t)15) : kSingleScratch;
  unsigned int* w = reinterpret_cast<unsigned int*>(smem);
  int* hist = reinterpret_cast<int*>(smem);
  unsigned short* par = reinterpret_cast<unsigned short*>(smem + w_bytes);
  unsigned short* lv16 = par;
  unsigned short* queue = par + (((size_t)n + 7) & ~(size_t)7);   // start nodes of the climb, at most n / 2
  unsigned short* lab = reinterpret_cast<unsigned short*>(
      smem + w_bytes + ((((size_t)n * 2) + 15) & ~(size_t)15) + (((size_t)n + 15) & ~(size_t)15));
  // where shared memory allows (no sub-forest labels, forest small enough): both children of every node,
  // packed, so that the second look at them does not go back to global memory
  unsigned int* lr = cache_children ? reinterpret_cast<unsigned int*>(lab) : nullptr;
  __shared__ int scan_tmp[32];
  __shared__ int s_err, s_maxlevel, s_qhead, s_qtail;
  const int tid = threadIdx.x;
  constexpr unsigned short kNoParent = 0xFFFF;
  constexpr unsigned int kDone = 0x80000000u;
  clear_status(st, keep_choice);
#ifdef TREELSTM_TRACE
  // phase stamps of thread 0 (cycles since the start) in the unused words of the control block
  const long long t_start = clock64();
#define TL_SCHED_STAMP(i) do { if (tid == 0) st->pad[i] = (int)(clock64() - t_start); } while (0)
#else
#define TL_SCHED_STAMP(i) do { } while (0)
#endif
  if (tid == 0) { s_err = 0; s_maxlevel = 0; s_qhead = 0; s_qtail = 0; }
  for (int k = tid; k < n; k += kSingleThreads) { w[k] = 0; par[k] = kNoParent; }
  __syncthreads();
  // A kernel launched behind this one as its programmatic dependent may start now.  The part of it
  // that comes before its own wait for this grid reads nothing this grid writes, except that it
  // uses the (now cleared) control block: its barrier counter, and the status word this grid may
  // still set.
  if (tid == 0) {
    __threadfence();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  TL_SCHED_STAMP(0);   // cleared
  // validate; children record their caller; leaves are complete at once (level 0)
  // Node j of this thread is tid + j * 1024 (at most 32 per thread); leaf_bits remembers which are
  // leaves so that later passes need not look at the child arrays again.
  unsigned int leaf_bits = 0;
  for (int j0 = 0; j0 * kSingleThreads + tid < n; j0 += 8) {   // eight nodes per trip: loads first
    int l[8], r[8], t[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = tid + (j0 + j) * kSingleThreads;
      l[j] = k < n ? left[k] : -1;
      r[j] = k < n ? right[k] : -1;
      t[j] = k < n ? token[k] : 0;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = tid + (j0 + j) * kSingleThreads;
      if (k >= n) break;
      int err = 0;
      if (l[j] < 0 && r[j] < 0) {
        if (l[j] != -1 || r[j] != -1) err = TREELSTM_ERR_INVALID_FOREST;
        else if (t[j] < 0 || t[j] >= vocab) err = TREELSTM_ERR_TOKEN_OUT_OF_RANGE;
        else { w[k] = kDone; leaf_bits |= 1u << (j0 + j); }
      } else if (l[j] < 0 || r[j] < 0 || l[j] >= n || r[j] >= n || l[j] == r[j] || l[j] == k || r[j] == k) {
        err = TREELSTM_ERR_INVALID_FOREST;
      } else {
        par[l[j]] = (unsigned short)k;
        par[r[j]] = (unsigned short)k;
        if (lr) lr[k] = (unsigned int)l[j] | ((unsigned int)r[j] << 16);
      }
      if (err) atomicMin(&s_err, err);
    }
  }
  __syncthreads();
  TL_SCHED_STAMP(1);   // validated and linked
  if (s_err == 0) {
    // a child claimed by two callers kept only one of them: checked at the caller
    for (int j0 = 0; j0 * kSingleThreads + tid < n; j0 += 8) {
      int l[8], r[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int k = tid + (j0 + j) * kSingleThreads;
        const bool internal = k < n && !((leaf_bits >> (j0 + j)) & 1u);
        if (lr) {
          const unsigned int both = internal ? lr[k] : 0xFFFFFFFFu;
          l[j] = internal ? (int)(both & 0xFFFFu) : -1;
          r[j] = internal ? (int)(both >> 16) : -1;
        } else {
          l[j] = internal ? left[k] : -1;
          r[j] = internal ? right[k] : -1;
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int k = tid + (j0 + j) * kSingleThreads;
        if (l[j] >= 0 && (par[l[j]] != k || par[r[j]] != k)) atomicMin(&s_err, (int)TREELSTM_ERR_INVALID_FOREST);
      }
    }
    // Every leaf reports to its caller.  A caller whose second child reports here is complete
    // (level 1) and goes into the queue of nodes to climb from; climbing starts only after all
    // leaves have reported, so no climb waits for a leaf its owner has not reached yet.
    for (unsigned int bits = leaf_bits; bits; bits &= bits - 1) {
      const int k = tid + (__ffs(bits) - 1) * kSingleThreads;
      const unsigned short p = par[k];
      if (p == kNoParent) continue;
      if (atomicExch(&w[p], 1u) != 0) {         // both children are leaves
        w[p] = kDone | 1u;
        queue[atomicAdd(&s_qtail, 1)] = p;
      }
    }
  }
  __syncthreads();
  TL_SCHED_STAMP(2);   // links checked, leaves reported
  if (s_err == 0) {
    // Climb: threads take start nodes from the queue until it is empty.
    for (;;) {
      const int q = atomicAdd(&s_qhead, 1);
      if (q >= s_qtail) break;
      int cur = queue[q], lvl = 1;
      for (int step = 0; step < n; ++step) {   // a path to the root has fewer than n edges
        const unsigned short p = par[cur];
        if (p == kNoParent) break;
        const unsigned int old = atomicExch(&w[p], (unsigned int)lvl + 1u);
        if (old == 0) break;                   // sibling subtree still unresolved
        lvl = 1 + max(lvl, (int)old - 1);
        w[p] = kDone | (unsigned int)lvl;
        cur = p;
      }
    }
  }
  __syncthreads();
  TL_SCHED_STAMP(3);   // climbed
  int local_max = 0;
  if (s_err == 0) {
    for (int k = tid; k < n; k += kSingleThreads) {
      const unsigned int wk = w[k];
      if (!(wk & kDone)) atomicMin(&s_err, (int)TREELSTM_ERR_INVALID_FOREST);   // on a cycle: never ready
      const int lvl = (int)(wk & 0x7FFFu);
      const unsigned short pk = par[k];
      lv16[k] = (unsigned short)(lvl | (pk == kNoParent ? 0x8000 : 0));
      if (n_parts > 0) {
        lab[k] = pk == kNoParent ? (unsigned short)k : pk;   // start of the pointer jumping
        if (slot) slot[k] = -1;
      }
      level[k] = lvl;
      local_max = max(local_max, lvl);
    }
    atomicMax(&s_maxlevel, local_max);
  }
  __syncthreads();
  if (s_err != 0) {
    if (tid == 0) { report(st, s_err); *n_levels_out = 0; }
    return;
  }
  const int n_levels = n > 0 ? s_maxlevel + 1 : 0;
  TL_SCHED_STAMP(4);   // levels written
  // The few-levels placement needs 2 KB per wavefront for its counts and 2 n bytes for the staged
  // order: the packed children's shared memory (no longer needed) takes the latter, or what the
  // dependency words leave free behind the counts.
  const size_t tab_bytes = (size_t)n_levels * kSingleThreads * 2;
  unsigned short* staged = lr != nullptr ? reinterpret_cast<unsigned short*>(lr)
                           : (tab_bytes + (size_t)n * 2 <= w_bytes ? reinterpret_cast<unsigned short*>(smem + tab_bytes) : nullptr);
  if (n_levels <= 32 && n_parts == 0 && staged != nullptr) {
    const int n_roots = place_few_levels(n, n_levels, lv16, order, level_offset, roots,
                                         reinterpret_cast<unsigned short*>(smem), staged, scan_tmp, st->pad + 8);
    if (tid == 0) {
      level_offset[n_levels] = n; st->n_levels = n_levels; *n_levels_out = n_levels;
      st->n_roots = n_roots;
    }
    TL_SCHED_STAMP(5);   // ordered
    return;
  }
  // canonical ready order: LSD radix on the level, 8 bits per pass, ties by node id
  int passes = 1;
  while (passes < 4 && (n_levels - 1) >> (8 * passes)) ++passes;
  for (int p = 0; p < passes; ++p) {
    int* dst = ((passes - 1 - p) & 1) ? order_tmp : order;
    const int* src = p == 0 ? nullptr : (dst == order ? order_tmp : order);
    const int shift = 8 * p;
    block_counting_pass(n, src, dst, [=](int item) { return ((lv16[item] & 0x7FFF) >> shift) & 255; },
                        hist, scan_tmp, passes == 1 ? level_offset : nullptr, passes == 1 ? n_levels : 0);
  }
  if (passes > 1) {   // wavefront boundaries from the sorted order
    for (int r = tid; r < n; r += kSingleThreads) {
      const int a = lv16[order[r]] & 0x7FFF;
      if (r == 0 || (lv16[order[r - 1]] & 0x7FFF) != a) level_offset[a] = r;
    }
  }
  if (tid == 0) { level_offset[n_levels] = n; st->n_levels = n_levels; *n_levels_out = n_levels; }
  if (n_parts > 0) {
    // lab[k] = root of k's tree: every node replaces its link by its link's link until all links
    // end at a root (a root links to itself); ceil(log2(depth)) + 1 rounds.  Updates are made in
    // place: a link read while it is being advanced is still an ancestor.
    for (int round = 0; round < 17; ++round) {
      int changed = 0;
      for (int k = tid; k < n; k += kSingleThreads) {
        const unsigned short a = lab[k], b = lab[a];
        if (b != a) { lab[k] = b; changed = 1; }
      }
      if (!__syncthreads_or(changed)) break;
    }
  }
  // roots (nodes without a caller) in ascending node id; the t-th root takes sub-forest t mod n_parts
  const int n_roots = block_compact(n, roots, [=](int item) { return (lv16[item] & 0x8000) != 0; }, scan_tmp,
                                    [=](int idx, int item) { if (n_parts > 0) lab[item] = (unsigned short)(idx % n_parts); });
  if (tid == 0) st->n_roots = n_roots;
  if (n_parts > 0) {
    // every other node takes its root's sub-forest (its own entry is read by nobody else: links
    // end at roots only)
    for (int k = tid; k < n; k += kSingleThreads)
      if (!(lv16[k] & 0x8000)) lab[k] = lab[lab[k]];
    __syncthreads();
    // stable pass over the ready order by sub-forest: ascending (sub-forest, level, node id)
    block_counting_pass(n, order, part_order, [=](int item) { return (int)lab[item]; }, hist, scan_tmp,
                        part_offset, n_parts);
    if (tid == 0) part_offset[n_parts] = n;
  }
}

// ------------------------------------------------------------------------------------------ //
// One cluster schedules the whole forest in its shared memory.
//
// The same algorithm as the single CTA's, with the nodes dealt out to the CTAs in contiguous id ranges (a power of two,
// so that a node's CTA is a shift) and the links, reports and climbs going through distributed shared memory.  What
// bounds the single CTA is its issue slots - every node takes part in half a dozen passes - and it takes 31 us for
// 14 k nodes; here the longest climb counts: two round trips per level, 300 to 650 cycles depending on whether a
// tree's nodes lie in one CTA's range.  Measured (trace build, cycles): 14.6 k nodes, 15 levels 25 k (single CTA 57 k);
// 57 k nodes 30 k (before: ten launches, 145 us); of it linking 3 to 5 k, climbs 10 k, ordering 8 to 10 k.
//
// Order: LSD passes of kClBits bits.  A warp owns a contiguous run of positions of the pass's input and ranks its
// items 32 at a time by matching bins; a warp per bin turns the warps' counts into prefixes, the CTAs exchange their
// totals per bin.  The items are staged in the order of the CTA's places, so that the stores to global memory run
// along whole lines.
constexpr int kClBits = 6, kClBins = 1 << kClBits, kClMax = 16, kClGroups = 8;
constexpr int kClMaxPer = 32 * 32 * kClGroups;           // nodes per CTA: a warp keeps its items' ranks in registers
constexpr unsigned int kClDone = 0x80000000u, kClNone = 0xFFFFFFFFu;
struct ClSmem {                                          // behind it: uint32 state[per], caller[per], uint16 staged[per]
  int hist[kClBins + 1][33];                             // items of a bin per warp, then before the warp; last row: roots
  int totals[kClMax][kClBins + 1];                       // items of a bin per CTA
  int local[kClBins + 1];                                // first staged place of a bin
  int place[kClBins + 1];                                // place in the output minus staged place
  int scan[8];
  int err, max_level, qhead, qtail;
};
inline int cl_shift(int n, int cs) {
  int sh = 5;
  while (((long long)cs << sh) < n) ++sh;
  return sh;
}
inline size_t cl_smem_bytes(int sh) { return round_up_sz(sizeof(ClSmem), 16) + ((size_t)10 << sh); }
__device__ __forceinline__ uint32_t cl_addr(uint32_t smem_addr, unsigned rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr), "r"(rank));
  return a;
}
__device__ __forceinline__ unsigned int cl_ld(uint32_t a) {
  unsigned int v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cl_st(uint32_t a, unsigned int v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned int cl_exch(uint32_t a, unsigned int v) {
  unsigned int old;
  asm volatile("atom.shared::cluster.exch.b32 %0, [%1], %2;" : "=r"(old) : "r"(a), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ void cl_min(uint32_t a, int v) {
  asm volatile("red.shared::cluster.min.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_max(uint32_t a, int v) {
  asm volatile("red.shared::cluster.max.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Called by all threads of all CTAs of one cluster.
__device__ __forceinline__ void
schedule_cluster(unsigned char* cl_smem, bool keep_choice, int n, const int* left, const int* right, const int* token,
                   int vocab, int* level, int* order, int* order_tmp, int* level_offset, int* roots, int* n_levels_out,
                   DevStatus* st, int sh) {
  ClSmem& sm = *reinterpret_cast<ClSmem*>(cl_smem);
  uint32_t cs, rank;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(cs));
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = 1 << sh, base = (int)rank << sh, mine = max(0, min(per, n - base));
  unsigned int* const state = reinterpret_cast<unsigned int*>(cl_smem + (sizeof(ClSmem) + 15) / 16 * 16);
  unsigned int* const caller = state + per;
  unsigned short* const queue = reinterpret_cast<unsigned short*>(caller + per);   // leaves whose callers start a climb; later staged items
  const uint32_t state_addr = (uint32_t)__cvta_generic_to_shared(state), to_caller = 4u << sh;   // distance of the two words of a node
  const uint32_t err_addr = cl_addr((uint32_t)__cvta_generic_to_shared(&sm.err), 0), max_addr = cl_addr((uint32_t)__cvta_generic_to_shared(&sm.max_level), 0);
#ifdef TREELSTM_TRACE
  const long long t_start = clock64();
#define TL_CL_STAMP(i) do { if (tid == 0 && rank == 0) st->pad[i] = (int)(clock64() - t_start); } while (0)
#else
#define TL_CL_STAMP(i) do { } while (0)
#endif
  if (rank == 0) clear_status(st, keep_choice);
  if (tid == 0) { sm.err = 0; sm.max_level = 0; sm.qhead = 0; sm.qtail = 0; }
  for (int k = tid; k < mine; k += kSingleThreads) { state[k] = 0u; caller[k] = kClNone; }
  if (rank == 0) __threadfence();
  cl_sync();
  TL_CL_STAMP(0);   // cleared
  // a kernel launched behind this one as its programmatic dependent may start now (see k_schedule_single)
  if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  auto node_at = [&](unsigned k) { return cl_addr(state_addr + 4u * (k & (unsigned)(per - 1)), k >> sh); };
  // validate; a child's word gets its caller (a second caller finds the first one there)
  for (int k0 = tid; k0 < mine; k0 += 4 * kSingleThreads) {
    int l[4], r[4], t[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = k0 + j * kSingleThreads;
      l[j] = k < mine ? left[base + k] : -1;
      r[j] = k < mine ? right[base + k] : -1;
      t[j] = k < mine ? token[base + k] : 0;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = k0 + j * kSingleThreads, id = base + k;
      if (k >= mine) break;
      int err = 0;
      if (l[j] < 0 && r[j] < 0) {
        if (l[j] != -1 || r[j] != -1) err = TREELSTM_ERR_INVALID_FOREST;
        else if (t[j] < 0 || t[j] >= vocab) err = TREELSTM_ERR_TOKEN_OUT_OF_RANGE;
        else state[k] = kClDone;
      } else if (l[j] < 0 || r[j] < 0 || l[j] >= n || r[j] >= n || l[j] == r[j] || l[j] == id || r[j] == id) {
        err = TREELSTM_ERR_INVALID_FOREST;
      } else {
        const unsigned int a = cl_exch(node_at((unsigned)l[j]) + to_caller, (unsigned int)id), b = cl_exch(node_at((unsigned)r[j]) + to_caller, (unsigned int)id);
        if (a != kClNone || b != kClNone) err = TREELSTM_ERR_INVALID_FOREST;
      }
      if (err) cl_min(err_addr, err);
    }
  }
  cl_sync();
  TL_CL_STAMP(1);   // validated and linked
  if ((int)cl_ld(err_addr) == 0) {
    // every leaf reports to its caller; a caller whose second child reports here starts a climb
    for (int k = tid; k < mine; k += kSingleThreads) {
      const unsigned int p = caller[k];
      if (state[k] != kClDone || p == kClNone) continue;
      const uint32_t a = node_at(p);
      const unsigned int old = cl_exch(a, 1u);           // 1 + the level of the other child, if that was there first
      if (old != 0u) {
        cl_st(a, kClDone | old);
        queue[atomicAdd(&sm.qtail, 1)] = (unsigned short)k;
      }
    }
    __syncthreads();
    TL_CL_STAMP(2);   // leaves reported
    for (;;) {
      const int q = atomicAdd(&sm.qhead, 1);
      if (q >= sm.qtail) break;
      const uint32_t first = node_at(caller[queue[q]]);
      unsigned int lvl = cl_ld(first) & ~kClDone, p = cl_ld(first + to_caller);
      for (int step = 0; p != kClNone && step < n; ++step) {   // a path to the root has fewer than n edges
        const uint32_t a = node_at(p);
        const unsigned int old = cl_exch(a, lvl + 1u);
        if (old == 0u) break;                            // sibling subtree still unresolved
        lvl = 1u + max(lvl, old - 1u);
        cl_st(a, kClDone | lvl);
        p = cl_ld(a + to_caller);
      }
    }
  }
  TL_CL_STAMP(3);
  cl_sync();
  TL_CL_STAMP(4);   // climbed
  // A warp's contiguous run of positions, 32 at a time: its items (positions within the CTA) and their levels.
  const int wper = (((mine + 31) / 32) + 31) & ~31;
  const int w_begin = min(mine, warp * wper), w_end = min(mine, w_begin + wper);
  {
    int top = 0, bad = 0;
    for (int k = w_begin + lane; k < w_end; k += 32) {
      const unsigned int v = state[k];
      bad |= !(v & kClDone);                             // on a cycle: never ready
      const int lvl = (int)(v & ~kClDone);
      level[base + k] = lvl;
      top = max(top, lvl);
    }
    top = __reduce_max_sync(kWarpMask, top);
    if (lane == 0) cl_max(max_addr, top);
    if (bad) cl_min(err_addr, (int)TREELSTM_ERR_INVALID_FOREST);
  }
  for (int i = tid; i < (kClBins + 1) * 33; i += kSingleThreads) (&sm.hist[0][0])[i] = 0;
  cl_sync();
  const int err = (int)cl_ld(err_addr), n_levels = (int)cl_ld(max_addr) + 1;
  TL_CL_STAMP(5);   // levels written
  if (err != 0) {
    if (rank == 0 && tid == 0) { report(st, err); *n_levels_out = 0; }
    cl_sync();                                           // rank 0's words are read until here
    return;
  }
  int passes = 1;
  while ((n_levels - 1) >> (kClBits * passes)) ++passes;
  for (int pass = 0; pass < passes; ++pass) {
    int* const dst = ((passes - 1 - pass) & 1) ? order_tmp : order;
    const int* const src = pass == 0 ? nullptr : (dst == order ? order_tmp : order);
    const int shift = kClBits * pass, bins = min(kClBins, ((n_levels - 1) >> shift) + 1);
    if (pass > 0) {                                      // this CTA's items of the last pass's output and their levels
      for (int k = tid; k < mine; k += kSingleThreads) {
        const int item = *(volatile const int*)(src + base + k);
        state[k] = (unsigned int)*(volatile const int*)(level + item);
        caller[k] = (unsigned int)item;
      }
      for (int i = tid; i < (kClBins + 1) * 33; i += kSingleThreads) (&sm.hist[0][0])[i] = 0;
      __syncthreads();
    }
    // rank of every item among the warp's items of its bin (and of every root among the warp's roots)
    unsigned int ranks[kClGroups];                       // rank | bin << 16 | root rank << 23, per group of 32
    int warp_roots = 0;
#pragma unroll
    for (int g = 0; g < kClGroups; ++g) {
      const int k = w_begin + 32 * g + lane;
      ranks[g] = 0u;
      if (w_begin + 32 * g >= w_end) continue;           // the same for the whole warp
      const bool valid = k < w_end;
      const int bin = valid ? (int)((state[k] & ~kClDone) >> shift) & (kClBins - 1) : kClBins;
      const bool root = pass == 0 && valid && caller[k] == kClNone;
      const unsigned peers = __match_any_sync(kWarpMask, bin), rmask = __ballot_sync(kWarpMask, root);
      const int before = valid ? sm.hist[bin][warp] : 0;
      __syncwarp();
      if (valid && lane == __ffs(peers) - 1) sm.hist[bin][warp] = before + __popc(peers);
      ranks[g] = (unsigned)(before + __popc(peers & lanemask_lt())) | ((unsigned)bin << 16) |
                 ((unsigned)(warp_roots + __popc(rmask & lanemask_lt())) << 23);
      warp_roots += __popc(rmask);
      __syncwarp();
    }
    if (lane == 0) sm.hist[kClBins][warp] = warp_roots;
    __syncthreads();
    for (int b = warp; b <= kClBins; b += 32) {          // counts of the warps -> prefixes; the bin's total to every CTA
      if (b >= bins && b != kClBins) continue;
      const int v = sm.hist[b][lane];
      int incl = v;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(kWarpMask, incl, d);
        if (lane >= d) incl += t;
      }
      sm.hist[b][lane] = incl - v;
      const int total = __shfl_sync(kWarpMask, incl, 31);
      if (lane < (int)cs) cl_st(cl_addr((uint32_t)__cvta_generic_to_shared(&sm.totals[rank][b]), lane), (unsigned int)total);
    }
    TL_CL_STAMP(6);   // counted
    cl_sync();
    TL_CL_STAMP(7);
    // places: bins before it in the whole forest, then CTAs before this one
    if (warp < 2) {
      const int b = tid;
      int all = 0, before = 0;
#pragma unroll
      for (int c = 0; c < kClMax; ++c) {
        const int v = c < (int)cs && b < bins ? sm.totals[c][b] : 0;
        all += v;
        before += c < (int)rank ? v : 0;
      }
      const int own = b < bins ? sm.totals[rank][b] : 0;
      int ga = all, la = own;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int x = __shfl_up_sync(kWarpMask, ga, d), y = __shfl_up_sync(kWarpMask, la, d);
        if (lane >= d) { ga += x; la += y; }
      }
      if (tid == 31) { sm.scan[0] = ga; sm.scan[1] = la; }
      asm volatile("bar.sync 1, 64;" ::: "memory");
      const int first = ga - all + (warp ? sm.scan[0] : 0), local = la - own + (warp ? sm.scan[1] : 0);
      sm.local[b] = local;
      sm.place[b] = first + before - local;
      if (rank == 0 && passes == 1 && b < bins) level_offset[b] = first;
    } else if (warp == 2 && pass == 0) {
      const int v = lane < (int)cs ? sm.totals[lane][kClBins] : 0;
      const int before = __reduce_add_sync(kWarpMask, lane < (int)rank ? v : 0), all = __reduce_add_sync(kWarpMask, v);
      if (lane == 0) {
        sm.place[kClBins] = before;
        if (rank == 0) st->n_roots = all;
      }
    }
    __syncthreads();
    const int root_at = sm.place[kClBins] + sm.hist[kClBins][warp];
#pragma unroll
    for (int g = 0; g < kClGroups; ++g) {
      const int k = w_begin + 32 * g + lane;
      if (k >= w_end) break;
      const int bin = (int)(ranks[g] >> 16) & (kClBins - 1);
      queue[sm.local[bin] + sm.hist[bin][warp] + (int)(ranks[g] & 0xFFFFu)] = (unsigned short)k;
      if (pass == 0 && caller[k] == kClNone) roots[root_at + (int)(ranks[g] >> 23)] = base + k;
    }
    __syncthreads();
    TL_CL_STAMP(8);   // staged
    for (int q = tid; q < mine; q += kSingleThreads) {
      const int k = queue[q];
      dst[sm.place[(int)((state[k] & ~kClDone) >> shift) & (kClBins - 1)] + q] = pass == 0 ? base + k : (int)caller[k];
    }
    if (pass + 1 < passes) {
      __threadfence();
      cl_sync();                                         // the next pass reads what every CTA has placed
    }
  }
  if (passes > 1) {                                      // wavefront boundaries from the sorted order
    __threadfence();
    cl_sync();
    for (int r = base + tid; r < base + mine; r += kSingleThreads) {
      const int a = *(volatile const int*)(level + *(volatile const int*)(order + r));
      if (r == 0 || *(volatile const int*)(level + *(volatile const int*)(order + r - 1)) != a) level_offset[a] = r;
    }
  }
  if (rank == 0 && tid == 0) { level_offset[n_levels] = n; st->n_levels = n_levels; *n_levels_out = n_levels; }
  TL_CL_STAMP(9);
  cl_sync();                                             // no CTA leaves while a peer may still read its words
}

size_t single_smem_bytes(int n, bool with_parts) {
  size_t w = (size_t)n * 4;
  w = w > kSingleScratch ? round_up_sz(w, 16) : kSingleScratch;
  return w + round_up_sz((size_t)n * 2, 16) + round_up_sz((size_t)n, 16) +
         (with_parts ? round_up_sz((size_t)n * 2, 16) : 0);
}
// The packed children of every node next to the rest, if that still fits one CTA's shared memory.
bool single_caches_children(int n, bool with_parts) {
  return !with_parts && single_smem_bytes(n, false) + (size_t)n * 4 + 16 <= single_smem_bytes(kSchedSingleMaxNodes, false);
}

}  // namespace
}  // namespace tl
