// Which trees a cluster takes and in which order it walks them: the pieces that every kernel whose clusters evaluate whole
// trees shares (trees_fp32.cu; trees_tc.cu has a plan of its own and takes the tables, the ranking and the choice from here).
//
// A cluster needs the internal nodes of its trees by depth, deepest last, and for every node the row of its caller.  For a TreeLSTM forward one CTA of
// the launch ahead works that out for all clusters, beside the leaves (plan_walks: 1 and 2 below, then nodes counted by cluster and depth), and a
// backward pass reads what its forward has walked (load_walk).  Everywhere else, and where that CTA's tables do not hold the forest, all CTAs of all
// clusters work it out for themselves from the child arrays, each the same way, since the rows of a cluster's lists are addresses in the shared
// memory of all its CTAs:
//   1. child table, caller of every node, a bit for every node that has a caller           (load_kids)
//   2. every internal node climbs to its root; trees ranked by size and dealt out to the clusters there and back (0 .. Q-1,
//      Q-1 .. 0, ...): the fullest cluster sets the time, and of 25 sentences on 15 clusters it held 85 to 96 nodes when trees
//      were dealt in the order of their ids, the largest tree alone (54) this way; greedy dealing to the least loaded cluster,
//      a serial chain, gives the same                                                      (deal_by_size)
//   3. one warp walks the cluster's trees from the roots down                              (walk_trees)
#pragma once

#include "common.cuh"

namespace tl {
namespace {

constexpr int kDealt = 512;                // trees that are dealt by size at most
struct ForestIn { int n, vocab; const int *left, *right, *token; };

constexpr int kSmemMax = 224 * 1024;
constexpr unsigned kFull = 0xffffffffu;

// ---- shared memory -------------------------------------------------------------------------------- //
// Offsets in 4-byte words.  What is left behind `state` holds the states of the cluster's nodes, if they fit.
struct TreesSmem {
  int buf, kids, child, list, start, par, leaf, leaf_par, state, state_words;
};
__host__ __device__ inline TreesSmem trees_smem(int n, int buf_words) {
  TreesSmem s{};
  int off = 0;
  auto take = [&](int words) { const int o = off; off += (words + 3) & ~3; return o; };
  s.buf = take(buf_words);
  s.kids = take(n);
  s.child = take(n / 32 + 1);             // a bit per node: it has a caller
  const int half = n / 4 + 8;             // uint16 entries for the internal nodes (fewer than n / 2)
  s.list = take(half);
  s.start = take(half);
  s.par = take(half);
  s.leaf = take(n / 2 + 8);               // (a forest of single-leaf trees has n leaves)
  s.leaf_par = take(n / 2 + 8);
  s.state = off;
  s.state_words = kSmemMax / 4 - off;
  return s;
}

// Child table entry of a node: left | right << 16 (ids below 32768), or the top bit and the token of a leaf.  Ids and
// tokens are clamped: nothing has been validated yet.
constexpr unsigned kLeafBit = 0x80000000u;
__device__ __forceinline__ bool is_leaf(unsigned kids) { return (kids & kLeafBit) != 0; }
// (up: if given, every node's caller, a root's itself.  Two callers of one child are no forest: which of them is found is a matter of timing, so
// the answer is true then, the same in every CTA.  internal: if given, zero before; how many nodes have children.)
__device__ __forceinline__ bool load_kids(const ForestIn& p, const TreesSmem& s, float* sm, unsigned short* up, int* internal) {
  unsigned* kids = reinterpret_cast<unsigned*>(sm + s.kids);
  unsigned* child = reinterpret_cast<unsigned*>(sm + s.child);
  for (int k = threadIdx.x; k < p.n / 32 + 1; k += blockDim.x) child[k] = 0u;
  if (up)
    for (int k = threadIdx.x; k < p.n; k += blockDim.x) up[k] = (unsigned short)k;
  __syncthreads();
  bool twice = false;
  int own = 0;
  constexpr int kAhead = 4;                // nodes whose loads are under way together (one after the other: 6 k cycles for 1.4 k nodes, this way 4.1 k)
#pragma unroll 1
  for (int k0 = threadIdx.x; k0 < p.n; k0 += kAhead * blockDim.x) {
    int l[kAhead], r[kAhead], t[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int k = min(k0 + j * (int)blockDim.x, p.n - 1);
      l[j] = p.left[k]; r[j] = p.right[k]; t[j] = p.token[k];
    }
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int k = k0 + j * (int)blockDim.x;
      if (k >= p.n) break;
      if (l[j] < 0) {
        kids[k] = kLeafBit | (unsigned)min(max(t[j], 0), p.vocab - 1);
        continue;
      }
      const unsigned a = (unsigned)min(l[j], p.n - 1), b = (unsigned)min(max(r[j], 0), p.n - 1);
      kids[k] = a | (b << 16);
      ++own;
      if (up) {
        up[a] = up[b] = (unsigned short)k;
        const unsigned had_a = atomicOr(child + (a >> 5), 1u << (a & 31)), had_b = atomicOr(child + (b >> 5), 1u << (b & 31));
        twice = twice || ((had_a >> (a & 31) | had_b >> (b & 31)) & 1u);
      } else {
        atomicOr(child + (a >> 5), 1u << (a & 31));
        atomicOr(child + (b >> 5), 1u << (b & 31));
      }
    }
  }
  if (internal) {
    own = __reduce_add_sync(kFull, own);
    if ((threadIdx.x & 31) == 0) atomicAdd(internal, own);
  }
  return __syncthreads_or(twice) != 0;
}

// The cluster's trees by depth: internal node number q is list[q], depth d is [start[d], start[d + 1]), the leaves are
// in leaf[]; par[q] and leaf_par[] say whose child a node is: 2 x number of the caller + side, kNoCaller for a root.  One
// warp; every CTA of the cluster gets the same lists.
constexpr unsigned short kNoCaller = 0xFFFF;
struct Walk { int depths, internal, leaves; };
// `few`: no more trees than clusters; `dealt`: if given, the cluster of every root (ascending ids), else root r goes to cluster r mod parts; `win`: if given, the walk
// may end where it reads zero.
__device__ __forceinline__ void walk_trees(const ForestIn& p, const TreesSmem& s, float* sm, int part, int parts, bool few, const unsigned char* dealt, const int* win, Walk* out) {
  const unsigned* kids = reinterpret_cast<const unsigned*>(sm + s.kids);
  const unsigned* child = reinterpret_cast<const unsigned*>(sm + s.child);
  unsigned short* list = reinterpret_cast<unsigned short*>(sm + s.list);
  unsigned short* start = reinterpret_cast<unsigned short*>(sm + s.start);
  unsigned short* par = reinterpret_cast<unsigned short*>(sm + s.par);
  unsigned short* leaf = reinterpret_cast<unsigned short*>(sm + s.leaf);
  unsigned short* leaf_par = reinterpret_cast<unsigned short*>(sm + s.leaf_par);
  const int lane = threadIdx.x & 31, n = p.n;
  const unsigned below = (1u << lane) - 1u;
  const int max_internal = n / 2, max_leaves = n;
  int count = 0, leaves = 0, depth = 0, lo = 0, rank0 = 0;
  auto scan = [&](int v) {                // inclusive over the lanes
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(kFull, v, d);
      if (lane >= d) v += t;
    }
    return v;
  };
  auto mine = [&](int rank) {
    if (__builtin_expect(dealt != nullptr, 0)) return (int)dealt[min(rank, kDealt - 1)] == part;
    return (few ? rank : rank % parts) == part;
  };
  for (int w0 = 0; w0 * 32 < n; w0 += 32) {   // roots: nodes without a caller, 32 words of 32 ids at a time
    const int w = w0 + lane, base = w * 32;
    unsigned m = base < n ? ~child[w] : 0u;
    if (base < n && n - base < 32) m &= (1u << (n - base)) - 1u;
    const int roots = __popc(m), incl = scan(roots);
    int rank = rank0 + incl - roots, mi = 0, ml = 0;
    rank0 += __shfl_sync(kFull, incl, 31);
    for (unsigned b = m; b; b &= b - 1, ++rank)
      if (mine(rank)) (is_leaf(kids[base + __ffs(b) - 1]) ? ml : mi) += 1;
    const int ii = scan(mi), il = scan(ml);
    int ci = count + ii - mi, cl = leaves + il - ml;
    rank = rank0 - __shfl_sync(kFull, incl, 31) + incl - roots;
    for (unsigned b = m; b; b &= b - 1, ++rank)
      if (mine(rank)) {
        const int node = base + __ffs(b) - 1;
        if (is_leaf(kids[node])) { leaf[cl] = (unsigned short)node; leaf_par[cl++] = kNoCaller; }
        else if (ci < max_internal) { list[ci] = (unsigned short)node; par[ci++] = kNoCaller; }
      }
    count = min(count + __shfl_sync(kFull, ii, 31), max_internal);
    leaves += __shfl_sync(kFull, il, 31);
  }
  bool fits = true;
  if (lane == 0) start[0] = 0;
  __syncwarp();
  while (lo < count && fits) {
    const int hi = count;
    if (win && hi - lo >= 512 && !__shfl_sync(kFull, *(const volatile int*)win, 0)) break;   // (narrow depths are not worth the look)
    ++depth;
    if (lane == 0) start[depth] = (unsigned short)hi;
    for (int i0 = lo; i0 < hi; i0 += 32) {
      const bool have = i0 + lane < hi;
      const unsigned kd = have ? kids[list[i0 + lane]] : 0u;
      const int l = (int)(kd & 0xFFFFu), r = (int)(kd >> 16);
      const bool ll = is_leaf(kids[l]), lr = is_leaf(kids[r]);
      const unsigned il = __ballot_sync(kFull, have && !ll), ir = __ballot_sync(kFull, have && !lr);
      const unsigned fl = __ballot_sync(kFull, have && ll), fr = __ballot_sync(kFull, have && lr);
      // only arrays that are no forest of trees can run over
      if (count + __popc(il) + __popc(ir) > max_internal || leaves + __popc(fl) + __popc(fr) > max_leaves) { fits = false; break; }
      if (have) {
        const int al = ll ? leaves + __popc(fl & below) : count + __popc(il & below);
        const int ar = lr ? leaves + __popc(fl) + __popc(fr & below) : count + __popc(il) + __popc(ir & below);
        (ll ? leaf : list)[al] = (unsigned short)l;
        (lr ? leaf : list)[ar] = (unsigned short)r;
        (ll ? leaf_par : par)[al] = (unsigned short)(2 * (i0 + lane));
        (lr ? leaf_par : par)[ar] = (unsigned short)(2 * (i0 + lane) + 1);
      }
      count += __popc(il) + __popc(ir);
      leaves += __popc(fl) + __popc(fr);
      __syncwarp();
    }
    lo = hi;
  }
  if (lane == 0) *out = fits ? Walk{depth, count, leaves} : Walk{0, 0, 0};
}


// What the clusters would have to walk, and (`win`) whether that is faster than wavefront by wavefront over the whole GPU;
// of up to kDealt trees, the cluster that each goes to.
constexpr int kMaxTreeClusters = 192, kClimbs = 3;
struct TreeLoads { int nodes[kMaxTreeClusters], depth[kMaxTreeClusters], win, internal, longer; unsigned char part[kDealt]; };
// Tables that are needed until the trees are dealt: callers by node id, roots before each word of the bit map, size and depth
// of the trees.  Behind the lists (where the states go afterwards) if there is room, else in their place.
struct TreeLinks { unsigned short* up; int *before, *size, *deep; };
__host__ __device__ inline int deal_words(int n) { return ((n + 1) / 2 + n / 32 + 4) / 4 * 4 + 2 * kDealt; }
__device__ __forceinline__ TreeLinks tree_links(float* at, int n) {
  TreeLinks t;
  t.up = reinterpret_cast<unsigned short*>(at);
  t.before = reinterpret_cast<int*>(at + (n + 1) / 2);
  t.size = reinterpret_cast<int*>(at + ((n + 1) / 2 + n / 32 + 4) / 4 * 4);
  t.deep = t.size + kDealt;
  return t;
}
__device__ __forceinline__ int roots_in_all(const TreeLinks& t, const unsigned* child, int n) {
  return t.before[(n - 1) >> 5] + __popc(~child[(n - 1) >> 5] & (0xFFFFFFFFu >> (31 - ((n - 1) & 31))));
}
// one warp
__device__ __forceinline__ void count_roots(const TreeLinks& t, const unsigned* child, int n, int lane) {
  int sum = 0;
  for (int w0 = 0; w0 * 32 < n; w0 += 32) {
    const int w = w0 + lane, roots = w * 32 < n ? __popc(~child[w]) : 0;   // (ids beyond n come last: nobody counts them)
    int incl = roots;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, d);
      if (lane >= d) incl += v;
    }
    if (w * 32 < n) t.before[w] = sum + incl - roots;
    sum += __shfl_sync(kFull, incl, 31);
  }
}
// The cluster of tree `q` when trees are dealt by size there and back (equal ones in the order of their ids; the sizes, a multiple of
// four of them, are zero behind the last tree).
__device__ __forceinline__ int dealt_to(const int* size, int slots, int q, int parts) {
  const int mine = size[q];
  int rank = 0;
#pragma unroll 1
  for (int s0 = 0; s0 < slots; s0 += 4) {
    const int4 v = *reinterpret_cast<const int4*>(size + s0);
    rank += (v.x > mine || (v.x == mine && s0 < q)) + (v.y > mine || (v.y == mine && s0 + 1 < q)) +
            (v.z > mine || (v.z == mine && s0 + 2 < q)) + (v.w > mine || (v.w == mine && s0 + 3 < q));
  }
  const int turn = rank / parts, in_turn = rank - turn * parts;
  return turn & 1 ? parts - 1 - in_turn : in_turn;
}
// one warp: the outcome, from the clusters' loads (counts of a sample: `share` internal nodes for each)
__device__ __forceinline__ bool clusters_win(const WalkCosts& costs, const TreeLoads& loads, int parts, float internal, float share, int lane) {
  float cost = 0.f;
  int waves = 0;
  for (int q = lane; q < parts; q += 32) {
    cost = fmaxf(cost, tree_cost(costs, share * (float)loads.nodes[q], (float)loads.depth[q], internal));
    waves = max(waves, loads.depth[q]);
  }
  waves = __reduce_max_sync(kFull, waves);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) cost = fmaxf(cost, __shfl_xor_sync(kFull, cost, d));
  return cost < grid_cost(costs, (float)waves, internal);
}
// The nodes of a sample - all, if there are no more than kClimbs a thread - climb to their roots, which gives the sizes and depths
// of the trees; the trees are dealt out (see the head of this file), and (`choose`) the clusters' loads say whether they win.  (The
// average load of a cluster says too little: one tree of 1024 leaves among 24 sentences, H = 150, was 4.5 times slower on
// clusters than over the whole GPU.)  Called by the threads from `first` on, a multiple of 32; barrier 1 is theirs.  Every CTA
// takes the same sample and comes to the same answer.  (This code runs once, and what is not in the instruction cache costs
// more than what it does: 25 sentences on 512 threads 10 k cycles, twice that with loops unrolled and all nodes climbing.)
__device__ __forceinline__ void deal_by_size(int n, const unsigned* kids, const unsigned* child, const TreeLinks& t, const WalkCosts& costs, int parts,
                                             bool dealt, bool choose, int first, TreeLoads* out, unsigned* found = nullptr) {
  const int tid = (int)threadIdx.x - first, nt = (int)blockDim.x - first, lane = tid & 31;
  auto sync = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory"); };
  const int internal = out->internal, trees = max(1, min(n - 2 * internal, kDealt)), slots = dealt ? trees : parts;   // (not dealt: the clusters' own)
  if (tid < 32) count_roots(t, child, n, lane);
#pragma unroll 1
  for (int q = tid; q < slots + 3; q += nt)
    if (q < kDealt) t.size[q] = t.deep[q] = 0;
#pragma unroll 1
  for (int q = tid; q < parts; q += nt) out->nodes[q] = out->depth[q] = 0;
  const int sample = min(n, nt * kClimbs);
  int at[kClimbs], depth[kClimbs];
  bool have[kClimbs];
#pragma unroll
  for (int q = 0; q < kClimbs; ++q) {
    const int i = tid + q * nt;
    have[q] = i < sample;
    at[q] = have[q] ? (int)((long long)i * n / sample) : 0;
    depth[q] = is_leaf(kids[at[q]]) ? 0 : 1;
  }
#pragma unroll 1
  for (int step = 0; step < n; ++step) {                     // (arrays that are no forest may hold a cycle)
    bool any = false;
#pragma unroll
    for (int q = 0; q < kClimbs; ++q) {
      const int up = t.up[at[q]];
      if (up != at[q]) { ++depth[q]; any = true; }
      at[q] = up;
    }
    if (!any) break;
  }
  if (found && sample == n)                                // (of all nodes: root | distance << 16)
#pragma unroll
    for (int q = 0; q < kClimbs; ++q)
      if (have[q]) found[tid + q * nt] = (unsigned)at[q] | (unsigned)(depth[q] - (is_leaf(kids[tid + q * nt]) ? 0 : 1)) << 16;
  sync();
#pragma unroll
  for (int q = 0; q < kClimbs; ++q) {
    const int rank = t.before[at[q] >> 5] + __popc(~child[at[q] >> 5] & ((1u << (at[q] & 31)) - 1u));   // (of a node on a cycle: some tree's)
    const int slot = !have[q] ? -1 : (dealt ? min(rank, trees - 1) : rank % parts);
    const unsigned peers = __match_any_sync(kFull, slot);
    const int deepest = __reduce_max_sync(peers, depth[q]);
    if (have[q] && lane == __ffs(peers) - 1) {
      atomicAdd(t.size + slot, __popc(peers));
      atomicMax(t.deep + slot, deepest);
    }
  }
  sync();
#pragma unroll 1
  for (int q = tid; q < slots; q += nt) {
    const int mine = t.size[q];
    int part = q;
    if (dealt) {
      part = dealt_to(t.size, slots, q, parts);
      out->part[q] = (unsigned char)part;
    }
    if (choose && mine) {
      atomicAdd(&out->nodes[part], mine);
      atomicMax(&out->depth[part], t.deep[q]);
    }
  }
  if (!choose) return;
  sync();
  if (tid < 32) {
    const bool win = clusters_win(costs, *out, parts, (float)internal, (float)internal / (float)sample, lane);
    if (lane == 0) *(volatile int*)&out->win = win;
  }
}

// Whether the trees are dealt by size: there are more than clusters, and no more than the tables hold.  Else tree t is cluster
// t mod parts's.
__device__ __forceinline__ bool deals_by_size(int n, int internal, int parts) {
  const int trees = n - 2 * internal;                                    // (arrays that are no forest: whatever that is)
  return trees > parts && trees <= kDealt;
}
// The tables of the forest, then what the cluster has to walk: nothing, if loads->win says that the forest is the next kernel's
// (`choose`).  A choice without a deal (`by_size`: there may be one) takes its time beside the walk.
__device__ __forceinline__ void deal_trees(const ForestIn& p, const WalkCosts& costs, const TreesSmem& s, float* sm, int part, int parts, bool choose, bool by_size, TreeLoads* loads, Walk* walk, long long* trace) {
  const int tid = (int)threadIdx.x, nt = (int)blockDim.x, n = p.n;
  if (!choose && !by_size) {                               // (the short forwards of the recursive cells: without the other's branches 1 us less)
    load_kids(p, s, sm, nullptr, nullptr);
    TL_STAMP(trace, kTraceLevels - 1, 5);
    if (tid < 32) walk_trees(p, s, sm, part, parts, false, nullptr, nullptr, walk);
    __syncthreads();
    return;
  }
  const unsigned* kids = reinterpret_cast<const unsigned*>(sm + s.kids);
  const unsigned* child = reinterpret_cast<const unsigned*>(sm + s.child);
  const bool beside = s.state_words >= deal_words(n);
  const TreeLinks links = tree_links(sm + (beside ? s.state : s.list), n);
  if (tid == 0) { loads->win = 1; loads->internal = 0; }
  const bool forest = !load_kids(p, s, sm, choose ? links.up : nullptr, choose || by_size ? &loads->internal : nullptr);   // (else the scheduler reports it, and the walk is bounded)
  TL_STAMP(trace, kTraceLevels - 1, 5);
  const bool dealt = forest && by_size && deals_by_size(n, loads->internal, parts), climb = forest && (dealt || choose);
  if (__builtin_expect(climb, 0)) {                        // (out of the way of what every call executes)
    if (!choose) {                                                       // the callers were not noted with the child table
#pragma unroll 1
      for (int k = tid; k < n; k += nt) links.up[k] = (unsigned short)k;
      __syncthreads();
#pragma unroll 1
      for (int k = tid; k < n; k += nt) {
        const unsigned kd = kids[k];
        if (!is_leaf(kd)) links.up[kd & 0xFFFFu] = links.up[kd >> 16] = (unsigned short)k;
      }
      __syncthreads();
    }
    const int first = dealt ? 0 : 32;
    if (tid >= first) deal_by_size(n, kids, child, links, costs, parts, dealt, choose, first, loads);
    if (dealt || !beside) __syncthreads();
  }
  TL_STAMP(trace, kTraceLevels - 1, 6);
  if (tid < 32) walk_trees(p, s, sm, part, parts, by_size && forest && n - 2 * loads->internal <= parts, dealt ? loads->part : nullptr, choose ? &loads->win : nullptr, walk);
  __syncthreads();
  if (choose) {
    if (tid == 0 && !loads->win) *walk = Walk{0, 0, 0};
    __syncthreads();
  }
}

// What the clusters of a forward walk, in the workspace: planned ahead of them by one CTA (plan_walks), or kept by them for the backward pass of the same forest,
// whose clusters would otherwise work it out again beside k_bwd_begin (34 k cycles there for 25 sentences, H = 150).  One block per cluster:
// header, then children, node and caller of every row, leaves and their callers, starts of the depths.  A block has room for four times the average
// (`cap` rows).  One tree's lists are one cluster's, whatever their length: the planning CTA, which knows all of them, puts longer ones behind the blocks, one after
// the other, and the header says where.  (Left to the clusters themselves, behind the leaves, the plan of one chain of 200 leaves
// had its forward take 656 us and not 604, H = 150, and 321 and not 270, H = 24.)  A cluster that keeps its own lists says that it has none if they are longer, and the backward pass deals anew.
struct SavedWalks { unsigned char* at; int cap; };
__host__ __device__ inline int saved_cap(int n, int parts) { return min(n / 2 + 2, 4 * (n / 2 / parts) + 64); }
__host__ __device__ inline size_t saved_block(int cap) { return (size_t)(16 + 18 * cap + 4 + 15) / 16 * 16; }
__host__ __device__ inline size_t longer_bytes(int n, int parts) { return 18 * (size_t)n + 48 * (size_t)parts; }   // of all longer blocks: each has room for as many rows as the cluster has leaves
struct SavedBlock {
  unsigned char* at;
  int cap;
  __device__ __forceinline__ int4* head() const { return reinterpret_cast<int4*>(at); }   // depths, rows, leaves, clusters | 16-byte units to where the rest is << 8 (zero: here)
  __device__ __forceinline__ uint2* row(int q) const { return reinterpret_cast<uint2*>(at + 16) + q; }   // children, node | caller << 16
  __device__ __forceinline__ unsigned* leaf(int q) const { return reinterpret_cast<unsigned*>(at + 16 + 8 * (size_t)cap) + q; }   // node | caller << 16
  __device__ __forceinline__ unsigned short* start(int d) const { return reinterpret_cast<unsigned short*>(at + 16 + 16 * (size_t)cap) + d; }
};
__device__ __forceinline__ SavedBlock saved_at(const SavedWalks& w, int part) { return {w.at + saved_block(w.cap) * part, w.cap}; }
// All threads, with the cluster's lists in shared memory.
__device__ __forceinline__ void save_walk(const SavedWalks& w, const TreesSmem& s, const float* sm, int part, int parts, const Walk& walk) {
  const SavedBlock b = saved_at(w, part);
  const bool fits = walk.internal <= w.cap && walk.leaves <= 2 * w.cap;
  if (threadIdx.x == 0) *b.head() = make_int4(walk.depths, walk.internal, walk.leaves, fits ? parts : 0);
  if (!fits) return;
  const unsigned short* list = reinterpret_cast<const unsigned short*>(sm + s.list);
#pragma unroll 1
  for (int q = threadIdx.x; q < walk.leaves || q <= walk.internal; q += blockDim.x) {
    if (q < walk.internal) *b.row(q) = make_uint2(reinterpret_cast<const unsigned*>(sm + s.kids)[list[q]], list[q] | (unsigned)reinterpret_cast<const unsigned short*>(sm + s.par)[q] << 16);
    if (q <= walk.depths) *b.start(q) = reinterpret_cast<const unsigned short*>(sm + s.start)[q];
    if (q < walk.leaves) *b.leaf(q) = reinterpret_cast<const unsigned short*>(sm + s.leaf)[q] | (unsigned)reinterpret_cast<const unsigned short*>(sm + s.leaf_par)[q] << 16;
  }
}
// The same from one CTA for all clusters, ahead of the kernel that walks (TreeLSTM forward: beside the leaves).  Behind deal_by_size, whose tables and
// outcome it takes (`climbed`: what its climbs found is where the places go, `at`); all threads.  `at`: what the tables leave of the CTA's shared memory, `words` of it.
// Every node finds its root and its distance from it by pointer jumping (in place: a word holds an ancestor and its distance, whichever it is; a step at a
// time, a chain of 8192 leaves took millions of cycles).  Internal nodes are counted by cluster and depth and take their places there (which one of a depth does
// not matter), then look up their callers' places.  Clusters without a tree have no counts: one tree's depths fit whatever their number.  Arrays
// that are no forest get empty lists (the scheduler reports them); lists that are not wanted or not to be had say so in all headers.
__device__ __forceinline__ void plan_walks(int n, const unsigned* kids, const unsigned* child, const TreeLinks& t, bool wanted, bool forest, bool dealt, bool climbed, int parts, int* at, int words,
                                           const SavedWalks& w, TreeLoads* loads) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  unsigned* const where = reinterpret_cast<unsigned*>(at);   // cluster | depth << 8; then a leaf's cluster | place << 8, an internal node's place | cluster << 16
  int* const next = at + n;
  const int busy = max(1, min(parts, n - 2 * loads->internal));   // clusters with a tree
  constexpr unsigned kNone = 0xFFFFFFFFu;
  __syncthreads();
  for (int q = tid; q < parts; q += nt) loads->nodes[q] = loads->depth[q] = 0;   // 16-byte units to the lists, leaves
  if (tid == 0) loads->internal = loads->longer = 0;         // deepest; 16-byte units in use behind the blocks
  __syncthreads();
  bool fits = wanted && forest && n + busy <= words && parts < 256;   // (as many depths as there is room for: below)
  if (fits) {
    if (!climbed) {                                          // root | distance << 16, as the climbs leave them
      for (int k = tid; k < n; k += nt) where[k] = (unsigned)t.up[k] | (t.up[k] != k ? 1u << 16 : 0u);
      __syncthreads();
      constexpr int kAhead = 4;
#pragma unroll 1
      for (int round = 0; round < 16; ++round) {             // (n < 2^15; arrays that are no forest may hold a cycle)
        bool any = false;
#pragma unroll 1
        for (int k0 = tid; k0 < n; k0 += kAhead * nt) {
          unsigned v[kAhead], u[kAhead];
#pragma unroll
          for (int j = 0; j < kAhead; ++j) v[j] = where[min(k0 + j * nt, n - 1)];
#pragma unroll
          for (int j = 0; j < kAhead; ++j) u[j] = where[v[j] & 0xFFFFu];
#pragma unroll
          for (int j = 0; j < kAhead; ++j)
            if (k0 + j * nt < n && (u[j] & 0xFFFFu) != (v[j] & 0xFFFFu)) {
              where[k0 + j * nt] = (u[j] & 0xFFFFu) | ((v[j] >> 16) + (u[j] >> 16)) << 16;
              any = true;
            }
        }
        if (!__syncthreads_or(any)) break;
      }
    }
    int deepest = 0;
#pragma unroll 1
    for (int k0 = tid; k0 < n; k0 += kClimbs * nt) {
      unsigned v[kClimbs];
#pragma unroll
      for (int j = 0; j < kClimbs; ++j) v[j] = where[min(k0 + j * nt, n - 1)];
#pragma unroll
      for (int j = 0; j < kClimbs; ++j) {
        const int k = k0 + j * nt;
        if (k >= n) continue;
        const int root = (int)(v[j] & 0xFFFFu), depth = (int)(v[j] >> 16);
        const int rank = t.before[root >> 5] + __popc(~child[root >> 5] & ((1u << (root & 31)) - 1u));
        const bool tree = !(child[root >> 5] >> (root & 31) & 1u);
        const unsigned part = dealt ? loads->part[min(rank, kDealt - 1)] : (unsigned)(rank % parts);
        where[k] = tree ? part | (unsigned)depth << 8 : kNone;
        if (tree && !is_leaf(kids[k])) deepest = max(deepest, depth + 1);
      }
    }
    deepest = __reduce_max_sync(kFull, deepest);
    if (lane == 0) atomicMax(&loads->internal, deepest);
  }
  __syncthreads();
  const int depths = loads->internal;
  fits = fits && n + busy * depths <= words;
  if (fits) {
    for (int q = tid; q < busy * depths; q += nt) next[q] = 0;
    __syncthreads();
#pragma unroll 1
    for (int k0 = 0; k0 < n; k0 += nt) {                     // (leaves take their places)
      const int k = min(k0 + tid, n - 1);
      const unsigned v = k0 + tid < n ? where[k] : kNone;
      const bool lf = v != kNone && is_leaf(kids[k]);
      if (v != kNone && !lf) atomicAdd(next + (v & 255u) * depths + (v >> 8), 1);
      const unsigned peers = __match_any_sync(kFull, lf ? (int)(v & 255u) : -1);
      int place = 0;
      if (lf && lane == __ffs(peers) - 1) place = atomicAdd(loads->depth + (v & 255u), __popc(peers));
      place = __shfl_sync(kFull, place, __ffs(peers) - 1) + __popc(peers & ((1u << lane) - 1u));
      if (lf) where[k] = (v & 255u) | (unsigned)place << 8;
    }
    __syncthreads();
    // (a tree has one more leaf than rows)
    const int units = (int)(saved_block(w.cap) / 16);
    for (int part = tid; part < parts; part += nt) {
      const int leaves = loads->depth[part];
      loads->nodes[part] = leaves > w.cap ? parts * units + atomicAdd(&loads->longer, (int)(saved_block(leaves) / 16)) : part * units;
    }
    __syncthreads();
    auto block_of = [&](int part) { return SavedBlock{w.at + 16 * (size_t)loads->nodes[part], max(w.cap, loads->depth[part])}; };
    for (int part = tid >> 5; part < busy; part += nt >> 5) {
      const SavedBlock b = block_of(part);
      int sum = 0, deep = 0;
      for (int d0 = 0; d0 < depths; d0 += 32) {
        const int d = d0 + lane, v = d < depths ? next[part * depths + d] : 0;
        int incl = v;
#pragma unroll
        for (int e = 1; e < 32; e <<= 1) {
          const int x = __shfl_up_sync(kFull, incl, e);
          if (lane >= e) incl += x;
        }
        if (d < depths) next[part * depths + d] = sum + incl - v;
        if (v) *b.start(d) = (unsigned short)(sum + incl - v);
        sum += __shfl_sync(kFull, incl, 31);
        deep += __popc(__ballot_sync(kFull, v != 0));        // (depths have no gaps)
      }
      if (lane == 0) {
        *b.start(deep) = (unsigned short)sum;
        const int at = loads->nodes[part];
        *saved_at(w, part).head() = make_int4(deep, sum, loads->depth[part], parts | (at == part * units ? 0 : at) << 8);
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int k = tid; k < n; k += nt) {
      const unsigned v = where[k];
      if (v == kNone || is_leaf(kids[k])) continue;
      const unsigned part = v & 255u;
      where[k] = (unsigned)atomicAdd(next + part * depths + (v >> 8), 1) | part << 16;
    }
    __syncthreads();
#pragma unroll 1
    for (int k = tid; k < n; k += nt) {
      const unsigned v = where[k], kd = kids[k];
      if (v == kNone) continue;
      const int up = t.up[k];
      unsigned code = kNoCaller;
      if (up != k) code = 2u * (where[up] & 0xFFFFu) + (unsigned)((kids[up] & 0xFFFFu) != (unsigned)k);
      const SavedBlock b = block_of((int)(is_leaf(kd) ? v & 255u : v >> 16));
      if (is_leaf(kd)) *b.leaf((int)(v >> 8)) = (unsigned)k | code << 16;
      else *b.row((int)(v & 0xFFFFu)) = make_uint2(kd, (unsigned)k | code << 16);
    }
  }
  // (All clusters' or none: one that deals anew keeps its lists where these would be.)
  for (int part = fits ? busy + tid : tid; part < parts; part += nt) *saved_at(w, part).head() = make_int4(0, 0, 0, !forest || fits ? parts : 0);
}
// All threads (of a small block each looks at several headers); false: there is nothing to load.  Of the child table only the entries of the cluster's internal nodes are filled.
// (The first entries are asked for together with the headers.)
__device__ __forceinline__ bool load_walk(const SavedWalks& w, const WalkCosts& costs, int n, int n_roots, const TreesSmem& s, float* sm, int part, int parts,
                                          bool choose, TreeLoads* loads, Walk* walk) {
  SavedBlock b = saved_at(w, part);
  struct Entry { uint2 row; unsigned leaf; unsigned short start; };
  auto read = [&](int q) { return Entry{*b.row(min(q, b.cap - 1)), *b.leaf(min(q, 2 * b.cap - 1)), *b.start(min(q, b.cap))}; };
  Entry e = read(threadIdx.x);
  bool ok = true;
#pragma unroll 1
  for (int q = threadIdx.x; q < parts; q += blockDim.x) {
    const int4 head = *saved_at(w, q).head();
    ok = ok && (head.w & 255) == parts;
    loads->nodes[q] = head.y;
    loads->depth[q] = head.x;
    if (q == part) { *walk = Walk{head.x, head.y, head.z}; loads->win = 1; loads->longer = head.w >> 8; }
  }
  if (!__syncthreads_and(ok)) return false;
  if (choose) {
    if (threadIdx.x < 32) {
      const bool win = clusters_win(costs, *loads, parts, (float)((n - n_roots) / 2), 1.f, threadIdx.x);
      __syncwarp();
      if (threadIdx.x == 0) {
        loads->win = win;
        if (!win) *walk = Walk{0, 0, 0};
      }
    }
    __syncthreads();
  }
  const Walk have = *walk;
  if (__builtin_expect(loads->longer != 0 && have.leaves > 0, 0)) {   // (none: the outcome is the whole GPU)
    b = {w.at + 16 * (size_t)loads->longer, have.leaves};
    e = read(threadIdx.x);
  }
#pragma unroll 1
  for (int q = threadIdx.x; q < have.leaves || q <= have.internal;) {
    if (q < have.internal) {
      reinterpret_cast<unsigned*>(sm + s.kids)[e.row.y & 0xFFFFu] = e.row.x;
      reinterpret_cast<unsigned short*>(sm + s.list)[q] = (unsigned short)e.row.y;
      reinterpret_cast<unsigned short*>(sm + s.par)[q] = (unsigned short)(e.row.y >> 16);
    }
    if (q <= have.depths) reinterpret_cast<unsigned short*>(sm + s.start)[q] = e.start;
    if (q < have.leaves) {
      reinterpret_cast<unsigned short*>(sm + s.leaf)[q] = (unsigned short)e.leaf;
      reinterpret_cast<unsigned short*>(sm + s.leaf_par)[q] = (unsigned short)(e.leaf >> 16);
    }
    q += blockDim.x;
    e = read(q);
  }
  __syncthreads();
  return true;
}

}  // namespace
}  // namespace tl
