// bf16 evaluation of narrow, deep forests: whole trees on thread-block clusters, beside the scheduler (sm_100a: tcgen05.mma,
// tensor memory, TMA, distributed shared memory).
//
// Paper: Section 2.2 - the trees of a batch are independent; Section 6.3 - on deep, narrow trees what counts is the time from
// "child finished" to "caller finished".  In the grid-wide kernel (gemm_tc.cu) that is 7.8 k cycles whatever the width: states to
// global memory, grid barrier, operand rows back through TMA, MMAs, cell update.  A cluster that has all of a tree needs none of
// the first three: the new bf16 h goes straight into the shared memory of the CTAs that multiply with it next.  And nothing waits
// for the schedule: a cluster needs only "children before parents", so it walks its trees by distance from the root, deepest
// first, which it finds from the child arrays itself (tt_decide, tt_lists).  The launch is the scheduler's: its first cluster
// schedules, the others evaluate meanwhile, or leave the forest to the grid-wide kernel behind (DevStatus::trees_fwd).
//
// One depth.  CTA r of a cluster owns hidden units [r U, (r + 1) U), U = 8 gpc, and keeps the packed recurrent weights of those
// units (40 gpc rows x 2 Hp) in tensor memory.  Weight rows are the M side of the MMA (tensor-memory lanes = gate rows), the
// depth's nodes the N side, so a depth of up to R nodes is one chain of MMAs.  By depth a node's inner children are always one
// step away: two operand buffers [h_l | h_r] of R rows, used in turn, are all the state there is.  A buffer is filled by
//   - pushes: each CTA sends its U units of a new h to the row of the caller in every CTA (st.async, the bytes counted on the
//     receiver's mbarrier);
//   - the filling warps, a depth ahead: rows of children that are leaves, from global memory, where the leaf phase put them.
// No CTA writes into a buffer that is still read: a push for depth d - 2 follows all pushes for d - 1, hence every CTA's MMAs of
// depth d (the argument is the same for the gate values, which take the buffer of the depth being finished).  There is no other
// signal between CTAs.  Cell states stay with the units' owner.
//
// Leaves first: tiles of 96 leaves of the cluster's trees, every CTA its own units, the same orientation (weights M, leaves N).
//
// Measured (H = 256, 11 nodes a depth): a depth takes 3.6 k cycles - 32 MMAs 1.1 k (34 cycles each whatever their width; 43 with the
// weights in shared memory), their retirement seen 0.35 k, gate values to shared memory 0.5 k, cell updates, pushes and their way
// 1.7 k (the interconnect moves about 8 bytes a cycle and CTA) - where the grid-wide kernel takes 7.8 k: 64 chains of 64 leaves
// 308 -> 180 us, 25 sentences (H = 150) 80 -> 43, one sentence from and to host arrays 70 -> 52.  Before the first depth: 23 k cycles for
// one sentence (trees and loads 8 k, lists 4.5 k, leaves 6 k, exchange 2 k), 30 k for the 25, 96 k for the 64 chains (41 k, 9 k, 39 k).
//
// Warp roles (1024 threads, as the scheduler's): warps 0-23 epilogue (warp w reads tensor-memory lane quadrant w mod 4), 24-30
// filling warps, 31 MMA issuer and tensor-memory owner; all of them gather and finish leaves.
#include "cluster_ptx.cuh"
#include "schedule.cuh"
#include "trees_plan.cuh"

namespace tl {
namespace {

constexpr int kT = kSingleThreads;
constexpr int kEpiWarps = 24, kFillWarps = 7, kMmaWarp = 31;
constexpr int kLeafTile = 96;
constexpr int kMaxInner = 1280, kMaxLeaves = 1536;        // nodes of a cluster
constexpr int kSmemDynamic = 222 * 1024;                  // (static shared memory of the scheduler and the plan beside it)
constexpr uint32_t kAcc0 = 256, kAccStep = 64, kAccLeaf = 384;   // tensor memory: weights, then accumulators of the depths (in turn), of the leaves
constexpr int kSampleNodes = 2048;                        // larger forests are looked at in a sample first
constexpr int kMaxTtNodes = 16384;
constexpr int kMaxTtParts = 32;                           // (a lane each)

// Shared memory of a CTA, bytes from the 1024-byte aligned base.  The plan's tables and the leaf phase use what the depths use
// later; the lists stay.
struct TtLayout {
  uint32_t x, c, rk, list, par, start, leaf, ltok, bars;
  uint32_t x_bytes, c_bytes;                              // of one of the two buffers
  uint32_t wx, wx_bytes, rows, rows_bytes, gates;         // leaf phase
  int R;
};
__host__ __device__ inline TtLayout tt_layout(int Hp, int Ep, int gpc) {
  TtLayout L{};
  const uint32_t kb = 2u * (uint32_t)Hp / kKBlock, kbl = (uint32_t)Ep / kKBlock, U = 8u * (uint32_t)gpc;
  L.bars = kSmemDynamic - 1024u - 256u;                   // alignment slack behind
  L.ltok = L.bars - 4u * kMaxLeaves;
  L.leaf = L.ltok - 2u * kMaxLeaves;
  L.start = L.leaf - 2u * (kMaxInner + 8);
  L.par = L.start - 2u * kMaxInner;
  L.list = L.par - 2u * kMaxInner;
  L.rk = L.list - 4u * kMaxInner;
  L.x = 0;
  const uint32_t per_row = 2u * (kb * 128u + 2u * U * 4u), room = L.rk;
  int R = 64;
  while (R > 0 && (uint32_t)R * per_row > room) R -= 16;
  L.R = R;
  L.x_bytes = (uint32_t)R * kb * 128u;
  L.c_bytes = (uint32_t)R * 2u * U * 4u;
  L.c = L.x + 2u * L.x_bytes;
  L.wx = 0;
  L.wx_bytes = kbl * (uint32_t)gpc * kGColsL * 128u;
  L.rows = (L.wx_bytes + 1023u) & ~1023u;
  L.rows_bytes = kbl * (uint32_t)kLeafTile * 128u;
  L.gates = L.rows + 2u * L.rows_bytes;
  return L;
}
// The plan's tables, offsets in 4-byte words: children by node (left | right << 16, or the top bit and the token of a leaf), for every node an
// ancestor and its distance (later tree | depth << 16, later the row), a bit for every node that has a caller, roots before each
// word of those, sizes of the trees; behind them, nodes of every cluster's depths.
struct TtTables { int kids, up, child, before, size, wide; };
__host__ __device__ inline TtTables tt_tables(int n) {
  TtTables t{};
  int at = 0;
  auto take = [&](int words) { const int o = at; at += (words + 3) & ~3; return o; };
  t.kids = take(n);
  t.up = take(n);
  t.child = take(n / 32 + 1);
  t.before = take(n / 32 + 1);
  t.size = take(kDealt);
  t.wide = at;
  return t;
}

struct TtParams {
  ForestIn f;
  int H, Hp, Ep, gpc;
  int* chk_counts;
  const __nv_bfloat16* emb_bf;
  const uint4* wp_t;                                      // recurrent weights as tensor memory takes them (tt_weight_at)
  const float *bp_h, *bp_x;
  float *h, *c, *gates;
  __nv_bfloat16* hb;                                      // [n][Hp]: bf16 h of the leaves
  DevStatus* st;
  long long wait_limit;
  WalkCosts costs;
  long long* trace;
};
struct TtSched {
  int on_cluster, sh, cache_children;
  int *parent, *level, *order, *order_tmp, *level_offset, *roots, *n_levels_out;
};

// The plan is made by the first `pt` threads of every CTA, in two steps.  An instruction that all 32 warps execute costs eight
// issue cycles and a barrier of them more than one of a few, so small forests get no more warps than they have work for.
__device__ __forceinline__ int tt_plan_threads(int n) { return n <= 512 ? (n + 31) & ~31 : (n <= 2048 ? 512 : kT); }
__device__ __forceinline__ void tt_sync(int pt) { asm volatile("bar.sync 1, %0;" ::"r"(pt) : "memory"); }
__device__ __forceinline__ bool tt_any(bool mine, int pt) {
  uint32_t any;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.or.pred p, 1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(any) : "r"((uint32_t)mine), "r"(pt) : "memory");
  return any != 0u;
}
struct TtPlan {
  unsigned *kids, *up, *child;
  int *before, *size, *wide;
  int n, pt, parts, trees;
  bool dealt;
  unsigned inner;                                          // bit j: node tid + j pt has children (n <= 32 pt)
  __device__ __forceinline__ TtPlan(float* sm, int n_, int parts_) : n(n_), pt(tt_plan_threads(n_)), parts(parts_), trees(0), dealt(false), inner(0u) {
    const TtTables T = tt_tables(n_);
    kids = reinterpret_cast<unsigned*>(sm + T.kids);
    up = reinterpret_cast<unsigned*>(sm + T.up);
    child = reinterpret_cast<unsigned*>(sm + T.child);
    before = reinterpret_cast<int*>(sm + T.before);
    size = reinterpret_cast<int*>(sm + T.size);
    wide = reinterpret_cast<int*>(sm + T.wide);
  }
  __device__ __forceinline__ bool no_caller(int k) const { return (child[k >> 5] >> (k & 31) & 1u) == 0u; }
  __device__ __forceinline__ int slot_of(int root) const {
    const int at = before[root >> 5] + __popc(~child[root >> 5] & ((1u << (root & 31)) - 1u));
    return dealt ? at : at % parts;
  }
};
// Trees, depths, loads.  loads->win = 0: the forest is the grid-wide kernel's - because that is faster (clusters_win), because a
// depth of some cluster has more nodes than a buffer holds, or because a node has two callers (the scheduler reports it).  Every
// CTA of every cluster comes to the same answer: they all count all nodes.
// Trees and depths come from pointer jumping (in place: a word holds an ancestor and its distance, whichever it is): 64 chains of
// 64 leaves took 107 k cycles with climbs.
__device__ __forceinline__ void tt_decide(TtPlan& t, const TtParams& p, const ForestIn& f, int R, int wide_words, TreeLoads* loads, long long* trace) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = t.n, pt = t.pt, parts = t.parts;
#pragma unroll 1
  for (int k = tid; k < n; k += pt) t.up[k] = (unsigned)k;
#pragma unroll 1
  for (int k = tid; k < kDealt; k += pt) t.size[k] = 0;
  if (warp == 0) {
    if (lane < parts) loads->nodes[lane] = loads->depth[lane] = 0;
    if (lane == 0) { loads->internal = 0; loads->win = 0; }
  }
  tt_sync(pt);
#pragma unroll 1
  for (int j0 = 0; j0 * pt + tid < n; j0 += 4) {           // ids are clamped: nothing has been validated yet
    int l[4], r[4], w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = tid + (j0 + j) * pt;
      l[j] = k < n ? __ldcg(f.left + k) : -1;
      r[j] = k < n ? __ldcg(f.right + k) : -1;
      w[j] = k < n ? __ldcg(f.token + k) : 0;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = tid + (j0 + j) * pt;
      if (k >= n) break;
      if (l[j] < 0) {
        t.kids[k] = kLeafBit | (unsigned)min(max(w[j], 0), f.vocab - 1);   // (its token: no trip to memory behind the lists; 25 sentences 40.6 -> 40.2 us)
      } else {
        const unsigned a = (unsigned)min(l[j], n - 1), b = (unsigned)min(max(r[j], 0), n - 1);
        t.kids[k] = a | (b << 16);
        t.up[a] = t.up[b] = (unsigned)k | 0x10000u;
        t.inner |= 1u << (j0 + j);
      }
    }
  }
  {
    const int own = __reduce_add_sync(kFull, __popc(t.inner));
    if (lane == 0 && own) atomicAdd(&loads->internal, own);
  }
  tt_sync(pt);
  const int internal = loads->internal;
  if (internal > parts * kMaxInner) return;
  if (n > kSampleNodes) {
    // Before most of the work that grows with the forest, a look at a sample (of arrays that are no forest the CTAs may see different
    // things here; those that go on find that below): if most of its nodes lie at a depth that must be wider than
    // the buffers, or if not even an equal deal would win, the forest is left here (the scheduler takes 30 k cycles, and what the
    // plan takes beyond that the grid-wide kernel waits for: 140 sentences, H = 256, 107 us and not 101).
    constexpr int kDepths = 64;
    if (tid < kDepths + 2) t.wide[tid] = 0;                // (nodes of the sample by depth, their number, the deepest)
    tt_sync(pt);
    const int from = (int)((long long)tid * n / pt);
    if (!is_leaf(t.kids[from])) {
      int at = from, depth = 0;
#pragma unroll 1
      for (; depth < kDepths - 1; ++depth) {
        const unsigned v = t.up[at];
        if (v >> 16 == 0u) break;
        at = (int)(v & 0xFFFFu);
      }
      atomicAdd(t.wide + depth, 1);
      atomicAdd(t.wide + kDepths, 1);
      atomicMax(t.wide + kDepths + 1, depth + 1);
    }
    tt_sync(pt);
    const float share = (float)internal / (float)(parts * max(t.wide[kDepths], 1));   // of one cluster, for a node of the sample
    const float nodes = share * (float)t.wide[kDepths], depth = (float)t.wide[kDepths + 1];
    // (a cluster's nodes of a depth scatter by about their root around the mean, and the widest counts: 180 sentences, H = 156, with 60 of 64
    // in the mean, were left only after the plan, 128 us; now at once. The last word holds all depths that are deeper.)
    const float seen = tid < kDepths - 1 ? (float)t.wide[tid] : 0.f, mean = share * (seen + 0.5f * sqrtf(seen));   // (what is seen scatters, too)
    const bool over = mean + sqrtf(mean) > (float)R;
    if (tt_any(over || 0.8f * tree_cost(p.costs, nodes, depth, (float)internal) > grid_cost(p.costs, depth, (float)internal), pt)) return;
  }
  // a node's word says whose child it is now: a child that two callers claim has one of them (no atomics: the bits of 32
  // neighbours are one word)
  bool twice = false;
#pragma unroll 1
  for (int j = 0; j * pt + warp * 32 < n; ++j) {
    const int k = tid + j * pt;
    const unsigned m = __ballot_sync(kFull, k < n && t.up[min(k, n - 1)] >> 16 != 0u);
    if (lane == 0) t.child[k >> 5] = m;
    if (t.inner >> j & 1u) {
      const unsigned kd = t.kids[k], a = kd & 0xFFFFu, b = kd >> 16;
      twice = twice || a == b || (t.up[a] & 0xFFFFu) != (unsigned)k || (t.up[b] & 0xFFFFu) != (unsigned)k;
    }
  }
  if (tt_any(twice, pt)) return;
  TL_STAMP(trace, kTraceLevels - 1, 1);
  const TreeLinks links{nullptr, t.before, nullptr, nullptr};
  if (warp == (pt >> 5) - 1) count_roots(links, t.child, n, lane);   // (the last to have nodes)
  // Small forests: up to kClimb steps at once - what others have found by then counts as one -, and again where that was not
  // enough; sentences are done after the first turn (five rounds of single steps took 3 k cycles of barriers).  Large ones, where a
  // step takes what a round does: a step at a time, four nodes of a thread side by side.
  constexpr int kClimb = 12;
  unsigned far = t.inner;                                  // nodes whose ancestor may not be the root yet
#pragma unroll 1
  for (int round = 0; round < 17 && n <= kSampleNodes; ++round) {   // (arrays that are no forest may hold a cycle)
    unsigned left = 0u;
#pragma unroll 1
    for (int j0 = 0; far >> j0; j0 += 3) {                 // three chains of reads under way
      unsigned v[3];
      bool go[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        go[j] = (far >> (j0 + j) & 1u) != 0u;
        v[j] = go[j] ? t.up[tid + (j0 + j) * pt] : 0u;
      }
#pragma unroll 1
      for (int step = 0; step < kClimb && (go[0] || go[1] || go[2]); ++step) {
        unsigned x[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) x[j] = t.up[v[j] & 0xFFFFu];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          go[j] = go[j] && ((v[j] ^ x[j]) & 0xFFFFu) != 0u;   // (an ancestor that is its own is a root)
          if (go[j]) v[j] = (x[j] & 0xFFFFu) | ((v[j] & 0xFFFF0000u) + (x[j] & 0xFFFF0000u));
        }
      }
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (far >> (j0 + j) & 1u) {
          t.up[tid + (j0 + j) * pt] = v[j];
          if (go[j]) left |= 1u << (j0 + j);
        }
    }
    far = left;
    if (!tt_any(far != 0u, pt)) break;
  }
#pragma unroll 1
  for (int round = 0; round < 17 && n > kSampleNodes; ++round) {
    bool moved = false;
#pragma unroll 1
    for (int j0 = 0; far >> j0; j0 += 4) {
      unsigned v[4], x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = far >> (j0 + j) & 1u ? t.up[tid + (j0 + j) * pt] : 0u;
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = t.up[v[j] & 0xFFFFu];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (!(far >> (j0 + j) & 1u)) continue;
        if (((v[j] ^ x[j]) & 0xFFFFu) != 0u) {
          t.up[tid + (j0 + j) * pt] = (x[j] & 0xFFFFu) | ((v[j] & 0xFFFF0000u) + (x[j] & 0xFFFF0000u));
          moved = true;
        } else {
          far &= ~(1u << (j0 + j));
        }
      }
    }
    if (!tt_any(moved, pt)) break;
  }
  t.trees = roots_in_all(links, t.child, n);
  t.dealt = t.trees > parts && t.trees <= kDealt;
  int deepest = -1;
#pragma unroll 1
  for (unsigned bits = t.inner; bits; bits &= bits - 1u) {
    const int k = tid + (__ffs(bits) - 1) * pt;
    const unsigned v = t.up[k];
    unsigned now = 0xFFFFFFFFu;                            // (ended on a cycle: nobody's node)
    if (t.no_caller((int)(v & 0xFFFFu))) {
      const int slot = t.slot_of((int)(v & 0xFFFFu));
      atomicAdd(t.size + slot, 1);
      deepest = max(deepest, (int)(v >> 16));
      now = (unsigned)slot | (v & 0xFFFF0000u);
    }
    t.up[k] = now;
  }
  deepest = __reduce_max_sync(kFull, deepest);
  if (lane == 0 && deepest >= 0) atomicMax(&loads->depth[0], deepest + 1);   // (here: of all clusters)
  tt_sync(pt);
  const int slots = t.dealt ? t.trees : parts;
#pragma unroll 1
  for (int q = tid; q < slots; q += pt) {
    const int mine = t.size[q], to = t.dealt ? dealt_to(t.size, slots, q, parts) : q;
    loads->part[q] = (unsigned char)to;
    if (mine) atomicAdd(&loads->nodes[to], mine);
  }
  // nodes of every cluster's depths, if there is room for them
  const int most = loads->depth[0], cells = parts * most;
#pragma unroll 1
  for (int q = tid; q < cells && q < wide_words; q += pt) t.wide[q] = 0;
  tt_sync(pt);
  TL_STAMP(trace, kTraceLevels - 1, 2);
  if (cells > wide_words) return;
#pragma unroll 1
  for (unsigned bits = t.inner; bits; bits &= bits - 1u) {
    const unsigned v = t.up[tid + (__ffs(bits) - 1) * pt];
    if (v != 0xFFFFFFFFu) atomicAdd(t.wide + loads->part[v & 0xFFFFu] * most + (v >> 16), 1);
  }
  tt_sync(pt);
  bool over = false;
#pragma unroll 1
  for (int q = tid; q < cells; q += pt) {
    const int w = t.wide[q], c = q / most;
    over = over || w > R;
    if (w && (q == (c + 1) * most - 1 || t.wide[q + 1] == 0)) loads->depth[c] = q - c * most + 1;   // (depths have no gaps)
    if (q == c * most && w == 0) loads->depth[c] = 0;
  }
  if (tt_any(over, pt)) return;
  if (warp == 0) {                                         // (loads->internal: from here on, cells per cluster)
    const bool bad = __any_sync(kFull, lane < parts && (loads->nodes[lane] > kMaxInner ||
                                                        loads->nodes[lane] + (t.trees + parts - 1) / parts + 1 > kMaxLeaves));
    // (of 70 forests with fewer nodes none was slower on clusters by more than 2 %)
    const bool win = n <= kSampleNodes || clusters_win(p.costs, *loads, parts, (float)internal, 1.f, lane);
    if (lane == 0) { loads->win = win && !bad; loads->internal = most; }
  }
}
// The cluster's lists: internal nodes by depth, their callers' rows and children, the leaves.  The place of a node among those of
// its depth does not matter, but all CTAs must agree on it (it is an address in all of them): the first one gives the places out,
// the others read its list.  All threads of the CTA; those behind the first pt only take part in the cluster's barrier.
__device__ __forceinline__ void tt_lists(const TtPlan& t, float* sm, const TtLayout& L, int part, int rank, TreeLoads* loads, Walk* walk) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = t.n, pt = t.pt;
  unsigned char* const base = reinterpret_cast<unsigned char*>(sm);
  unsigned short* const list = reinterpret_cast<unsigned short*>(base + L.list);
  unsigned short* const par = reinterpret_cast<unsigned short*>(base + L.par);
  unsigned short* const start = reinterpret_cast<unsigned short*>(base + L.start);
  unsigned short* const leaf = reinterpret_cast<unsigned short*>(base + L.leaf);
  unsigned* const rk = reinterpret_cast<unsigned*>(base + L.rk);
  int* const next = t.wide + loads->internal * part;       // next place in a depth
  const int mine = loads->nodes[part], depths = loads->depth[part];
  if (tid < pt) {
    if (warp == 0) {
      int sum = 0;
#pragma unroll 1
      for (int d0 = 0; d0 < depths; d0 += 32) {
        const int d = d0 + lane, v = d < depths ? next[d] : 0;
        int incl = v;
#pragma unroll
        for (int e = 1; e < 32; e <<= 1) {
          const int x = __shfl_up_sync(kFull, incl, e);
          if (lane >= e) incl += x;
        }
        if (d < depths) { next[d] = sum + incl - v; start[d] = (unsigned short)(sum + incl - v); }
        sum += __shfl_sync(kFull, incl, 31);
      }
      if (lane == 0) start[depths] = (unsigned short)mine;
    }
#pragma unroll 1
    for (int q = tid; q < mine; q += pt) par[q] = kNoCaller;
    tt_sync(pt);
    if (tid == 0) loads->internal = 0;                     // (from here on: leaves of the cluster)
    tt_sync(pt);
    if (rank == 0)
#pragma unroll 1
      for (unsigned bits = t.inner; bits; bits &= bits - 1u) {
        const int k = tid + (__ffs(bits) - 1) * pt;
        const unsigned v = t.up[k];
        if (v != 0xFFFFFFFFu && loads->part[v & 0xFFFFu] == part) list[atomicAdd(next + (v >> 16), 1)] = (unsigned short)k;
      }
#pragma unroll 1
    for (int w = warp; w * 32 < n; w += pt >> 5) {         // trees of one leaf
      const int k = w * 32 + lane;
      if (~t.child[w] >> lane & 1u && k < n && is_leaf(t.kids[k]) && loads->part[t.slot_of(k)] == part)
        leaf[atomicAdd(&loads->internal, 1)] = (unsigned short)k;
    }
  }
  cluster_barrier();
  if (tid >= pt) return;
  if (rank != 0) {
    const uint32_t from = map_to_cta(smem_u32(list), 0);
#pragma unroll 1
    for (int q = tid; q < (mine + 1) / 2; q += pt) {
      unsigned v;
      asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(from + 4u * (uint32_t)q) : "memory");
      reinterpret_cast<unsigned*>(list)[q] = v;
    }
    tt_sync(pt);
  }
#pragma unroll 1
  for (int q = tid; q < mine; q += pt) t.up[list[q]] = (unsigned)q;
  tt_sync(pt);
#pragma unroll 1
  for (int q0 = warp * 32; q0 < mine; q0 += pt) {
    const int q = q0 + lane;
    const unsigned kd = q < mine ? t.kids[list[q]] : 0u;
    const int l = (int)(kd & 0xFFFFu), r = (int)(kd >> 16);
    const bool ll = q < mine && is_leaf(t.kids[l]), lr = q < mine && is_leaf(t.kids[r]);
    const unsigned ml = __ballot_sync(kFull, ll), mr = __ballot_sync(kFull, lr);
    int at = 0;
    if (lane == 0) at = atomicAdd(&loads->internal, __popc(ml) + __popc(mr));
    at = __shfl_sync(kFull, at, 0);
    if (q < mine) {
      rk[q] = kd | (ll ? 0x8000u : 0u) | (lr ? 0x80000000u : 0u);
      const unsigned below = (1u << lane) - 1u;
      if (ll) leaf[at + __popc(ml & below)] = (unsigned short)l;
      else par[t.up[l]] = (unsigned short)(2 * q);
      if (lr) leaf[at + __popc(ml) + __popc(mr & below)] = (unsigned short)r;
      else par[t.up[r]] = (unsigned short)(2 * q + 1);
    }
  }
  tt_sync(pt);
  const int leaves = loads->internal;
  unsigned* const ltok = reinterpret_cast<unsigned*>(base + L.ltok);
#pragma unroll 1
  for (int e = tid; e < leaves; e += pt) ltok[e] = t.kids[leaf[e]] & ~kLeafBit;
  if (tid == 0) *walk = Walk{depths, mine, leaves};
}

__global__ void __launch_bounds__(kT, 1) k_schedule_trees_tc(const __grid_constant__ CUtensorMap wx_map, const __grid_constant__ TtParams p, const __grid_constant__ TtSched q) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Walk s_walk;
  __shared__ TreeLoads s_loads;
  const int cs = (int)cluster_size();
  ForestIn f = p.f;
  wait_for_last(f.left, f.right, f.token);
  if ((int)blockIdx.x < cs) {
    if (q.on_cluster)
      schedule_cluster(smem_raw, true, f.n, f.left, f.right, f.token, f.vocab, q.level, q.order, q.order_tmp, q.level_offset, q.roots, q.n_levels_out, p.st, q.sh);
    else if (blockIdx.x == 0)
      schedule_single(smem_raw, true, f.n, f.left, f.right, f.token, f.vocab, q.parent, q.level, q.order, q.order_tmp, q.level_offset, q.roots, q.n_levels_out,
                      p.st, 0, nullptr, nullptr, nullptr, q.cache_children);
    else
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    return;
  }
  // (Nothing decided: the kernel behind, which comes up with what it needs unless it reads otherwise.  One thread speaks for its CTA, behind what it has stored.)
  if (threadIdx.x == 0) {
    if ((int)blockIdx.x == cs) {
      p.st->trees_fwd = 0;
      __threadfence();
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  const int rank = (int)cluster_rank(), part = (int)blockIdx.x / cs - 1, parts = (int)gridDim.x / cs - 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = f.n, H = p.H, Hp = p.Hp, Ep = p.Ep, gpc = p.gpc, U = 8 * gpc, U0 = rank * U;
  const TtLayout L = tt_layout(Hp, Ep, gpc);
  const uint32_t raw_addr = smem_u32(smem_raw), base = (raw_addr + 1023u) & ~1023u;
  unsigned char* const base_ptr = smem_raw + (base - raw_addr);
  float* const sm = reinterpret_cast<float*>(base_ptr);
#ifdef TREELSTM_TRACE
  long long* const trace = part == 0 && rank == 0 && tid == 0 ? p.trace : nullptr;
  long long* const trace_cta = part == 0 && rank == 0 ? p.trace : nullptr;
#else
  long long* const trace = nullptr;
#endif
  TL_STAMP(trace, kTraceLevels - 1, 0);
  TtPlan t(sm, n, parts);
  if (tid < t.pt) tt_decide(t, p, f, L.R, (int)L.rk / 4 - tt_tables(n).wide, &s_loads, trace);
  __syncthreads();
  const bool taken = s_loads.win != 0;
  if (part == 0 && rank == 0 && tid == 0 && taken) p.st->trees_fwd = 1;
  if (!taken) return;
  TL_STAMP(trace, kTraceLevels - 1, 3);
  uint64_t* const bars = reinterpret_cast<uint64_t*>(base_ptr + L.bars);
  // bars: 0 W_x  1 TF (MMAs of a depth retired)  2, 3 XF (operands of a depth complete)  4, 5 EP (epilogue has read a depth's
  //       buffers)  6 EB (meeting point of the epilogue warps)  7 drain;  leaves: 8, 9 LF (rows there)  10, 11 LE (rows read)
  //       12, 13 LT (MMAs retired)  14, 15 LD (accumulator read)
  const uint32_t bar0 = smem_u32(bars), WXb = bar0, TFb = bar0 + 8, XF0 = bar0 + 16, EP0 = bar0 + 32, EBb = bar0 + 48, drainb = bar0 + 56, LF0 = bar0 + 64,
                 LE0 = bar0 + 80, LT0 = bar0 + 96, LD0 = bar0 + 112;
  uint32_t* const s_tmem = reinterpret_cast<uint32_t*>(bars + 16);
  volatile int* const s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
  if (tid == kT - 1) {
    mbar_init(WXb, 1);
    mbar_init(TFb, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(XF0 + 8 * b, 1 + kFillWarps);
      mbar_init(EP0 + 8 * b, kEpiWarps);
      mbar_init(LF0 + 8 * b, kEpiWarps + kFillWarps);
      mbar_init(LE0 + 8 * b, 1);
      mbar_init(LT0 + 8 * b, 1);
      mbar_init(LD0 + 8 * b, kEpiWarps);
    }
    mbar_init(EBb, kEpiWarps);
    mbar_init(drainb, 1);
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == kMmaWarp) tmem_alloc(smem_u32(s_tmem), 512);
  tt_lists(t, sm, L, part, rank, &s_loads, &s_walk);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  TL_STAMP(trace, kTraceLevels - 1, 4);

  const Walk walk = s_walk;
  const unsigned short* list = reinterpret_cast<const unsigned short*>(base_ptr + L.list);
  const unsigned short* par = reinterpret_cast<const unsigned short*>(base_ptr + L.par);
  const unsigned short* start = reinterpret_cast<const unsigned short*>(base_ptr + L.start);
  const unsigned short* leaf = reinterpret_cast<const unsigned short*>(base_ptr + L.leaf);
  const unsigned* const rk = reinterpret_cast<const unsigned*>(base_ptr + L.rk);   // children of a row: left | right << 16, bits 15 and 31: a leaf
  unsigned* const ltok = reinterpret_cast<unsigned*>(base_ptr + L.ltok);                // token of a leaf
  const int m_rows = gpc * kGColsI, l_rows = gpc * kGColsL, kb_int = 2 * Hp / kKBlock, kb_leaf = Ep / kKBlock, R = L.R;

  const uint32_t tmem = *s_tmem;
  const int quad = warp & 3, m = quad * 32 + lane;         // gate row of this thread
  uint32_t tf_phase = 0;
  bool ok = true;

  // ---- leaves ---------------------------------------------------------------------------------------- //
  const int tiles = (walk.leaves + kLeafTile - 1) / kLeafTile;
  const int r0 = tid / U, u0 = tid - r0 * U;               // epilogue: the thread's first node of a pass and unit (further nodes: the same
  const bool real = U0 + u0 < H;                           // unit, since U divides the epilogue's threads)
  const int hc = row_pitch(H), step = kEpiWarps * 32 / U;
  uint32_t eb_phase = 0;
  auto meet = [&]() {                                      // the epilogue warps
    __syncwarp();
    if (lane == 0) mbar_arrive(EBb);
    const bool met = mbar_wait(EBb, eb_phase, s_abort, p.wait_limit, p.st);
    eb_phase ^= 1u;
    return __all_sync(kFullMask, met) != 0;
  };
  // Embedding rows of a tile in the layout of a swizzled K-major operand: a row per warp and turn, 16 bytes a lane, all of a warp's
  // rows asked for at once.  (By seven warps alone a tile took 6.9 k cycles: a warp has about four such requests under way.)
  auto gather = [&](int t2) {
    const int rows = min(kLeafTile, walk.leaves - t2 * kLeafTile), cpr = Ep / 8;
    const uint32_t dst = base + L.rows + (uint32_t)(t2 & 1) * L.rows_bytes;
#pragma unroll 1
    for (int r = warp; r < rows; r += kEpiWarps + kFillWarps) {
      const uint4* const src = reinterpret_cast<const uint4*>(p.emb_bf + (size_t)ltok[t2 * kLeafTile + r] * Ep);
#pragma unroll 1
      for (int c0 = lane; c0 < cpr; c0 += 32)
        cp_async16(dst + (uint32_t)(c0 >> 3) * (kLeafTile * 128u) + (uint32_t)r * 128u + (uint32_t)(((c0 & 7) ^ (r & 7)) << 4), src + c0, 16u);
    }
  };
  auto gathered = [&](int t2) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(LF0 + 8 * (t2 & 1));
  };
  if (warp == kMmaWarp) {
    const bool issue = elect_one();
    if (lane == 0 && tiles > 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the plan's tables were here
      mbar_arrive_expect_tx(WXb, L.wx_bytes);
      tma_load_3d(base + L.wx, &wx_map, 0, rank * l_rows, 0, WXb);
    }
    __syncwarp();
    const uint32_t idesc = umma_idesc(kLeafTile);
#pragma unroll 1
    for (int t2 = 0; t2 < tiles; ++t2) {
      const int b = t2 & 1;
      ok = (t2 > 0 || mbar_wait(WXb, 0, s_abort, p.wait_limit, p.st)) && mbar_wait(LF0 + 8 * b, (uint32_t)(t2 >> 1) & 1u, s_abort, p.wait_limit, p.st) &&
           (t2 < 2 || mbar_wait(LD0 + 8 * b, (uint32_t)((t2 - 2) >> 1) & 1u, s_abort, p.wait_limit, p.st));
      ok = __all_sync(kFullMask, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem + (b ? kAccLeaf : kAcc0), x_addr = base + L.rows + (uint32_t)b * L.rows_bytes;
      for (int kb = 0; kb < kb_leaf; ++kb) {
        const uint64_t a_desc = umma_desc(base + L.wx + (uint32_t)kb * (uint32_t)l_rows * 128u);
        const uint64_t b_desc = umma_desc(x_addr + (uint32_t)kb * (kLeafTile * 128u));
#pragma unroll
        for (int k = 0; k < kKBlock / 16; ++k)
          if (issue) umma_bf16(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, !(kb == 0 && k == 0));
      }
      if (issue) { umma_commit(LE0 + 8 * b); umma_commit(LT0 + 8 * b); }
    }
  } else if (warp >= kEpiWarps) {
#pragma unroll 1
    for (int t2 = 0; t2 < tiles; ++t2) {
      ok = t2 < 2 || mbar_wait(LE0 + 8 * (t2 & 1), (uint32_t)((t2 - 2) >> 1) & 1u, s_abort, p.wait_limit, p.st);
      ok = __all_sync(kFullMask, ok);
      if (!ok) break;
      gather(t2);
      gathered(t2);
    }
  } else {
    // The recurrent weights, meanwhile, to tensor memory: lane = gate row, a column = two contraction indices.  An MMA whose
    // weights come from there reads only the nodes' rows from shared memory.
    if (tiles > 0) { gather(0); gathered(0); }
    if (quad * 32 < m_rows && walk.depths > 0) {
      const int pitch = (m_rows + 31) / 32 * 32;           // 16-byte pieces: [8 columns][half][lane]
      const uint4* const src = p.wp_t + ((size_t)rank * (Hp / 8) * 2) * pitch + m;
      const uint32_t to = tmem + ((uint32_t)(quad * 32) << 16);
#pragma unroll 1
      for (int c0 = warp >> 2; c0 < Hp / 8; c0 += 2 * (kEpiWarps / 4)) {
        const int c1 = min(c0 + kEpiWarps / 4, Hp / 8 - 1);   // (twice the last columns: the same values)
        const uint4 a0 = __ldg(src + (size_t)(2 * c0) * pitch), a1 = __ldg(src + (size_t)(2 * c0 + 1) * pitch);
        const uint4 b0 = __ldg(src + (size_t)(2 * c1) * pitch), b1 = __ldg(src + (size_t)(2 * c1 + 1) * pitch);
        tmem_st8(to + (uint32_t)(8 * c0), a0, a1);
        tmem_st8(to + (uint32_t)(8 * c1), b0, b1);
      }
      tmem_st_wait();
      tc_fence_before();
    }
    const float bias = m < l_rows ? __ldg(p.bp_x + rank * l_rows + m) : 0.f;
    const bool is_tanh = m % kGColsL >= 16;
    const float a_in = is_tanh ? 1.f : 0.5f, a_add = is_tanh ? 0.f : 0.5f;
    float* const gsm = reinterpret_cast<float*>(base_ptr + L.gates);
#pragma unroll 1
    for (int t2 = 0; t2 < tiles; ++t2) {
      const int b = t2 & 1, rows = min(kLeafTile, walk.leaves - t2 * kLeafTile);
      if (t2 + 1 < tiles) gather(t2 + 1);                  // (the MMAs of the tile before the last have retired)
      ok = mbar_wait(LT0 + 8 * b, (uint32_t)(t2 >> 1) & 1u, s_abort, p.wait_limit, p.st);
      if (t2 + 1 < tiles) gathered(t2 + 1);
      ok = __all_sync(kFullMask, ok);
      if (!ok) break;
      tc_fence_after();
      if (quad * 32 < l_rows) {
#pragma unroll 1
        for (int col0 = (warp >> 2) * 8; col0 < rows; col0 += 2 * kEpiWarps) {
          uint32_t v[8];
          tmem_ld8(tmem + (b ? kAccLeaf : kAcc0) + ((uint32_t)(quad * 32) << 16) + (uint32_t)col0, v);
          tmem_ld_wait();
          if (m < l_rows) {
#pragma unroll
            for (int j = 0; j < 8; ++j) gsm[(col0 + j) * l_rows + m] = fmaf(a_in, act_tanh(a_in * (__uint_as_float(v[j]) + bias)), a_add);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(LD0 + 8 * b);
      ok = meet();
      if (!ok) break;
#pragma unroll 1
      for (int r = r0; r < rows; r += step) {
        const int node = leaf[t2 * kLeafTile + r];
        const float* const g = gsm + r * l_rows + (u0 >> 3) * kGColsL + (u0 & 7);
        const float gi = g[0], go = g[8], gu = g[16];
        const float cv = gi * gu;
        const float hv = go * act_tanh(cv);
        p.hb[(size_t)node * Hp + U0 + u0] = __float2bfloat16_rn(real ? hv : 0.f);
        if (real) {
          p.h[(size_t)node * H + U0 + u0] = hv;
          p.c[(size_t)node * H + U0 + u0] = cv;
          count_write(p.chk_counts, node, 1);
          if (p.gates) {
            float* gp = p.gates + (size_t)node * 5 * hc + U0 + u0;
            gp[0] = gi; gp[hc] = 0.f; gp[2 * hc] = 0.f; gp[3 * hc] = go; gp[4 * hc] = gu;
          }
        }
      }
      if (t2 + 1 < tiles) ok = meet();                     // the gate values may be overwritten
      if (!ok) break;
    }
  }
  ok = __syncthreads_or(!ok) == 0;
  TL_STAMP(trace, kTraceLevels - 1, 5);
  const int D = ok ? walk.depths : 0;
  // the leaves' rows are read by all CTAs of the cluster; every CTA's barriers exist
  __threadfence();
  cluster_barrier();
  TL_STAMP(trace, kTraceLevels - 1, 6);

  // ---- depths, deepest first -------------------------------------------------------------------------- //
  if (warp == kMmaWarp) {
    const bool issue = elect_one();
    bool alive = true;
#pragma unroll 1
    for (int i = 0; i < D; ++i) {
      const int d = D - 1 - i, b = i & 1, w = start[d + 1] - start[d];
      alive = alive && mbar_wait_cluster(XF0 + 8 * b, (uint32_t)(i >> 1) & 1u, s_abort, p.wait_limit, p.st);
      alive = __all_sync(kFullMask, alive);
      if (!alive) break;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // pushed pieces are read by the tensor core
      tc_fence_after();
#ifdef TREELSTM_TRACE
      if (lane == 0) TL_STAMP(trace_cta, i, 0);
#endif
      const uint32_t idesc = umma_idesc((w + 15) & ~15);
      const uint32_t x_addr = base + L.x + (uint32_t)b * L.x_bytes, d_tmem = tmem + kAcc0 + (uint32_t)b * kAccStep;
      for (int kb = 0; kb < kb_int; ++kb) {
        const uint64_t b_desc = umma_desc(x_addr + (uint32_t)kb * (uint32_t)R * 128u);
#pragma unroll
        for (int k = 0; k < kKBlock / 16; ++k)
          if (issue) umma_bf16_tmem(d_tmem, tmem + (uint32_t)(kb * 32 + k * 8), b_desc + 2 * k, idesc, !(kb == 0 && k == 0));
      }
      if (issue) umma_commit(TFb);
#ifdef TREELSTM_TRACE
      if (lane == 0) TL_STAMP(trace_cta, i, 1);
#endif
    }
  } else if (warp >= kEpiWarps) {
    const int fw = warp - kEpiWarps, chunks = Hp / 8;
    bool alive = true;
#pragma unroll 1
    for (int i = 0; i < D; ++i) {
      const int d = D - 1 - i, b = i & 1, lo = start[d], w = start[d + 1] - lo;
      if (i >= 2) alive = mbar_wait(EP0 + 8 * b, (uint32_t)((i - 2) >> 1) & 1u, s_abort, p.wait_limit, p.st);
      alive = __all_sync(kFullMask, alive);
      if (!alive) break;
      if (fw == 0 && lane == 0)
        mbar_arrive_expect_tx(XF0 + 8 * b, i > 0 ? (uint32_t)(start[d + 2] - start[d + 1]) * (uint32_t)(2 * Hp) : 0u);
      unsigned char* const xb = base_ptr + L.x + (uint32_t)b * L.x_bytes;
      float* const cb = reinterpret_cast<float*>(base_ptr + L.c + (uint32_t)b * L.c_bytes);
#pragma unroll 1
      for (int pr = fw; pr < 2 * w; pr += kFillWarps) {
        const int r = pr >> 1, side = pr & 1;
        const unsigned kd = side ? rk[lo + r] >> 16 : rk[lo + r] & 0xFFFFu;
        if (!(kd & 0x8000u)) continue;
        const int node = (int)(kd & 0x7FFFu);
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        float cv = 0.f;
        if (lane < chunks) v = __ldcg(reinterpret_cast<const uint4*>(p.hb + (size_t)node * Hp) + lane);
        if (lane < U && U0 + lane < H) cv = __ldcg(p.c + (size_t)node * H + U0 + lane);
        if (lane < chunks) {
          const int ch = side * chunks + lane;
          *reinterpret_cast<uint4*>(xb + (uint32_t)(ch >> 3) * (uint32_t)R * 128u + (uint32_t)r * 128u + (uint32_t)(((ch & 7) ^ (r & 7)) << 4)) = v;
        }
        if (lane < U) cb[pr * U + lane] = cv;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(XF0 + 8 * b);
    }
  } else {
    const float bias = m < m_rows ? __ldg(p.bp_h + rank * m_rows + m) : 0.f;
    const bool is_tanh = m % kGColsI >= 32;                // rows 32..39 of a group: candidate u
    const float a_in = is_tanh ? 1.f : 0.5f, a_add = is_tanh ? 0.f : 0.5f;
    // the peers this lane sends to (cs is 8 or 16), eight lanes a piece of eight units
    uint32_t px[2], pf[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint32_t peer = (uint32_t)min((lane & 7) + 8 * k, cs - 1);
      px[k] = map_to_cta(base + L.x, peer);
      pf[k] = map_to_cta(XF0, peer);
    }
    bool alive = true;
#pragma unroll 1
    for (int i = 0; i < D; ++i) {
      const int d = D - 1 - i, b = i & 1, nb = b ^ 1, lo = start[d], w = start[d + 1] - lo, nlo = d > 0 ? start[d - 1] : 0;
      // where the results of this thread's first node go, while the MMAs run
      uint32_t to = 0;
      int c_to = 0, node = 0;
      auto target = [&](int r) {                           // r < w; to: in the next buffer of every CTA, or no caller
        node = list[lo + r];
        const unsigned code = par[lo + r];
        const int rn = (int)(code >> 1) - nlo, side = (int)(code & 1u), k = side * Hp + U0 + (u0 & ~7);
        to = code == kNoCaller ? ~0u : (uint32_t)nb * L.x_bytes + (uint32_t)(k / kKBlock) * (uint32_t)R * 128u + (uint32_t)rn * 128u +
                                           ((((uint32_t)(k % kKBlock) >> 3) ^ ((uint32_t)rn & 7u)) << 4);
        c_to = (2 * rn + side) * U + u0;
      };
      if (r0 < w) target(r0);
      // (XF has completed; waiting for it makes the filling warps' cell states this thread's to read)
      alive = mbar_wait(TFb, tf_phase, s_abort, p.wait_limit, p.st) && mbar_wait(XF0 + 8 * b, (uint32_t)(i >> 1) & 1u, s_abort, p.wait_limit, p.st);
      tf_phase ^= 1u;
      alive = __all_sync(kFullMask, alive);
      if (!alive) break;
      TL_STAMP(trace, i, 2);
      tc_fence_after();
      float* const gsm = reinterpret_cast<float*>(base_ptr + L.x + (uint32_t)b * L.x_bytes);   // gate values [node][m_rows]
      if (quad * 32 < m_rows) {
#pragma unroll 1
        for (int col0 = (warp >> 2) * 4; col0 < w; col0 += kEpiWarps) {
          uint32_t v[4];
          tmem_ld4(tmem + kAcc0 + ((uint32_t)(quad * 32) << 16) + (uint32_t)b * kAccStep + (uint32_t)col0, v);
          tmem_ld_wait();
          if (m < m_rows) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float z = __uint_as_float(v[j]) + bias;
              if (col0 + j < w) gsm[(col0 + j) * m_rows + m] = fmaf(a_in, act_tanh(a_in * z), a_add);
            }
          }
        }
      }
      tc_fence_before();
      alive = meet();
      if (!alive) break;
      TL_STAMP(trace, i, 3);
      const float* const cb = reinterpret_cast<const float*>(base_ptr + L.c + (uint32_t)b * L.c_bytes);
      float* const c_next = reinterpret_cast<float*>(base_ptr + L.c + (uint32_t)nb * L.c_bytes);
#pragma unroll 1
      for (int rw = warp * 32 / U, r = r0; rw < w; rw += step, r += step) {   // (rw: the warp's first node)
        const bool have = r < w;
        if (r != r0 && have) target(r);
        const int rr = have ? r : 0;
        const float* const g = gsm + rr * m_rows + (u0 >> 3) * kGColsI + (u0 & 7);
        const float gi = g[0], gfl = g[8], gfr = g[16], go = g[24], gu = g[32];
        const float cl = cb[2 * rr * U + u0], cr = cb[(2 * rr + 1) * U + u0];
        const float cn = gi * gu + gfl * cl + gfr * cr;
        const float hn = go * act_tanh(cn);
        const __nv_bfloat16 h16 = __float2bfloat16_rn(real ? hn : 0.f);
        const unsigned mine = (unsigned)*reinterpret_cast<const unsigned short*>(&h16);
        const unsigned two = mine | (__shfl_down_sync(kFullMask, mine, 1) << 16);
        uint4 v;
        v.x = __shfl_sync(kFullMask, two, lane & ~7);
        v.y = __shfl_sync(kFullMask, two, (lane & ~7) + 2);
        v.z = __shfl_sync(kFullMask, two, (lane & ~7) + 4);
        v.w = __shfl_sync(kFullMask, two, (lane & ~7) + 6);
        if (have && to != ~0u) {
          st_async16(px[0] + to, v, pf[0] + 8u * (uint32_t)nb);
          if (cs > 8) st_async16(px[1] + to, v, pf[1] + 8u * (uint32_t)nb);
          c_next[c_to] = real ? cn : 0.f;
        }
        if (have && real) {
          p.h[(size_t)node * H + U0 + u0] = hn;
          p.c[(size_t)node * H + U0 + u0] = cn;
          count_write(p.chk_counts, node, 1);
          if (p.gates) {
            float* gp = p.gates + (size_t)node * 5 * hc + U0 + u0;
            gp[0] = gi; gp[hc] = gfl; gp[2 * hc] = gfr; gp[3 * hc] = go; gp[4 * hc] = gu;
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(EP0 + 8 * b);
      TL_STAMP(trace, i, 4);
    }
  }
  // teardown
  tc_fence_before();
  __syncthreads();
  if (*s_abort) {
    // a wait expired: give what was requested a bounded time to land, the MMAs a bounded time to retire
    if (tid == 0) mbar_drain(WXb, 0);
    if (warp == kMmaWarp && elect_one()) { umma_commit(drainb); mbar_drain(drainb, 0); }
    __syncthreads();
  }
  cluster_barrier();                                       // no CTA may leave while a peer can still write into its shared memory
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// Recurrent weights as the CTAs put them into tensor memory: [rank][eight columns][half][lane] pieces of eight contraction
// indices, lane = gate row of the rank ((u / 8) 40 + gate 8 + u % 8), so that a warp reads whole lines (by rows of 1 KB it took
// 7 k cycles).
__global__ void k_pack_tt(int H, int E, int Hp, int gpc, const float* W, __nv_bfloat16* out) {
  const int m_rows = gpc * kGColsI, pitch = (m_rows + 31) / 32 * 32, cs = Hp / (8 * gpc);
  const size_t J = 5 * (size_t)H, total = (size_t)cs * (Hp / 4) * pitch * 8;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const int e = (int)(i % 8), m = (int)(i / 8 % pitch), piece = (int)(i / 8 / pitch % (Hp / 4)), rank = (int)(i / 8 / pitch / (Hp / 4));
    const int k = piece * 8 + e, kk = k < Hp ? k : k - Hp, u = rank * 8 * gpc + (m / kGColsI) * 8 + m % 8, g = m % kGColsI / 8;
    float v = 0.f;
    if (m < m_rows && u < H && kk < H) v = W[(size_t)(E + (k < Hp ? 0 : H) + kk) * J + g * H + u];
    out[i] = __float2bfloat16_rn(v);
  }
}

// Fitted to whole calls with the choice fixed either way (1 to 500 trees of up to 8 400 nodes together: sentences, chains, balanced;
// H = 120, 150, 256).  Forward in us, whole GPU against clusters: chain of 64 leaves, H = 256, 215 against 122, 64 of them 306 against
// 178, H = 150 327 against 145; 25 sentences 86 against 53 and 87 against 47; 200 balanced trees of 16 leaves 52 against 59 and 62
// against 68.  (A cluster's leaves are as many as its nodes; the clusters of eight CTAs, H = 129 to 192, take twice as long over each.)
WalkCosts tt_costs(int Hp) {
  if (Hp > 192) return {19.6f, 0.075f, 1.62f, 0.f, 18.f, 4.1f, 0.007f};
  if (Hp > 128) return {18.4f, 0.19f, 1.5f, 0.f, 19.f, 4.3f, 0.0075f};
  return {19.5f, 0.08f, 1.33f, 0.f, 18.f, 3.9f, 0.0035f};
}

int tt_smem_ok(const treelstm* ctx) {
  const TtLayout L = tt_layout(ctx->Hp, ctx->Ep, ctx->sf.groups_per_cta);
  const uint32_t gates_end = L.gates + (uint32_t)kLeafTile * (uint32_t)(ctx->sf.groups_per_cta * kGColsL) * 4u;
  // (an MMA reads 128 weight rows from the start of a K block, whatever lies behind the CTA's own)
  const uint32_t m_rows = (uint32_t)(ctx->sf.groups_per_cta * kGColsI);
  return L.R >= 16 && gates_end <= L.rk && L.wx_bytes + 128u * 128u <= L.rk && m_rows <= 128u && m_rows * 4u <= 2u * (uint32_t)ctx->Hp * 2u && ctx->Hp <= (int)kAcc0;
}

}  // namespace

// CTAs of a cluster and unit groups of a CTA, as the sub-forest kernel has them; 0: these sizes have none.
static int tt_groups(const treelstm* ctx) {
  const int groups = ctx->Hp / kUnitGroup, cs = groups % 16 == 0 ? 16 : 8;
  return ctx->precision == TREELSTM_BF16 && groups <= 3 * cs && groups % cs == 0 && ctx->Hp <= (int)kAcc0 ? groups / cs : 0;
}
size_t trees_tc_bytes(const treelstm* ctx) {
  const int gpc = tt_groups(ctx);
  return gpc ? (size_t)(ctx->Hp / (8 * gpc)) * (ctx->Hp / 4) * ((gpc * kGColsI + 31) / 32 * 32) * 16 : 0;
}
int pack_trees_tc(treelstm* ctx, cudaStream_t stream) {
  const int gpc = tt_groups(ctx);
  if (!gpc) return TREELSTM_OK;
  k_pack_tt<<<512, 256, 0, stream>>>(ctx->H, ctx->E, ctx->Hp, gpc, ctx->W, ctx->Wp_t);
  TL_CUDA(ctx, cudaGetLastError());
  return TREELSTM_OK;
}

// Whether and how this context's forests can go to clusters beside the scheduler.  After subforest_plan.
void init_trees_tc(treelstm* ctx) {
  auto& t = ctx->ttc;
  t = {};
  if (!ctx->sf.ok || ctx->sf.groups_per_cta != tt_groups(ctx) || !tt_smem_ok(ctx)) return;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ctx->sf.cluster_size; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  cfg.gridDim = dim3(ctx->sf.cluster_size); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = kSmemDynamic;
  cfg.attrs = &at; cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaFuncSetAttribute(k_schedule_trees_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemDynamic) != cudaSuccess ||
      cudaFuncSetAttribute(k_schedule_trees_tc, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&clusters, k_schedule_trees_tc, &cfg) != cudaSuccess || clusters < 2) {
    cudaGetLastError();
    return;
  }
  t.parts = clusters - 1 < kMaxTtParts ? clusters - 1 : kMaxTtParts;
  const TtLayout L = tt_layout(ctx->Hp, ctx->Ep, ctx->sf.groups_per_cta);
  int n = kMaxTtNodes;
  while (n > 0 && 4u * (uint32_t)tt_tables(n).wide + 4u * (uint32_t)(n / 2) > L.rk) n -= 256;
  t.max_nodes = n;
}

// Forests that the clusters are asked about: persistent mode with the library's own choice of kernels (no option that asks for
// one of them), tables that fit, a scheduler that the launch contains.
bool trees_tc_asked(const treelstm* ctx, int n, int flags) {
  return ctx->ttc.parts > 0 && (flags & TREELSTM_PERSISTENT) && !(flags & TREELSTM_SUBFORESTS) && ctx->opt.tail_width > 0 && ctx->opt.tail_min_levels == 0 &&
         ctx->opt.max_ctas == 0 && !ctx->opt.time_kernel && n >= 1 && n <= ctx->ttc.max_nodes && ctx->opt.sched_single_cta_max >= kSchedSingleMaxNodes;
}

// A forest that the clusters leave has a depth of more than R nodes, or more nodes than their lists hold.  One of no more than R nodes has neither whatever
// its shape, and the kernels behind, which would look and exit, are not launched: one sentence of 30 words from and to host arrays, H = 256, 53.0 -> 50.2 us.
bool trees_tc_always_take(const treelstm* ctx, int n) { return n <= tt_layout(ctx->Hp, ctx->Ep, ctx->sf.groups_per_cta).R; }

int launch_schedule_trees_tc(treelstm* ctx, int n, const int32_t* left, const int32_t* right, const int32_t* token, float* h, float* c, int32_t* level,
                             int32_t* order, int32_t* level_offset, int32_t* n_levels_out, bool save_gates, void* ws, const WsLayout& lay, cudaStream_t stream) {
  char* base = static_cast<char*>(ws);
  const int cs = ctx->sf.cluster_size;
  TtParams p{};
  p.f = {n, ctx->vocab, left, right, token};
  p.H = ctx->H; p.Hp = ctx->Hp; p.Ep = ctx->Ep; p.gpc = ctx->sf.groups_per_cta;
  p.chk_counts = check_counters(ws, lay);
  p.emb_bf = ctx->emb_bf; p.wp_t = reinterpret_cast<const uint4*>(ctx->Wp_t);
  p.bp_h = ctx->bp_h; p.bp_x = ctx->bp_x;
  p.h = h; p.c = c;
  p.gates = save_gates ? reinterpret_cast<float*>(base + lay.gates) : nullptr;
  p.hb = reinterpret_cast<__nv_bfloat16*>(base + lay.ain);
  p.st = reinterpret_cast<DevStatus*>(base + lay.status);
  p.wait_limit = ctx->opt.wait_limit_kcycles * 1024;
  p.costs = tt_costs(ctx->Hp);
#ifdef TREELSTM_TRACE
  p.trace = reinterpret_cast<long long*>(base + lay.trace) + kTraceSlots * kTraceLevels;
#endif
  TtSched q{};
  q.on_cluster = n >= kClusterMinNodes;
  q.sh = cl_shift(n, cs);
  q.cache_children = single_caches_children(n, false);
  q.parent = reinterpret_cast<int*>(base + lay.parent);
  q.level = level; q.order = order; q.order_tmp = reinterpret_cast<int*>(base + lay.order_tmp);
  q.level_offset = level_offset; q.roots = reinterpret_cast<int*>(base + lay.roots); q.n_levels_out = n_levels_out;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1] = behind_last(ctx, stream);
  cfg.gridDim = dim3(cs * (1 + ctx->ttc.parts)); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = kSmemDynamic; cfg.stream = stream;
  cfg.attrs = at; cfg.numAttrs = 2;
  TL_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_schedule_trees_tc, ctx->sf_maps.wx[0], p, q));
  ctx->launches += 1;
  return TREELSTM_OK;
}

}  // namespace tl
