// dW = In^T dZ and db = sum dZ of the training step on the tensor cores, at fp32 accuracy.
//
// Paper, Section 4.2.2: the weight gradient of the recursive body sums one outer product
// in_n (x) dz_n per invocation n.  That sum is the only large contraction of a training step
// ((E + 2H) x 5H outputs, contraction over all nodes) and has no dependency between wavefronts, so
// it runs once, after the last wavefront, as a dense GEMM: tcgen05.mma with fp32 accumulators in
// tensor memory.  The fp32 path owes its callers fp32 results, and bf16 operands carry 8 mantissa
// bits, so every operand value v is split into three bf16 pieces v = v0 + v1 + v2 (v0 = bf16(v),
// v1 = bf16(v - v0), v2 = bf16(v - v0 - v1): together the 24 bits of v) and six products are
// accumulated: a0 b0 + a0 b1 + a1 b0 + a1 b1 + a0 b2 + a2 b0; the three that are left out are below
// 2^-24 of |a b|.
//
// Work item = (part, 128 input rows, 128 gate columns, a run of 64-node blocks).  part 0: the leaves,
// input rows = embedding units (In = embedding row of the leaf's token); part 1: the internal nodes,
// input rows = [h_l | h_r].  One more input row holds ones: its output row is db.  A CTA builds its
// operand tiles in shared memory itself, straight from the fp32 arrays (gathered through the
// schedule), in the layout the tensor core reads: K-major rows of 128 bytes, 128-byte swizzle - the
// node index is the contraction index, so this is a transposition, done on the fly: a thread takes one
// input row (or gate column) and eight consecutive nodes, which is one 16-byte piece of that layout.
// Two stages of tiles: block b + 1 is built while the MMAs of block b run.  Partial sums of the node
// runs meet in dW by atomic adds (dW and db are cleared before), whole rows at a time through a
// shared-memory copy of the accumulator.
#include "split_tc.cuh"

namespace tl {
namespace {

constexpr int kDwThreads = 512;
constexpr int kDwTile = kSpTile;                 // rows of either operand tile (UMMA M and N)
constexpr int kDwBlock = kSpBlock;               // nodes per block of the contraction (one swizzle span of bf16)
constexpr int kDwStageBytes = kSpStageBytes;     // A and B, three pieces each: 96 KB
constexpr int kDwStages = 2;
constexpr int kDwMaxRun = 16;                    // blocks per work item at most (index tables in shared memory)
constexpr int kDwSmemBytes = kDwStages * kDwStageBytes + 1024;   // + alignment slack

struct DwParams {
  int n, n_leaves, H, E, vocab;
  int run;                      // 64-node blocks per work item
  const int *order, *token, *left, *right;
  const int* level_offset;      // level_offset[1] = number of leaves (the host may not know it)
  const float *emb, *h, *dz, *W;
  const int* tok_slot;          // row of every token in dEmb_rows (third kind of work item only)
  float *dW, *db, *dEmb_rows;   // dEmb_rows == nullptr: the leaves' input gradients are not formed here
  DevStatus* st;
  StatusOut out;
  long long wait_limit;
  BwdImages img;                // operands split beforehand (forests that went to the grid-wide wavefront kernel)
  int after_trees;              // the tree kernels took the forest if the control block says so, and img holds nothing
};

// One operand tile (128 rows x 64 nodes, three pieces) of block `kb` of the work item, in two steps: the
// fp32 values into registers (tile_load: nothing but loads, so all of a block's are in flight together),
// then split, packed and stored into shared memory (tile_store).
// kKind 0: input rows of the leaves (embedding units, then the row of ones), 1: input rows of the internal
// nodes ([h_l | h_r], then the row of ones), 2: gate columns (dz).  row0: first row of the tile within its
// operand.  s_node / s_ia / s_ib: per node of the item its id and where its input row comes from (token; left,
// right child); entries behind the item's last node are 0 and their values are discarded.  Warp w takes the
// nodes 8 (w mod 8) .. + 7 of the block, lane l the rows l and l + 32 of the tile's lower (w < 8) or upper half.
template <int kKind>
__device__ __forceinline__ void tile_load(const DwParams& p, int row0, const int* s_node, const int* s_ia,
                                          const int* s_ib, int kb, float (&v)[2][8]) {
  const int warp = (threadIdx.x >> 5) & 7, half = threadIdx.x >> 8, lane = threadIdx.x & 31;
  const int H = p.H, E = p.E, J = 5 * H;
  const int rows = kKind == 0 ? E : (kKind == 1 ? 2 * H : J);
#pragma unroll
  for (int rg = 0; rg < 2; ++rg) {
    const int fc = min(row0 + half * 64 + rg * 32 + lane, rows - 1);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = kb * kDwBlock + 8 * warp + i;
      const float* src;
      if (kKind == 0) src = p.emb + (size_t)s_ia[k] * E + fc;
      else if (kKind == 1) src = p.h + (size_t)(fc < H ? s_ia[k] : s_ib[k]) * H + (fc < H ? fc : fc - H);
      else src = p.dz + (size_t)s_node[k] * J + fc;
      v[rg][i] = kKind == 0 ? __ldg(src) : *src;
    }
  }
}
template <int kKind>
__device__ __forceinline__ void tile_store(const DwParams& p, unsigned char* tile, int row0, int valid_nodes,
                                           const float (&v)[2][8]) {
  const int warp = (threadIdx.x >> 5) & 7, half = threadIdx.x >> 8, lane = threadIdx.x & 31;
  const int rows = kKind == 0 ? p.E : (kKind == 1 ? 2 * p.H : 5 * p.H);   // row `rows` of an input operand is the ones
#pragma unroll
  for (int rg = 0; rg < 2; ++rg) {
    const int r = half * 64 + rg * 32 + lane, f = row0 + r;
    float x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool node_ok = 8 * warp + i < valid_nodes;
      x[i] = node_ok && f < rows ? v[rg][i] : 0.f;
      if (kKind != 2 && node_ok && f == rows) x[i] = 1.f;
    }
    split_store8(tile, r, warp, x);
  }
}

// The third kind of work item, dEmb_rows += dz_leaves W_x^T, contracts over the gate columns, which are
// contiguous in both operands (a leaf's dz row, a row of W): no transposition, a thread takes four
// consecutive columns - half of a 16-byte piece - of four rows, sixteen lanes a row's whole block (eight columns a thread, one after
// the other, had a warp touch 32 sectors with every load: 7.3 k cycles a block, this way 6.6 k).  row_ptr(r): start of tile row r in
// global memory; j0: first column of the block; J: columns in a row; pairs: rows are even and start on 8-byte boundaries.
template <class RowFn>
__device__ __forceinline__ void rows_load(RowFn row_ptr, int j0, int J, bool pairs, float (&v)[2][8]) {
  const int j = j0 + 4 * (threadIdx.x & 15);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float* row = row_ptr((threadIdx.x >> 4) + 32 * i);
    float* x = &v[i >> 1][4 * (i & 1)];
    if (pairs) {
      const float2 a = *reinterpret_cast<const float2*>(row + min(j, J - 2)), b = *reinterpret_cast<const float2*>(row + min(j + 2, J - 2));
      x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) x[e] = row[min(j + e, J - 1)];
    }
  }
}
__device__ __forceinline__ void rows_store(unsigned char* tile, int rows_valid, int j0, int J, const float (&v)[2][8]) {
  const int c = threadIdx.x & 15;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = (threadIdx.x >> 4) + 32 * i;
    float x[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) x[e] = r < rows_valid && j0 + 4 * c + e < J ? v[i >> 1][4 * (i & 1) + e] : 0.f;
    uint32_t w0[2], w1[2], w2[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) split3_pair(x[2 * e], x[2 * e + 1], w0[e], w1[e], w2[e]);
    unsigned char* dst = tile + swz_piece(r, c >> 1) + 8 * (c & 1);
    *reinterpret_cast<uint2*>(dst) = make_uint2(w0[0], w0[1]);
    *reinterpret_cast<uint2*>(dst + kSpTileBytes) = make_uint2(w1[0], w1[1]);
    *reinterpret_cast<uint2*>(dst + 2 * kSpTileBytes) = make_uint2(w2[0], w2[1]);
  }
}
// A finished tile from its copy in shared memory to the outputs: rows [0, rows) of `cols` columns, row r to out_of(r), in adds of V floats
// (5.5 to 6.5 k cycles one by one, H = 150, 4.2 to 5.5 k in pairs).
template <int V, class OutFn>
__device__ __forceinline__ void add_rows(const float* staged, int stride, int rows, int cols, OutFn out_of) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int r = warp; r < rows; r += kDwThreads / 32) {
    float* out = out_of(r);
#pragma unroll
    for (int i = 0; i < kDwTile / (32 * V); ++i) {
      const int c = V * (lane + 32 * i);
      if (c >= cols) continue;                               // (cols is a multiple of V)
      const float* x = staged + (size_t)r * stride + c;
      if constexpr (V == 4) atomicAdd(reinterpret_cast<float4*>(out + c), *reinterpret_cast<const float4*>(x));
      else if constexpr (V == 2) atomicAdd(reinterpret_cast<float2*>(out + c), *reinterpret_cast<const float2*>(x));
      else atomicAdd(out + c, *x);
    }
  }
}
template <class OutFn>
__device__ __forceinline__ void add_rows(const float* staged, int stride, int rows, int cols, int width, uintptr_t address, OutFn out_of) {   // `width` floats a row of the output
  if (width % 4 == 0 && address % 16 == 0) add_rows<4>(staged, stride, rows, cols, out_of);
  else if (width % 2 == 0 && address % 8 == 0) add_rows<2>(staged, stride, rows, cols, out_of);
  else add_rows<1>(staged, stride, rows, cols, out_of);
}

struct DwShape {
  int rows[2], nodes[2], first_pos[2], m_tiles[2], runs[2], items[3], n_tiles;
  // third kind (input gradients of the leaves): tiles of 128 leaves x 128 embedding units, contraction over
  // the 64-column blocks of the gate columns that are not all forget gates (those are zero for a leaf)
  int leaf_tiles, e_tiles, kblocks, skip_first, skip_count, runs2;
};
__host__ __device__ inline DwShape dw_shape(int n, int n_leaves, int H, int E, int run, bool leaf_dinput) {
  DwShape s;
  s.rows[0] = E; s.rows[1] = 2 * H;
  s.nodes[0] = n_leaves; s.nodes[1] = n - n_leaves;
  s.first_pos[0] = 0; s.first_pos[1] = n_leaves;
  s.n_tiles = (5 * H + kDwTile - 1) / kDwTile;
  for (int q = 0; q < 2; ++q) {
    s.m_tiles[q] = (s.rows[q] + 1 + kDwTile - 1) / kDwTile;   // + 1: the row of ones
    const int blocks = (s.nodes[q] + kDwBlock - 1) / kDwBlock;
    s.runs[q] = (blocks + run - 1) / run;
    s.items[q] = s.m_tiles[q] * s.n_tiles * s.runs[q];
  }
  const int all = (5 * H + kDwBlock - 1) / kDwBlock;
  s.skip_first = (H + kDwBlock - 1) / kDwBlock;              // first block that starts inside [H, 3H)
  const int skip_end = 3 * H / kDwBlock;                     // first block that ends outside it
  s.skip_count = skip_end > s.skip_first ? skip_end - s.skip_first : 0;
  s.kblocks = all - s.skip_count;
  s.leaf_tiles = (n_leaves + kDwTile - 1) / kDwTile;
  s.e_tiles = (E + kDwTile - 1) / kDwTile;
  s.runs2 = (s.kblocks + run - 1) / run;
  s.items[2] = leaf_dinput ? s.leaf_tiles * s.e_tiles * s.runs2 : 0;
  return s;
}
// The number of 64-wide blocks per work item: as few as give every CTA of the grid at most one item.  A whole warp, a lane per number.
__device__ __forceinline__ int dw_run(int n, int n_leaves, int H, int E, bool leaf_dinput, int ctas) {
  const DwShape s = dw_shape(n, n_leaves, H, E, min((int)(threadIdx.x & 31) + 1, kDwMaxRun), leaf_dinput);
  const unsigned fits = __ballot_sync(0xffffffffu, s.items[0] + s.items[1] + s.items[2] <= ctas);
  return min(fits ? __ffs(fits) : kDwMaxRun, kDwMaxRun);
}

// The sums over the nodes where the wavefront kernel has left both operands split (BwdImages): no thread touches a
// value before the accumulator.  One thread asks for the units of a block, one issues its MMAs, two stages; bound by the
// shared-memory reads of the MMAs (8 KB per 64 cycles of tensor pipe) and the 96 KB of a block on their way in.
// (Splitting inside this kernel instead converts every value of dz once per row tile: 335 us for 14.6 k nodes,
// H = 256, tensor pipe 24 % active, 43 % of the issue slots taken by conversions; this way 87 us.)
__device__ void dw_from_images(const DwParams& p, int n_leaves, unsigned char* tiles, uint32_t full_bar0, uint32_t empty_bar0,
                               uint32_t acc_bar, uint32_t tmem_base, int* s_abort_) {
  volatile int* s_abort = s_abort_;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = p.H, E = p.E, J = 5 * H;
  const int gp = gate_pitch(H), ju = img_units(5 * gp), xu[2] = {img_units(E + 1), img_units(2 * H + 1)};
  // column tiles; the leaves' forget gates are zero: tiles inside them [skip_lo, skip_lo + skip) are left out
  const int skip_lo = (gp + kDwTile - 1) / kDwTile, skip = max(0, 3 * gp / kDwTile - skip_lo);
  const int all_tiles = (5 * gp + kDwTile - 1) / kDwTile, n_tiles[2] = {all_tiles - skip, all_tiles};
  const int m_tiles[2] = {(E + 1 + kDwTile - 1) / kDwTile, (2 * H + 1 + kDwTile - 1) / kDwTile};
  const int pb_lo[2] = {0, n_leaves / 64}, pb_hi[2] = {(n_leaves + 63) / 64, p.n > n_leaves ? (p.n + 63) / 64 : n_leaves / 64};
  // runs of blocks as long as leave every CTA about two items (each ends in an atomic add per output)
  int run = 1, items[2];
  for (;; run *= 2) {
    for (int q = 0; q < 2; ++q) items[q] = m_tiles[q] * n_tiles[q] * ((pb_hi[q] - pb_lo[q] + run - 1) / run);
    if (items[0] + items[1] <= 2 * (int)gridDim.x || run >= 256) break;
  }
  const uint32_t tiles_addr = smem_u32(tiles), idesc = umma_idesc_mn(kDwTile);
  uint32_t put = 0, got = 0;             // blocks asked for / multiplied so far (thread 0 / thread 32)
  uint32_t done = 0;
  bool failed = false;
  for (int item = blockIdx.x; item < items[0] + items[1] && !failed; item += gridDim.x, ++done) {
    const int part = item < items[0] ? 0 : 1;
    int it = item - (part ? items[0] : 0);
    int nt = it % n_tiles[part]; it /= n_tiles[part];
    if (!part && nt >= skip_lo) nt += skip;
    const int mt = it % m_tiles[part], b0 = pb_lo[part] + it / m_tiles[part] * run;
    const int nblk = min(run, pb_hi[part] - b0);
    bool ok = true;
    if (tid == 0) {
      const unsigned char* xi = p.img.x[part];
      for (int b = 0; b < nblk && ok; ++b, ++put) {
        const uint32_t stage = put & 1u, dst = tiles_addr + stage * kDwStageBytes, bar = full_bar0 + 8 * stage;
        if (put >= 2) ok = mbar_wait(empty_bar0 + 8 * stage, ((put >> 1) - 1) & 1u, s_abort, p.wait_limit, p.st);
        if (!ok) break;
        const size_t pb = b0 + b;
        // (the last tile of either operand may have one unit only: the other half keeps what it holds, its outputs are dropped)
        const int ma = min(2, xu[part] - 2 * mt), mb = min(2, ju - 2 * nt);
        mbar_arrive_expect_tx(bar, (uint32_t)(ma + mb) * kUnitBytes);
        bulk_load(dst, xi + (pb * xu[part] + 2 * mt) * kUnitBytes, (uint32_t)ma * kUnitBytes, bar);
        bulk_load(dst + kSpOperandBytes, p.img.dz + (pb * ju + 2 * nt) * kUnitBytes, (uint32_t)mb * kUnitBytes, bar);
      }
    } else if (warp == 1) {
      const bool issue = elect_one();
      for (int b = 0; b < nblk && ok; ++b, ++got) {
        const uint32_t stage = got & 1u, src = tiles_addr + stage * kDwStageBytes;
        ok = __all_sync(0xffffffffu, mbar_wait(full_bar0 + 8 * stage, (got >> 1) & 1u, s_abort, p.wait_limit, p.st));
        if (!ok) break;
        tc_fence_after();
        split_mmas_mn(tmem_base, src, src + kSpOperandBytes, idesc, b == 0, issue);
        if (issue) umma_commit(empty_bar0 + 8 * stage);
        if (issue && b == nblk - 1) umma_commit(acc_bar);
      }
    }
    __syncwarp();
    ok = mbar_wait(acc_bar, done & 1u, s_abort, p.wait_limit, p.st) && ok;
    if (__syncthreads_or(!ok)) { failed = true; break; }
    tc_fence_after();
    // tensor memory -> row segments: a warp reads 32 rows x 32 columns, lane = row; adds go out along the row through a transposition
    {
      const int quad = warp & 3, quarter = warp >> 2;
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(quarter * 32);
      float v[32];
      split_sum(taddr, v);
      tc_fence_before();
      constexpr int kRowStride = kDwTile + 4;
      float* stage_out = reinterpret_cast<float*>(tiles);   // both stages are idle: every block asked for has been multiplied
      float* dst = stage_out + (size_t)(quad * 32 + lane) * kRowStride + quarter * 32;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *reinterpret_cast<float4*>(dst + 4 * i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      __syncthreads();
      const int rows = part ? 2 * H : E, m0 = mt * kDwTile;
      auto column = [&](int c) {                              // of dW; none behind a gate's last unit
        const int gate = (nt * kDwTile + c) / gp, u = nt * kDwTile + c - gate * gp;
        return gate < 5 && u < H ? gate * H + u : -1;
      };
      auto row_of = [&](int f) { return f == rows ? p.db : p.dW + (size_t)((part ? E : 0) + f) * J; };
      const int r_end = min(kDwTile, rows + 1 - m0);
      if (H % 4 == 0 && ((reinterpret_cast<uintptr_t>(p.dW) | reinterpret_cast<uintptr_t>(p.db)) & 15) == 0) {
        const int j = column(4 * lane);
        if (j >= 0)
          for (int r = warp; r < r_end; r += kDwThreads / 32)
            atomicAdd(reinterpret_cast<float4*>(row_of(m0 + r) + j), *reinterpret_cast<const float4*>(stage_out + (size_t)r * kRowStride + 4 * lane));
      } else {
        int j[kDwTile / 32];
#pragma unroll
        for (int i = 0; i < kDwTile / 32; ++i) j[i] = column(lane + 32 * i);
        for (int r = warp; r < r_end; r += kDwThreads / 32) {
          float* out = row_of(m0 + r);
#pragma unroll
          for (int i = 0; i < kDwTile / 32; ++i)
            if (j[i] >= 0) atomicAdd(out + j[i], stage_out[(size_t)r * kRowStride + lane + 32 * i]);
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the next item's bulk copies overwrite the staging rows
    __syncthreads();
  }
}

__device__ __forceinline__ void dweight(DwParams& p) {
  extern __shared__ unsigned char dw_dyn[];
  __shared__ int s_node[kDwMaxRun * kDwBlock], s_ia[kDwMaxRun * kDwBlock], s_ib[kDwMaxRun * kDwBlock];
  __shared__ __align__(8) uint64_t s_bars[2 * kDwStages + 2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  // What the forward has left (status, level table, order) is final before this kernel comes up.
  if (__syncthreads_or(ld_volatile(&p.st->status) != 0)) {   // the forward failed: nothing here may be trusted
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* tiles = dw_dyn + ((1024u - (smem_u32(dw_dyn) & 1023u)) & 1023u);
  const uint32_t tiles_addr = smem_u32(tiles);
  const uint32_t stage_bar0 = smem_u32(&s_bars[0]), acc_bar = smem_u32(&s_bars[kDwStages]),
                 drain_bar = smem_u32(&s_bars[kDwStages + 1]);
  if (tid == 0) {
    for (int s = 0; s < kDwStages; ++s) mbar_init(stage_bar0 + 8 * s, 1);
    for (int s = 0; s < kDwStages; ++s) mbar_init(smem_u32(&s_bars[kDwStages + 2 + s]), 1);
    mbar_init(acc_bar, 1);
    mbar_init(drain_bar, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(smem_u32(&s_tmem), kSpTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = s_tmem;
  const int H = p.H, E = p.E, J = 5 * H;
  const int n_leaves = p.st->n_levels > 0 ? min(p.n, max(0, p.level_offset[1])) : 0;
  const bool leaf_dinput = p.dEmb_rows != nullptr;
  // (Where the host knows that the operands are split, nothing is set up here: it would be behind the kernel ahead, 2 us of a step of 256 sentences.)
  const bool images = p.img.dz != nullptr && !p.after_trees;
  int run = 1;                           // the host does not know the number of leaves
  DwShape sh{};
  if (!images) {
    run = dw_run(p.n, n_leaves, H, E, leaf_dinput, (int)gridDim.x);
    sh = dw_shape(p.n, n_leaves, H, E, run, leaf_dinput);
  }
  const uint32_t idesc = umma_idesc(kDwTile);
  const int n_items = sh.items[0] + sh.items[1] + sh.items[2];
  int part = 0, m0 = 0, j0 = 0, pos0 = 0, pos_end = 0, nblk = 0, kb0 = 0, rows_here = 0;   // of the CTA's item
  auto take = [&](int item) {            // its place and its tables
    part = item < sh.items[0] ? 0 : (item < sh.items[0] + sh.items[1] ? 1 : 2);
    int it = item - (part > 0 ? sh.items[0] : 0) - (part > 1 ? sh.items[1] : 0);
    pos0 = pos_end = kb0 = rows_here = 0;
    if (part < 2) {
      const int nt = it % sh.n_tiles; it /= sh.n_tiles;
      const int mt = it % sh.m_tiles[part], ri = it / sh.m_tiles[part];
      m0 = mt * kDwTile; j0 = nt * kDwTile;
      pos0 = sh.first_pos[part] + ri * run * kDwBlock;
      pos_end = min(sh.first_pos[part] + sh.nodes[part], pos0 + run * kDwBlock);
      nblk = (pos_end - pos0 + kDwBlock - 1) / kDwBlock;
      // the item's nodes and where their input rows come from
      for (int t = tid; t < nblk * kDwBlock; t += kDwThreads) {
        int node = 0, ia = 0, ib = 0;
        if (pos0 + t < pos_end) {
          node = chk(p.st, p.order[pos0 + t], p.n);
          if (part == 0) ia = chk(p.st, p.token[node], p.vocab);
          else { ia = chk(p.st, p.left[node], p.n); ib = chk(p.st, p.right[node], p.n); }
        }
        s_node[t] = node; s_ia[t] = ia; s_ib[t] = ib;
      }
    } else {
      const int et = it % sh.e_tiles; it /= sh.e_tiles;
      const int lt = it % sh.leaf_tiles, ri = it / sh.leaf_tiles;
      m0 = lt * kDwTile;                 // first leaf (position in the ready order: the leaves are wavefront 0)
      j0 = et * kDwTile;                 // first embedding unit
      rows_here = min(kDwTile, n_leaves - m0);
      kb0 = ri * run;                    // first of the item's blocks among those that are not skipped
      nblk = min(run, sh.kblocks - kb0);
      // the tile's leaves and their rows of dEmb_rows
      for (int t = tid; t < kDwTile; t += kDwThreads) {
        int node = 0, slot = 0;
        if (t < rows_here) {
          node = chk(p.st, p.order[m0 + t], p.n);
          slot = chk(p.st, p.tok_slot[chk(p.st, p.token[node], p.vocab)], n_leaves);
        }
        s_node[t] = node; s_ia[t] = slot;
      }
    }
  };
  // The first item's tables hold rows of the embedding gradient (tok_slot), which k_bwd_begin or, where that is the kernel ahead, k_bwd_persistent numbers.
  // Behind the tree kernels they are read ahead of the wait: k_bwd_begin has ended when k_trees_backward lets this kernel come up, and a kernel between
  // those two lets go at its end only and leaves the rows alone.  Else the kernel ahead is waited for first.
  if (!p.after_trees) asm volatile("griddepcontrol.wait;" ::: "memory");
  if ((int)blockIdx.x < n_items) take(blockIdx.x);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const bool stop = __syncthreads_or(ld_volatile(&p.st->status) != 0) != 0;   // (a label out of range)
  if (!stop && (images || (p.img.dz != nullptr && !p.st->trees_bwd))) {
    dw_from_images(p, n_leaves, tiles, stage_bar0, smem_u32(&s_bars[kDwStages + 2]), acc_bar, tmem_base, &s_abort);
    tc_fence_before();
    __syncthreads();
    if (s_abort) {                         // what was asked for gets a bounded time to land, the MMAs a bounded time to retire
      if (warp == 1 && elect_one()) { umma_commit(drain_bar); mbar_drain(drain_bar, 0); }
      if (tid == 0) for (int s = 0; s < kDwStages; ++s) mbar_drain(stage_bar0 + 8 * s, 0);
      __syncthreads();
    }
    if (warp == 0) {
      tc_fence_after();
      tmem_dealloc(tmem_base, kSpTmemCols);
    }
    return;
  }
  uint32_t built = 0, items_done = 0;   // blocks built / items finished by this CTA so far (barrier phases)
  bool failed = false;
  for (int item = blockIdx.x; item < n_items && !failed && !stop; item += gridDim.x) {
    if (item != (int)blockIdx.x) take(item);
    __syncthreads();
    // The fp32 values of block b + 1 are on their way into registers while block b is split, stored and multiplied.
    auto block_col = [&](int b) {        // part 2: first gate column of the block
      const int kb = kb0 + b;
      return (kb < sh.skip_first ? kb : kb + sh.skip_count) * kDwBlock;
    };
    float va[2][8], vb[2][8], na[2][8], nb[2][8];
    auto load_block = [&](int b) {
      if (part == 0) tile_load<0>(p, m0, s_node, s_ia, s_ib, b, na);
      else if (part == 1) tile_load<1>(p, m0, s_node, s_ia, s_ib, b, na);
      else rows_load([&](int r) { return p.dz + (size_t)s_node[r] * J; }, block_col(b), J, J % 2 == 0, na);   // (dz and W: the library's, on 256-byte boundaries)
      if (part < 2) tile_load<2>(p, j0, s_node, s_ia, s_ib, b, nb);
      else rows_load([&](int r) { return p.W + (size_t)min(j0 + r, E - 1) * J; }, block_col(b), J, J % 2 == 0, nb);
    };
    load_block(0);
    for (int b = 0; b < nblk; ++b, ++built) {
      const uint32_t stage = built & 1u, use = built >> 1;
      unsigned char* st_tiles = tiles + stage * kDwStageBytes;
      const int valid_nodes = min(kDwBlock, pos_end - pos0 - b * kDwBlock);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int e = 0; e < 8; ++e) { va[i][e] = na[i][e]; vb[i][e] = nb[i][e]; }
      if (b + 1 < nblk) load_block(b + 1);
      bool ok = true;
      if (use >= 1)   // the MMAs that read this stage two blocks ago must have retired before it is overwritten
        ok = mbar_wait(stage_bar0 + 8 * stage, (use - 1) & 1u, &s_abort, p.wait_limit, p.st);
      if (__syncthreads_or(!ok)) { failed = true; break; }
      if (part == 0) tile_store<0>(p, st_tiles, m0, valid_nodes, va);
      else if (part == 1) tile_store<1>(p, st_tiles, m0, valid_nodes, va);
      else rows_store(st_tiles, rows_here, block_col(b), J, va);
      if (part < 2) tile_store<2>(p, st_tiles + kSpOperandBytes, j0, valid_nodes, vb);
      else rows_store(st_tiles + kSpOperandBytes, min(kDwTile, E - j0), block_col(b), J, vb);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy stores -> visible to the tensor core
      tc_fence_before();
      __syncthreads();
      if (warp == 0) {
        const bool issue = elect_one();
        tc_fence_after();
        const uint32_t a_addr = tiles_addr + stage * kDwStageBytes;
        split_mmas(tmem_base, a_addr, a_addr + kSpOperandBytes, idesc, b == 0, issue);
        if (issue) umma_commit(stage_bar0 + 8 * stage);
        if (issue && b == nblk - 1) umma_commit(acc_bar);
      }
    }
    if (failed) break;
    // the accumulator: tensor memory -> registers -> shared memory (whole rows) -> atomic adds of row segments
    const bool acc_ok = mbar_wait(acc_bar, items_done & 1u, &s_abort, p.wait_limit, p.st);
    if (__syncthreads_or(!acc_ok)) { failed = true; break; }
    ++items_done;
    tc_fence_after();
    constexpr int kRowStride = kDwTile + 4;                 // floats; 16-byte stores of a warp's 32 rows spread over all banks
    float* stage_out = reinterpret_cast<float*>(tiles);     // every MMA that read the operand stages has retired
    {
      const int quad = warp & 3, quarter = warp >> 2;       // a warp reads the tensor-memory lanes of quadrant (warp id mod 4)
      const int r = quad * 32 + lane;
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(quarter * 32);
      float v[32];
      split_sum(taddr, v);
      tc_fence_before();
      float* dst = stage_out + (size_t)r * kRowStride + quarter * 32;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *reinterpret_cast<float4*>(dst + 4 * i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
    __syncthreads();
    const int rows_valid = part < 2 ? min(kDwTile, sh.rows[part] + 1 - m0) : rows_here;
    const int cols_valid = part < 2 ? min(kDwTile, J - j0) : min(kDwTile, E - j0);
    if (part < 2)
      add_rows(stage_out, kRowStride, rows_valid, cols_valid, J, reinterpret_cast<uintptr_t>(p.dW) | reinterpret_cast<uintptr_t>(p.db),
               [&](int r) { return m0 + r == sh.rows[part] ? p.db + j0 : p.dW + (size_t)((part ? E : 0) + m0 + r) * J + j0; });
    else                                                     // leaves with the same token share a row
      add_rows(stage_out, kRowStride, rows_valid, cols_valid, E, reinterpret_cast<uintptr_t>(p.dEmb_rows),
               [&](int r) { return p.dEmb_rows + (size_t)s_ia[r] * E + j0; });
    __syncthreads();   // the next item overwrites the index tables, the stages and the accumulator
  }
  // teardown: MMAs still in flight after a failed wait get a bounded time to retire before tensor memory goes back
  tc_fence_before();
  __syncthreads();
  if (failed && warp == 0 && elect_one()) {
    umma_commit(drain_bar);
    mbar_drain(drain_bar, 0);
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kSpTmemCols);
  }
}
__global__ void __launch_bounds__(kDwThreads, 1) k_bwd_dweight_tc(DwParams p) {
  dweight(p);
  publish_status(p.st, p.out);
}

}  // namespace

// W -> its split image (see wsp_bytes)
__global__ void k_split_w(int H, int E, const float* W, unsigned char* out) {
  const int J = 5 * H, gp = gate_pitch(H), kbs = wsp_kblocks(H), tx = wsp_tiles_x(E), tiles = tx + wsp_tiles_h(H);
  const int total = tiles * kbs * kSpTile * 8;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < total; q += gridDim.x * blockDim.x) {
    const int c = q & 7, r = (q >> 3) % kSpTile, kb = (q >> 3) / kSpTile % kbs, t = (q >> 3) / kSpTile / kbs;
    const int row = t < tx ? t * kSpTile + r : (t - tx) * kSpTile + r;
    const bool in = row < (t < tx ? E : 2 * H);
    float x[8];
    for (int e = 0; e < 8; ++e) {
      const int j = kb * kSpBlock + 8 * c, gate = j / gp, u = j - gate * gp + e;
      x[e] = in && gate < 5 && u < H ? W[(size_t)(t < tx ? row : E + row) * J + gate * H + u] : 0.f;
    }
    split_store8(out + (size_t)(t * kbs + kb) * kSpOperandBytes, r, c, x);
  }
}
size_t wide_backward_bytes(const treelstm* ctx) {
  if (ctx->cell != 0 || ctx->H > 512 || ctx->E > 1024) return 0;
  return round_up_sz(wsp_bytes(ctx->H, ctx->E), 1024);
}
int pack_wide_backward(treelstm* ctx, cudaStream_t stream) {
  if (!ctx->wsp) return TREELSTM_OK;
  k_split_w<<<592, 256, 0, stream>>>(ctx->H, ctx->E, ctx->W, ctx->wsp);
  TL_CUDA(ctx, cudaGetLastError());
  return TREELSTM_OK;
}
// bytes of the images of n positions x `features` features (one unit row more than needed: tiles of 128 positions)
size_t image_bytes(int n, int features) { return (size_t)((n + 63) / 64 + 1) * img_units(features) * kUnitBytes; }

int init_dweight_tc_attributes(treelstm* ctx) {
  TL_CUDA(ctx, cudaFuncSetAttribute(k_bwd_dweight_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmemBytes));
  return TREELSTM_OK;
}

// dW, db (and dEmb_rows, if given: then tok_slot holds every token's row) must have been cleared on the
// stream before; dz holds the gate gradients of every node.
int launch_dweight_tc(treelstm* ctx, int n, const int32_t* order, const int32_t* level_offset, const int32_t* token,
                      const int32_t* left, const int32_t* right, const float* h, const float* dz, float* dW, float* db,
                      const int* tok_slot, float* dEmb_rows, DevStatus* st, const BwdImages* img, bool after_trees, cudaStream_t stream) {
  DwParams p;
  if (img) p.img = *img;
  p.after_trees = after_trees ? 1 : 0;
  p.n = n; p.n_leaves = 0; p.H = ctx->H; p.E = ctx->E; p.vocab = ctx->vocab; p.run = 0;
  p.order = order; p.level_offset = level_offset; p.token = token; p.left = left; p.right = right;
  p.emb = ctx->emb; p.h = h; p.dz = dz; p.W = ctx->W; p.dW = dW; p.db = db; p.st = st;
  p.tok_slot = tok_slot; p.dEmb_rows = dEmb_rows;
  p.wait_limit = ctx->opt.wait_limit_kcycles * 1024;
  if (n == 0) return TREELSTM_OK;
  p.out = {ctx->bwd_status, expect_status(ctx, stream)};
  // The host does not know how the nodes divide into leaves and internal nodes (the level table stayed on the
  // device), so the kernel sizes its work items itself from the grid it finds: one CTA per SM unless even
  // single-block items are fewer (counted for the division that gives the most).
  int items = 0;
  for (int nl = 0; nl <= n; nl += (n > 8 ? n / 8 : 1)) {
    const DwShape s = dw_shape(n, nl, p.H, p.E, 1, dEmb_rows != nullptr);
    const int c = s.items[0] + s.items[1] + s.items[2];
    if (c > items) items = c;
  }
  const int grid = items < ctx->sm_count ? items : ctx->sm_count;
  // (as the programmatic dependent of whatever is ahead: it comes up while that ends)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3(kDwThreads); cfg.dynamicSmemBytes = kDwSmemBytes; cfg.stream = stream;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization; at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at; cfg.numAttrs = 1;
  TL_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_bwd_dweight_tc, p));
  ctx->launches += 1;
  return TREELSTM_OK;
}

}  // namespace tl
