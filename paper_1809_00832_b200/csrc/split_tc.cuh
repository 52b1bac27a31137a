// fp32 contractions on the tensor cores: every operand value v is split into three bf16 pieces v = v0 + v1 + v2
// (v0 = bf16(v), v1 = bf16(v - v0), v2 = bf16(v - v0 - v1): together the 24 bits of v) and six of the nine products
// of pieces are accumulated in fp32; the three that are left out are below 2^-24 of |a b|.  Operand tiles are
// 128 rows x 64 contraction indices, one 16 KB tile per piece, K-major rows of 128 bytes with the 128-byte swizzle.
#pragma once

#include "tc_ptx.cuh"

namespace tl {

constexpr int kSpTile = 128, kSpBlock = 64, kSpPieces = 3;
constexpr int kSpTileBytes = kSpTile * 128;
constexpr int kSpOperandBytes = kSpPieces * kSpTileBytes;     // one operand of one block: 48 KB
constexpr int kSpStageBytes = 2 * kSpOperandBytes;

// (x, y) -> three words of two bf16 pieces each (x in the low half): x = x0 + x1 + x2, y likewise
__device__ __forceinline__ void split3_pair(float x, float y, uint32_t& w0, uint32_t& w1, uint32_t& w2) {
  auto pack = [](float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
  };
  w0 = pack(x, y);
  x -= __uint_as_float(w0 << 16);  y -= __uint_as_float(w0 & 0xFFFF0000u);
  w1 = pack(x, y);
  x -= __uint_as_float(w1 << 16);  y -= __uint_as_float(w1 & 0xFFFF0000u);
  w2 = pack(x, y);
}
// byte offset of the 16-byte piece (row r, contraction indices 8 c .. 8 c + 7) inside a tile
__device__ __forceinline__ uint32_t swz_piece(int r, int c) {
  return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4));
}
// eight values of row r -> their place in the three tiles
__device__ __forceinline__ void split_store8(unsigned char* tiles, int r, int c, const float (&x)[8]) {
  uint32_t w0[4], w1[4], w2[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) split3_pair(x[2 * e], x[2 * e + 1], w0[e], w1[e], w2[e]);
  unsigned char* dst = tiles + swz_piece(r, c);
  *reinterpret_cast<uint4*>(dst) = make_uint4(w0[0], w0[1], w0[2], w0[3]);
  *reinterpret_cast<uint4*>(dst + kSpTileBytes) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
  *reinterpret_cast<uint4*>(dst + 2 * kSpTileBytes) = make_uint4(w2[0], w2[1], w2[2], w2[3]);
}
// The MMAs of one block (a whole warp, issued by its elected lane): (piece of A, piece of B).  The tensor core cuts a sum
// off where it leaves its 24 bits, towards zero: every MMA into an accumulator may cost it half a last place, always in the
// same direction.  So the five small products, 2^-8 and less of the first, have an accumulator of their own, the product
// of the first pieces three (by step), and the four meet once, rounded (split_sum).  dW of 58 trees of 128 leaves, H = 198, is
// 6.5e-7 of its norm off the fp64 result (in runs of few blocks with one accumulator: 3.2e-6; in long ones 1e-5), at the same time.
constexpr int kSpTmemCols = 4 * kSpTile;
__device__ __forceinline__ void split_mmas(uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, uint32_t idesc, bool first_block, bool issue) {
#pragma unroll
  for (int k = 0; k < kSpBlock / 16; ++k)     // UMMA K = 16 bf16 = 32 bytes = 2 descriptor units
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int pa = (0x010120 >> (4 * q)) & 0xF, pb = (0x001102 >> (4 * q)) & 0xF;
      if (issue) umma_bf16(d_tmem + (q == 5 ? k % 3 : 3) * kSpTile, umma_desc(a_addr + pa * kSpTileBytes) + 2 * k,
                           umma_desc(b_addr + pb * kSpTileBytes) + 2 * k, idesc, !(first_block && (q == 5 ? k < 3 : k == 0 && q == 0)));
    }
}
// 32 columns of the finished sums of this thread's row
__device__ __forceinline__ void split_sum(uint32_t taddr, float (&x)[32]) {
#pragma unroll
  for (int h = 0; h < 32; h += 16) {
    uint32_t v[4][16];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i) tmem_ld4(taddr + q * kSpTile + h + 4 * i, v[q] + 4 * i);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; ++i)
      x[h + i] = (__uint_as_float(v[0][i]) + __uint_as_float(v[1][i])) + (__uint_as_float(v[2][i]) + __uint_as_float(v[3][i]));
  }
}
// bytes (a multiple of 16) from global to shared memory, counted on an mbarrier
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// whether the 128 columns of tile t are a leaf's forget gates, all of them (zero: not computed with)
__host__ __device__ inline bool forget_tile(int t, int gp) { return t * 128 >= gp && (t + 1) * 128 <= 3 * gp; }

// W split once, in the layout of the tiles: rows of W in tiles of 128 (the input rows [0, E) first, then the 2H state
// rows), columns in blocks of 64; block (tile, kb) is kSpOperandBytes at ((tile * kblocks) + kb).
__host__ __device__ inline int wsp_kblocks(int H) { return (5 * gate_pitch(H) + kSpBlock - 1) / kSpBlock; }
__host__ __device__ inline int wsp_tiles_x(int E) { return (E + kSpTile - 1) / kSpTile; }
__host__ __device__ inline int wsp_tiles_h(int H) { return (2 * H + kSpTile - 1) / kSpTile; }
__host__ __device__ inline size_t wsp_bytes(int H, int E) {
  return (size_t)(wsp_tiles_x(E) + wsp_tiles_h(H)) * wsp_kblocks(H) * kSpOperandBytes;
}

// Images of the operands of the backward pass: units of 64 positions (ready order) x 64 features, each piece one 8 KB
// tile of 64 rows of 128 bytes; unit (pb, fb) is kUnitBytes at pb * units_per_row + fb.  A unit is K-major where the
// contraction runs over the features (dz W^T) and MN-major where it runs over the positions (In^T dz).
constexpr int kUnitPieceBytes = 64 * 128, kUnitBytes = kSpPieces * kUnitPieceBytes;
__host__ __device__ inline int img_units(int features) { return (features + 63) / 64; }
struct BwdImages {                       // nullptr: not kept
  unsigned char *dz = nullptr, *x[2] = {nullptr, nullptr};   // x[0]: embedding rows and a one, x[1]: [h_l | h_r] and a one
  const unsigned char* w = nullptr;      // W split (wsp layout)
};
__device__ __forceinline__ void split_store8_unit(unsigned char* unit, int r, int c, const float (&x)[8]) {
  uint32_t w0[4], w1[4], w2[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) split3_pair(x[2 * e], x[2 * e + 1], w0[e], w1[e], w2[e]);
  unsigned char* dst = unit + swz_piece(r, c);
  *reinterpret_cast<uint4*>(dst) = make_uint4(w0[0], w0[1], w0[2], w0[3]);
  *reinterpret_cast<uint4*>(dst + kUnitPieceBytes) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
  *reinterpret_cast<uint4*>(dst + 2 * kUnitPieceBytes) = make_uint4(w2[0], w2[1], w2[2], w2[3]);
}
// MN-major operand of two units side by side (128 of the outer dimension): rows of 128 bytes run along it, groups of
// eight contraction indices 1024 bytes apart, the second unit kUnitBytes further
__device__ __forceinline__ uint64_t umma_desc_mn(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFF) >> 4);
  d |= (uint64_t)(kUnitBytes >> 4) << 16; // leading byte offset: next 64 of the outer dimension
  d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset: next eight contraction indices
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;                 // SWIZZLE_128B
  return d;
}
__device__ __forceinline__ uint32_t umma_idesc_mn(int n) { return umma_idesc(n) | (1u << 15) | (1u << 16); }
// one block (64 positions) of In^T dz: both operands MN-major, [unit][piece] in shared memory
__device__ __forceinline__ void split_mmas_mn(uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, uint32_t idesc, bool first_block, bool issue) {
#pragma unroll
  for (int k = 0; k < 4; ++k)            // 16 positions = two groups of eight
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int pa = (0x010120 >> (4 * q)) & 0xF, pb = (0x001102 >> (4 * q)) & 0xF;
      if (issue) umma_bf16(d_tmem + (q == 5 ? k % 3 : 3) * kSpTile, umma_desc_mn(a_addr + pa * kUnitPieceBytes) + 128 * k,
                           umma_desc_mn(b_addr + pb * kUnitPieceBytes) + 128 * k, idesc, !(first_block && (q == 5 ? k < 3 : k == 0 && q == 0)));
    }
}

}  // namespace tl
