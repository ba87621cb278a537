// fwd_tc.cuh -- what the tensor-core forward scans (fwd_tc.cu, fwd_pair.cu)
// share: the operand-tile writers and the tensor maps.
#pragma once
#include "chunk_common.cuh"
#include "tc_common.cuh"

namespace rdn {
namespace fwdtc {

using namespace tc;

constexpr int D = 128;
constexpr int kTcThreads = 512;
constexpr int kGroups = kTcThreads / 128;  // threads sharing a value column
static_assert(kGroups == 4, "each group owns 16 of a chunk's 64 token columns");

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t *>(&v);
}

// Write 16 consecutive values (columns c0..c0+15 of row r) of a K-major SW128
// tile whose 64-column blocks are blk_bytes apart.
__device__ __forceinline__ void st_row16(uint8_t *tile, uint32_t blk_bytes, int r, int c0,
                                         const float (&v)[16]) {
  uint8_t *blk = tile + (c0 >> 6) * blk_bytes;
  const int cc = c0 & 63;
  uint4 a, b;
  a.x = pack_bf16(v[0], v[1]);
  a.y = pack_bf16(v[2], v[3]);
  a.z = pack_bf16(v[4], v[5]);
  a.w = pack_bf16(v[6], v[7]);
  b.x = pack_bf16(v[8], v[9]);
  b.y = pack_bf16(v[10], v[11]);
  b.z = pack_bf16(v[12], v[13]);
  b.w = pack_bf16(v[14], v[15]);
  *reinterpret_cast<uint4 *>(blk + sw128(r, cc)) = a;
  *reinterpret_cast<uint4 *>(blk + sw128(r, cc + 8)) = b;
}

// Same, split into bf16 hi + lo parts (split_pack_bf16) in two tiles.
__device__ __forceinline__ void st_row16_split(uint8_t *hi, uint8_t *lo, int r, int c0,
                                               const float (&v)[16]) {
  uint32_t h[8], l[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) split_pack_bf16(v[2 * i], v[2 * i + 1], h[i], l[i]);
  const int cc = c0 & 63;
  *reinterpret_cast<uint4 *>(hi + sw128(r, cc)) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4 *>(hi + sw128(r, cc + 8)) = make_uint4(h[4], h[5], h[6], h[7]);
  *reinterpret_cast<uint4 *>(lo + sw128(r, cc)) = make_uint4(l[0], l[1], l[2], l[3]);
  *reinterpret_cast<uint4 *>(lo + sw128(r, cc + 8)) = make_uint4(l[4], l[5], l[6], l[7]);
}

// D (+)= (A_hi + A_lo)(B_hi + B_lo)^T without the lo*lo term: three MMAs
// over K = 64 for K-major 128B-swizzled tiles.
__device__ __forceinline__ void mma_split3(uint32_t d, uint32_t a_hi, uint32_t a_lo,
                                           uint32_t b_hi, uint32_t b_lo, uint32_t idesc,
                                           bool accumulate_first) {
  mma_tile(d, a_hi, 0, b_hi, 0, 4, idesc, accumulate_first);
  mma_tile(d, a_hi, 0, b_lo, 0, 4, idesc, true);
  mma_tile(d, a_lo, 0, b_hi, 0, 4, idesc, true);
}

// Tensor maps (CUtensorMap, 64-byte aligned) over v, k, q as [tokens][H][D]
// with a 64-token x 64-column box (make_tile_map); ok: they are valid.
struct FwdMaps {
  alignas(64) unsigned char v[128];
  alignas(64) unsigned char k[128];
  alignas(64) unsigned char q[128];
  bool ok;
  alignas(64) unsigned char o[128];  // (fwd_pair.cu: bf16 results)
  bool o_ok;
};

}  // namespace fwdtc

// The scan over a CTA pair per (sequence, head) (fwd_pair.cu).
cudaError_t launch_fwd_pair(const FwdParams &p, const fwdtc::FwdMaps &maps, bool rdnv, cudaStream_t s);

}  // namespace rdn
