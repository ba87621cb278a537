// bwd_tc.cuh -- what the tensor-core backward kernels (bwd_tc.cu, bwd_chain.cu)
// share: their parameters, operand-tile writers, and the barriers and phases of
// a CTA.
#pragma once
#include "chunk_common.cuh"
#include "tc_common.cuh"

namespace rdn {
namespace bwdtc {

using namespace tc;

constexpr int D = 128;
constexpr int NTC = 512;  // bwd_chain's element-wise threads (4 warps per TMEM lane quadrant)

struct TcBwdParams {
  FwdParams f;          // inputs; f.ws = prep records (shared-memory images)
  const void *dO;
  const float *dST, *dRT;
  const float *Sc, *Rc;  // chunk-start states [B,H,NC,D,D]
  void *dv;
  float *dS0, *dR0;
  uint8_t *Ebuf, *E2buf; // [B*H*NC][32 KB]: images of E^T, E2^T (rows j, columns t; hi | lo)
  float *dX2buf, *dXbuf; // [B*H*NC][64][128]
  uint8_t *gimg;         // [B*H*NC][128 KB]: gradients w.r.t. each chunk's end states as
                         // bf16 images (rows j): dS hi | dR hi | dS lo | dR lo, 32 KB each
  unsigned long long *mask;  // [B*H*NC][128]: bit t = clip inactive (|x| <= c)
  void *dq, *dk;             // outputs of bwd_post
  float *dg, *dbeta, *dgamma;
  // RLA: the records carry T_beta = T_gamma = I and the deltas are absent
  // (E = V, E2 = r), so the terms through -Gam K S0, -Gam K R0 and the
  // gradients of A_beta, A_gamma drop out; the chunk-start state enters the
  // recomputed prediction with a lo part (RLA's S is not contracted)
  bool rla;
  bool f32g;    // dq, dk, dv stored in fp32 (RDN_FLAG_F32_OUT), else bf16
  bool f32qk;   // dq, dk stored in fp32 whatever f32g (for a step that follows)
  // tensor maps (CUtensorMap, 64-byte aligned) over k, q, dO as [tokens][H][D]
  // with a 64-token x 64-column box (make_tile_map); tma: they are valid
  alignas(64) unsigned char map_k[128];
  alignas(64) unsigned char map_q[128];
  alignas(64) unsigned char map_do[128];
  bool tma;
  alignas(64) unsigned char map_dv[128];  // and over dv (bf16); dv_ok: it is valid
  bool dv_ok;
};

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t *>(&v);
}

// Row r, columns c0..c0+15 of a K-major SW128 tile (64-col blocks blk apart).
__device__ __forceinline__ void put16(uint8_t *tile, uint32_t blk, int r, int c0,
                                      const float (&v)[16]) {
  uint8_t *b = tile + (c0 >> 6) * blk;
  const int cc = c0 & 63;
  uint4 x, y;
  x.x = pack2(v[0], v[1]); x.y = pack2(v[2], v[3]); x.z = pack2(v[4], v[5]); x.w = pack2(v[6], v[7]);
  y.x = pack2(v[8], v[9]); y.y = pack2(v[10], v[11]); y.z = pack2(v[12], v[13]); y.w = pack2(v[14], v[15]);
  *reinterpret_cast<uint4 *>(b + sw128(r, cc)) = x;
  *reinterpret_cast<uint4 *>(b + sw128(r, cc + 8)) = y;
}
// hi / lo split (split_pack_bf16) of 16 values into two single-block tiles
__device__ __forceinline__ void put16s(uint8_t *hi, uint8_t *lo, int r, int c0,
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
// the same for 8 values (one 16-byte chunk of each tile)
__device__ __forceinline__ void put8s(uint8_t *hi, uint8_t *lo, int r, int c0,
                                      const float (&v)[8]) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) split_pack_bf16(v[2 * i], v[2 * i + 1], h[i], l[i]);
  *reinterpret_cast<uint4 *>(hi + sw128(r, c0)) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4 *>(lo + sw128(r, c0)) = make_uint4(l[0], l[1], l[2], l[3]);
}
// K-major A and B (single block, K = 64), split both
__device__ __forceinline__ void mma_s3_kk(uint32_t d, uint32_t a_hi, uint32_t a_lo, uint32_t b_hi,
                                          uint32_t b_lo, uint32_t idesc, bool acc_first) {
  mma_tile(d, a_hi, 0, b_hi, 0, 4, idesc, acc_first);
  mma_tile(d, a_hi, 0, b_lo, 0, 4, idesc, true);
  mma_tile(d, a_lo, 0, b_hi, 0, 4, idesc, true);
}

// Common per-CTA machinery: mbarriers (MMA, copies A, B, C, and D for the
// drain), TMEM, phases.  Thread 0 counts the copy phases it arms on A, B, C
// and the ones it has seen complete, so that a CTA whose bounded wait gave up
// can wait (again with a limit) for every copy and MMA still in flight before
// it releases its shared memory and TMEM (ctl_drain).
struct Ctl {
  uint64_t *bar, *barA, *barB, *barC, *barD;
  volatile int *flag;
  uint32_t phase, phA, phB;
  uint32_t armA, armB, armC, seenA, seenB, seenC;  // (thread 0) copy phases on A, B, C
};

__device__ __forceinline__ void ctl_init(Ctl &k, uint8_t *base, int tid) {
  k.bar = reinterpret_cast<uint64_t *>(base);
  k.barA = k.bar + 1;
  k.barB = k.bar + 2;
  k.barC = k.bar + 3;
  k.flag = reinterpret_cast<volatile int *>(base + 32);
  k.barD = reinterpret_cast<uint64_t *>(base + 40);
  k.phase = k.phA = k.phB = 0;
  k.armA = k.armB = k.armC = k.seenA = k.seenB = k.seenC = 0;
  if (tid == 0) {
    mbar_init(k.bar, 1);
    mbar_init(k.barA, 1);
    mbar_init(k.barB, 1);
    mbar_init(k.barC, 1);
    mbar_init(k.barD, 1);
    fence_mbar_init();
    *k.flag = 0;
  }
}

// the barrier and counters of copy barrier W (0: A, 1: B, 2: C)
template <int W>
__device__ __forceinline__ uint64_t *ctl_bar(Ctl &k) {
  return W == 0 ? k.barA : (W == 1 ? k.barB : k.barC);
}
template <int W>
__device__ __forceinline__ uint32_t &ctl_armed(Ctl &k) {
  return W == 0 ? k.armA : (W == 1 ? k.armB : k.armC);
}
template <int W>
__device__ __forceinline__ uint32_t &ctl_seen(Ctl &k) {
  return W == 0 ? k.seenA : (W == 1 ? k.seenB : k.seenC);
}
// (thread 0) arm a copy phase of barrier W for `bytes`
template <int W>
__device__ __forceinline__ void ctl_arm(Ctl &k, uint32_t bytes) {
  mbar_expect_tx(ctl_bar<W>(k), bytes);
  ++ctl_armed<W>(k);
}
// wait for a copy phase of barrier W (thread 0 counts it)
template <int W>
__device__ __forceinline__ bool ctl_wait(Ctl &k, uint32_t parity, int tid) {
  const bool ok = mbar_wait(ctl_bar<W>(k), parity);
  if (ok && tid == 0) ++ctl_seen<W>(k);
  return ok;
}
template <int W>
__device__ __forceinline__ void ctl_drain_copies(Ctl &k) {
  for (; ctl_seen<W>(k) < ctl_armed<W>(k); ++ctl_seen<W>(k))
    mbar_wait(ctl_bar<W>(k), ctl_seen<W>(k) & 1u);
}
// (thread 0, after a wait gave up) every MMA this thread issued (one commit
// covers them) and every armed copy phase, with bounded waits
__device__ __forceinline__ void ctl_drain(Ctl &k) {
  mma_commit(k.barD);
  mbar_wait(k.barD, 0);
  ctl_drain_copies<0>(k);
  ctl_drain_copies<1>(k);
  ctl_drain_copies<2>(k);
}

template <int W>
__device__ __forceinline__ void load_slot(Ctl &k, uint8_t *dst, const void *src, uint32_t bytes) {
  ctl_arm<W>(k, bytes);
  bulk_g2s(dst, src, bytes, ctl_bar<W>(k));
}

// One MMA phase: publish shared-memory writes, issue (thread 0), wait.
template <typename F>
__device__ __forceinline__ bool phase_run(Ctl &k, int tid, F issue) {
  fence_async_smem();
  fence_before_sync();
  __syncthreads();
  if (tid == 0) {
    fence_after_sync();
    if (!issue()) *k.flag = 1;
    mma_commit(k.bar);
  }
  const bool ok = mbar_wait(k.bar, k.phase);
  k.phase ^= 1u;
  if (!ok) *k.flag = 1;
  __syncthreads();
  fence_after_sync();
  return *k.flag == 0;
}

// The same, running `during` (work the MMAs do not touch) between the issue
// and the wait.
template <typename F, typename G>
__device__ __forceinline__ bool phase_run_with(Ctl &k, int tid, F issue, G during) {
  fence_async_smem();
  fence_before_sync();
  __syncthreads();
  if (tid == 0) {
    fence_after_sync();
    if (!issue()) *k.flag = 1;
    mma_commit(k.bar);
  }
  __syncwarp();  // (TMEM accesses take whole warps)
  during();
  const bool ok = mbar_wait(k.bar, k.phase);
  k.phase ^= 1u;
  if (!ok) *k.flag = 1;
  __syncthreads();
  fence_after_sync();
  return *k.flag == 0;
}

// The same phase in two halves, for work that overlaps the MMAs: publish and
// issue ...
template <typename F>
__device__ __forceinline__ void phase_issue(Ctl &k, int tid, F issue) {
  fence_async_smem();
  fence_before_sync();
  __syncthreads();
  if (tid == 0) {
    fence_after_sync();
    if (!issue()) *k.flag = 1;
    mma_commit(k.bar);
  }
  __syncwarp();  // (TMEM accesses take whole warps)
}
// ... then wait for them (every thread).
__device__ __forceinline__ bool phase_wait(Ctl &k) {
  const bool ok = mbar_wait(k.bar, k.phase);
  k.phase ^= 1u;
  if (!ok) *k.flag = 1;
  __syncthreads();
  fence_after_sync();
  return *k.flag == 0;
}

// thread 0: wait for a slot's bulk copy
template <int W>
__device__ __forceinline__ bool slot_wait(Ctl &k, uint32_t &ph) {
  const bool ok = ctl_wait<W>(k, ph, 0);
  ph ^= 1u;
  return ok;
}

__device__ __forceinline__ const uint8_t *rec_bytes(const FwdParams &p, size_t chunk) {
  return reinterpret_cast<const uint8_t *>(p.ws + chunk * kRecFloats);
}

}  // namespace bwdtc

// The gradients carried between chunks (bwd_chain.cu).
cudaError_t launch_bwd_chain(const bwdtc::TcBwdParams &P, cudaStream_t s);

}  // namespace rdn
