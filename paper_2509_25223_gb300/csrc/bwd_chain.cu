// bwd_chain.cu -- the sequential part of the tensor-core backward (bwd_tc.cu):
// the gradients carried between chunks, chunks in reverse, one CTA per
// (sequence, head).  With dR, dS the gradients w.r.t. a chunk's end states,
//
//   A  K dR; M2^T (gamma dO), Mq^T dO      dE2 = M2^T dOa + diag(wR) K dR
//   B  dX2 = T_gamma^T dE2                 dP  = -mask * dX2, dKR = -Gam dX2
//   C  Ap^T dP                             dE  = Mq^T dO + Ap^T dP + diag(wS) K dS
//   D  dX  = T_beta^T dE                   dKS = Gprev dP - Gam dX, dv = -dP + dX
//   E  dS_prev = Gam_C dS + Q^T dQS + K^T dKS   (dQS = Gam dO)
//      dR_prev = Gam_C dR + K^T dKR + Q^T dQR   (dQR = Gam gamma dO)
//
// Only the first product of each step stands on the chain of dependent steps;
// the others run behind them: Mq^T dO behind A, K dS behind B, K^T dKR behind C,
// the two products with Q behind D, and the next chunk's M2^T (gamma dO) behind
// E.  Nor do the stores stand on it: dX2 is staged behind C, dX and dv behind E,
// where dR (complete before E) is also made into the next chunk's operand; dS is
// during the next A.
//
// The 16 element-wise warps form 4 groups of 128 threads: thread j of a group
// owns value column j = TMEM lane j, group g the tokens [16g, 16g + 16) (and
// the key columns [16g, 16g + 16) and [64 + 16g, 80 + 16g)).  The products are issued
// by a warp of their own and the copies by another: an issuing thread is held for
// most of its products' time, and the stores of the gradients' images (128 KB a
// chunk, read from shared memory at about 30 bytes a cycle) outlast two steps of
// the chain.  What a chain product multiplies (dE2, dP, dE, dKS) is an operand in
// TMEM, written in place by the thread that forms it: for its 16 tokens 8
// columns of bf16 hi parts and then 8 of lo parts, within the 16 columns that
// it alone reads.
//
// Measured (a chunk; before, with every product and copy issued by an element-wise
// thread and every step waited for in full): 128 heads, T = 4096: 8.9 us (11.8),
// 570 us a call (755); packed, 157 chunks the longest: 7.8 us (11.7); RLA,
// T = 2048: 7.5 us.  A pair of CTAs a head took 7.4 us, so that there is none any
// more.  A CTA moves 340 KB a chunk from and to HBM: with 128 of them 4.9 TB/s of
// the 6.9 a copy reaches; with few the chain of steps bounds it, of which the
// copies through shared memory (30 bytes a cycle out, 42 in) are the longest part.
//
// TMEM (512 columns): [0,128) dS   [128,256) dR   [256,320) K dR, then dE2, dP, dE
// and dKS   [320,384) K dS, then dQR   [384,448) M2^T dO, then dX2, Ap^T dP, dX
// [448,512) Mq^T dO, then dQS.
#include "bwd_tc.cuh"

namespace rdn {
namespace {

using namespace bwdtc;

// shared-memory carve-up (bytes from the 1024-aligned dynamic base)
constexpr uint32_t SM_KQ = 0;        // K rows 0..63, Q rows 64..127, two 64-column blocks
// the carried gradients' bf16 tiles (rows j, two 16 KB blocks; hi and lo), the A
// operands of K dR, K dS, which also leave as images for bwd_post.  In between
// they hold dX2 (DRH) and dX (DSH), fp32 [t][j], on their way out, and dKR (DRL,
// [j][t] hi | lo).
constexpr uint32_t SM_DRH = 32768, SM_DRL = 65536, SM_DSH = 98304, SM_DSL = 131072;
constexpr uint32_t SM_SLOTA = 163840;  // diag(gamma) M2 -> T_gamma -> T_beta (hi | lo)
constexpr uint32_t SM_SLOTB = 180224;  // Mq -> Ap (hi | lo)
constexpr uint32_t SM_DO = 196608;   // dO, exact bf16, rows t (two 8 KB column blocks)
constexpr uint32_t SM_DV = 212992;   // dv on its way out (likewise)
constexpr uint32_t SM_VEC = 229376;  // two chunks' gates, fp32: Gam, Gprev, wS, wR, gamma, GamC
constexpr int kVec = 324;
constexpr uint32_t SM_BAR = SM_VEC + 2 * kVec * 4;
constexpr int kBars = 15;
constexpr uint32_t SM_SLOT = SM_BAR + 8 * kBars;
constexpr uint32_t SM_FLAG = SM_SLOT + 4;
constexpr size_t kChainSmem = SM_FLAG + 4;
static_assert(kChainSmem <= 232448, "shared memory");

constexpr uint32_t T_DS = 0, T_DR = 128, T_R1 = 256, T_R2 = 320, T_R3 = 384, T_R4 = 448;

constexpr int kChainThreads = NTC + 64, kOneMore = NTC + 32;
// named barriers on which the element-wise warps hand operands to the issuing
// warp (B, C, D, E), to the copying warp (DS, DX) or to both (DX2, Q)
constexpr int kBarB = 1, kBarC = 2, kBarDX2 = 3, kBarD = 4, kBarQ = 5, kBarE = 6, kBarDX = 7,
              kBarDS = 8;

// kGeneric: the RLA mode and the variant flags (TcBwdParams::rla, FwdParams::mods)
// are read; the RDN method's instance has them folded away
template <bool kGeneric>
__global__ void __launch_bounds__(kChainThreads, 1)
    bwd_chain_kernel(const __grid_constant__ TcBwdParams P) {
  extern __shared__ __align__(1024) uint8_t sm[];
  const uint32_t sb = smem_u32(sm);
  const FwdParams &p = P.f;
  if (sb & 1023u) {
    if (threadIdx.x == 0 && p.err) atomicExch(p.err, RDN_ERR_CUDA);
    return;
  }
  uint64_t *bar = reinterpret_cast<uint64_t *>(sm + SM_BAR);  // the chain's products
  uint64_t *barA = bar + 1, *barB = bar + 2;  // slot A / slot B bulk copies
  uint64_t *barO = bar + 3, *barT = bar + 4;  // a whole chunk's dO / K, Q tiles
  // products done with slot A (T_gamma, T_beta), slot B (Ap), slot A (M2), slot B (Mq)
  uint64_t *barSA = bar + 5, *barSB = bar + 6, *barF = bar + 7, *barM = bar + 14;
  uint64_t *barK = bar + 8;   // ... and with K, Q
  uint64_t *barG = bar + 9;   // the copies out have read: dR's tiles; dS's and dX2; dX
  uint64_t *barR = bar + 12;  // dR is complete
  uint64_t *barD = bar + 13;  // the drain after a wait that gave up
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + SM_SLOT);
  volatile int *flag = reinterpret_cast<volatile int *>(sm + SM_FLAG);

  const bool rla = kGeneric && P.rla;
  const unsigned mods = kGeneric ? p.mods : 0u;
  const bool tnh = mods & RDN_FLAG_TANH_RESIDUAL;
  const bool plain = mods & RDN_FLAG_PLAIN_COMBINE;  // (no gamma_t in the output)
  const bool dec_res = mods & RDN_FLAG_DECAYED_RESIDUAL;
  // the stateless correction: the chunk-end R is not carried into the next
  // chunk nor read out there, so the gradient carried back to it is zero
  // (dR_prev = 0; a chunk's own dR is the upstream dRT for the last chunk)
  const bool stl = mods & RDN_FLAG_STATELESS_AUX;
  const int tid = threadIdx.x, warp = tid >> 5, j = tid & 127;
  const int g16 = (warp >> 2) * 16;  // this thread's token (and key) columns start
  const int H = p.H, sq = seq_at(p, blockIdx.x / H), h = blockIdx.x % H;
  const SeqSpan sp = seq_span(p, sq, h);  // this (sequence, head)'s tokens and records
  const long long tok0 = sp.tok0;
  const int NC = sp.nc, T = sp.len;
  const size_t st_base = ((size_t)sq * H + h) * D * D;
  // Chunks before the last are whole: with tensor maps the copying warp brings
  // their tiles by tiled bulk copies.  The last one, which may be ragged, comes by
  // cp.async with zero fill.
  const bool tma = P.tma;
  auto dv_tiles = [&](int c) { return P.dv_ok && T - c * 64 >= 64; };
  // the waits on the MMAs: normally about a second; a test (p.inject) skips the
  // first product's completion signal and waits about 5 ms for it instead
  const long long limit = p.inject == 2 ? 10000000ll : 2000000000ll;

  if (tid == 0) {
    for (int b = 0; b < kBars; ++b) mbar_init(bar + b, 1);
    fence_mbar_init();
    *flag = 0;
  }
  if (warp == 0) tmem_alloc(slot, 512);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tm = *slot;

  if (warp == NTC / 32) {
    // =============================================== the issuing warp (lane 0)
    bool one = (tid & 31) == 0;
    bool skip_commit = p.inject == 2;
    uint32_t na = 0;  // copies to slot A waited for
    const uint32_t i64 = idesc_bf16(128, 64), i128 = idesc_bf16(128, 128);
    // wait for a copy by the copying warp; when it gave up, nothing more is issued
    // or completed (no barrier is armed again before its phase is complete)
    auto wait_copy = [&](uint64_t *b, uint32_t ph) {
      if (mbar_wait(b, ph)) return true;
      *flag = 1;
      return one = false;
    };
    // M2^T (gamma dO), Mq^T dO; dO is the MN-major A operand
    auto m2_product = [&] {
      if (!wait_copy(barA, na & 1u)) return;
      ++na;
      mma_tile_mnmn(tm + T_R3, sb + SM_DO, 8192, sb + SM_SLOTA, 16384, 4, i64, false);
      mma_tile_mnmn(tm + T_R3, sb + SM_DO, 8192, sb + SM_SLOTA + 8192, 16384, 4, i64, true);
      mma_commit(barF);
    };
    auto mq_product = [&] {
      if (!wait_copy(barB, 0)) return;
      mma_tile_mnmn(tm + T_R4, sb + SM_DO, 8192, sb + SM_SLOTB, 16384, 4, i64, false);
      mma_tile_mnmn(tm + T_R4, sb + SM_DO, 8192, sb + SM_SLOTB + 8192, 16384, 4, i64, true);
      mma_commit(barM);
    };
    // R3 = image^T times the operand in R1, both hi + lo (three products)
    auto r1_image = [&](uint32_t img) {
#pragma unroll
      for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_bf16_ta(tm + T_R3, tm + T_R1 + 16 * kk + (u == 2 ? 8 : 0),
                      sdesc_sw128_mn(img + (u == 1 ? 8192u : 0u) + 2048u * kk, 16384),
                      i64 | kBMajorMN, u || kk ? 1u : 0u);
    };
    // d += K^T or Q^T (rows of `kq`) times the operand in column `op`, hi, then lo
    auto op_rows = [&](uint32_t d, uint32_t op, uint32_t kq) {
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
        mma_bf16_ta(tm + d, tm + op + 16 * (kk & 3) + (kk >> 2) * 8,
                    sdesc_sw128_mn(kq + (kk & 3) * 2048, 16384), i128 | kBMajorMN, 1u);
    };
    bool alive = true;
    for (int c = NC - 1; c >= 0; --c) {
      const uint32_t it = (uint32_t)(NC - 1 - c);
      __syncthreads();
      fence_after_sync();
      if (*flag) {
        alive = false;
        break;
      }
      if (one && (it == 0 || !tma)) m2_product();
      if (one) {  // A: K dR; Mq^T dO behind it
        mma_tile(tm + T_R1, sb + SM_DRH, 16384, sb + SM_KQ, 16384, 8, i64, false);
        mma_tile(tm + T_R1, sb + SM_DRL, 16384, sb + SM_KQ, 16384, 8, i64, true);
        if (!skip_commit) mma_commit(bar);
        skip_commit = false;
        mq_product();
      }
      __syncwarp();
      bar_sync(kBarB, kOneMore);
      fence_after_sync();
      if (one && wait_copy(barA, na & 1u)) {  // B: T_gamma^T dE2; K dS behind it
        ++na;
        r1_image(sb + SM_SLOTA);
        mma_commit(bar);
        mma_commit(barSA);
        mma_tile(tm + T_R2, sb + SM_DSH, 16384, sb + SM_KQ, 16384, 8, i64, false);
        mma_tile(tm + T_R2, sb + SM_DSL, 16384, sb + SM_KQ, 16384, 8, i64, true);
      }
      __syncwarp();
      bar_sync(kBarC, kOneMore);
      fence_after_sync();
      if (one && wait_copy(barB, 1)) {  // C: Ap^T dP
        r1_image(sb + SM_SLOTB);
        mma_commit(bar);
        mma_commit(barSB);
      }
      __syncwarp();
      bar_sync(kBarDX2, kChainThreads);
      fence_after_sync();
      if (one && !rla && !stl) {  // dR += K^T dKR
        mma_tile_kmn(tm + T_DR, sb + SM_DRL, 0, sb + SM_KQ, 16384, 4, i128, true);
        mma_tile_kmn(tm + T_DR, sb + SM_DRL + 16384, 0, sb + SM_KQ, 16384, 4, i128, true);
      }
      __syncwarp();
      bar_sync(kBarD, kOneMore);
      fence_after_sync();
      if (one && wait_copy(barA, na & 1u)) {  // D: T_beta^T dE
        ++na;
        r1_image(sb + SM_SLOTA);
        mma_commit(bar);
        mma_commit(barSA);
      }
      __syncwarp();
      bar_sync(kBarQ, kChainThreads);
      fence_after_sync();
      if (one) {  // dR += Q^T dQR, dS += Q^T dQS
        if (!stl) op_rows(T_DR, T_R2, sb + SM_KQ + 8192);
        mma_commit(barR);
        op_rows(T_DS, T_R4, sb + SM_KQ + 8192);
      }
      __syncwarp();
      bar_sync(kBarE, kOneMore);
      fence_after_sync();
      if (one) {  // E: dS += K^T dKS (hi, then lo); the next chunk's M2^T (gamma dO)
        op_rows(T_DS, T_R1, sb + SM_KQ);
        mma_commit(bar);
        mma_commit(barK);
        if (c > 0 && tma && wait_copy(barO, it & 1u)) m2_product();
      }
      __syncwarp();
    }
    __syncthreads();
    if ((!alive || *flag) && (tid & 31) == 0) {  // a wait gave up: drain the products, bounded
      if (p.err) atomicExch(p.err, RDN_ERR_TIMEOUT);
      mma_commit(barD);
      mbar_wait(barD, 0);
    }
    __syncwarp();
    fence_before_sync();
    __syncthreads();
    return;
  }
  if (warp == NTC / 32 + 1) {
    // =============================================== the copying warp
    const bool one = (tid & 31) == 0;
    const int ln = tid & 31;
    uint32_t armA = 0, armB = 0, armO = 0, armT = 0;  // copies armed on the barriers
    auto rec_of = [&](int c) { return rec_bytes(p, (size_t)(sp.rbase + c)); };
    auto load_a = [&](const uint8_t *src) {
      ++armA;
      mbar_expect_tx(barA, 16384);
      bulk_g2s(sm + SM_SLOTA, src, 16384, barA);
    };
    auto load_b = [&](const uint8_t *apmq, uint32_t half) {  // Ap (0) or Mq (8192), hi | lo
      ++armB;
      mbar_expect_tx(barB, 16384);
      bulk_g2s(sm + SM_SLOTB, apmq + half, 8192, barB);
      bulk_g2s(sm + SM_SLOTB + 8192, apmq + 16384 + half, 8192, barB);
    };
    // a chunk's gates, lane l those of tokens l and l + 32
    float gt[5][2], gc = 0.f;
    auto load_gates = [&](int c) {
      const float *rc = p.ws + (size_t)(sp.rbase + c) * kRecFloats + OFF_VEC;
      const int t0 = c * 64, n = min(64, T - t0);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int t = ln + 32 * u;
        gt[0][u] = rc[V_GAM + t];
        gt[1][u] = rc[V_GPREV + t];
        gt[2][u] = rc[V_WS + t];
        gt[3][u] = rc[V_WR + t];
        gt[4][u] = t < n ? p.gamma[(size_t)(tok0 + t0 + t) * H + h] : 0.f;
      }
      gc = rc[V_GAMC];
    };
    auto put_gates = [&](int c) {
      float *g = reinterpret_cast<float *>(sm + SM_VEC) + kVec * (c & 1);
#pragma unroll
      for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int u = 0; u < 2; ++u) g[64 * i + ln + 32 * u] = gt[i][u];
      if (ln == 0) g[320] = gc;
    };
    // L2 prefetch of a chunk's record and tiles, one chunk ahead of their copies
    auto prefetch_chunk = [&](int c) {
      static_assert((kRecFloats * 4) % 16 == 0 && kRecFloats * 4 > 65536, "record");
      prefetch_l2_bulk(rec_of(c), 65536);
      prefetch_l2_bulk(rec_of(c) + 65536, kRecFloats * 4 - 65536);
      if (!tma) return;
      const int row = (int)(tok0 + (long long)c * 64);
      for (int kb = 0; kb < 2; ++kb) {
        tma_prefetch_3d(P.map_do, 64 * kb, h, row);
        tma_prefetch_3d(P.map_k, 64 * kb, h, row);
        tma_prefetch_3d(P.map_q, 64 * kb, h, row);
      }
    };
    if (NC > 0) {
      if (one) {
        load_a(rec_of(NC - 1) + IMG_M2);
        load_b(rec_of(NC - 1) + IMG_APMQ, 8192);
      }
      load_gates(NC - 1);
      put_gates(NC - 1);
    }
    bool alive = true, good = true;  // good: (lane 0) no wait of this warp gave up
    // (a wait that gave up leaves its phase incomplete, which takes no further
    // arrival: nothing is armed after it)
    auto await = [&](uint64_t *b, uint32_t ph) {
      if (!mbar_wait(b, ph, limit)) {
        good = false;
        *flag = 1;
      }
    };
    for (int c = NC - 1; c >= 0; --c) {
      const uint32_t it = (uint32_t)(NC - 1 - c), ph = it & 1u;
      const size_t chunk = (size_t)(sp.rbase + c);
      const bool tma_next = tma && c > 0;
      if (one && tma && it > 0) {  // this chunk's tiles
        await(barO, (armO - 1) & 1u);
        await(barT, (armT - 1) & 1u);
      }
      __syncwarp();
      __syncthreads();
      if (*flag) {
        alive = false;
        break;
      }
      if (one) {
        // (the copy engine takes copies in turn: what the chain waits for first)
        await(barF, ph);
        if (good) load_a(rec_of(c) + IMG_TG);
        // the images of the gradients w.r.t. this chunk's end states, for bwd_post
        uint8_t *g = P.gimg + chunk * 131072;
        bulk_s2g(g + 32768, sm + SM_DRH, 32768);
        bulk_s2g(g + 98304, sm + SM_DRL, 32768);
        bulk_commit();
        if (it > 0) {
          bulk_wait_read_all_but_last();
          mbar_arrive(barG + 2);  // dS's tiles over the chunk before's dX
        }
        bulk_wait_read();
        mbar_arrive(barG);  // dX2 and dKR may come over dR's tiles
      }
      __syncwarp();
      if (c > 0) load_gates(c - 1);
      if (one && c > 0) prefetch_chunk(c - 1);
      __syncwarp();
      bar_sync(kBarDS, kOneMore);
      if (one) {
        await(barM, ph);
        if (good) load_b(rec_of(c) + IMG_APMQ, 0);
        bulk_s2g(P.gimg + chunk * 131072, sm + SM_DSH, 32768);
        bulk_s2g(P.gimg + chunk * 131072 + 65536, sm + SM_DSL, 32768);
        bulk_commit();
        await(barSA, 0);
        if (good) load_a(rec_of(c) + IMG_TB);
      }
      __syncwarp();
      if (c > 0) put_gates(c - 1);  // (its set was last read for chunk c + 1)
      bar_sync(kBarDX2, kChainThreads);
      if (one) {
        bulk_s2g(P.dX2buf + chunk * 64 * D, sm + SM_DRH, 32768);
        bulk_commit();
        bulk_wait_read();
        mbar_arrive(barG + 1);  // dX may come over dS's tiles, dR's tiles over dX2
      }
      __syncwarp();
      bar_sync(kBarQ, kChainThreads);
      if (one) {
        if (good && tma_next) {  // dO has been read
          const int row = (int)(tok0 + (long long)(c - 1) * 64);
          ++armO;
          mbar_expect_tx(barO, 16384);
          for (int kb = 0; kb < 2; ++kb)
            tma_load_3d(sm + SM_DO + kb * 8192, P.map_do, 64 * kb, h, row, barO);
        }
        await(barSB, ph);
        if (good && c > 0) load_b(rec_of(c - 1) + IMG_APMQ, 8192);
        await(barSA, 1);
        if (good && c > 0) load_a(rec_of(c - 1) + IMG_M2);
      }
      __syncwarp();
      bar_sync(kBarDX, kOneMore);
      if (one) {
        await(barK, ph);
        if (good && tma_next) {
          const int row = (int)(tok0 + (long long)(c - 1) * 64);
          ++armT;
          mbar_expect_tx(barT, 32768);
          for (int kb = 0; kb < 2; ++kb) {
            tma_load_3d(sm + SM_KQ + kb * 16384, P.map_k, 64 * kb, h, row, barT);
            tma_load_3d(sm + SM_KQ + kb * 16384 + 8192, P.map_q, 64 * kb, h, row, barT);
          }
        }
        bulk_s2g(P.dXbuf + chunk * 64 * D, sm + SM_DSH, 32768);
        if (dv_tiles(c))
          for (int kb = 0; kb < 2; ++kb)
            tma_store_3d(P.map_dv, 64 * kb, h, (int)(tok0 + (long long)c * 64), sm + SM_DV + 8192 * kb);
        bulk_commit();
      }
      __syncwarp();
    }
    if (one) bulk_wait_all();
    __syncthreads();
    if ((!alive || *flag) && one) {  // every copy armed has landed, bounded
      if (armA) mbar_wait(barA, (armA - 1) & 1u);
      if (armB) mbar_wait(barB, (armB - 1) & 1u);
      if (armO) mbar_wait(barO, (armO - 1) & 1u);
      if (armT) mbar_wait(barT, (armT - 1) & 1u);
    }
    __syncwarp();
    fence_before_sync();
    __syncthreads();
    return;
  }

  // ================================================= the 16 element-wise warps
  const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
  // a warp's wait: one lane polls (512 polling threads take shared-memory
  // bandwidth from the products' operands)
  auto warp_wait = [&](uint64_t *b, uint32_t parity) {
    if ((tid & 31) == 0 && !mbar_wait(b, parity, limit)) *flag = 1;
    __syncwarp();
  };
  uint32_t phase = 0;  // chain phases waited for (parity)
  auto wait_chain = [&] {
    warp_wait(bar, phase);
    phase ^= 1u;
    fence_after_sync();
  };
  // hand this warp's shared-memory writes and TMEM accesses on
  auto publish = [&](int id, int count) {
    fence_async_smem();
    fence_before_sync();
    bar_arrive(id, count);
  };
  // this thread's 16 tokens of a chain operand (hi | lo) in its columns of `col`
  auto put_op = [&](uint32_t col, const float (&v)[16]) {
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) split_pack_bf16(v[2 * i], v[2 * i + 1], hi[i], lo[i]);
    tmem_st8x2(tm + lane + col + g16, hi, tm + lane + col + g16 + 8, lo);
  };
  // a carried gradient's bf16 hi + lo tiles (rows j), 16 of its key columns
  auto put_grad16 = [&](uint32_t hi, uint32_t lo, int c0, const float (&g)[16]) {
    put16s(sm + hi + (c0 >> 6) * 16384, sm + lo + (c0 >> 6) * 16384, j, c0, g);
  };
  // a complete gradient's tiles, the A operands of the next chunk's K dR, K dS, and
  // its TMEM copy times f in place (the chunk's products accumulate onto that);
  // once the barrier's phase is complete
  auto next_tiles = [&](uint32_t col, uint32_t hi, uint32_t lo, float f, uint64_t *b, uint32_t par) {
    warp_wait(b, par);
    fence_after_sync();
    float x[16], y[16];
    tmem_ld16x2(tm + lane + col + g16, x, tm + lane + col + g16 + 64, y);
    put_grad16(hi, lo, g16, x);
    put_grad16(hi, lo, g16 + 64, y);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      x[i] *= f;
      y[i] *= f;
    }
    tmem_st16x2(tm + lane + col + g16, x, tm + lane + col + g16 + 64, y);
  };
  auto rec_gamc = [&](int c) { return p.ws[(size_t)(sp.rbase + c) * kRecFloats + OFF_VEC + V_GAMC]; };
  for (int c0 = g16; c0 < D; c0 += 64) {  // upstream gradients of the final states
    float s[16], r[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      s[i] = P.dST ? P.dST[st_base + (size_t)(c0 + i) * D + j] : 0.f;
      r[i] = P.dRT ? P.dRT[st_base + (size_t)(c0 + i) * D + j] : 0.f;
    }
    put_grad16(SM_DSH, SM_DSL, c0, s);
    put_grad16(SM_DRH, SM_DRL, c0, r);
    // (TMEM: times the chunk's total decay, its products accumulate onto that)
    const float f = NC > 0 ? rec_gamc(NC - 1) : 1.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      s[i] *= f;
      r[i] *= stl && NC > 0 ? 0.f : f;
    }
    tmem_st16x2(tm + lane + T_DS + c0, s, tm + lane + T_DR + c0, r);
  }
  // a chunk's tiles (rows t, exact bf16, zero past the end), asynchronous
  auto fetch = [&](int c) {
    const __nv_bfloat16 *q = (const __nv_bfloat16 *)p.q, *k = (const __nv_bfloat16 *)p.k,
                        *dO = (const __nv_bfloat16 *)P.dO;
    const int t0 = c * 64, n = min(64, T - t0);
    for (int e = tid; e < 64 * 16; e += NTC) {
      const int t = e >> 4, ch = e & 15;
      const bool vld = t < n;
      const size_t off = ((size_t)(tok0 + t0 + (vld ? t : 0)) * H + h) * D + ch * 8;
      const int blk = ch >> 3, cc = (ch & 7) * 8;
      cp_async16(sm + SM_KQ + blk * 16384 + sw128(t, cc), k + off, vld);
      cp_async16(sm + SM_KQ + blk * 16384 + sw128(64 + t, cc), q + off, vld);
      cp_async16(sm + SM_DO + blk * 8192 + sw128(t, cc), dO + off, vld);
    }
  };
  if (NC > 0) fetch(NC - 1);

  bool alive = true;
  for (int c = NC - 1; c >= 0 && alive; --c) {
    const uint32_t ph = (uint32_t)(NC - 1 - c) & 1u;
    const size_t chunk = (size_t)(sp.rbase + c);
    if (!tma || c == NC - 1) cp_async_wait_all();
    fence_async_smem();
    fence_before_sync();
    __syncthreads();  // (with the copying warp, which has waited for the tiles)
    fence_after_sync();
    if (*flag) {
      alive = false;
      break;
    }
    // bit i: clip inactive at t = g16 + i ([g16, g16 + 16) of the column's word,
    // little-endian); or the tanh residual's derivative there (grad_q16)
    unsigned m = 0;
    uint4 dd[2];
    if (!tnh) {
      m = reinterpret_cast<const uint16_t *>(P.mask + chunk * D + j)[g16 >> 4];
    } else {
      const uint4 *src = reinterpret_cast<const uint4 *>(
          reinterpret_cast<const uint16_t *>(P.mask) + (chunk * D + j) * 64 + g16);
      dd[0] = src[0];
      dd[1] = src[1];
    }
    const float *Gam = reinterpret_cast<const float *>(sm + SM_VEC) + kVec * (c & 1);
    const float *Gprev = Gam + 64, *wS = Gam + 128, *wR = Gam + 192, *gamv = Gam + 256;
    auto dO = [&](int t) {  // dO[t, j] from the tile
      return __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(
          sm + SM_DO + (j >> 6) * 8192 + sw128(t, j & 63)));
    };
    // while A runs: dS's tiles, and in TMEM dS times this chunk's total decay
    if (c < NC - 1) next_tiles(T_DS, SM_DSH, SM_DSL, Gam[320], barG + 2, ph ^ 1u);
    wait_chain();
    {  // dE2 = M2^T dOa + wR K dR
      float x[16], y[16], w[16];
      tmem_ld16x2(tm + lane + T_R1 + g16, x, tm + lane + T_R3 + g16, y);
      lds16(wR + g16, w);
#pragma unroll
      for (int i = 0; i < 16; ++i) y[i] += w[i] * x[i];
      put_op(T_R1, y);
    }
    publish(kBarB, kOneMore);
    bar_arrive(kBarDS, kOneMore);
    wait_chain();
    float dP[16];  // t in [g16, g16 + 16)
    {  // dX2 -> dP = -mask dX2, dKR = -Gam dX2; dX2 itself (fp32 [t][j]) for bwd_post
      float x[16], g[16];
      tmem_ld16(tm + lane + T_R3 + g16, x);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        if (tnh) {  // the derivative of c tanh(x / c) instead of the mask
          const uint32_t w = reinterpret_cast<const uint32_t *>(dd)[i >> 1];
          dP[i] = -grad_uq16((i & 1) ? w >> 16 : w & 0xffffu) * x[i];
        } else {
          dP[i] = ((m >> i) & 1u) ? -x[i] : 0.f;
        }
      }
      put_op(T_R1, dP);
      publish(kBarC, kOneMore);
      float *stg = reinterpret_cast<float *>(sm + SM_DRH);
      lds16(Gam + g16, g);
      warp_wait(barG, ph);  // (dR's tiles have left)
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        stg[(g16 + i) * D + j] = x[i];
        x[i] *= -g[i];
      }
      if (!rla && !stl) put16s(sm + SM_DRL, sm + SM_DRL + 16384, j, g16, x);
    }
    publish(kBarDX2, kChainThreads);
    wait_chain();
    {  // dE = dE_partial + Ap^T dP
      float x[16], y[16], w[16];
      tmem_ld16x2(tm + lane + T_R2 + g16, x, tm + lane + T_R4 + g16, y);
      lds16(wS + g16, w);
#pragma unroll
      for (int i = 0; i < 16; ++i) y[i] += w[i] * x[i];
      tmem_ld16(tm + lane + T_R3 + g16, x);
#pragma unroll
      for (int i = 0; i < 16; ++i) y[i] += x[i];
      put_op(T_R1, y);
    }
    publish(kBarD, kOneMore);
    {  // dQR, dQS (Q unscaled), over K dS and Mq^T dO
      float x[16], w[16], d[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) d[i] = dO(g16 + i);
      if (!stl) {
        lds16(Gam + g16, x);
        lds16(gamv + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = p.scale * x[i] * (plain ? 1.f : w[i]) * d[i];
        put_op(T_R2, x);
      }
      // the base read-out Gam Q S0 (plain combine: Gprev Q S0)
      lds16(plain ? Gprev + g16 : Gam + g16, x);
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] = p.scale * x[i] * d[i];
      put_op(T_R4, x);
    }
    publish(kBarQ, kChainThreads);
    wait_chain();
    {  // dX -> dv = -dP + dX; dKS = Gprev dP - Gam dX; dX (fp32 [t][j]) for bwd_post
      float *stg = reinterpret_cast<float *>(sm + SM_DSH);
      float x[16], w[16], g[16];
      tmem_ld16(tm + lane + T_R3 + g16, x);
      // the prediction's state term: Gprev K S0 (decayed residual: Gam K S0)
      lds16(dec_res ? Gam + g16 : Gprev + g16, w);
      lds16(Gam + g16, g);
#pragma unroll
      for (int i = 0; i < 16; ++i) w[i] = w[i] * dP[i] - (rla ? 0.f : g[i] * x[i]);
      put_op(T_R1, w);
      publish(kBarE, kOneMore);
      warp_wait(barG + 1, ph);  // (dS's tiles have left, and dX2)
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        stg[(g16 + i) * D + j] = x[i];
        x[i] -= dP[i];
      }
      if (dv_tiles(c)) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          *reinterpret_cast<__nv_bfloat16 *>(sm + SM_DV + (j >> 6) * 8192 + sw128(g16 + i, j & 63)) =
              __float2bfloat16_rn(x[i]);
      }
      publish(kBarDX, kOneMore);
      if (!dv_tiles(c)) {  // fp32 gradients, the ragged last chunk
        const int t0 = c * 64, n = min(64, T - t0);
        const size_t row = ((size_t)(tok0 + t0 + g16) * H + h) * D + j;
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (g16 + i < n) {
            if (P.f32g) ((float *)P.dv)[row + (size_t)i * H * D] = x[i];
            else ((__nv_bfloat16 *)P.dv)[row + (size_t)i * H * D] = __float2bfloat16_rn(x[i]);
          }
      }
    }
    // while E runs: dR's tiles, and in TMEM dR times the next chunk's total decay
    if (c > 0) {
      const float f = reinterpret_cast<const float *>(sm + SM_VEC)[kVec * ((c - 1) & 1) + 320];
      next_tiles(T_DR, SM_DRH, SM_DRL, stl ? 0.f : f, barR, ph);
    }
    wait_chain();
    if (!tma && c > 0) fetch(c - 1);
  }
  __syncthreads();
  if (*flag) alive = false;
  if (alive) {
    for (int c0 = g16; c0 < D; c0 += 64) {
      float s[16], r[16];
      tmem_ld16x2(tm + lane + T_DS + c0, s, tm + lane + T_DR + c0, r);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        if (P.dS0) P.dS0[st_base + (size_t)(c0 + i) * D + j] = s[i];
        if (P.dR0) P.dR0[st_base + (size_t)(c0 + i) * D + j] = r[i];
      }
    }
  }
  cp_async_wait_all();
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tm, 512);
}

}  // namespace

cudaError_t launch_bwd_chain(const TcBwdParams &P, cudaStream_t s) {
  auto kern = P.rla || P.f.mods != 0 ? bwd_chain_kernel<true> : bwd_chain_kernel<false>;
  const cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kChainSmem);
  if (e != cudaSuccess) return e;
  RDN_LAUNCH("bwd_chain", s, kern<<<P.f.nseq * P.f.H, kChainThreads, kChainSmem, s>>>(P));
  return cudaGetLastError();
}

}  // namespace rdn
