// bwd_pair.cu -- the tensor-core backward chain of bwd_tc.cu over a pair of
// CTAs (a cluster of two SMs) per (sequence, head), for calls whose sequences
// are too few to fill the chip.
//
// The gradient of R never reads the gradient of S: CTA 1 carries dR, forms
// dX2 and copies it (32 KB, the fp32 tile it stages for bwd_post anyway) into
// CTA 0's shared memory; CTA 0 carries dS and forms dP, dX and dv, one chunk
// behind.  Each has three phases a chunk where the one-CTA chain
// has five:
//
//   CTA 1:  K dR, M2^T dOa             |  dX2, dR += Q^T dQR  |  dR += K^T dKR
//   CTA 0:  K dS, Mq^T dO, Ap^T dP     |  dX,  dS += Q^T dQS  |  dS += K^T dKS
//
// (operands and arithmetic as in bwd_tc.cu, in the same order: the results are
// the same bits).  The hand-over has a pair of mbarriers (`full` in CTA 0, the
// copy's bytes; `empty` in CTA 1, one arrival per warp of CTA 0 once it holds
// the values in registers, after which CTA 1 also rewrites what it copied
// from); its waits are bounded like every other, and the two CTAs meet at the
// cluster's barrier before either releases its shared memory.
//
// Measured: B = 2, H = 16, T = 2000 (RLA), 0.385 ms in one CTA per head,
// 0.289 ms in pairs.
#include "bwd_tc.cuh"

namespace rdn {
namespace {

using namespace bwdtc;

// shared memory (bytes from the 1024-aligned base)
constexpr uint32_t KQ = 0;
constexpr uint32_t GH = 32768, GL = 65536;  // the carried gradient's hi, lo tiles; then scratch
constexpr uint32_t F = 98304;    // scratch tile pair (hi | lo): CTA 1 dE2, dX2's staging; CTA 0 dP, dE, dKS
constexpr uint32_t X = 131072;   // CTA 1: dQR tile pair; CTA 0: the hand-over buffer
constexpr uint32_t SLOTA = 163840;  // CTA 1: diag(gamma) M2; CTA 0: Mq
constexpr uint32_t SLOTB = 180224;  // CTA 1: T_gamma; CTA 0: Ap
constexpr uint32_t SLOTC = 196608;  // CTA 0: T_beta
constexpr uint32_t DOT = 212992;    // dO, exact bf16, rows t
constexpr uint32_t VEC = 229376;    // Gam Gprev wS wR gamma (5 x 64)
constexpr uint32_t CTL = VEC + 5 * 64 * 4;
constexpr uint32_t BARX = CTL + 48;  // CTA 0: full; CTA 1: empty
constexpr uint32_t SLOT = BARX + 8;
constexpr size_t SMEM = SLOT + 16;
static_assert(SMEM <= 232448, "shared memory");
constexpr uint32_t HALF = 16384;  // a scratch pair's lo part
constexpr uint32_t T_G = 0, T_R1 = 128, T_R2 = 192, T_R3 = 256;

template <bool kGeneric>  // (as bwd_chain_kernel's)
__global__ void __launch_bounds__(NTC, 1) bwd_pair_kernel(const __grid_constant__ TcBwdParams P) {
  extern __shared__ __align__(1024) uint8_t sm[];
  const uint32_t sb = smem_u32(sm);
  const FwdParams &p = P.f;
  const bool rla = kGeneric && P.rla;
  const unsigned mods = kGeneric ? p.mods : 0u;
  if (!picked(p)) return;
  if (sb & 1023u) {  // (the same in both CTAs)
    if (threadIdx.x == 0 && p.err) atomicExch(p.err, RDN_ERR_CUDA);
    return;
  }
  float *vec = reinterpret_cast<float *>(sm + VEC);
  float *Gam = vec, *Gprev = vec + 64, *wS = vec + 128, *wR = vec + 192, *gamv = vec + 256;
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + SLOT);
  uint64_t *barX = reinterpret_cast<uint64_t *>(sm + BARX);
  const int tid = threadIdx.x, warp = tid >> 5, j = tid & 127;
  const uint32_t rank = cluster_rank();
  const bool base = rank == 0;  // CTA 0: dS; CTA 1: dR
  const int g16 = (warp >> 2) * 16;  // this thread's token (and key) columns start
  const int H = p.H, sq = seq_at(p, (blockIdx.x >> 1) / H), h = (blockIdx.x >> 1) % H;
  const SeqSpan sp = seq_span(p, sq, h);
  const long long tok0 = sp.tok0;
  const int NC = sp.nc, T = sp.len;
  const __nv_bfloat16 *q = (const __nv_bfloat16 *)p.q, *k = (const __nv_bfloat16 *)p.k,
                      *dOp = (const __nv_bfloat16 *)P.dO;
  __nv_bfloat16 *dv = (__nv_bfloat16 *)P.dv;
  const size_t st_base = ((size_t)sq * H + h) * D * D;
  const bool tnh = kGeneric && (mods & RDN_FLAG_TANH_RESIDUAL);
  const bool stl = kGeneric && (mods & RDN_FLAG_STATELESS_AUX);
  const bool plain = mods & RDN_FLAG_PLAIN_COMBINE;
  const bool dec_res = mods & RDN_FLAG_DECAYED_RESIDUAL;

  Ctl K;
  ctl_init(K, sm + CTL, tid);
  if (p.inject == 2) {  // (a test: the first phase's signal is skipped, the wait gives up)
    K.limit = 10000000ll;
    K.skip = !base;
  }
  if (tid == 0) {
    mbar_init(barX, base ? 1 : NTC / 32);
    fence_mbar_init();
    if (base) mbar_expect_tx(barX, 32768);
  }
  if (warp == 0) tmem_alloc(slot, 512);
  auto load_a = [&](size_t ck) {  // (thread 0) CTA 1: M2; CTA 0: Mq and Ap
    const uint8_t *r = rec_bytes(p, ck);
    if (!base) {
      load_slot<0>(K, sm + SLOTA, r + IMG_M2, 16384);
      return;
    }
    ctl_arm<0>(K, 32768);
    bulk_g2s(sm + SLOTA, r + IMG_APMQ + 8192, 8192, K.barA);
    bulk_g2s(sm + SLOTA + 8192, r + IMG_APMQ + 16384 + 8192, 8192, K.barA);
    bulk_g2s(sm + SLOTB, r + IMG_APMQ, 8192, K.barA);
    bulk_g2s(sm + SLOTB + 8192, r + IMG_APMQ + 16384, 8192, K.barA);
  };
  const uint32_t slot_t = base ? SLOTC : SLOTB;
  auto load_t = [&](size_t ck) {  // (thread 0) T_gamma / T_beta
    load_slot<1>(K, sm + slot_t, rec_bytes(p, ck) + (base ? IMG_TB : IMG_TG), 16384);
  };
  if (tid == 0 && NC > 0) {
    load_a((size_t)(sp.rbase + NC - 1));
    load_t((size_t)(sp.rbase + NC - 1));
  }
  fence_before_sync();
  __syncthreads();
  cluster_sync();  // the partner's barriers exist before anything arrives on them
  fence_after_sync();
  const uint32_t tm = *slot;
  const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
  const uint32_t peer_bar = map_rank(barX, rank ^ 1u);
  const uint32_t peer_x = map_rank(sm + X, 0u);

  auto put_grad16 = [&](int c0, const float (&g)[16]) {
    put16s(sm + GH + (c0 >> 6) * 16384, sm + GL + (c0 >> 6) * 16384, j, c0, g);
  };
  auto scale_grad = [&](float f) {  // the TMEM copy times the chunk's total decay, in place
    float x[16], y[16];
    tmem_ld16x2(tm + lane + T_G + g16, x, tm + lane + T_G + g16 + 64, y);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      x[i] *= f;
      y[i] *= f;
    }
    tmem_st16(tm + lane + T_G + g16, x);
    tmem_st16(tm + lane + T_G + g16 + 64, y);
  };
  {  // the upstream gradient of the final state
    const float *up = base ? P.dST : P.dRT;
    for (int c0 = g16; c0 < D; c0 += 64) {
      float s[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) s[i] = up ? up[st_base + (size_t)(c0 + i) * D + j] : 0.f;
      tmem_st16(tm + lane + T_G + c0, s);
      put_grad16(c0, s);
    }
    fence_async_smem();
  }
  // a chunk's K, Q, dO tiles: whole chunks by tensor-map copies on barrier C
  // (armed with dO's), the last, which may be ragged, by cp.async with zero fill
  auto fetch_kq = [&](int c) {
    const int t0 = c * 64, n = min(64, T - t0);
    for (int e = tid; e < 64 * 16; e += NTC) {
      const int t = e >> 4, chn = e & 15;
      const bool vld = t < n;
      const size_t off = ((size_t)(tok0 + t0 + (vld ? t : 0)) * H + h) * D + chn * 8;
      const int blk = chn >> 3, cc = (chn & 7) * 8;
      cp_async16(sm + KQ + blk * 16384 + sw128(t, cc), k + off, vld);
      cp_async16(sm + KQ + blk * 16384 + sw128(64 + t, cc), q + off, vld);
    }
  };
  auto fetch_do = [&](int c) {
    const int t0 = c * 64, n = min(64, T - t0);
    for (int e = tid; e < 64 * 16; e += NTC) {
      const int t = e >> 4, chn = e & 15;
      const bool vld = t < n;
      const size_t off = ((size_t)(tok0 + t0 + (vld ? t : 0)) * H + h) * D + chn * 8;
      cp_async16(sm + DOT + (chn >> 3) * 8192 + sw128(t, (chn & 7) * 8), dOp + off, vld);
    }
  };
  const bool tma = P.tma;
  uint32_t tma_ph = 0, tma_arms = 0, tma_seen = 0;  // phases waited for; (thread 0) armed, seen
  auto next_do = [&](int cc) {
    if (!tma) {
      fetch_do(cc);
    } else if (tid == 0) {
      const int row = (int)(tok0 + (long long)cc * 64);
      ++tma_arms;
      mbar_expect_tx(K.barC, 49152);
      for (int kb = 0; kb < 2; ++kb) tma_load_3d(sm + DOT + kb * 8192, P.map_do, 64 * kb, h, row, K.barC);
    }
  };
  auto next_kq = [&](int cc) {
    if (!tma) {
      fetch_kq(cc);
    } else if (tid == 0) {
      const int row = (int)(tok0 + (long long)cc * 64);
      for (int kb = 0; kb < 2; ++kb) {
        tma_load_3d(sm + KQ + kb * 16384, P.map_k, 64 * kb, h, row, K.barC);
        tma_load_3d(sm + KQ + kb * 16384 + 8192, P.map_q, 64 * kb, h, row, K.barC);
      }
    }
  };
  struct Pre {  // a chunk's gate vectors (threads 0..63) and this thread's mask bits (CTA 0)
    float gam_, gprev, ws_, wr_, g_, gamc;
    unsigned m;
    uint4 d0, d1;  // the tanh residual's derivative at this thread's 16 tokens (grad_q16)
  };
  auto fetch_pre = [&](int c) {
    const size_t ck = (size_t)(sp.rbase + c);
    const int t0 = c * 64, n = min(64, T - t0);
    const float *rf = p.ws + ck * kRecFloats;
    Pre x;
    x.gam_ = x.gprev = x.ws_ = x.wr_ = x.g_ = 0.f;
    x.m = 0u;
    x.d0 = x.d1 = make_uint4(0u, 0u, 0u, 0u);
    if (tid < 64) {
      x.gam_ = rf[OFF_VEC + V_GAM + tid];
      x.gprev = rf[OFF_VEC + V_GPREV + tid];
      x.ws_ = rf[OFF_VEC + V_WS + tid];
      x.wr_ = rf[OFF_VEC + V_WR + tid];
      x.g_ = tid < n ? p.gamma[(size_t)(tok0 + t0 + tid) * H + h] : 0.f;
    }
    x.gamc = rf[OFF_VEC + V_GAMC];
    if (base) {
      if (!tnh) {
        x.m = reinterpret_cast<const uint16_t *>(P.mask + ck * D + j)[g16 >> 4];
      } else {
        const uint4 *dp_ = reinterpret_cast<const uint4 *>(
            reinterpret_cast<const uint16_t *>(P.mask) + (ck * D + j) * 64 + g16);
        x.d0 = dp_[0];
        x.d1 = dp_[1];
      }
    }
    return x;
  };
  Pre pre{};
  if (NC > 0) {
    fetch_kq(NC - 1);
    fetch_do(NC - 1);
    pre = fetch_pre(NC - 1);
  }
  auto dO = [&](int t) {  // dO[t, j] from the tile
    return __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(
        sm + DOT + (j >> 6) * 8192 + sw128(t, j & 63)));
  };
  const uint32_t i64 = idesc_bf16(128, 64), i128 = idesc_bf16(128, 128);

  bool ok = true;
  uint32_t hand = 0;    // chunks done so far
  uint32_t handed = 0;  // (CTA 1, thread 0) copies to CTA 0 issued
  for (int c = NC - 1; c >= 0 && ok; --c, ++hand) {
    const size_t chunk = (size_t)(sp.rbase + c);
    const int t0 = c * 64, n = min(64, T - t0);
    __syncthreads();
    if (tid == 0) {  // the gradient w.r.t. this chunk's end state, for bwd_post
      bulk_s2g(P.gimg + chunk * 131072 + (base ? 0 : 32768), sm + GH, 32768);
      bulk_commit();
      bulk_s2g(P.gimg + chunk * 131072 + (base ? 65536 : 98304), sm + GL, 32768);
      bulk_commit();
    }
    if (tid < 64) {
      Gam[tid] = pre.gam_;
      Gprev[tid] = pre.gprev;
      wS[tid] = pre.ws_;
      wR[tid] = pre.wr_;
      gamv[tid] = pre.g_;
    }
    const float GamC = pre.gamc;
    const unsigned m = pre.m;  // bit i: clip inactive at t = g16 + i
    const uint4 dd0 = pre.d0, dd1 = pre.d1;
    if (!tma || c == NC - 1) cp_async_wait_all();
    if (tma && c < NC - 1) {
      if (mbar_wait(K.barC, tma_ph & 1u))
        tma_seen = tma_ph + 1;
      else
        *K.flag = 1;
      ++tma_ph;
    }
    float dP[16];  // t in [g16, g16 + 16)
    if (base) {    // dX2 of this chunk from CTA 1; dP = -mask dX2, also as a tile pair
      const bool got = mbar_wait_cluster(barX, hand & 1u, K.limit);
      if (!got) *K.flag = 1;
      const float *x2 = reinterpret_cast<const float *>(sm + X);
#pragma unroll
      for (int i = 0; i < 16; ++i) dP[i] = x2[(g16 + i) * D + j];
      // (a phase that has not completed takes no further arrival)
      if (got && tid == 0 && c > 0) mbar_expect_tx(barX, 32768);
      __syncwarp();
      if (got && (tid & 31) == 0) mbar_arrive_remote_relaxed(peer_bar);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        if (tnh) {  // the derivative of c tanh(x / c) instead of the mask
          const uint32_t w = (i < 8 ? reinterpret_cast<const uint32_t *>(&dd0)
                                    : reinterpret_cast<const uint32_t *>(&dd1))[(i & 7) >> 1];
          dP[i] = -grad_uq16((i & 1) ? w >> 16 : w & 0xffffu) * dP[i];
        } else {
          dP[i] = ((m >> i) & 1u) ? -dP[i] : 0.f;
        }
      }
      put16s(sm + F, sm + F + HALF, j, g16, dP);
    }
    __syncthreads();
    if (*K.flag) {
      ok = false;
      break;
    }
    if (!base) {
      // ---- K dR, M2^T (gamma dO); dR (TMEM) times Gam_C meanwhile
      ok = phase_run_with(K, tid, [&] {
        if (!slot_wait<0>(K, K.phA)) return false;
        mma_tile(tm + T_R1, sb + GH, 16384, sb + KQ, 16384, 8, i64, false);
        mma_tile(tm + T_R1, sb + GL, 16384, sb + KQ, 16384, 8, i64, true);
        mma_tile_mnmn(tm + T_R3, sb + DOT, 8192, sb + SLOTA, 16384, 4, i64, false);
        mma_tile_mnmn(tm + T_R3, sb + DOT, 8192, sb + SLOTA + 8192, 16384, 4, i64, true);
        return true;
      }, [&] { scale_grad(stl ? 0.f : GamC); });
      if (!ok) break;
      if (tid == 0 && c > 0) load_a(chunk - 1);
      {  // dE2 = M2^T dOa + wR K dR; dQR = Gam gamma dO
        float x[16], y[16], w[16];
        tmem_ld16x2(tm + lane + T_R1 + g16, x, tm + lane + T_R3 + g16, y);
        lds16(wR + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) y[i] += w[i] * x[i];
        // (the previous chunk's dX2 has left F)
        if (hand > 0 && !mbar_wait_cluster(barX, (hand - 1) & 1u, K.limit)) *K.flag = 1;
        put16s(sm + F, sm + F + HALF, j, g16, y);
        lds16(Gam + g16, x);
        lds16(gamv + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i)  // (Q unscaled)
          x[i] = stl ? 0.f : p.scale * x[i] * (plain ? 1.f : w[i]) * dO(g16 + i);
        put16s(sm + X, sm + X + HALF, j, g16, x);
      }
      // ---- dX2 = T_gamma^T dE2; dR += Q^T dQR
      ok = phase_run(K, tid, [&] {
        if (!slot_wait<1>(K, K.phB)) return false;
        mma_s3_kmn(tm + T_R3, sb + F, sb + F + HALF, sb + slot_t, sb + slot_t + 8192, 16384, i64, false);
        mma_tile_kmn(tm + T_G, sb + X, 0, sb + KQ + 8192, 16384, 4, i128, true);
        mma_tile_kmn(tm + T_G, sb + X + HALF, 0, sb + KQ + 8192, 16384, 4, i128, true);
        bulk_wait_read_all_but_last();  // the hi tiles are scratch after this phase
        return true;
      });
      if (!ok) break;
      if (c > 0) {
        if (tid == 0) load_t(chunk - 1);
        next_do(c - 1);
      }
      {  // dKR = -Gam dX2; dX2 (fp32 [t][j]) staged for CTA 0 and for bwd_post
        float *stg = reinterpret_cast<float *>(sm + F);
        float x[16], dkr[16];
        tmem_ld16(tm + lane + T_R3 + g16, x);
        lds16(Gam + g16, dkr);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          stg[(g16 + i) * D + j] = x[i];
          dkr[i] = (rla || stl) ? 0.f : -dkr[i] * x[i];
        }
        put16s(sm + GH, sm + GH + HALF, j, g16, dkr);
      }
      // ---- dR += K^T dKR
      ok = phase_run(K, tid, [&] {
        bulk_s2s(peer_x, sm + F, 32768, peer_bar);  // (published by this barrier)
        ++handed;
        bulk_s2g(P.dX2buf + chunk * 64 * D, sm + F, 32768);
        bulk_commit();
        mma_tile_kmn(tm + T_G, sb + GH, 0, sb + KQ, 16384, 4, i128, true);
        mma_tile_kmn(tm + T_G, sb + GH + HALF, 0, sb + KQ, 16384, 4, i128, true);
        bulk_wait_read();  // the staging and the lo tiles are rewritten next
        return true;
      });
      if (!ok) break;
    } else {
      // ---- K dS, Mq^T dO, Ap^T dP; dS (TMEM) times Gam_C meanwhile
      ok = phase_run_with(K, tid, [&] {
        if (!slot_wait<0>(K, K.phA)) return false;
        mma_tile(tm + T_R1, sb + GH, 16384, sb + KQ, 16384, 8, i64, false);
        mma_tile(tm + T_R1, sb + GL, 16384, sb + KQ, 16384, 8, i64, true);
        mma_tile_mnmn(tm + T_R2, sb + DOT, 8192, sb + SLOTA, 16384, 4, i64, false);
        mma_tile_mnmn(tm + T_R2, sb + DOT, 8192, sb + SLOTA + 8192, 16384, 4, i64, true);
        mma_s3_kmn(tm + T_R3, sb + F, sb + F + HALF, sb + SLOTB, sb + SLOTB + 8192, 16384, i64, false);
        bulk_wait_read_all_but_last();  // the hi tiles are scratch after this phase
        return true;
      }, [&] { scale_grad(GamC); });
      if (!ok) break;
      if (tid == 0 && c > 0) load_a(chunk - 1);
      {  // dE = Mq^T dO + wS K dS + Ap^T dP; dQS = Gam dO
        float x[16], y[16], w[16];
        tmem_ld16x2(tm + lane + T_R1 + g16, x, tm + lane + T_R2 + g16, y);
        lds16(wS + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) y[i] += w[i] * x[i];
        tmem_ld16(tm + lane + T_R3 + g16, x);
#pragma unroll
        for (int i = 0; i < 16; ++i) y[i] += x[i];
        put16s(sm + F, sm + F + HALF, j, g16, y);
        lds16(plain ? Gprev + g16 : Gam + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = p.scale * w[i] * dO(g16 + i);
        put16s(sm + GH, sm + GH + HALF, j, g16, w);
      }
      // ---- dX = T_beta^T dE; dS += Q^T dQS
      ok = phase_run(K, tid, [&] {
        if (!slot_wait<1>(K, K.phB)) return false;
        mma_s3_kmn(tm + T_R3, sb + F, sb + F + HALF, sb + slot_t, sb + slot_t + 8192, 16384, i64, false);
        mma_tile_kmn(tm + T_G, sb + GH, 0, sb + KQ + 8192, 16384, 4, i128, true);
        mma_tile_kmn(tm + T_G, sb + GH + HALF, 0, sb + KQ + 8192, 16384, 4, i128, true);
        bulk_wait_read();  // the lo tiles are scratch after this phase
        return true;
      });
      if (!ok) break;
      if (c > 0) {
        if (tid == 0) load_t(chunk - 1);
        next_do(c - 1);
      }
      {  // dX -> dv = -dP + dX; dKS = Gprev dP - Gam dX; dX (fp32) and dv staged
        float *stg = reinterpret_cast<float *>(sm + GL);
        __nv_bfloat16 *dvs = reinterpret_cast<__nv_bfloat16 *>(sm + GH);
        float *dvs32 = reinterpret_cast<float *>(sm + GH);
        float x[16], dks[16], gm[16];
        tmem_ld16(tm + lane + T_R3 + g16, x);
        lds16(dec_res ? Gam + g16 : Gprev + g16, dks);
        lds16(Gam + g16, gm);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int t = g16 + i;
          stg[t * D + j] = x[i];
          if (P.f32g)
            dvs32[t * D + j] = x[i] - dP[i];
          else
            dvs[t * D + j] = __float2bfloat16_rn(x[i] - dP[i]);
          dks[i] = dks[i] * dP[i] - (rla ? 0.f : gm[i] * x[i]);
        }
        put16s(sm + F, sm + F + HALF, j, g16, dks);
      }
      // ---- dS += K^T dKS; the staged dX and dv leave meanwhile
      ok = phase_run_with(K, tid, [&] {
        bulk_s2g(P.dXbuf + chunk * 64 * D, sm + GL, 32768);
        bulk_commit();
        mma_tile_kmn(tm + T_G, sb + F, 0, sb + KQ, 16384, 4, i128, true);
        mma_tile_kmn(tm + T_G, sb + F + HALF, 0, sb + KQ, 16384, 4, i128, true);
        return true;
      }, [&] {
        if (P.f32g) {  // dv rows, 16 bytes at a time
          float *dvf = (float *)P.dv;
          for (int e = tid; e < 64 * 32; e += NTC) {
            const int t = e >> 5, chn = e & 31;
            if (t < n)
              *reinterpret_cast<uint4 *>(dvf + ((size_t)(tok0 + t0 + t) * H + h) * D + chn * 4) =
                  *reinterpret_cast<const uint4 *>(sm + GH + t * 512 + chn * 16);
          }
        } else {
          for (int e = tid; e < 64 * 16; e += NTC) {
            const int t = e >> 4, chn = e & 15;
            if (t < n)
              *reinterpret_cast<uint4 *>(dv + ((size_t)(tok0 + t0 + t) * H + h) * D + chn * 8) =
                  *reinterpret_cast<const uint4 *>(sm + GH + t * 256 + chn * 16);
          }
        }
        if (tid == 0) bulk_wait_read();  // the staging is rewritten next (the gradient tiles)
      });
      if (!ok) break;
    }
    if (c > 0) {  // the next chunk's inputs, while this one finishes
      next_kq(c - 1);
      pre = fetch_pre(c - 1);
    }
    // the carried gradient's tiles (complete in TMEM)
#pragma unroll 1
    for (int c0 = g16; c0 < D; c0 += 64) {
      float s[16];
      tmem_ld16(tm + lane + T_G + c0, s);
      put_grad16(c0, s);
    }
    fence_async_smem();  // the tiles are read by the MMAs and by a bulk copy
  }
  __syncthreads();
  if (*K.flag) ok = false;
  // the last copy to CTA 0 has been taken
  if (!base && ok && NC > 0 && !mbar_wait_cluster(barX, (uint32_t)(NC - 1) & 1u, K.limit) &&
      tid == 0 && p.err)
    atomicExch(p.err, RDN_ERR_TIMEOUT);
  if (ok) {
    float *out = base ? P.dS0 : P.dR0;
    for (int c0 = g16; c0 < D && out; c0 += 64) {
      float s[16];
      tmem_ld16(tm + lane + T_G + c0, s);
#pragma unroll
      for (int i = 0; i < 16; ++i) out[st_base + (size_t)(c0 + i) * D + j] = s[i];
    }
  } else if (tid == 0) {
    if (p.err) atomicExch(p.err, RDN_ERR_TIMEOUT);
    // no copy into this CTA's shared memory or MMA outlives it (bounded waits)
    ctl_drain(K);
    for (; tma_seen < tma_arms; ++tma_seen) mbar_wait(K.barC, tma_seen & 1u);
    if (handed) mbar_wait_cluster(barX, (handed - 1) & 1u, K.limit);
  }
  cp_async_wait_all();
  if (tid == 0) bulk_wait_all();
  fence_before_sync();
  __syncthreads();
  cluster_sync();  // the partner may still write here, or arrive on a barrier
  if (warp == 0) tmem_dealloc(tm, 512);
}

}  // namespace

cudaError_t launch_bwd_pair(const bwdtc::TcBwdParams &P, cudaStream_t s) {
  auto kern = P.rla || P.f.mods != 0 ? bwd_pair_kernel<true> : bwd_pair_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * P.f.nseq * P.f.H);
  cfg.blockDim = dim3(NTC);
  cfg.dynamicSmemBytes = SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 2;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  RDN_LAUNCH("bwd_chain_pair", s, e = cudaLaunchKernelEx(&cfg, kern, P));
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace rdn
