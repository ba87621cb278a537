// fwd_pair.cu -- the tensor-core forward scan of fwd_tc.cu over a pair of CTAs
// (a cluster of two SMs) per (sequence, head), for calls whose sequences are
// too few to fill the chip.
//
// The scan is a chain of dependent phases per chunk, so a single sequence is
// bound by their latencies and not by any pipe.  The base recurrence never
// reads the auxiliary one: CTA 0 carries S, forms E, the clipped residual r
// and the base output Ob, and sends r and Ob (32 fp32 values a thread, the
// same thread mapping on both sides) into CTA 1's shared memory; CTA 1 carries
// R and finishes the output, one chunk behind.  Each has three phases a chunk
// where the one-CTA scan has six:
//
//   CTA 0:  MMA1 [KS | QS]  |  MMA2 E  |  MMA3 [P | Ob], MMA4 S        -> r, Ob
//   CTA 1:  MMA5 [KR | QR]  |  MMA6 E2 |  MMA7 Ob += .., MMA8 R        -> o
//
// (phases, operands and arithmetic as in fwd_tc.cu, in the same order: the
// results are the same bits).  The hand-over is one 64 KB buffer in CTA 1,
// filled by two bulk copies from CTA 0's shared memory, with a pair of
// mbarriers: `full` in CTA 1 (the copies' bytes), `empty` in CTA 0 (one arrival
// per warp of CTA 1 once it holds the values in registers; CTA 0 then also
// reuses what it copied from).  Both waits are bounded like every other; a CTA
// that gave up stops, its partner's waits then run out too, and the two meet
// at the cluster's barrier before either releases its shared memory.
//
// Measured: B = 2, H = 16, T = 16384 with states, 2.24 ms in one CTA per head,
// 1.59 ms in pairs; B = 1, T = 777, 0.123 and 0.095 ms.
#include "fwd_tc.cuh"

namespace rdn {
namespace {

using namespace fwdtc;

// shared memory (bytes from the 1024-aligned base); both CTAs:
constexpr uint32_t SM_ST = 0;        // the carried state's bf16 copy, two 64-column blocks
constexpr uint32_t SM_KQ = 32768;    // [K ; Q], 128 rows x 128
constexpr uint32_t SM_XE = 65536;    // X^T then E^T (X2^T then E2^T), hi | lo; CTA 0: from a
constexpr uint32_t SM_XE_LO = 81920; // chunk's end to the next MMA1 the state's lo part
constexpr uint32_t SM_W = 98304;     // (wS E)^T / (wR E2)^T, hi | lo; then CTA 0: Ob, fp32, to
constexpr uint32_t SM_W_LO = 114688; // be handed over; CTA 1: the o tile
constexpr uint32_t SM_SLOTA = 131072;  // T_beta / T_gamma image (hi | lo)
constexpr uint32_t SM_SLOTB = 147456;  // CTA 0: [Ap ; Mq] image, 32 KB; CTA 1: M2 image, 16 KB
// CTA 0: r, fp32, to be handed over (32 KB), V;  CTA 1: the hand-over buffer (r | Ob)
constexpr uint32_t SM_RES = 180224, SM_V = 212992;
constexpr uint32_t SM_X = 163840;
constexpr uint32_t SM_VEC = 229376;  // 5 x 64 fp32: Gam Gprev wS wR gamma
constexpr uint32_t SM_BAR = SM_VEC + 5 * 64 * 4;  // MMA, slot A, slot B, drain, tiles, hand-over
constexpr uint32_t SM_SLOT = SM_BAR + 48;
constexpr uint32_t SM_FLAG = SM_SLOT + 4;
constexpr size_t kPairSmem = SM_FLAG + 4;
static_assert(SM_X + 65536 == SM_VEC && SM_V + 16384 == SM_VEC, "carve-up");
static_assert(kPairSmem <= 232448, "shared memory");

// TMEM columns: the state, the read-outs D1 (CTA 0: KS | QS, ..; CTA 1: E2 |
// Ob) and CTA 1's KR | QR
constexpr uint32_t T_ST = 0, T_D1 = 128, T_X = 256;

template <bool RDNV, bool kGeneric>
__global__ void __launch_bounds__(kTcThreads, 1)
    fwd_pair_kernel(FwdParams p, const __grid_constant__ FwdMaps maps) {
  extern __shared__ __align__(1024) uint8_t sm[];
  const uint32_t sbase = smem_u32(sm);
  if (sbase & 1023u) {  // (the same in both CTAs)
    if (threadIdx.x == 0 && p.err) atomicExch(p.err, RDN_ERR_CUDA);
    return;
  }
  float *vec = reinterpret_cast<float *>(sm + SM_VEC);
  float *Gam = vec, *Gprev = vec + 64, *wS = vec + 128, *wR = vec + 192, *gamv = vec + 256;
  uint64_t *bar = reinterpret_cast<uint64_t *>(sm + SM_BAR);
  uint64_t *barA = bar + 1, *barB = bar + 2, *barD = bar + 3, *barE = bar + 4;
  uint64_t *barX = bar + 5;  // CTA 1: full; CTA 0: empty
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + SM_SLOT);
  volatile int *flag = reinterpret_cast<volatile int *>(sm + SM_FLAG);

  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t rank = cluster_rank();
  const bool base = rank == 0;     // CTA 0: S; CTA 1: R
  const int j = tid & 127;         // value column == TMEM lane
  const int g16 = (warp >> 2) * 16;  // this thread's token (and state) columns start
  const int bh = blockIdx.x >> 1;
  const int h = bh % p.H;
  const SeqSpan sp = seq_span(p, bh / p.H, h);
  const long long tok0 = sp.tok0;
  const int T = sp.len, H = p.H, NC = sp.nc;
  const __nv_bfloat16 *q = (const __nv_bfloat16 *)p.q;
  const __nv_bfloat16 *k = (const __nv_bfloat16 *)p.k;
  const __nv_bfloat16 *v = (const __nv_bfloat16 *)p.v;
  __nv_bfloat16 *o = (__nv_bfloat16 *)p.o;
  const float clip = p.clip;
  // (the variants: fwd_tc.cu)
  const bool dec_res = kGeneric && (p.mods & RDN_FLAG_DECAYED_RESIDUAL);
  const bool plain = kGeneric && (p.mods & RDN_FLAG_PLAIN_COMBINE);
  const bool tnh = kGeneric && (p.mods & RDN_FLAG_TANH_RESIDUAL);
  const bool stl = kGeneric && (p.mods & RDN_FLAG_STATELESS_AUX);
  const size_t st_base = (size_t)bh * D * D;

  if (tid == 0) {
    for (int b = 0; b < 5; ++b) mbar_init(bar + b, 1);
    mbar_init(barX, base ? kTcThreads / 32 : 1);
    fence_mbar_init();
    if (!base) mbar_expect_tx(barX, 65536);
    *flag = 0;
  }
  if (warp == 0) tmem_alloc(slot, 512);
  fence_before_sync();
  __syncthreads();
  cluster_sync();  // the partner's barriers exist before anything arrives on them
  fence_after_sync();
  const uint32_t tm = *slot;
  const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
  uint32_t phase = 0, phA = 0, phB = 0;  // phA/phB: tracked by thread 0 only
  bool pendA = false, pendB = false;     // (thread 0) a slot copy armed and not yet waited for
  const long long limit = p.inject == 1 ? 10000000ll : 2000000000ll;
  bool skip_commit = p.inject == 1 && base;
  const uint32_t peer_bar = map_rank(barX, rank ^ 1u);
  const uint32_t peer_x = map_rank(sm + SM_X, 1u);

  auto rec_of = [&](int c) {
    return reinterpret_cast<const uint8_t *>(p.ws + (size_t)(sp.rbase + c) * kRecFloats);
  };
  auto load_a = [&](int c) {  // (thread 0) T_beta / T_gamma
    mbar_expect_tx(barA, 16384);
    bulk_g2s(sm + SM_SLOTA, rec_of(c) + (base ? IMG_TB : IMG_TG), 16384, barA);
    pendA = true;
  };
  auto load_b = [&](int c) {  // (thread 0) [Ap ; Mq] / M2
    const uint32_t bytes = base ? 32768u : 16384u;
    mbar_expect_tx(barB, bytes);
    bulk_g2s(sm + SM_SLOTB, rec_of(c) + (base ? IMG_APMQ : IMG_M2), bytes, barB);
    pendB = true;
  };
  auto wait_a = [&]() {
    if (!mbar_wait(barA, phA)) return false;
    phA ^= 1u;
    pendA = false;
    return true;
  };
  auto wait_b = [&]() {
    if (!mbar_wait(barB, phB)) return false;
    phB ^= 1u;
    pendB = false;
    return true;
  };
  if (tid == 0 && NC > 0) {
    if (RDNV) load_a(0);
    load_b(0);
  }
  // a chunk's tiles: by tensor-map copies on barrier E where the chunk is whole
  // (not the first, not the last), by cp.async with zero fill otherwise
  auto fetch_v = [&](int c) {
    const int t0 = c * 64, n = min(64, T - t0);
    for (int e = tid; e < 64 * 16; e += kTcThreads) {
      const int t = e >> 4, ch = e & 15;
      const bool vld = t < n;
      const size_t off = ((size_t)(tok0 + t0 + (vld ? t : 0)) * H + h) * D + ch * 8;
      cp_async16(sm + SM_V + (ch >> 3) * 8192 + sw128(t, (ch & 7) * 8), v + off, vld);
    }
  };
  auto fetch_kq = [&](int c) {
    const int t0 = c * 64, n = min(64, T - t0);
    for (int e = tid; e < 64 * 16; e += kTcThreads) {
      const int t = e >> 4, ch = e & 15;
      const bool vld = t < n;
      const size_t off = ((size_t)(tok0 + t0 + (vld ? t : 0)) * H + h) * D + ch * 8;
      const int blk = ch >> 3, cc = (ch & 7) * 8;
      cp_async16(sm + SM_KQ + blk * 16384 + sw128(t, cc), k + off, vld);
      cp_async16(sm + SM_KQ + blk * 16384 + sw128(64 + t, cc), q + off, vld);
    }
  };
  auto by_tma = [&](int cc) { return maps.ok && cc > 0 && cc < NC - 1; };
  uint32_t phE = 0;    // phases of barrier E waited for
  bool pendE = false;  // (thread 0) a phase armed and not yet waited for
  // V is free a phase earlier than K, Q: CTA 0 arms barrier E with V's copy,
  // CTA 1, which reads no V, with K's and Q's
  auto next_v = [&](int cc) {
    if (!by_tma(cc)) {
      fetch_v(cc);
    } else if (tid == 0) {
      const int row = (int)(tok0 + (long long)cc * 64);
      mbar_expect_tx(barE, 49152);
      pendE = true;
      for (int kb = 0; kb < 2; ++kb) tma_load_3d(sm + SM_V + kb * 8192, maps.v, 64 * kb, h, row, barE);
    }
  };
  auto next_kq = [&](int cc) {
    if (!by_tma(cc)) {
      fetch_kq(cc);
    } else if (tid == 0) {
      const int row = (int)(tok0 + (long long)cc * 64);
      if (!base) {
        mbar_expect_tx(barE, 32768);
        pendE = true;
      }
      for (int kb = 0; kb < 2; ++kb) {
        tma_load_3d(sm + SM_KQ + kb * 16384, maps.k, 64 * kb, h, row, barE);
        tma_load_3d(sm + SM_KQ + kb * 16384 + 8192, maps.q, 64 * kb, h, row, barE);
      }
    }
  };
  if (NC > 0) {
    if (base) fetch_v(0);
    fetch_kq(0);
  }

  // a state's bf16 copy, and CTA 0's also its lo part, 16 columns
  auto put_state = [&](int c0, const float (&s)[16]) {
    st_row16(sm + SM_ST, 16384, j, c0, s);
    if (base) {
      float lo[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) lo[i] = s[i] - __bfloat162float(__float2bfloat16_rn(s[i]));
      st_row16(sm + SM_XE, SM_XE_LO - SM_XE, j, c0, lo);
    }
  };
  const float *init = base ? p.S0 : p.R0;
  float *chunks = base ? p.S_chunks : p.R_chunks;
  for (int c0 = g16; c0 < D; c0 += 64) {
    float s[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) s[i] = init ? init[st_base + (size_t)(c0 + i) * D + j] : 0.f;
    tmem_st16(tm + lane + T_ST + c0, s);
    put_state(c0, s);
    if (chunks && NC > 0)
#pragma unroll
      for (int i = 0; i < 16; ++i)
        chunks[(size_t)sp.rbase * D * D + (size_t)(c0 + i) * D + j] = s[i];
  }

  auto run_phase = [&](auto issue, auto during) -> bool {
    fence_async_smem();
    fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      fence_after_sync();
      if (!issue()) *flag = 1;
      if (!skip_commit) mma_commit(bar);
      skip_commit = false;
    }
    during();
    const bool ok = mbar_wait(bar, phase, limit);
    phase ^= 1u;
    if (!ok) *flag = 1;
    __syncthreads();
    fence_after_sync();
    return *flag == 0;
  };
  auto nothing = [] {};
  // L2 prefetch of what this CTA reads of a chunk's record and rows
  auto prefetch_chunk = [&](int c) {
    const int t0_ = c * 64, n_ = min(64, T - t0_);
    if (tid == 0) {
      const uint8_t *r = rec_of(c);
      prefetch_l2_bulk(r + (base ? IMG_TB : IMG_TG), base ? 49152 : 32768);
      static_assert(IMG_APMQ == IMG_TB + 16384 && IMG_M2 == IMG_TG + 16384, "contiguous images");
      prefetch_l2_bulk(r + OFF_VEC * 4, (kRecFloats - OFF_VEC) * 4);
    }
    if (tid < 384) {
      const int rr = tid >> 1, t = rr & 63, w = rr >> 6;
      const __nv_bfloat16 *src = w == 0 ? k : (w == 1 ? q : v);
      if (t < n_ && (base || w < 2))
        prefetch_l2_line(src + ((size_t)(tok0 + t0_ + t) * H + h) * D + (tid & 1) * 64);
    } else if (!base && tid < 416) {
      const int t = 2 * (tid - 384);
      if (t < n_) prefetch_l2_line(p.gamma + (size_t)(tok0 + t0_ + t) * H + h);
    }
  };
  // the state's TMEM copy times the chunk's total decay, in place, its values
  // before that to the chunk-start states (fwd_tc.cu's scale_state)
  auto scale_state = [&](float f, float *start) {
    float x[16], y[16];
    tmem_ld16x2(tm + lane + T_ST + g16, x, tm + lane + T_ST + g16 + 64, y);
    if (start) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        start[(size_t)(g16 + i) * D + j] = x[i];
        start[(size_t)(g16 + 64 + i) * D + j] = y[i];
      }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      x[i] *= f;
      y[i] *= f;
    }
    tmem_st16(tm + lane + T_ST + g16, x);
    tmem_st16(tm + lane + T_ST + g16 + 64, y);
  };
  struct Pre {  // a chunk's gate values (threads 0..63) and its total decay
    float gm, gp, w, g, gc;
  };
  auto fetch_pre = [&](int c) {
    const float *rc = p.ws + (size_t)(sp.rbase + c) * kRecFloats;
    const int t0_ = c * 64, n_ = min(64, T - t0_);
    Pre x;
    x.gm = x.gp = x.w = x.g = 0.f;
    if (tid < 64) {
      x.gm = rc[OFF_VEC + V_GAM + tid];
      x.w = rc[OFF_VEC + (base ? V_WS : V_WR) + tid];
      if (base) x.gp = rc[OFF_VEC + V_GPREV + tid];
      else x.g = tid < n_ ? p.gamma[(size_t)(tok0 + t0_ + tid) * H + h] : 0.f;
    }
    x.gc = rc[OFF_VEC + V_GAMC];
    return x;
  };
  Pre pre{};
  if (NC > 0) pre = fetch_pre(0);

  // CTA 0, thread 0 (after a barrier that published them): r and Ob -> CTA 1
  uint32_t handed = 0;
  auto hand_over = [&] {
    ++handed;
    bulk_s2s(peer_x, sm + SM_RES, 32768, peer_bar);
    bulk_s2s(peer_x + 32768, sm + SM_W, 32768, peer_bar);
  };

  bool alive = true;
  for (int c = 0; c < NC && alive; ++c) {
    const int t0 = c * 64;
    const int n = min(64, T - t0);
    const size_t ci = (size_t)(sp.rbase + c);  // chunk index of the saved intermediates
    if (c + 1 < NC) prefetch_chunk(c + 1);
    if (by_tma(c)) {
      if (!mbar_wait(barE, phE & 1u)) *flag = 1;
      ++phE;
      if (tid == 0) pendE = false;
    } else {
      cp_async_wait_all();
    }
    float *start = (chunks && c > 0) ? chunks + ci * D * D : nullptr;
    if (tid < 64) {  // (last read before the previous chunk's last barrier)
      Gam[tid] = pre.gm;
      if (base) {
        Gprev[tid] = pre.gp;
        wS[tid] = pre.w;
      } else {
        wR[tid] = pre.w;
        gamv[tid] = pre.g;
      }
    }
    const float GamC = pre.gc;
    if (c + 1 < NC) pre = fetch_pre(c + 1);  // in flight during this chunk
    if (base) fence_async_smem();            // r and Ob of the previous chunk
    __syncthreads();
    if (*flag) {
      alive = false;
      break;
    }
    if (base) {
      if (tid == 0 && c > 0) hand_over();
      // ---- MMA1: D1 = S^T [K ; Q]^T (S as hi + lo)
      alive = run_phase([&] {
        mma_tile(tm + T_D1, sbase + SM_ST, 16384, sbase + SM_KQ, 16384, 8, idesc_bf16(128, 128), false);
        mma_tile(tm + T_D1, sbase + SM_XE, SM_XE_LO - SM_XE, sbase + SM_KQ, 16384, 8, idesc_bf16(128, 128), true);
        return true;
      }, [&] { scale_state(GamC, start); });
      if (!alive) break;
      float gks[16], vv[16];
      {
        float x[16], gm[16], gp[16];
        tmem_ld16x2(tm + lane + T_D1 + 64 + g16, x, tm + lane + T_D1 + g16, gks);
        lds16(plain ? Gprev + g16 : Gam + g16, gm);
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] *= gm[i] * p.scale;  // Ob accumulates onto Gam scale QS
        tmem_st16(tm + lane + T_D1 + 64 + g16, x);
        lds16(Gam + g16, gm);
        lds16(Gprev + g16, gp);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          vv[i] = __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(
              sm + SM_V + (j >> 6) * 8192 + sw128(g16 + i, j & 63)));
          x[i] = vv[i] - gm[i] * gks[i];
          gks[i] *= dec_res ? gm[i] : gp[i];
        }
        if (RDNV) {
          st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, x);
        } else {
          tmem_st16(tm + lane + T_D1 + g16, gks);
        }
      }
      if (RDNV) {  // ---- MMA2: E^T = X^T T_beta^T
        alive = run_phase([&] {
          if (!wait_a()) return false;
          mma_split3(tm + T_D1, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTA,
                     sbase + SM_SLOTA + 8192, idesc_bf16(128, 64), false);
          return true;
        }, nothing);
        if (!alive) break;
        if (tid == 0 && c + 1 < NC) load_a(c + 1);
      } else {
        __syncthreads();  // (every thread has read its V)
      }
      if (c + 1 < NC) next_v(c + 1);
      {
        float e[16], w[16];
        if (RDNV) {
          tmem_ld16(tm + lane + T_D1 + g16, e);
          tmem_st16(tm + lane + T_D1 + g16, gks);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) e[i] = vv[i];
        }
        lds16(wS + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] *= e[i];
        st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, e);
        // (the previous chunk's hand-over has left W and the r staging)
        if (c > 0 && !mbar_wait_cluster(barX, (uint32_t)(c - 1) & 1u, limit)) *flag = 1;
        st_row16_split(sm + SM_W, sm + SM_W_LO, j, g16, w);
      }
      // ---- MMA3: D1 += E^T [Ap;Mq]^T;  MMA4: S += (wS E)^T K
      alive = run_phase([&] {
        if (!wait_b()) return false;
        mma_split3(tm + T_D1, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTB,
                   sbase + SM_SLOTB + 16384, idesc_bf16(128, 128), true);
        if (p.sv_E) {  // keep the E^T image (hi | lo) for the backward
          static_assert(SM_XE_LO == SM_XE + 16384, "contiguous");
          bulk_s2g(p.sv_E + ci * 32768, sm + SM_XE, 32768);
          bulk_commit();
        }
        mma_tile_kmn(tm + T_ST, sbase + SM_W, 0, sbase + SM_KQ, 16384, 4, idesc_bf16(128, 128), true);
        mma_tile_kmn(tm + T_ST, sbase + SM_W_LO, 0, sbase + SM_KQ, 16384, 4, idesc_bf16(128, 128), true);
        return true;
      }, [&] {
        if (tid == 0 && p.sv_E) bulk_wait_read();  // the E^T tiles are rewritten next
      });
      if (!alive) break;
      if (c + 1 < NC) {
        if (tid == 0) load_b(c + 1);
        next_kq(c + 1);
      }
      // ---- S (= Gam_C S + U) -> its bf16 copies; r = clip(V - P); r, Ob -> CTA 1
      {
        float s0[16], s1[16];
        tmem_ld16x2(tm + lane + T_ST + g16, s0, tm + lane + T_ST + g16 + 64, s1);
        put_state(g16, s0);
        put_state(g16 + 64, s1);
      }
      {
        float pp[16], ob[16], r[16];
        tmem_ld16x2(tm + lane + T_D1 + g16, pp, tm + lane + T_D1 + 64 + g16, ob);
        if (!tnh) {
          unsigned msk = 0u;  // bit i: |x| <= c at t = g16 + i
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float x = vv[i] - pp[i];
            if (fabsf(x) <= clip) msk |= 1u << i;
            r[i] = clampf(x, clip);
          }
          if (p.sv_mask) reinterpret_cast<uint16_t *>(p.sv_mask + ci * D + j)[g16 >> 4] = (uint16_t)msk;
        } else {
          uint32_t dg[8];
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            const float x0 = vv[i] - pp[i], x1 = vv[i + 1] - pp[i + 1];
            r[i] = resid_map(x0, clip, true);
            r[i + 1] = resid_map(x1, clip, true);
            dg[i / 2] = grad_q16(resid_grad(x0, clip, true)) |
                        (grad_q16(resid_grad(x1, clip, true)) << 16);
          }
          if (p.sv_mask) {
            uint4 *dst = reinterpret_cast<uint4 *>(reinterpret_cast<uint16_t *>(p.sv_mask) +
                                                   (ci * D + j) * 64 + g16);
            dst[0] = make_uint4(dg[0], dg[1], dg[2], dg[3]);
            dst[1] = make_uint4(dg[4], dg[5], dg[6], dg[7]);
          }
        }
        float4 *xr = reinterpret_cast<float4 *>(sm + SM_RES) + tid;
        float4 *xo = reinterpret_cast<float4 *>(sm + SM_W) + tid;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          xr[512 * i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
          xo[512 * i] = make_float4(ob[4 * i], ob[4 * i + 1], ob[4 * i + 2], ob[4 * i + 3]);
        }
      }
    } else {
      // ---- MMA5: X = R^T [K ; Q]^T
      alive = run_phase([&] {
        if (p.sv_E2) bulk_wait_read();  // the E2^T tiles of the previous chunk are rewritten next
        mma_tile(tm + T_X, sbase + SM_ST, 16384, sbase + SM_KQ, 16384, 8, idesc_bf16(128, 128), false);
        return true;
      }, [&] { scale_state(stl ? 0.f : GamC, start); });
      if (!alive) break;
      float r[16];
      const bool got = mbar_wait_cluster(barX, (uint32_t)c & 1u, limit);
      if (!got) *flag = 1;
      {
        float ob[16];
        const float4 *x = reinterpret_cast<const float4 *>(sm + SM_X) + tid;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 a = x[512 * i], b = x[512 * (4 + i)];
          r[4 * i] = a.x; r[4 * i + 1] = a.y; r[4 * i + 2] = a.z; r[4 * i + 3] = a.w;
          ob[4 * i] = b.x; ob[4 * i + 1] = b.y; ob[4 * i + 2] = b.z; ob[4 * i + 3] = b.w;
        }
        // (a phase that has not completed takes no further arrival)
        if (got && tid == 0 && c + 1 < NC) mbar_expect_tx(barX, 65536);
        __syncwarp();
        if (got && (tid & 31) == 0) mbar_arrive_remote(peer_bar);
        tmem_st16(tm + lane + T_D1 + 64 + g16, ob);
      }
      if (RDNV) {  // ---- X2 = r - Gam KR;  MMA6: E2^T = X2^T T_gamma^T
        {
          float x[16], gm[16];
          tmem_ld16(tm + lane + T_X + g16, x);
          lds16(Gam + g16, gm);
#pragma unroll
          for (int i = 0; i < 16; ++i) x[i] = stl ? r[i] : r[i] - gm[i] * x[i];
          st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, x);
        }
        alive = run_phase([&] {
          if (!wait_a()) return false;
          mma_split3(tm + T_D1, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTA,
                     sbase + SM_SLOTA + 8192, idesc_bf16(128, 64), false);
          return true;
        }, nothing);
        if (!alive) break;
        if (tid == 0 && c + 1 < NC) load_a(c + 1);
      }
      {
        float e[16], w[16];
        if (RDNV) {
          tmem_ld16(tm + lane + T_D1 + g16, e);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) e[i] = r[i];
        }
        lds16(wR + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] *= e[i];
        st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, e);
        st_row16_split(sm + SM_W, sm + SM_W_LO, j, g16, w);
      }
      // ---- MMA7: Ob += E2^T (gamma M2)^T;  MMA8: R += (wR E2)^T K
      alive = run_phase([&] {
        if (!wait_b()) return false;
        mma_split3(tm + T_D1 + 64, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTB,
                   sbase + SM_SLOTB + 8192, idesc_bf16(128, 64), true);
        if (p.sv_E2) {
          bulk_s2g(p.sv_E2 + ci * 32768, sm + SM_XE, 32768);
          bulk_commit();
        }
        mma_tile_kmn(tm + T_ST, sbase + SM_W, 0, sbase + SM_KQ, 16384, 4, idesc_bf16(128, 128), true);
        mma_tile_kmn(tm + T_ST, sbase + SM_W_LO, 0, sbase + SM_KQ, 16384, 4, idesc_bf16(128, 128), true);
        return true;
      }, nothing);
      if (!alive) break;
      if (c + 1 < NC) {
        if (tid == 0) load_b(c + 1);
        next_kq(c + 1);
      }
      // ---- R -> its bf16 copy; o = Ob + gamma Gam QR, staged in W's place
      {
        float r0[16], r1[16];
        tmem_ld16x2(tm + lane + T_ST + g16, r0, tm + lane + T_ST + g16 + 64, r1);
        put_state(g16, r0);
        put_state(g16 + 64, r1);
      }
      {
        __nv_bfloat16 *ostg = reinterpret_cast<__nv_bfloat16 *>(sm + SM_W);
        float *ostg32 = reinterpret_cast<float *>(sm + SM_W);
        static_assert(SM_W_LO == SM_W + 16384, "fp32 o staging spans W and its lo part");
        float ob[16], oa[16], gm[16], gv[16];
        tmem_ld16x2(tm + lane + T_D1 + 64 + g16, ob, tm + lane + T_X + 64 + g16, oa);
        lds16(Gam + g16, gm);
        lds16(gamv + g16, gv);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int t = g16 + i;
          const float gg = plain ? 1.f : gv[i];
          const float ov = stl ? ob[i] : fmaf(gg * gm[i] * p.scale, oa[i], ob[i]);
          if (p.f32out)
            ostg32[t * D + j] = ov;
          else
            ostg[t * D + j] = __float2bfloat16_rn(ov);
        }
      }
      __syncthreads();  // the o tile
      if (p.f32out) {
        float *of = (float *)p.o;
        for (int e = tid; e < 64 * 32; e += kTcThreads) {
          const int t = e >> 5, ch = e & 31;
          if (t < n)
            *reinterpret_cast<uint4 *>(of + ((size_t)(tok0 + t0 + t) * H + h) * D + ch * 4) =
                *reinterpret_cast<const uint4 *>(sm + SM_W + t * 512 + ch * 16);
        }
      } else {
        for (int e = tid; e < 64 * 16; e += kTcThreads) {
          const int t = e >> 4, ch = e & 15;
          if (t < n)
            *reinterpret_cast<uint4 *>(o + ((size_t)(tok0 + t0 + t) * H + h) * D + ch * 8) =
                *reinterpret_cast<const uint4 *>(sm + SM_W + t * 256 + ch * 16);
        }
      }
    }
  }

  if (tid == 0 && p.sv_E) bulk_wait_all();
  if (base) fence_async_smem();
  __syncthreads();
  if (*flag) alive = false;  // (a wait of the last chunk)
  if (base && alive && NC > 0) {  // the last chunk's r and Ob, until CTA 1 holds them
    if (tid == 0) hand_over();
    if (!mbar_wait_cluster(barX, (uint32_t)(NC - 1) & 1u, limit) && tid == 0 && p.err)
      atomicExch(p.err, RDN_ERR_TIMEOUT);
  }
  if (alive) {  // final state
    float *fin = base ? p.ST : p.RT;
    for (int c0 = g16; c0 < D && fin; c0 += 64) {
      float s[16];
      tmem_ld16(tm + lane + T_ST + c0, s);
#pragma unroll
      for (int i = 0; i < 16; ++i) fin[st_base + (size_t)(c0 + i) * D + j] = s[i];
    }
  } else {
    // a bounded wait gave up: drain what is in flight (fwd_tc.cu), bounded
    if (tid == 0) {
      if (p.err) atomicExch(p.err, RDN_ERR_TIMEOUT);
      mma_commit(barD);
      mbar_wait(barD, 0);
      if (pendA) mbar_wait(barA, phA);
      if (pendB) mbar_wait(barB, phB);
      if (pendE) mbar_wait(barE, phE & 1u);
      if (handed) mbar_wait_cluster(barX, (handed - 1) & 1u, limit);
      bulk_wait_all();
    }
    cp_async_wait_all();
  }
  fence_before_sync();
  __syncthreads();
  cluster_sync();  // the partner may still write here, or arrive on a barrier
  if (warp == 0) tmem_dealloc(tm, 512);
}

}  // namespace

cudaError_t launch_fwd_pair(const FwdParams &p, const fwdtc::FwdMaps &maps, bool rdnv, cudaStream_t s) {
  const bool generic = p.mods != 0;
  auto kern = rdnv ? (generic ? fwd_pair_kernel<true, true> : fwd_pair_kernel<true, false>)
                   : (generic ? fwd_pair_kernel<false, true> : fwd_pair_kernel<false, false>);
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPairSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * p.nseq * p.H);
  cfg.blockDim = dim3(kTcThreads);
  cfg.dynamicSmemBytes = kPairSmem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 2;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  RDN_LAUNCH("fwd_tc_pair", s, e = cudaLaunchKernelEx(&cfg, kern, p, maps));
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace rdn
