// bwd_tc.cu -- tensor-core (tcgen05 / TMEM) backward of the chunkwise RDN
// forward, bf16 inputs, d_k = d_v = 128; RLA (TcBwdParams::rla) and the variant
// flags are modes of separate kernel instances.
//
// Reverse mode of the chunk algebra of chunk_fwd.cu, split by what depends on
// the gradients carried between chunks:
//
//  1. bwd_recompute (parallel, one CTA per chunk): from the chunk-start
//     states rebuild E, E2 and the clip mask (the forward's pieces for one
//     chunk).  It does not run when the forward saved them.
//  2. bwd_chain (sequential over chunks, one CTA per (b,h); bwd_chain.cu): the
//     gradients carried between chunks, dX2, dX and dv.  No forward quantity
//     other than the clip mask enters this chain.
//  3. bwd_post (parallel, one CTA per chunk): every product that reduces over
//     the value dimension -- the state terms of dK, dQ, the five C x C
//     gradients, the per-row gate terms -- and then the gradients of the chunk
//     matrices' entries turned into dq, dk, dg, dbeta, dgamma.
//
// Orientation: value column j = TMEM lane j, owned by thread j of a group of
// 128 threads, for every column quantity (X, E, dO, dX2, ...), which is kept as a bf16 hi + lo tile
// [j][t] (K-major for products over t).  Products over j use the same tiles
// as MN-major operands.  The chunk matrices come from chunk_prep's images
// (bf16 hi + lo); products with them are three MMAs (hi*hi + hi*lo + lo*hi).
// States and carried gradients enter their products as bf16 hi + lo as well.
#include "bwd_tc.cuh"

namespace rdn {
namespace {

using namespace bwdtc;

constexpr int NT = 128;   // threads per CTA of bwd_recompute

// bwd_post's per-token sums kept in shared memory from where they are formed
// to the gate pass (floats): the read-out part of d gamma, dwS, dwR (C each).
struct A8 {
  static constexpr int V_DGAM_OUT = 0, V_DWS = C, V_DWR = 2 * C;
  static constexpr int FLOATS = 3 * C;
};

// ======================================================================== 1
// bwd_recompute: the forward pieces of one chunk from its start states.
namespace rc {
constexpr uint32_t SA = 0, RA = 32768, B1 = 65536, SLOTA = 98304, SLOTB = 114688;
constexpr uint32_t XE = 147456, XE_LO = 163840, VEC = 180224;
constexpr uint32_t CTL = VEC + 7 * 64 * 4;
constexpr uint32_t SLOT = CTL + 48;
constexpr uint32_t SA_LO = 183296;  // S0 - bf16(S0), two 16 KB blocks
static_assert(SA_LO >= SLOT + 16 && SA_LO % 1024 == 0, "layout");
constexpr size_t SMEM = SA_LO + 32768;
constexpr uint32_t T_D1 = 0, T_D3 = 128, T_X = 256;
}  // namespace rc

__global__ void __launch_bounds__(NT, 1) bwd_recompute_kernel(TcBwdParams P) {
  using namespace rc;
  extern __shared__ __align__(1024) uint8_t sm[];
  const uint32_t sb = smem_u32(sm);
  const FwdParams &p = P.f;
  if (sb & 1023u) {
    if (threadIdx.x == 0 && p.err) atomicExch(p.err, RDN_ERR_CUDA);
    return;
  }
  float *vec = reinterpret_cast<float *>(sm + VEC);
  float *Gam = vec, *Gprev = vec + 64, *gamv = vec + 320;
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + SLOT);
  const int tid = threadIdx.x, warp = tid >> 5, j = tid;
  const size_t chunk = blockIdx.x;
  if ((long long)chunk >= total_records(p)) return;  // (packed sequences: the grid is a bound)
  const int H = p.H;
  int sq, h, c;
  rec_decode(p, (long long)chunk, sq, h, c);
  const SeqSpan sp = seq_span(p, sq, h);
  const long long tok0 = sp.tok0;
  const int T = sp.len;
  const int t0 = c * 64, n = min(64, T - t0);
  const __nv_bfloat16 *k = (const __nv_bfloat16 *)p.k, *v = (const __nv_bfloat16 *)p.v;
  const uint8_t *rec = rec_bytes(p, chunk);
  const float clip = p.clip;

  Ctl K;
  ctl_init(K, sm + CTL, tid);
  if (warp == 0) tmem_alloc(slot, 512);
  if (tid == 0) {
    load_slot<0>(K, sm + SLOTA, rec + IMG_TB, 16384);
    load_slot<1>(K, sm + SLOTB, rec + IMG_APMQ, 32768);
  }
  if (tid < 64) {
    Gam[tid] = reinterpret_cast<const float *>(rec)[OFF_VEC + V_GAM + tid];
    Gprev[tid] = reinterpret_cast<const float *>(rec)[OFF_VEC + V_GPREV + tid];
    gamv[tid] = tid < n ? p.gamma[(size_t)(tok0 + t0 + tid) * H + h] : 0.f;
  }
  // chunk-start states -> bf16 A operands (row j = column j of [i][j])
  {
    const float *S0 = P.Sc + chunk * D * D, *R0 = P.Rc + chunk * D * D;
    for (int c0 = 0; c0 < D; c0 += 16) {
      float s[16], r[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        s[i] = S0[(size_t)(c0 + i) * D + j];
        r[i] = R0[(size_t)(c0 + i) * D + j];
      }
      put16(sm + SA, 16384, j, c0, s);
      put16(sm + RA, 16384, j, c0, r);
      {  // S0 - bf16(S0), as the forward scan's read-outs use it
#pragma unroll
        for (int i = 0; i < 16; ++i) s[i] -= __bfloat162float(__float2bfloat16_rn(s[i]));
        put16(sm + SA_LO, 16384, j, c0, s);
      }
    }
  }
  __syncthreads();
  // B1 = K (64 rows, exact bf16); the forward scan's arithmetic: unscaled
  // read-outs, gates applied in fp32
  for (int e = tid; e < 64 * 16; e += NT) {
    const int t = e >> 4, ch = e & 15;
    const bool vld = t < n;
    const size_t off = ((size_t)(tok0 + t0 + (vld ? t : 0)) * H + h) * D + ch * 8;
    cp_async16(sm + B1 + (ch >> 3) * 16384 + sw128(t, (ch & 7) * 8), k + off, vld);
  }
  cp_async_wait_all();
  fence_async_smem();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tm = *slot;
  const uint32_t lane = (uint32_t)(warp * 32) << 16;
  auto vval = [&](int t) -> float {
    return t < n ? __bfloat162float(v[((size_t)(tok0 + t0 + t) * H + h) * D + j]) : 0.f;
  };

  bool ok = phase_run(K, tid, [&] {  // KS, KR
    mma_tile(tm + T_D1, sb + SA, 16384, sb + B1, 16384, 8, idesc_bf16(128, 64), false);
    mma_tile(tm + T_D1, sb + SA_LO, 16384, sb + B1, 16384, 8, idesc_bf16(128, 64), true);
    mma_tile(tm + T_D3, sb + RA, 16384, sb + B1, 16384, 8, idesc_bf16(128, 64), false);
    return true;
  });
  float r[64];
  if (ok) {  // X = V - Gam KS -> E = T_beta X; D1 <- Gprev KS (P accumulates onto it)
#pragma unroll
    for (int c0 = 0; c0 < 64; c0 += 16) {
      float ks[16], x[16];
      tmem_ld16(tm + lane + T_D1 + c0, ks);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        x[i] = vval(c0 + i) - (P.rla ? 0.f : Gam[c0 + i] * ks[i]);
        ks[i] *= (p.mods & RDN_FLAG_DECAYED_RESIDUAL) ? Gam[c0 + i] : Gprev[c0 + i];
      }
      tmem_st16(tm + lane + T_D1 + c0, ks);
      put16s(sm + XE, sm + XE_LO, j, c0, x);
    }
    ok = phase_run(K, tid, [&] {
      if (!slot_wait<0>(K, K.phA)) return false;
      mma_s3_kk(tm + T_X, sb + XE, sb + XE_LO, sb + SLOTA, sb + SLOTA + 8192, idesc_bf16(128, 64),
                 false);
      return true;
    });
  }
  if (ok) {
    if (tid == 0) load_slot<0>(K, sm + SLOTA, rec + IMG_TG, 16384);
    __syncwarp();  // (TMEM accesses take whole warps)
#pragma unroll
    for (int c0 = 0; c0 < 64; c0 += 16) {
      float e[16];
      tmem_ld16(tm + lane + T_X + c0, e);
      put16s(sm + XE, sm + XE_LO, j, c0, e);
    }
    ok = phase_run(K, tid, [&] {  // D1 += E Ap^T -> P (the Ap rows of the [Ap ; Mq] image)
      if (!slot_wait<1>(K, K.phB)) return false;
      mma_s3_kk(tm + T_D1, sb + XE, sb + XE_LO, sb + SLOTB, sb + SLOTB + 16384,
                 idesc_bf16(128, 64), true);
      static_assert(XE_LO == XE + 16384, "contiguous");
      bulk_s2g(P.Ebuf + chunk * 32768, sm + XE, 32768);  // the E^T image, for bwd_post
      bulk_commit();
      bulk_wait_read();
      return true;
    });
  }
  if (ok) {
    // the clip mask, or with the tanh residual its derivative ([j][t], grad_q16)
    const bool tnh = p.mods & RDN_FLAG_TANH_RESIDUAL;
    uint16_t *drow = reinterpret_cast<uint16_t *>(P.mask) + (chunk * D + j) * 64;
    unsigned long long m = 0ull;
#pragma unroll
    for (int c0 = 0; c0 < 64; c0 += 16) {
      float pp[16], kr[16];
      tmem_ld16(tm + lane + T_D1 + c0, pp);
      tmem_ld16(tm + lane + T_D3 + c0, kr);
      float x2[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int t = c0 + i;
        const float x = vval(t) - pp[i];
        if (fabsf(x) <= clip) m |= 1ull << t;
        r[t] = resid_map(x, clip, tnh);
        if (tnh) drow[t] = (uint16_t)grad_q16(resid_grad(x, clip, true));
        x2[i] = r[t] - ((P.rla || (p.mods & RDN_FLAG_STATELESS_AUX)) ? 0.f : Gam[t] * kr[i]);
      }
      put16s(sm + XE, sm + XE_LO, j, c0, x2);
    }
    if (!tnh) P.mask[chunk * D + j] = m;
    ok = phase_run(K, tid, [&] {  // E2 = T_gamma X2
      if (!slot_wait<0>(K, K.phA)) return false;
      mma_s3_kk(tm + T_X, sb + XE, sb + XE_LO, sb + SLOTA, sb + SLOTA + 8192, idesc_bf16(128, 64),
                 false);
      return true;
    });
  }
  if (ok) {  // the E2^T image, for bwd_post
#pragma unroll
    for (int c0 = 0; c0 < 64; c0 += 16) {
      float e[16];
      tmem_ld16(tm + lane + T_X + c0, e);
      put16s(sm + XE, sm + XE_LO, j, c0, e);
    }
    fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      bulk_s2g(P.E2buf + chunk * 32768, sm + XE, 32768);
      bulk_commit();
      bulk_wait_all();
    }
  } else if (tid == 0) {
    if (p.err) atomicExch(p.err, RDN_ERR_TIMEOUT);
    ctl_drain(K);  // no copy or MMA of this CTA outlives it
  }
  if (tid == 0) bulk_wait_all();
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tm, 512);
}

// ======================================================================== 3
// bwd_post: everything that reduces over the value dimension, followed by the
// chunk-matrix part of the gradients, one persistent CTA of 512 threads per SM
// walking the chunks.  Thread (j, qd) owns value column j = TMEM lane j and quarter qd of
// the chunk's tokens (or of the key rows of a state).
//
// dK and dQ are accumulated transposed in TMEM (lane = key dimension d,
// column t for dK_t, 64 + t for dQ_t):
//   P2  R0 [dKR ; dQR]^T        P3  S0 [dKS ; dQS]^T
//   P4  dR (diag(wR) E2)^T + dS (diag(wS) E)^T        (dK columns only)
//   P7  K^T [dKK + dKK^T ; dQK]^T, and Q^T dQK kept apart (scaled at read-out)
// The per-token gate terms are sums over the value columns of the read-outs K S0,
// Q S0, K R0, Q R0 (P1) and K dR, K dS (P4) against the gradients in fp32.  They
// cancel: summed over the key index of P2's and P3's products instead (Q . (R0 dO^T)
// for dO . (Q R0)), which saves 64 of a chunk's 226 products and 4 % of the time,
// the gradients enter as bf16 hi + lo pairs, and dbeta was 4.7 % further from 64
// bits on the training pass, 51 to 81 % with upstream state gradients of unit size.
// The C x C gradients (P5) and the Gram matrices K K^T, Q K^T go through
// shared memory for the element-wise pass over (t, i) of Eqs. for T, M2, Mq, Ap.
// Q enters the tensor-core products unscaled; the scale is applied to the
// fp32 results.
//
// What bounds it: latencies.  A chunk takes about 50k cycles of an SM, in which
// the products take 14k and HBM is at 2.6 TB/s; shared memory (227 KB) holds one
// chunk at a time, so that its phases follow one another.  8192 chunks 1399 us,
// packed (32,768 tokens, 16 heads) 1480, RLA, 1024 chunks 207 (245 without an
// instance of its own).
namespace po {
constexpr int NTP = 512;
constexpr uint32_t SA = 0, SB = 65536;  // state images: hi 2 x 16 KB | lo 2 x 16 KB, rows j
constexpr uint32_t XH = 131072, XL = 147456, YH = 163840, YL = 180224;  // [j][t] atoms
constexpr uint32_t KQ = 196608;         // K rows 0..63, Q rows 64..127, 2 x 16 KB
constexpr uint32_t VEC = 229376;        // Gam Gprev wS wR gamma dGam dGprev (7 x 64), dGamC
constexpr uint32_t RED = VEC + 7 * 64 * 4 + 16;  // the 16 warps' <dS, S0> + <dR, R0> parts
constexpr uint32_t PARK = RED + 16 * 4;           // per-token sums kept to the gate pass (A8)
constexpr uint32_t CTL = PARK + A8::FLOATS * 4;
constexpr uint32_t SLOT = CTL + 48;
constexpr size_t SMEM = SLOT + 16;
static_assert(SMEM <= 232448, "shared memory");
// element-wise pass: fp32 C x C tiles (row stride 65) over the state images
constexpr int LDC = 65, TILE = 64 * LDC;
constexpr int F_DM2 = 0, F_DMQ = TILE, F_DAB = 2 * TILE, F_KK = 3 * TILE, F_DAG = 4 * TILE,
              F_DAP = 5 * TILE, F_QK = 6 * TILE, F_VEC = 7 * TILE;
static_assert((F_VEC + 9 * 64 + 6 * 8 * 64) * 4 <= (int)XH, "finish scratch");
// TMEM columns
constexpr uint32_t T_KS = 0, T_KR = 128, T_DKQ = 256, T_D2 = 384;
constexpr uint32_t T_KDR = 0, T_KDS = 64, T_U1 = 128, T_U2 = 192;  // P4, after the read-outs
// P5 (after the read-outs and P4): two 128-column products and the Gram one
// (past the dK, dQ accumulators)
constexpr uint32_t T_P5A = 0, T_P5B = 128, T_GR = 448;
}  // namespace po

// Sums over the 128 value columns: thread (j, qd) holds v[t - 16 qd] for the
// tokens t of its quarter.  Warp 4 qd + w covers columns [32 w, 32 w + 32);
// after the warp's transposed reduction lane 2 i holds its sum for token
// 16 qd + i.  Each warp leaves its part (16 floats) at part[16 warp, +16), so
// that several sums share the barriers ...
__device__ __forceinline__ void warp_row_part(const float (&v)[16], float *part, int tid) {
  const float o = warp_transpose_reduce16(v);
  const int warp = tid >> 5, lane = tid & 31;
  if (!(lane & 1)) part[warp * 16 + (lane >> 1)] = o;
}
// ... and, after a barrier, token t's total is the sum of its four warps' parts.
__device__ __forceinline__ float row_total(const float *part, int t) {
  const int g = t >> 4, i = t & 15;
  return part[(4 * g) * 16 + i] + part[(4 * g + 1) * 16 + i] + part[(4 * g + 2) * 16 + i] +
         part[(4 * g + 3) * 16 + i];
}

// kGeneric: the RLA mode and the variant flags (TcBwdParams::rla, FwdParams::mods)
// are read; the two methods' instances (kRla) have them folded away, which keeps
// their values in registers (beside 227 KB of shared memory the first-level
// cache is too small for spilled ones: 200 bytes a thread cost 10 % of the time)
template <bool kRla, bool kGeneric>
__global__ void __launch_bounds__(po::NTP, 1) bwd_post_kernel(TcBwdParams P) {
  using namespace po;
  extern __shared__ __align__(1024) uint8_t sm[];
  const uint32_t sb = smem_u32(sm);
  const FwdParams &p = P.f;
  if (sb & 1023u) {
    if (threadIdx.x == 0 && p.err) atomicExch(p.err, RDN_ERR_CUDA);
    return;
  }
  float *vec = reinterpret_cast<float *>(sm + VEC);
  float *Gam = vec, *Gprev = vec + 64, *wS = vec + 128, *wR = vec + 192, *gamv = vec + 256;
  float *dGamS = vec + 320, *dGprevS = vec + 384, *dGamC = vec + 448;
  float *red = reinterpret_cast<float *>(sm + RED);
  float *park = reinterpret_cast<float *>(sm + PARK);
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + SLOT);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j = tid & 127, qd = tid >> 7, tb = 16 * qd;
  const int H = p.H;
  const size_t nct = (size_t)total_records(p);
  const float scale = p.scale;
  const bool rla = kGeneric ? P.rla : kRla;
  // residual against a_t S_{t-1} k_t; o = S_{t-1} q_t + R_t q_t
  const bool dec_res = kGeneric && (p.mods & RDN_FLAG_DECAYED_RESIDUAL);
  const bool plain = kGeneric && (p.mods & RDN_FLAG_PLAIN_COMBINE);
  // the tanh residual: dP = -(1 - (r/c)^2) dX2 from the stored derivative
  const bool tnh = kGeneric && (p.mods & RDN_FLAG_TANH_RESIDUAL);
  // the stateless correction: R0 enters nothing (its read-outs, its P2 and
  // <dR, R0> terms are zero), wR is a constant one-hot (no gate gradient
  // through it) and M2 is diag(q_t . k_t) (no decay, no rate)
  const bool stl = kGeneric && (p.mods & RDN_FLAG_STATELESS_AUX);
  const __nv_bfloat16 *q = (const __nv_bfloat16 *)p.q, *k = (const __nv_bfloat16 *)p.k,
                      *dOp = (const __nv_bfloat16 *)P.dO;
  Ctl K;
  ctl_init(K, sm + CTL, tid);
  if (warp == 0) tmem_alloc(slot, 512);
  fence_before_sync();
  __syncthreads();  // barriers initialised, TMEM allocated
  fence_after_sync();
  const uint32_t tm = *slot;
  // A chunk's inputs are fetched in two parts, each during the previous chunk
  // (this CTA loops over chunks): the chunk-start states, fp32, staged where
  // their images go; then dX2, dX (fp32 [t][j], staged in the pair's place
  // until P2) and the K, Q tile.
  auto fetch_states = [&](size_t ck) {
    if (tid == 0) {
      ctl_arm<0>(K, 131072);
      bulk_g2s(sm + SA, P.Sc + ck * D * D, 65536, K.barA);
      bulk_g2s(sm + SB, P.Rc + ck * D * D, 65536, K.barA);
    }
  };
  auto fetch_rest = [&](size_t ck) {
    if (tid == 0) {
      ctl_arm<2>(K, 65536);
      bulk_g2s(sm + XH, P.dX2buf + ck * 64 * D, 32768, K.barC);
      bulk_g2s(sm + YH, P.dXbuf + ck * 64 * D, 32768, K.barC);
    }
    int s_, h_, cc_;
    rec_decode(p, (long long)ck, s_, h_, cc_);
    const SeqSpan sp_ = seq_span(p, s_, h_);
    const long long tok0_ = sp_.tok0;
    const int t0_ = cc_ * 64, n_ = min(64, sp_.len - t0_);
    for (int e = tid; e < 64 * 16; e += NTP) {  // K, Q (exact bf16), asynchronous
      const int t = e >> 4, chn = e & 15;
      const bool vld = t < n_;
      const size_t off = ((size_t)(tok0_ + t0_ + (vld ? t : 0)) * H + h_) * D + chn * 8;
      const int blk = chn >> 3, cc = (chn & 7) * 8;
      cp_async16(sm + KQ + blk * 16384 + sw128(t, cc), k + off, vld);
      cp_async16(sm + KQ + blk * 16384 + sw128(64 + t, cc), q + off, vld);
    }
  };
  if (blockIdx.x < nct) {
    fetch_states(blockIdx.x);
    fetch_rest(blockIdx.x);
  }
  // the previous chunk's dq, dk from TMEM to HBM (row = its first token row *
  // H + h; n = its valid tokens, -1 = none pending)
  long long dkq_row = 0;
  int dkq_n = -1;
  auto store_dkq = [&]() {
    __nv_bfloat16 *dk = (__nv_bfloat16 *)P.dk, *dq = (__nv_bfloat16 *)P.dq;
    const uint32_t tl = (uint32_t)((warp & 3) * 32) << 16;
    float a[16], d2[16], qv[16];
    tmem_ld16x2(tm + tl + T_DKQ + tb, a, tm + tl + T_D2 + tb, d2);
    tmem_ld16(tm + tl + T_DKQ + 64 + tb, qv);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int t = tb + i;
      if (t < dkq_n) {
        const size_t off = (size_t)(dkq_row + (long long)t * H) * D + j;
        if (P.f32qk) {
          ((float *)P.dk)[off] = a[i] + scale * d2[i];
          ((float *)P.dq)[off] = scale * qv[i];
        } else {
          dk[off] = __float2bfloat16_rn(a[i] + scale * d2[i]);
          dq[off] = __float2bfloat16_rn(scale * qv[i]);
        }
      }
    }
    dkq_n = -1;
  };
  bool ok = true;
  uint32_t it = 0;  // chunks done by this CTA: the parity of barrier B
  for (size_t chunk = blockIdx.x; chunk < nct && ok; chunk += gridDim.x, ++it) {
  const size_t next = chunk + gridDim.x;
  int sq, h, c;
  rec_decode(p, (long long)chunk, sq, h, c);
  const SeqSpan sp = seq_span(p, sq, h);
  const long long tok0 = sp.tok0;
  const int t0 = c * 64, n = min(64, sp.len - t0);
  const float *recf = p.ws + chunk * kRecFloats;
  const float *S0 = P.Sc + chunk * D * D, *R0 = P.Rc + chunk * D * D;
  const uint8_t *gimg = P.gimg + chunk * 131072;  // dS hi | dR hi | dS lo | dR lo
  // this thread's tokens of dX2, dX (from the staging) and dO: read after P1 is
  // issued, so that the MMA issue does not wait behind them
  float x2v[16], xv[16], dov[16];
  // this thread's key rows of a state: [32 qd, 32 qd + 32), the columns
  // [32 (qd & 1), +32) of 64-row block qd >> 1 of the image
  const uint32_t kblk = (uint32_t)(qd >> 1) * 16384u;
  const int kc0 = 32 * (qd & 1);
  // fp32 [i][j] state staged at `base` -> rows j of its (hi | lo) image at
  // `base` (every thread reads its values before any writes)
  auto stage_to_image = [&](uint32_t base) {
    const float *st = reinterpret_cast<const float *>(sm + base);
    float v[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = st[(32 * qd + i) * D + j];
    __syncthreads();
#pragma unroll
    for (int c0 = 0; c0 < 32; c0 += 16) {
      float w[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) w[i] = v[c0 + i];
      put16s(sm + base + kblk, sm + base + 32768 + kblk, j, kc0 + c0, w);
    }
  };
  // sum over this thread's entries of (image at base, hi + lo) * x[i][j]
  auto dot_image = [&](uint32_t base, const float (&x)[32]) {
    float s = 0.f;
#pragma unroll
    for (int k8 = 0; k8 < 4; ++k8) {
      const int c8 = (kc0 >> 3) + k8;
      const uint32_t o = base + kblk + j * 128 + (((c8 ^ (j & 7)) & 7) << 4);
      const uint4 hv = *reinterpret_cast<const uint4 *>(sm + o);
      const uint4 lv = *reinterpret_cast<const uint4 *>(sm + o + 32768);
      const __nv_bfloat16 *hb = reinterpret_cast<const __nv_bfloat16 *>(&hv);
      const __nv_bfloat16 *lb = reinterpret_cast<const __nv_bfloat16 *>(&lv);
#pragma unroll
      for (int e = 0; e < 8; ++e)
        s += (__bfloat162float(hb[e]) + __bfloat162float(lb[e])) * x[k8 * 8 + e];
    }
    return s;
  };
  // this thread's 16 tokens of a [j][t] atom pair (hi, lo)
  auto put_tok = [&](const float (&x)[16], uint32_t hi, uint32_t lo) {
    put16s(sm + hi, sm + lo, j, tb, x);
  };
  const uint32_t tm_lane = (uint32_t)((warp & 3) * 32) << 16;
  const uint32_t i128 = idesc_bf16(128, 128), i64 = idesc_bf16(128, 64);

  cp_async_wait_all();  // K, Q tile (published by the barriers below)
  if (!ctl_wait<0>(K, 0, tid)) *K.flag = 1;  // phase_run below reports it to every thread
#pragma unroll 1
  for (int s2 = 0; s2 < 2; ++s2) stage_to_image(s2 ? SB : SA);  // images of S0, R0
  // ---- P1: read-outs [K S0 | Q S0] and [K R0 | Q R0] (lanes j, columns t')
  phase_issue(K, tid, [&] {
    const uint32_t t_ = *slot;
    mma_tile<true>(t_ + T_KS, sb + SA, 16384, sb + KQ, 16384, 8, i128, false);
    mma_tile<true>(t_ + T_KS, sb + SA + 32768, 16384, sb + KQ, 16384, 8, i128, true);
    mma_tile<true>(t_ + T_KR, sb + SB, 16384, sb + KQ, 16384, 8, i128, false);
    mma_tile<true>(t_ + T_KR, sb + SB + 32768, 16384, sb + KQ, 16384, 8, i128, true);
    return true;
  });
  // while P1 runs: this thread's dO and the gate vectors (loads first, their
  // latency under the stores), the previous chunk's dq, dk, then dX2 and dX
  // from their staging
  const unsigned long long m = tnh ? 0ull : P.mask[chunk * D + j] >> tb;
  const uint16_t *drow = reinterpret_cast<const uint16_t *>(P.mask) + (chunk * D + j) * 64 + tb;
  __nv_bfloat16 dob[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int t = tb + i;
    dob[i] = t < n ? dOp[((size_t)(tok0 + t0 + t) * H + h) * D + j] : __float2bfloat16(0.f);
  }
  float gvv[5];
  if (tid < 64) {
    gvv[0] = recf[OFF_VEC + V_GAM + tid];
    gvv[1] = recf[OFF_VEC + V_GPREV + tid];
    gvv[2] = recf[OFF_VEC + V_WS + tid];
    gvv[3] = recf[OFF_VEC + V_WR + tid];
    gvv[4] = tid < n ? p.gamma[(size_t)(tok0 + t0 + tid) * H + h] : 0.f;
  }
  __syncwarp();  // (TMEM accesses take whole warps)
  if (dkq_n >= 0) store_dkq();
#pragma unroll
  for (int i = 0; i < 16; ++i) dov[i] = __bfloat162float(dob[i]);
  if (tid < 64) {
    Gam[tid] = gvv[0];
    Gprev[tid] = gvv[1];
    wS[tid] = gvv[2];
    wR[tid] = gvv[3];
    gamv[tid] = gvv[4];
  }
  if (!ctl_wait<2>(K, 0, tid)) *K.flag = 1;
  {
    const float *x2s = reinterpret_cast<const float *>(sm + XH);
    const float *xs = reinterpret_cast<const float *>(sm + YH);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      x2v[i] = x2s[(tb + i) * D + j];
      xv[i] = xs[(tb + i) * D + j];
    }
  }
  ok = phase_wait(K);  // (its barrier also publishes the gate vectors)
  auto dp_of = [&](int i) {
    if (tnh) return -grad_uq16(drow[i]) * x2v[i];
    return ((m >> i) & 1ull) ? -x2v[i] : 0.f;
  };
  if (ok) {  // per-token gate terms: dGam, dGprev, and <dR,R0> + <dS,S0>
    // the three sums' warp parts go where dX2 was staged (read into x2v above)
    float *part = reinterpret_cast<float *>(sm + XH);
    float rv[16];
    {
      float qs[16], qr[16];
      tmem_ld16x2(tm + tm_lane + T_KS + 64 + tb, qs, tm + tm_lane + T_KR + 64 + tb, qr);
      if (stl) {
#pragma unroll
        for (int i = 0; i < 16; ++i) qr[i] = 0.f;
      }
      // d gamma_t from the read-out: dO_t . (Gam_t Q R0)_t (the rest of Oa_t in P6)
      lds16(Gam + tb, rv);
#pragma unroll
      for (int i = 0; i < 16; ++i) rv[i] = plain ? 0.f : scale * rv[i] * dov[i] * qr[i];
      warp_row_part(rv, part, tid);
      lds16(gamv + tb, rv);
#pragma unroll
      for (int i = 0; i < 16; ++i)  // (plain combine: Gprev Q S0 and no gamma_t)
        rv[i] = plain ? scale * dov[i] * qr[i] : scale * dov[i] * (qs[i] + rv[i] * qr[i]);
    }
    {
      float ks[16], kr[16];
      tmem_ld16x2(tm + tm_lane + T_KS + tb, ks, tm + tm_lane + T_KR + tb, kr);
      if (stl) {
#pragma unroll
        for (int i = 0; i < 16; ++i) kr[i] = 0.f;
      }
      if (!rla) {
#pragma unroll
        for (int i = 0; i < 16; ++i) rv[i] -= x2v[i] * kr[i] + xv[i] * ks[i];
      }
      // the prediction's state term: Gprev K S0 (decayed residual: Gam K S0)
      if (dec_res) {
#pragma unroll
        for (int i = 0; i < 16; ++i) rv[i] += dp_of(i) * ks[i];
      }
      warp_row_part(rv, part + 256, tid);
#pragma unroll
      for (int i = 0; i < 16; ++i) rv[i] = dec_res ? 0.f : dp_of(i) * ks[i];
      if (plain) {  // the base read-out's gate is Gprev
        float qs[16];
        tmem_ld16(tm + tm_lane + T_KS + 64 + tb, qs);
#pragma unroll
        for (int i = 0; i < 16; ++i) rv[i] += scale * dov[i] * qs[i];
      }
    }
    warp_row_part(rv, part + 512, tid);
    __syncthreads();
    if (tid < 192) {
      const int w = tid >> 6, t = tid & 63;
      const float tot = row_total(part + 256 * w, t);
      if (w == 0)
        park[A8::V_DGAM_OUT + t] = tot;
      else
        (w == 1 ? dGamS : dGprevS)[t] = tot;
    }
    __syncthreads();  // (P2's operands go where the parts are)
    // ---- P2: dK, dQ += R0 [dKR ; dQR]^T, dKR = -Gam dX2, dQR = Gam gamma dO
    float x[16], y[16];
    lds16(Gam + tb, x);
    lds16(gamv + tb, y);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      y[i] = stl ? 0.f : (plain ? 1.f : y[i]) * x[i] * dov[i];
      x[i] = (rla || stl) ? 0.f : -x[i] * x2v[i];
    }
    put_tok(x, XH, XL);
    put_tok(y, YH, YL);
    ok = phase_run(K, tid, [&] {
      mma_tile_mnmn<true>(tm + T_DKQ, sb + SB, 16384, sb + XH, 32768, 8, i128, false);
      mma_tile_mnmn<true>(tm + T_DKQ, sb + SB, 16384, sb + XL, 32768, 8, i128, true);
      mma_tile_mnmn<true>(tm + T_DKQ, sb + SB + 32768, 16384, sb + XH, 32768, 8, i128, true);
      return true;
    });
  }
  if (ok && tid == 0) {  // R0's image is done with: dR's image into its place
    ctl_arm<1>(K, 65536);
    bulk_g2s(sm + SB, gimg + 32768, 32768, K.barB);
    bulk_g2s(sm + SB + 32768, gimg + 98304, 32768, K.barB);
  }
  __syncwarp();  // (TMEM accesses take whole warps)
  // <dR, R0> + <dS, S0> into dGamC, each computed while MMAs run: the states
  // are re-read from L2 (not through L1, which holds the prefetched dO rows),
  // the gradients' images are in the states' places
  float gdot = 0.f;
  auto dot_state = [&](const float *st, uint32_t img) {
    float x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = __ldcg(st + (size_t)(32 * qd + i) * D + j);
    return dot_image(img, x);
  };
  if (ok) {  // ---- P3: dK, dQ += S0 [dKS ; dQS]^T, dKS = Gprev dP - Gam dX, dQS = Gam dO;
             // meanwhile <dR, R0>
    float x[16], y[16];
    lds16(dec_res ? Gam + tb : Gprev + tb, x);
    lds16(Gam + tb, y);
    float gq[16];  // the base read-out's gate: Gam (plain combine: Gprev)
    lds16(plain ? Gprev + tb : Gam + tb, gq);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      x[i] = x[i] * dp_of(i) - (rla ? 0.f : y[i] * xv[i]);
      y[i] = gq[i] * dov[i];
    }
    put_tok(x, XH, XL);
    put_tok(y, YH, YL);
    ok = phase_run_with(K, tid, [&] {
      mma_tile_mnmn<true>(tm + T_DKQ, sb + SA, 16384, sb + XH, 32768, 8, i128, true);
      mma_tile_mnmn<true>(tm + T_DKQ, sb + SA, 16384, sb + XL, 32768, 8, i128, true);
      mma_tile_mnmn<true>(tm + T_DKQ, sb + SA + 32768, 16384, sb + XH, 32768, 8, i128, true);
      return true;
    }, [&] {
      if (!ctl_wait<1>(K, it & 1u, tid)) *K.flag = 1;  // dR's image
      gdot = stl ? 0.f : dot_state(R0, SB);
    });
  }
  if (ok && tid == 0) {  // and dS's image into S0's; the E2^T, E^T images into the pair's
    ctl_arm<0>(K, 65536);
    bulk_g2s(sm + SA, gimg, 32768, K.barA);
    bulk_g2s(sm + SA + 32768, gimg + 65536, 32768, K.barA);
    ctl_arm<2>(K, 65536);
    bulk_g2s(sm + XH, P.E2buf + chunk * 32768, 32768, K.barC);  // hi at XH, lo at XL
    bulk_g2s(sm + YH, P.Ebuf + chunk * 32768, 32768, K.barC);   // hi at YH, lo at YL
  }
  __syncwarp();  // (TMEM accesses take whole warps)
  // this thread's 16 tokens of row j of a (hi | lo) image of a [j][t] matrix
  auto image_row = [&](uint32_t base, float (&out)[16]) {
#pragma unroll
    for (int k8 = 0; k8 < 2; ++k8) {
      const int c8 = (tb >> 3) + k8;
      const uint32_t o = base + j * 128 + (((c8 ^ (j & 7)) & 7) << 4);
      const uint4 hv = *reinterpret_cast<const uint4 *>(sm + o);
      const uint4 lv = *reinterpret_cast<const uint4 *>(sm + o + 16384);
      const __nv_bfloat16 *hb = reinterpret_cast<const __nv_bfloat16 *>(&hv);
      const __nv_bfloat16 *lb = reinterpret_cast<const __nv_bfloat16 *>(&lv);
#pragma unroll
      for (int e = 0; e < 8; ++e) out[k8 * 8 + e] = __bfloat162float(hb[e]) + __bfloat162float(lb[e]);
    }
  };
  if (ok) {  // ---- P4: dR E2^T, dS E^T (scaled by wR, wS per token below); K dR, K dS read-outs;
             // meanwhile <dS, S0> and the dGamC reduction
    if (!ctl_wait<2>(K, 1, tid)) *K.flag = 1;  // the E images, for every thread
    if (!ctl_wait<0>(K, 1, tid)) *K.flag = 1;  // dS's image
    phase_issue(K, tid, [&] {
      mma_tile_mnmn<true>(tm + T_U1, sb + SB, 16384, sb + XH, 16384, 8, i64, false);
      mma_tile_mnmn<true>(tm + T_U1, sb + SB, 16384, sb + XL, 16384, 8, i64, true);
      mma_tile_mnmn<true>(tm + T_U1, sb + SB + 32768, 16384, sb + XH, 16384, 8, i64, true);
      mma_tile_mnmn<true>(tm + T_U2, sb + SA, 16384, sb + YH, 16384, 8, i64, false);
      mma_tile_mnmn<true>(tm + T_U2, sb + SA, 16384, sb + YL, 16384, 8, i64, true);
      mma_tile_mnmn<true>(tm + T_U2, sb + SA + 32768, 16384, sb + YH, 16384, 8, i64, true);
      // (K dR)^T, (K dS)^T (lanes j, columns t; K exact)
      mma_tile<true>(tm + T_KDR, sb + SB, 16384, sb + KQ, 16384, 8, i64, false);
      mma_tile<true>(tm + T_KDR, sb + SB + 32768, 16384, sb + KQ, 16384, 8, i64, true);
      mma_tile<true>(tm + T_KDS, sb + SA, 16384, sb + KQ, 16384, 8, i64, false);
      mma_tile<true>(tm + T_KDS, sb + SA + 32768, 16384, sb + KQ, 16384, 8, i64, true);
      return true;
    });
    gdot += dot_state(S0, SA);
#pragma unroll
    for (int off = 16; off; off >>= 1) gdot += __shfl_xor_sync(0xffffffffu, gdot, off);
    if (lane == 0) red[warp] = gdot;
    ok = phase_wait(K);  // (its barrier publishes the parts)
    if (ok && tid == 0) {
      float s = 0.f;
      for (int w = 0; w < NTP / 32; ++w) s += red[w];
      *dGamC = s;
    }
    __syncwarp();
  }
  if (ok) {
    // dK += diag(wR) E2 dR^T + diag(wS) E dS^T  (lanes i, columns t of this half)
    {
      float a[16], u1[16], u2[16], wr[16], ws[16];
      tmem_ld16x2(tm + tm_lane + T_DKQ + tb, a, tm + tm_lane + T_U1 + tb, u1);
      tmem_ld16(tm + tm_lane + T_U2 + tb, u2);
      lds16(wR + tb, wr);
      lds16(wS + tb, ws);
#pragma unroll
      for (int i = 0; i < 16; ++i) a[i] = fmaf(wr[i], u1[i], fmaf(ws[i], u2[i], a[i]));
      tmem_st16(tm + tm_lane + T_DKQ + tb, a);
    }
    // dwR_t = sum_j (K dR)[t,j] E2[t,j], dwS_t = sum_j (K dS)[t,j] E[t,j]; the
    // warp parts where dS's image was
    float *part = reinterpret_cast<float *>(sm + SA);
#pragma unroll 1
    for (int w = 0; w < 2; ++w) {
      float ev[16], rv[16];
      image_row(w == 0 ? XH : YH, ev);
      tmem_ld16(tm + tm_lane + (w == 0 ? T_KDR : T_KDS) + tb, rv);
#pragma unroll
      for (int i = 0; i < 16; ++i) rv[i] = (w == 0 && stl) ? 0.f : rv[i] * ev[i];
      warp_row_part(rv, part + 256 * w, tid);
    }
    __syncthreads();
    if (tid < 128) {  // read in the gate pass
      const int w = tid >> 6, t = tid & 63;
      park[(w == 0 ? A8::V_DWR : A8::V_DWS) + t] = row_total(part + 256 * w, t);
    }
    __syncthreads();  // (P5's operands go where the parts are)
  }
  // ---- P5: C x C gradients (lanes t' of a stacked pair, columns s of [E2 ; E])
  //   [dO ; dX2] [E2 ; E]^T -> dO E2^T | dO E^T ; dX2 E2^T | (unused)
  //   [dX ; dP] [E2 ; E]^T  -> (unused) | dX E^T ; (unused) | dP E^T
  //   and the Gram matrices [K ; Q] K^T, all in one phase: 128-column
  //   products take about the issue time of 64-column ones
  // images: E2 at XH (hi | lo), E at YH (hi | lo), 32 KB apart; the pair
  // [dO ; dX2] at SA (dO atom hi SA, lo SA + 16 KB; dX2 atom hi SA + 32 KB, lo
  // SA + 48 KB) and [dX ; dP] at SB the same way (dR's image is done with)
  // token tid's g and beta for the element-wise pass, loaded while P5 runs
  float g_t = 0.f, beta_t = 0.f;
  if (ok) {
    if (tid < n) {
      const size_t off = (size_t)(tok0 + t0 + tid) * H + h;
      g_t = p.g[off];
      beta_t = p.beta[off];
    }
    float y[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) y[i] = dp_of(i);
    put_tok(xv, SB, SB + 16384);
    put_tok(y, SB + 32768, SB + 49152);
    put_tok(dov, SA, SA + 16384);  // gamma_t enters in the element-wise pass
    put_tok(x2v, SA + 32768, SA + 49152);
    static_assert(YH - XH == 32768 && YL - XL == 32768, "the [E2 ; E] atoms");
    ok = phase_run(K, tid, [&] {
      mma_tile_mnmn<true>(tm + T_P5A, sb + SA, 32768, sb + XH, 32768, 8, i128, false);
      mma_tile_mnmn<true>(tm + T_P5A, sb + SA, 32768, sb + XL, 32768, 8, i128, true);
      mma_tile_mnmn<true>(tm + T_P5A, sb + SA + 16384, 32768, sb + XH, 32768, 8, i128, true);
      mma_tile_mnmn<true>(tm + T_P5B, sb + SB, 32768, sb + XH, 32768, 8, i128, false);
      mma_tile_mnmn<true>(tm + T_P5B, sb + SB, 32768, sb + XL, 32768, 8, i128, true);
      mma_tile_mnmn<true>(tm + T_P5B, sb + SB + 16384, 32768, sb + XH, 32768, 8, i128, true);
      mma_tile<true>(tm + T_GR, sb + KQ, 16384, sb + KQ, 16384, 8, i64, false);
      return true;
    });
  }
  // the next chunk's states into L2 while the element-wise pass and P7 run
  // (their copies into shared memory start once the element-wise pass is done
  // with the region, while P7 runs)
  if (ok && tid == 0 && next < nct) {
    prefetch_l2_bulk(P.Sc + next * D * D, 65536);
    prefetch_l2_bulk(P.Rc + next * D * D, 65536);
  }
  __syncwarp();  // (TMEM accesses take whole warps)
  // ---- element-wise pass over (t, i): the gradients of the chunk matrices'
  // entries turned into gradients of K K^T, Q K^T and of the gates
  float *F = reinterpret_cast<float *>(sm);
  float *cum = F + F_VEC, *cprev = cum + 64, *bet = cum + 128, *gam = cum + 192, *gg = cum + 256,
        *dcum = cum + 320, *dcprev = cum + 384, *dbet = cum + 448, *dgam = cum + 512;
  float *prt = cum + 576;  // [6][8][64] partial sums
  float o_dg = 0.f, o_dbeta = 0.f, o_dgamma = 0.f;  // this thread's token's gate gradients
  if (ok) {
    {
      const int r = j & 63;
      {
        float g1[16], g2[16], g3[16], gr[16];
        // g1: dO E2^T (rows t < 64) | dX2 E2^T; g2: dO E^T | dP E^T; g3: dX E^T
        tmem_ld16x2(tm + tm_lane + T_P5A + tb, g1,
                    tm + tm_lane + (j < 64 ? T_P5A : T_P5B) + 64 + tb, g2);
        tmem_ld16x2(tm + tm_lane + T_P5B + 64 + tb, g3, tm + tm_lane + T_GR + tb, gr);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int e = r * LDC + tb + i;
          if (j < 64) {
            F[F_DM2 + e] = g1[i];
            F[F_DMQ + e] = g2[i];
            F[F_DAB + e] = rla ? 0.f : -g3[i];
            F[F_KK + e] = gr[i];
          } else {
            F[F_DAG + e] = (rla || stl) ? 0.f : -g1[i];  // (no T_gamma to differentiate)
            F[F_DAP + e] = g2[i];
            F[F_QK + e] = scale * gr[i];
          }
        }
      }
    }
    if (tid < 64) {
      gg[tid] = g_t;
      bet[tid] = beta_t;
      gam[tid] = gamv[tid];
    }
    __syncthreads();
    if (warp == 0) {  // in-chunk cumulative log-decay
      float a = gg[lane], a2 = gg[32 + lane];
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const float ua = __shfl_up_sync(0xffffffffu, a, off);
        const float ub = __shfl_up_sync(0xffffffffu, a2, off);
        if (lane >= off) {
          a += ua;
          a2 += ub;
        }
      }
      a2 += __shfl_sync(0xffffffffu, a, 31);
      cum[lane] = a;
      cum[32 + lane] = a2;
      cprev[lane] = a - gg[lane];
      cprev[32 + lane] = a2 - gg[32 + lane];
    }
    __syncthreads();
    {  // row pass: thread (t, eighth) over i in [8 q8, 8 q8 + 8)
      const int t = tid & 63, q8 = tid >> 6;
      const float ct = cum[t], cpt = cprev[t];
      const float gt = gam[t];
      float rowc = 0.f, rowp = 0.f, dgo = 0.f;
#pragma unroll
      for (int ii = 0; ii < 8; ++ii) {
        const int i = 8 * q8 + ii, e = t * LDC + i;
        float dkk = 0.f, dqk = 0.f, cg = 0.f, cb = 0.f, cm = 0.f;
        if (i <= t) {
          const float dec = __expf(ct - cum[i]);
          const float kk = F[F_KK + e], qk = F[F_QK + e], bi = bet[i], gi = gam[i];
          if (stl) {  // M2 = diag(Q K^T): the diagonal only, no decay, no rate
            if (i == t) {
              const float g1 = F[F_DM2 + e];
              if (!plain) dgo += qk * g1;
              dqk += plain ? g1 : gt * g1;
            }
          } else {  // M2: inclusive, gamma, Q K^T; G1 holds dO E2^T, dM2 = gamma_t dO E2^T
            const float g1 = F[F_DM2 + e];
            if (!plain) dgo += dec * gi * qk * g1;  // d gamma_t += (M2 E2)_t . dO_t
            const float dm = plain ? g1 : gt * g1;
            const float G = dm * dec * gi * qk;
            rowc += G;
            cg += G;
            cm += dm * dec * qk;
            dqk += dm * dec * gi;
          }
          if (i < t) {
            const float decp = __expf(cpt - cum[i]);
            {  // Ap: strict, beta, K K^T, previous-token decay (decayed residual: to t)
              const float dA = dec_res ? dec : decp;
              const float dm = F[F_DAP + e];
              const float G = dm * dA * bi * kk;
              if (dec_res) rowc += G; else rowp += G;
              cg += G;
              cb += dm * dA * kk;
              dkk += dm * dA * bi;
            }
            {  // Mq: strict, beta, Q K^T (plain combine: decay to t-1)
              const float dA = plain ? decp : dec;
              const float dm = F[F_DMQ + e];
              const float G = dm * dA * bi * qk;
              if (plain) rowp += G; else rowc += G;
              cg += G;
              cb += dm * dA * qk;
              dqk += dm * dA * bi;
            }
            {  // A_beta, A_gamma: strict, K K^T
              const float da = F[F_DAB + e], dg2 = F[F_DAG + e];
              const float Gb = da * dec * bi * kk, Gg = dg2 * dec * gi * kk;
              rowc += Gb + Gg;
              cg += Gb + Gg;
              cb += da * dec * kk;
              cm += dg2 * dec * kk;
              dkk += da * dec * bi + dg2 * dec * gi;
            }
          }
        }
        F[F_KK + e] = dkk;
        F[F_QK + e] = dqk;
        F[F_DM2 + e] = cg;
        F[F_DMQ + e] = cb;
        F[F_DAB + e] = cm;
      }
      prt[0 * 512 + q8 * 64 + t] = rowc;
      prt[1 * 512 + q8 * 64 + t] = rowp;
      prt[5 * 512 + q8 * 64 + t] = dgo;
    }
    __syncthreads();
    {  // column pass: thread (i, eighth) over t in [8 q8, 8 q8 + 8)
      const int i = tid & 63, q8 = tid >> 6;
      float sg = 0.f, sbv = 0.f, smv = 0.f;
#pragma unroll
      for (int tt = 0; tt < 8; ++tt) {
        const int e = (8 * q8 + tt) * LDC + i;
        sg += F[F_DM2 + e];
        sbv += F[F_DMQ + e];
        smv += F[F_DAB + e];
      }
      prt[2 * 512 + q8 * 64 + i] = sg;
      prt[3 * 512 + q8 * 64 + i] = sbv;
      prt[4 * 512 + q8 * 64 + i] = smv;
    }
    __syncthreads();
    if (tid < 64) {
      const int i = tid;
      float s5[6];
#pragma unroll
      for (int w = 0; w < 6; ++w) {
        float a = 0.f;
#pragma unroll
        for (int q8 = 0; q8 < 8; ++q8) a += prt[w * 512 + q8 * 64 + i];
        s5[w] = a;
      }
      const float cC = cum[63];
      const float eC = __expf(cC - cum[i]);
      const float dwS = park[A8::V_DWS + i], dwR = park[A8::V_DWR + i];
      dbet[i] = s5[3] + dwS * eC;
      dgam[i] = s5[4] + s5[5] + park[A8::V_DGAM_OUT + i] + dwR * eC;
      dcum[i] = s5[0] - s5[2] - (dwS * bet[i] + dwR * gam[i]) * eC + dGamS[i] * __expf(cum[i]);
      dcprev[i] = s5[1] + dGprevS[i] * __expf(cprev[i]);
    }
    __syncthreads();
    if (warp == 0) {  // chunk-end terms land on cum_C = cum[63] (padding has g = 0)
      const float cC = cum[63];
      float s = 0.f;
      for (int t = lane; t < 64; t += 32)
        s += (park[A8::V_DWS + t] * bet[t] + park[A8::V_DWR + t] * gam[t]) *
             __expf(cC - cum[t]);
#pragma unroll
      for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      if (lane == 0) dcum[63] += s + *dGamC * __expf(cC);
      __syncwarp();
      // dg_s = sum_{t >= s} dcum_t + sum_{t > s} dcprev_t (reverse scans)
      float a = dcum[63 - lane], a2 = dcum[31 - lane];
      float pa = dcprev[63 - lane], pb = dcprev[31 - lane];
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const float ua = __shfl_up_sync(0xffffffffu, a, off), ub = __shfl_up_sync(0xffffffffu, a2, off);
        const float upa = __shfl_up_sync(0xffffffffu, pa, off), upb = __shfl_up_sync(0xffffffffu, pb, off);
        if (lane >= off) {
          a += ua;
          a2 += ub;
          pa += upa;
          pb += upb;
        }
      }
      a2 += __shfl_sync(0xffffffffu, a, 31);
      pb += __shfl_sync(0xffffffffu, pa, 31);
      gg[63 - lane] = a + (pa - dcprev[63 - lane]);
      gg[31 - lane] = a2 + (pb - dcprev[31 - lane]);
    }
    {  // B operand [dKK + dKK^T ; dQK] (rows t, columns i), hi | lo
      const int t = tid & 63, q8 = tid >> 6;
      float v[8], w[8];
#pragma unroll
      for (int ii = 0; ii < 8; ++ii) {
        const int i = 8 * q8 + ii;
        v[ii] = i == t ? 2.f * F[F_KK + t * LDC + t] : F[F_KK + t * LDC + i] + F[F_KK + i * LDC + t];
        w[ii] = F[F_QK + t * LDC + i];
      }
      put8s(sm + XH, sm + XL, t, 8 * q8, v);
      put8s(sm + XH, sm + XL, 64 + t, 8 * q8, w);
    }
    // ---- P7: dK, dQ += K^T [dKK + dKK^T ; dQK]^T ; D2 = Q^T dQK
    phase_issue(K, tid, [&] {
      mma_tile_mnk<true>(tm + T_DKQ, sb + KQ, 16384, sb + XH, 4, i128, true);
      mma_tile_mnk<true>(tm + T_DKQ, sb + KQ, 16384, sb + XL, 4, i128, true);
      mma_tile_mnmn<true>(tm + T_D2, sb + KQ + 8192, 16384, sb + XH + 8192, 16384, 4, i64, false);
      mma_tile_mnmn<true>(tm + T_D2, sb + KQ + 8192, 16384, sb + XL + 8192, 16384, 4, i64, true);
      return true;
    });
    if (tid < n) {  // the vectors live where the next chunk's states are staged
      o_dg = gg[tid];
      o_dbeta = dbet[tid];
      o_dgamma = dgam[tid];
    }
    __syncthreads();
    if (next < nct) fetch_states(next);  // the state images and the fp32 tiles are done with
    if (next < nct) {  // the next chunk's dO rows, mask words and gate vectors into L1
      int s_, h_, cc_;
      rec_decode(p, (long long)next, s_, h_, cc_);
      const SeqSpan sp_ = seq_span(p, s_, h_);
      const long long tok0_ = sp_.tok0;
      const int t0_ = cc_ * 64, n_ = min(64, sp_.len - t0_);
      if (tid < 128) {  // 64 rows of 256 bytes
        const int t = tid >> 1;
        if (t < n_) prefetch_l1_line(dOp + ((size_t)(tok0_ + t0_ + t) * H + h_) * D + (tid & 1) * 64);
      } else if (tid < 136) {  // 128 mask words
        if (!tnh) prefetch_l1_line(P.mask + next * D + (tid - 128) * 16);
      } else if (tid < 148) {  // the record's 6 x 64 gate floats
        prefetch_l1_line(p.ws + next * kRecFloats + OFF_VEC + (tid - 136) * 32);
      } else if (tid < 180) {  // gamma, one line per two tokens
        const int t = 2 * (tid - 148);
        if (t < n_) prefetch_l1_line(p.gamma + (size_t)(tok0_ + t0_ + t) * H + h_);
      }
    }
    ok = phase_wait(K);
    if (ok && next < nct) fetch_rest(next);  // K, Q and the pair region are done with
  }
  if (ok) {
    if (tid < n) {
      const size_t off = (size_t)(tok0 + t0 + tid) * H + h;
      P.dg[off] = o_dg;
      P.dbeta[off] = o_dbeta;
      P.dgamma[off] = o_dgamma;
    }
    // dq, dk of this chunk: read out and stored during the next chunk's P1
    // (T_DKQ, T_D2 keep them until its P2), or after the last chunk
    dkq_row = (tok0 + t0) * H + h;
    dkq_n = n;
  }
  }  // chunks
  __syncwarp();  // (TMEM accesses take whole warps)
  if (ok && dkq_n >= 0) store_dkq();
  if (!ok && tid == 0) {
    if (p.err) atomicExch(p.err, RDN_ERR_TIMEOUT);
    ctl_drain(K);  // no bulk copy or MMA of this CTA outlives it
  }
  cp_async_wait_all();  // (nor a cp.async of a chunk not reached)
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tm, 512);
}

}  // namespace


size_t bwd_tc_extra_bytes(long long nrec, bool deriv) {
  const size_t nct = (size_t)nrec;
  return nct * (4 * 64 * D * sizeof(float) + 2 * (size_t)D * D * sizeof(float) +
                mask_bytes_per_chunk(D, deriv, true));
}

cudaError_t launch_bwd_tc(const FwdParams &f, const void *dO, const float *dST, const float *dRT,
                          const float *Sc, const float *Rc, void *dq, void *dk, void *dv, float *dg,
                          float *dbeta, float *dgamma, float *dS0, float *dR0, char *extra,
                          bool rla, bool grad_f32, bool dqk_f32, cudaStream_t s) {
  TcBwdParams P;
  P.rla = rla;
  P.f32g = grad_f32;
  P.f32qk = grad_f32 || dqk_f32;
  P.dq = dq;
  P.dk = dk;
  P.dg = dg;
  P.dbeta = dbeta;
  P.dgamma = dgamma;
  P.f = f;
  P.dO = dO;
  P.dST = dST;
  P.dRT = dRT;
  P.Sc = Sc;
  P.Rc = Rc;
  P.dv = dv;
  P.dS0 = dS0;
  P.dR0 = dR0;
  const size_t nct = (size_t)f.nrec;  // record slots (packed sequences: a bound)
  float *x = reinterpret_cast<float *>(extra);
  P.Ebuf = reinterpret_cast<uint8_t *>(x);
  P.E2buf = reinterpret_cast<uint8_t *>(x + nct * 64 * D);
  P.dX2buf = x + 2 * nct * 64 * D;
  P.dXbuf = x + 3 * nct * 64 * D;
  P.gimg = reinterpret_cast<uint8_t *>(x + 4 * nct * 64 * D);
  P.mask = reinterpret_cast<unsigned long long *>(P.gimg + nct * 131072);
  // the chain's tiles of whole chunks by tensor-map copies (else cp.async)
  const long long rows = (long long)f.B * f.T;
  P.tma = make_tile_map(P.map_k, f.k, D, f.H, rows) && make_tile_map(P.map_q, f.q, D, f.H, rows) &&
          make_tile_map(P.map_do, dO, D, f.H, rows);
  P.dv_ok = !grad_f32 && make_tile_map(P.map_dv, dv, D, f.H, rows);
  const bool saved = f.sv_E && f.sv_E2 && f.sv_mask;  // E, E2, mask kept by the forward
  if (saved) {
    P.Ebuf = f.sv_E;
    P.E2buf = f.sv_E2;
    P.mask = f.sv_mask;
  }
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(bwd_recompute_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)rc::SMEM)) != cudaSuccess)
    return e;
  auto post = f.mods != 0 ? bwd_post_kernel<false, true>
                          : (rla ? bwd_post_kernel<true, false> : bwd_post_kernel<false, false>);
  if ((e = cudaFuncSetAttribute(post, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)po::SMEM)) != cudaSuccess)
    return e;
  if (!saved) {
    RDN_LAUNCH("bwd_recompute", s, bwd_recompute_kernel<<<(unsigned)nct, NT, rc::SMEM, s>>>(P));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if ((e = launch_bwd_chain(P, s)) != cudaSuccess) return e;
  int nsm = 0;
  if ((e = sm_count(&nsm)) != cudaSuccess) return e;
  const unsigned post_grid = (unsigned)(nct < (size_t)nsm ? nct : (size_t)nsm);  // one CTA per SM
  RDN_LAUNCH("bwd_post", s, post<<<post_grid, po::NTP, po::SMEM, s>>>(P));
  return cudaGetLastError();
}

}  // namespace rdn
