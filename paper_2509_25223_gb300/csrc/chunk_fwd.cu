// chunk_fwd.cu -- chunkwise-parallel forward of RLA / RDN (Section 3.4),
// fp32 SIMT path.
//
// Chunk algebra (C = 64 tokens; b_t = in-chunk cumulative log-decay,
// Gam_t = exp(b_t), Gprev_t = exp(b_{t-1}), b_0 = 0; states stored [d_k][d_v]):
//
//   RDN writes the delta rule as S_t = a_t S_{t-1} + beta_t k_t e_t^T with the
//   delta error e_t = v_t - a_t S_{t-1}^T k_t (Section 2.2).  Unrolling the
//   chunk gives (I + A) E = V - diag(Gam) K S0 with the strictly lower
//   A[t,i] = exp(b_t - b_i) beta_i (k_t.k_i), so E = T (V - diag(Gam) K S0),
//   T = (I + A)^-1 (the UT form of the WY representation).  RLA: E = V.
//
//   P   = diag(Gprev) K S0 + Ap E,   Ap[t,i] = exp(b_{t-1}-b_i) beta_i (k_t.k_i), i<t
//         (P_t = S_{t-1}^T k_t, the undecayed prediction of Section 3.3)
//   Ob  = diag(Gam) Q S0 + Mq E,     Mq[t,i] = exp(b_t-b_i) beta_i (q_t.k_i), i<t
//         (Ob_t = a_t S_{t-1}^T q_t, the base prediction)
//   S_C = Gam_C S0 + K^T diag(beta_i exp(b_C - b_i)) E
//   r   = clip(V - P, -c, c)                                   (Section 3.3)
//   the auxiliary pass repeats this with values r, rate gamma, state R; its
//   read-out includes token t:  Oa = diag(Gam) Q R0 + M2 E2,
//         M2[t,i] = exp(b_t-b_i) gamma_i (q_t.k_i), i<=t
//   o   = Ob + diag(gamma) Oa.
//
// Kernel 1 (chunk_prep): one CTA per chunk -- everything that does not depend
// on the state: the Gram matrices, the masked/decayed matrices Ap, Mq, M2 and
// (RDN) the two unit-lower inverses T_beta, T_gamma by forward substitution.
// Kernel 2 (chunk_scan): one CTA per (b, h, 8- to 32-column slice of d_v) -- the
// sequential pass over chunks carrying S and R slices in shared memory.  Each
// value column is independent (the clip is elementwise), so slicing d_v is
// exact; only the prep work is shared between slices.
#include <type_traits>

#include "chunk_common.cuh"
#include "simt.cuh"
#include "status.cuh"

namespace rdn {
namespace {

// ---------------------------------------------------------------- kernel 1
// Two CTAs of 256 threads per SM.  Thread (ty, tx) holds rows 4 ty .. 4 ty + 3
// and columns tx + 16 j of both Gram products (they share the operand K), goes
// from its accumulators to the decayed matrices without a pass through shared
// memory, and only A_beta, A_gamma stay there for the inverses; T_beta,
// T_gamma take the place of K and Q.  Bound by shared-memory loads and the
// inverses' chain: 2048 chunks of d = 64 in 0.124 ms (0.402 ms with scalar
// operand loads, every matrix in shared memory and one CTA per SM).
template <int DK>
struct PrepSm {  // float offsets
  static constexpr int LDK = DK + 4, LDA = C + 1, LDT = C + 4;
  static constexpr int K = 0, Q = K + C * LDK, TB = 0, TG = C * LDT;  // (T over K, Q)
  static constexpr int AB = 2 * C * LDK, AG = AB + C * LDA, VEC = AG + C * LDA;
  static constexpr int FLOATS = VEC + 7 * C;
  static_assert(2 * LDT <= 2 * LDK, "T fits over K and Q");
};

template <int DK, bool RDNV, typename InT>
__global__ void __launch_bounds__(kThreads, 2) chunk_prep_kernel(FwdParams p) {
  using SM = PrepSm<DK>;
  constexpr int LDK = SM::LDK, LDA = SM::LDA, LDT = SM::LDT;
  extern __shared__ __align__(16) float sm[];
  float *Ks = sm + SM::K, *Qs = sm + SM::Q, *Ab = sm + SM::AB, *Ag = sm + SM::AG;
  simt::Cum &cum = *reinterpret_cast<simt::Cum *>(sm + SM::VEC);
  float *bet = sm + SM::VEC + 4 * C, *gam = bet + C, *gg = gam + C;

  const long long chunk = blockIdx.x;
  if (chunk >= total_records(p)) return;  // (packed sequences: the grid covers the bound)
  int sq, h, c;
  rec_decode(p, chunk, sq, h, c);
  const SeqSpan sp = seq_span(p, sq, h);
  const int t0 = c * C;
  const int n = min(C, sp.len - t0);
  const int tid = threadIdx.x, tx = (tid & 31) >> 1, ty = 2 * (tid >> 5) + (tid & 1);

  {
    simt::RowTile<InT, DK, kThreads> kt, qt;
    const size_t off = ((size_t)(sp.tok0 + t0) * p.H + h) * DK;
    kt.fetch((const InT *)p.k + off, (size_t)p.H * DK, n);
    qt.fetch((const InT *)p.q + off, (size_t)p.H * DK, n);
    if (tid < 32) {  // gates of tokens tid, tid + 32 and the cumulative decay
      float g2[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int t = tid + 32 * u;
        const bool ok = t < n;
        const size_t go = (size_t)(sp.tok0 + t0 + (ok ? t : 0)) * p.H + h;
        g2[u] = ok ? p.g[go] : 0.f;
        gg[t] = g2[u];
        bet[t] = ok ? p.beta[go] : 0.f;
        gam[t] = ok ? p.gamma[go] : 0.f;
      }
      simt::cum64(g2[0], g2[1], cum);
    }
    kt.put(Ks, LDK, 1.f);
    qt.put(Qs, LDK, p.scale);
  }
  __syncthreads();
  float kk[4][4], qk[4][4];
  simt::mm_nt<4, 4, DK>(Ks + 4 * ty * LDK, LDK, Ks + tx * LDK, 16 * LDK, kk);
  simt::mm_nt<4, 4, DK>(Qs + 4 * ty * LDK, LDK, Ks + tx * LDK, 16 * LDK, qk);
  float *rec = p.ws + (size_t)chunk * kRecFloats;
  // variants: the decayed residual predicts with a_t S_{t-1} k_t, so Ap takes
  // the decay to t (not t-1); the plain combine reads S_{t-1} q_t, so Mq takes
  // the decay to t-1; the stateless correction reads r_t (q_t.k_t) alone
  const bool dec_res = p.mods & RDN_FLAG_DECAYED_RESIDUAL;
  const bool plain = p.mods & RDN_FLAG_PLAIN_COMBINE;
  const bool stl = p.mods & RDN_FLAG_STATELESS_AUX;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int t = 4 * ty + a, i = tx + 16 * b;
      float ap = 0.f, mq = 0.f, m2 = 0.f, ab = 0.f, ag = 0.f;
      if (i <= t) {
        const float dec = expf(cum.to(t, i));
        m2 = stl ? (i == t ? qk[a][b] : 0.f) : dec * gam[i] * qk[a][b];
        if (i < t) {
          const float decp = expf(cum.before(t, i));
          ap = (dec_res ? dec : decp) * bet[i] * kk[a][b];
          mq = (plain ? decp : dec) * bet[i] * qk[a][b];
          ab = dec * bet[i] * kk[a][b];
          ag = dec * gam[i] * kk[a][b];
        }
      }
      const int e = t * C + i;
      rec[OFF_AP + e] = ap;
      rec[OFF_MQ + e] = mq;
      rec[OFF_M2 + e] = m2;
      if (RDNV) {
        Ab[t * LDA + i] = ab;
        Ag[t * LDA + i] = ag;
      }
    }
  if (tid < C) {
    const int t = tid;
    const float end = expf(cum.to(C - 1, t));
    rec[OFF_VEC + V_GAM + t] = expf(cum.hi[t]);
    rec[OFF_VEC + V_GPREV + t] = expf(cum.phi[t]);
    rec[OFF_VEC + V_ALPHA + t] = expf(gg[t]);
    rec[OFF_VEC + V_WS + t] = bet[t] * end;
    // (stateless correction: R at the chunk end is k r^T of its last token)
    rec[OFF_VEC + V_WR + t] = stl ? (t == n - 1 ? 1.f : 0.f) : gam[t] * end;
    if (t == 0) rec[OFF_VEC + V_GAMC] = expf(cum.hi[C - 1]);
  }
  if (RDNV) {
    // threads 0..127 invert I + A_beta, threads 128..255 I + A_gamma
    __syncthreads();
    const int g = tid & 127;
    const float *A = tid < 128 ? Ab : Ag;
    float *Tm = sm + (tid < 128 ? SM::TB : SM::TG);
    // the blocks above the diagonal that the products read: (0, 1) and (2, 3)
    for (int e = g; e < 2 * 16 * 16; e += 128) {
      const int b = e >> 8, r = (e >> 4) & 15, cc = e & 15;
      Tm[(32 * b + r) * LDT + 32 * b + 16 + cc] = 0.f;
    }
    for (int stage = 0; stage <= 4; ++stage) {
      if (stage) __syncthreads();
      inv64_stage<LDA, LDT, LDT>(stage, A, Tm, Tm + 32, g);
    }
    __syncthreads();
    for (int e = tid; e < 2 * C * C / 4; e += kThreads) {
      const int m = e / (C * C / 4), t = (e / (C / 4)) % C, i = 4 * (e % (C / 4));
      const float4 x = *reinterpret_cast<const float4 *>(sm + (m ? SM::TG : SM::TB) + t * LDT + i);
      const float4 y = make_float4(i <= t ? x.x : 0.f, i + 1 <= t ? x.y : 0.f,
                                   i + 2 <= t ? x.z : 0.f, i + 3 <= t ? x.w : 0.f);
      *reinterpret_cast<float4 *>(rec + (m ? OFF_TG : OFF_TB) + t * C + i) = y;
    }
  }
}

// ---------------------------------------------------------------- kernel 2
// One CTA per (sequence, head, DVS value columns), the chunks in sequence.
// Thread (warp w, lane (lm, ln)) owns columns TN ln .. + TN and rows
// 32 i + LM w + lm of every 64-row product (i = 0, 1; for the stacked 128-row
// products i = 0, 1 are the K (or Ap) rows, 2, 3 the Q (or Mq) rows), so that a
// chunk's read-outs, predictions and outputs stay in its registers from one
// product to the next; only what the next product reads as its right operand
// (X, E, wS E, then X2, E2, wR E2) goes through shared memory.  Four phases a
// chunk: [KS; QS], [KR; QR] | E | [Ap; Mq] E and S's update | E2 | M2 E2 and R's
// update.  The upper halves of the triangular blocks are skipped.  The chunk
// matrices arrive by cp.async a phase or more ahead, in three slots; the next
// chunk's K, Q, V and gate vectors wait in registers over the last phase.
// Bound by the FMA pipe and the phases' latencies: B = 4, H = 16, T = 2048,
// d = 64 in 0.396 ms (1.079 ms with scalar operand loads), B = 2, H = 8,
// T = 1000, d = 128 fp32 in 0.181 ms (0.718), B = 1, H = 2, T = 256, d = 64 in
// 0.023 ms (0.085, on 4 CTAs).
// REC: one chunk per CTA from the chunk-start states p.S_chunks, p.R_chunks,
// writing only what the backward reads (E, E2 and the residual's mask).
template <int DK, int DVS, int NT>
struct ScanSm {  // float offsets
  static constexpr int LDK = DK + 4, LDM = C + 4;
  static constexpr int K = 0, Q = K + C * LDK, MAT = Q + C * LDK;  // MAT: 3 slots
  static constexpr int S = MAT + 3 * C * LDM, R = S + DK * DVS, V = R + DK * DVS;
  static constexpr int X = V + C * DVS, E = X + C * DVS, W = E + C * DVS, VEC = W + C * DVS;
  static constexpr int GM = VEC + 6 * C, FLOATS = GM + C;
};

template <int DK, bool RDNV, typename InT, int DVS, int NT, bool REC>
__global__ void __launch_bounds__(NT, NT == 128 ? 2 : 1) chunk_scan_kernel(FwdParams p) {
  using namespace simt;
  using SM = ScanSm<DK, DVS, NT>;
  constexpr int DV = DK, LDK = SM::LDK, LDM = SM::LDM;
  constexpr int TN = 32 * DVS / NT, LN = DVS / TN, LM = 32 / LN, TMU = DK / 32;
  static_assert(LM * (NT / 32) == 32, "row blocks of 32");
  extern __shared__ __align__(16) float sm[];
  float *Ks = sm + SM::K, *Qs = sm + SM::Q, *Ss = sm + SM::S, *Rs = sm + SM::R;
  float *Vs = sm + SM::V, *Xs = sm + SM::X, *Es = sm + SM::E, *Ws = sm + SM::W;
  float *vec = sm + SM::VEC, *gms = sm + SM::GM;
  float *mat[3] = {sm + SM::MAT, sm + SM::MAT + C * LDM, sm + SM::MAT + 2 * C * LDM};

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int lm, ln;
  lane_mn<LN>(lane, lm, ln);
  const int r0 = LM * warp + lm, n0 = TN * ln;
  int sq, h, c0 = 0, c1;
  if (REC) {
    if ((long long)blockIdx.x >= total_records(p)) return;
    rec_decode(p, blockIdx.x, sq, h, c0);
    c1 = c0 + 1;
  } else {
    sq = seq_at(p, blockIdx.x / p.H);
    h = blockIdx.x % p.H;
  }
  const SeqSpan sp = seq_span(p, sq, h);
  if (!REC) c1 = sp.nc;
  const int j0 = blockIdx.y * DVS;
  const float clip = p.clip;
  const bool dec_res = p.mods & RDN_FLAG_DECAYED_RESIDUAL;
  const bool plain = p.mods & RDN_FLAG_PLAIN_COMBINE;
  const bool tnh = p.mods & RDN_FLAG_TANH_RESIDUAL;
  const bool stl = p.mods & RDN_FLAG_STATELESS_AUX;
  const bool rdn_aux = RDNV && !stl;  // the auxiliary pass runs the delta rule

  const size_t sbase = REC ? (size_t)blockIdx.x * DK * DV : (size_t)(sq * (size_t)p.H + h) * DK * DV;
  {
    const float *S0 = REC ? p.S_chunks : p.S0, *R0 = REC ? p.R_chunks : p.R0;
    for (int e = tid; e < DK * DVS / 4; e += NT) {
      const size_t off = sbase + (size_t)(e / (DVS / 4)) * DV + j0 + 4 * (e % (DVS / 4));
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4 *>(Ss + 4 * e) = S0 ? *reinterpret_cast<const float4 *>(S0 + off) : z;
      *reinterpret_cast<float4 *>(Rs + 4 * e) = R0 ? *reinterpret_cast<const float4 *>(R0 + off) : z;
    }
  }

  RowTile<InT, DK, NT> kt, qt;
  RowTile<InT, DVS, NT> vt;
  constexpr int VU = 6 * C / NT + (6 * C % NT != 0);
  float vr[VU], gr = 0.f;
  auto fetch = [&](int c) {  // chunk c's K, Q, V, gate vectors
    const int n = min(C, sp.len - c * C);
    const size_t row = (size_t)(sp.tok0 + c * C) * p.H + h;
    kt.fetch((const InT *)p.k + row * DK, (size_t)p.H * DK, n);
    qt.fetch((const InT *)p.q + row * DK, (size_t)p.H * DK, n);
    vt.fetch((const InT *)p.v + row * DV + j0, (size_t)p.H * DV, n);
    const float *rec = p.ws + (size_t)(sp.rbase + c) * kRecFloats;
#pragma unroll
    for (int u = 0; u < VU; ++u) {
      const int e = tid + u * NT;
      vr[u] = e <= V_GAMC ? rec[OFF_VEC + e] : 0.f;
    }
    if (tid < C) gr = tid < n ? p.gamma[row + (size_t)tid * p.H] : 0.f;
  };
  auto mats = [&](int c) { return p.ws + (size_t)(sp.rbase + c) * kRecFloats; };
  if (c0 < c1) {
    fetch(c0);
    if (RDNV) cp_mat<NT>(mat[0], LDM, mats(c0) + OFF_TB);
    cp_commit();
    cp_mat<NT>(mat[1], LDM, mats(c0) + OFF_AP);
    if (!REC) cp_mat<NT>(mat[2], LDM, mats(c0) + OFF_MQ);
    cp_commit();
  }

  for (int c = c0; c < c1; ++c) {
    const int t0 = c * C;
    const int n = min(C, sp.len - t0);
    const bool more = c + 1 < c1;
    kt.put(Ks, LDK, 1.f);
    qt.put(Qs, LDK, p.scale);
    vt.put(Vs, DVS, 1.f);
#pragma unroll
    for (int u = 0; u < VU; ++u)
      if (tid + u * NT < 6 * C) vec[tid + u * NT] = vr[u];
    if (tid < C) gms[tid] = gr;
    __syncthreads();
    const float *Gam = vec + V_GAM, *Gprev = vec + V_GPREV, *wS = vec + V_WS, *wR = vec + V_WR;
    const float GamC = vec[V_GAMC];
    const size_t rec = (size_t)(sp.rbase + c);
    if (!REC && p.S_chunks) {
      float *sc = p.S_chunks + rec * DK * DV + j0, *rc = p.R_chunks + rec * DK * DV + j0;
      for (int e = tid; e < DK * DVS / 4; e += NT) {
        const size_t off = (size_t)(e / (DVS / 4)) * DV + 4 * (e % (DVS / 4));
        *reinterpret_cast<float4 *>(sc + off) = *reinterpret_cast<const float4 *>(Ss + 4 * e);
        *reinterpret_cast<float4 *>(rc + off) = *reinterpret_cast<const float4 *>(Rs + 4 * e);
      }
    }
    // ---- [K; Q] S and [K; Q] R
    float a1[4][TN], a2[4][TN];
    zero(a1);
    zero(a2);
    {
      const float *A = Ks + r0 * LDK;
      constexpr int MS = REC ? 3 : 15, MR = (RDNV ? 3 : 0) | (REC ? 0 : 12);
      if (stl) mm_ak<4, TN, MS>(A, 32 * LDK, Ss + n0, DVS, 0, DK, a1);
      else mm_ak2<4, TN, MS, MR>(A, 32 * LDK, Ss + n0, Rs + n0, DVS, DK, a1, a2);
    }
    float vv[2][TN];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int t = r0 + 32 * i;
      ldv<TN>(Vs + t * DVS + n0, vv[i]);
      float x[TN];
#pragma unroll
      for (int j = 0; j < TN; ++j)  // RDN: X = V - Gam K S; RLA (E = V): wS E
        x[j] = RDNV ? fmaf(-Gam[t], a1[i][j], vv[i][j]) : wS[t] * vv[i][j];
      stv<TN>((RDNV ? Xs : Ws) + t * DVS + n0, x);
    }
    const float *E = Vs;
    wait_groups<1>();  // (T_beta, and the M_q fetched before it)
    __syncthreads();
    // ---- E = T_beta X, wS E
    if (RDNV) {
      float e[2][TN];
      zero(e);
      const float *A = mat[0] + r0 * LDM;
      mm_ak<2, TN, 3>(A, 32 * LDM, Xs + n0, DVS, 0, 32, e);
      mm_ak<2, TN, 2>(A, 32 * LDM, Xs + n0, DVS, 32, 64, e);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = r0 + 32 * i;
        stv<TN>(Es + t * DVS + n0, e[i]);
        if (p.sv_E) stv<TN>((float *)p.sv_E + (rec * C + t) * DV + j0 + n0, e[i]);
#pragma unroll
        for (int j = 0; j < TN; ++j) e[i][j] *= wS[t];
        stv<TN>(Ws + t * DVS + n0, e[i]);
      }
      E = Es;
      wait_groups<0>();
      __syncthreads();
    } else {
      if (p.sv_E)
#pragma unroll
        for (int i = 0; i < 2; ++i)
          stv<TN>((float *)p.sv_E + (rec * C + r0 + 32 * i) * DV + j0 + n0, vv[i]);
      wait_groups<0>();
      __syncthreads();
    }
    if (rdn_aux) cp_mat<NT>(mat[0], LDM, mats(c) + OFF_TG);
    cp_commit();
    // ---- [Ap; Mq] E: the prediction, the residual, the base output; S's update
    float ob[2][TN], r[2][TN];
    {
      float pm[4][TN];
      zero(pm);
      const float *A = mat[1] + r0 * LDM;
      mm_ak<4, TN, REC ? 3 : 15>(A, 32 * LDM, E + n0, DVS, 0, 32, pm);
      mm_ak<4, TN, REC ? 2 : 10>(A, 32 * LDM, E + n0, DVS, 32, 64, pm);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = r0 + 32 * i;
        const float gp = dec_res ? Gam[t] : Gprev[t], gq = plain ? Gprev[t] : Gam[t];
        float x2[TN], dr[TN];
        uint32_t in = 0;  // bit j: |x| <= c
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          // P_t = S_{t-1}^T k_t (decayed residual: a_t S_{t-1}^T k_t)
          const float x = vv[i][j] - fmaf(gp, a1[i][j], pm[i][j]);
          r[i][j] = resid_map(x, clip, tnh);  // Section 3.3
          ob[i][j] = fmaf(gq, a1[2 + i][j], pm[2 + i][j]);
          x2[j] = fmaf(-Gam[t], a2[i][j], r[i][j]);
          in |= (fabsf(x) <= clip ? 1u : 0u) << j;
          if (tnh) dr[j] = resid_grad(x, clip, true);
        }
        if (rdn_aux) stv<TN>(Xs + t * DVS + n0, x2);
        if (p.sv_mask) {
          if (tnh) {
            stv<TN>((float *)p.sv_mask + (rec * C + t) * DV + j0 + n0, dr);
          } else {  // the row's DVS bits: one byte per 8 columns
            in <<= n0 & 7;
#pragma unroll
            for (int b = 0; 1 << b < 8 / TN; ++b)  // (bit b of ln is lane bit 2 b)
              in |= __shfl_xor_sync(0xffffffffu, in, 1 << 2 * b);
            if (n0 % 8 == 0)
              ((uint8_t *)p.sv_mask)[((rec * C + t) * DV + j0 + n0) >> 3] = (uint8_t)in;
          }
        }
      }
      if (!REC) {
        const int m0 = TMU * r0;
        float u[TMU][TN];
        zero(u);
        mm_am<TMU, TN>(Ks + m0, LDK, Ws + n0, DVS, C, u);  // K^T diag(wS) E
#pragma unroll
        for (int i = 0; i < TMU; ++i) {
          float s[TN];
          ldv<TN>(Ss + (m0 + i) * DVS + n0, s);
#pragma unroll
          for (int j = 0; j < TN; ++j) s[j] = fmaf(GamC, s[j], u[i][j]);
          stv<TN>(Ss + (m0 + i) * DVS + n0, s);
        }
      }
    }
    wait_groups<0>();  // T_gamma
    __syncthreads();
    if (!REC) {
      cp_mat<NT>(mat[1], LDM, mats(c) + OFF_M2);
      cp_commit();
      if (more) cp_mat<NT>(mat[2], LDM, mats(c + 1) + OFF_MQ);
      cp_commit();
    }
    // ---- E2 = T_gamma X2, wR E2
    if (rdn_aux) {
      zero(r);
      const float *A = mat[0] + r0 * LDM;
      mm_ak<2, TN, 3>(A, 32 * LDM, Xs + n0, DVS, 0, 32, r);
      mm_ak<2, TN, 2>(A, 32 * LDM, Xs + n0, DVS, 32, 64, r);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int t = r0 + 32 * i;
      if (p.sv_E2) stv<TN>((float *)p.sv_E2 + (rec * C + t) * DV + j0 + n0, r[i]);
      if (REC) continue;
      stv<TN>(Es + t * DVS + n0, r[i]);
#pragma unroll
      for (int j = 0; j < TN; ++j) r[i][j] *= wR[t];
      stv<TN>(Ws + t * DVS + n0, r[i]);
    }
    if (REC) break;
    wait_groups<1>();  // M2
    __syncthreads();
    if (more) {
      if (RDNV) cp_mat<NT>(mat[0], LDM, mats(c + 1) + OFF_TB);
      fetch(c + 1);
    }
    cp_commit();
    // ---- o = Ob + gamma (Gam Q R + M2 E2); R's update
    {
      float oa[2][TN];
      zero(oa);
      const float *A = mat[1] + r0 * LDM;
      mm_ak<2, TN, 3>(A, 32 * LDM, Es + n0, DVS, 0, 32, oa);
      mm_ak<2, TN, 2>(A, 32 * LDM, Es + n0, DVS, 32, 64, oa);
      InT *o = (InT *)p.o;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = r0 + 32 * i;
        if (t < n) {
          const float gm = plain ? 1.f : gms[t];
          const size_t off = ((size_t)(sp.tok0 + t0 + t) * p.H + h) * DV + j0 + n0;
          float y[TN];
#pragma unroll
          for (int j = 0; j < TN; ++j)
            y[j] = fmaf(gm, fmaf(Gam[t], a2[2 + i][j], oa[i][j]), ob[i][j]);
          if constexpr (sizeof(InT) == 4) {
            stv<TN>((float *)o + off, y);
          } else {
            uint32_t w[TN / 2 ? TN / 2 : 1];
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) {
              const __nv_bfloat162 b2 = __floats2bfloat162_rn(y[2 * j], y[2 * j + 1]);
              w[j] = *reinterpret_cast<const uint32_t *>(&b2);
            }
            if constexpr (TN == 4) *reinterpret_cast<uint2 *>(o + off) = make_uint2(w[0], w[1]);
            else *reinterpret_cast<uint32_t *>(o + off) = w[0];
          }
        }
      }
      const int m0 = TMU * r0;
      float u[TMU][TN];
      zero(u);
      mm_am<TMU, TN>(Ks + m0, LDK, Ws + n0, DVS, C, u);  // K^T diag(wR) E2
#pragma unroll
      for (int i = 0; i < TMU; ++i) {
        float s[TN];
        ldv<TN>(Rs + (m0 + i) * DVS + n0, s);
#pragma unroll
        for (int j = 0; j < TN; ++j) s[j] = fmaf(stl ? 0.f : GamC, s[j], u[i][j]);
        stv<TN>(Rs + (m0 + i) * DVS + n0, s);
      }
    }
    __syncthreads();  // every buffer of this chunk is free
    if (more) cp_mat<NT>(mat[1], LDM, mats(c + 1) + OFF_AP);
    cp_commit();
  }
  if (REC) return;
  __syncthreads();
  for (int e = tid; e < DK * DVS / 4; e += NT) {
    const size_t off = sbase + (size_t)(e / (DVS / 4)) * DV + j0 + 4 * (e % (DVS / 4));
    if (p.ST) *reinterpret_cast<float4 *>(p.ST + off) = *reinterpret_cast<const float4 *>(Ss + 4 * e);
    if (p.RT) *reinterpret_cast<float4 *>(p.RT + off) = *reinterpret_cast<const float4 *>(Rs + 4 * e);
  }
}

template <int DK, bool RDNV, typename InT, int DVS, int NT, bool REC>
cudaError_t launch_scan_t(const FwdParams &p, cudaStream_t s) {
  auto scan = chunk_scan_kernel<DK, RDNV, InT, DVS, NT, REC>;
  constexpr int smem = (int)sizeof(float) * ScanSm<DK, DVS, NT>::FLOATS;
  const cudaError_t e = cudaFuncSetAttribute(scan, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const dim3 grid(REC ? (unsigned)p.nrec : (unsigned)(p.nseq * p.H), DK / DVS);
  RDN_LAUNCH(REC ? "chunk_recompute" : "chunk_scan", s, scan<<<grid, NT, smem, s>>>(p));
  return cudaGetLastError();
}

template <int DK, bool RDNV, typename InT>
cudaError_t launch_scan(const FwdParams &p, cudaStream_t s) {
  int nsm = 0;
  const cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const int dvs = scan_columns(DK, (long long)p.nseq * p.H, nsm);
  if constexpr (DK == 64)
    return dvs == 16 ? launch_scan_t<64, RDNV, InT, 16, 128, false>(p, s)
                     : launch_scan_t<64, RDNV, InT, 8, 128, false>(p, s);
  else
    return dvs == 32   ? launch_scan_t<128, RDNV, InT, 32, 256, false>(p, s)
           : dvs == 16 ? launch_scan_t<128, RDNV, InT, 16, 256, false>(p, s)
                       : launch_scan_t<128, RDNV, InT, 8, 256, false>(p, s);
}

template <int DK, bool RDNV, typename InT>
cudaError_t launch_prep_t(const FwdParams &p, cudaStream_t s) {
  cudaError_t e;
  if (p.qk_norm) {  // q, k are raw: the prologue kernel writes the normalised copies first
    rdn_prologue_args pa{};
    pa.rows = (long long)p.B * p.T * p.H;
    pa.D = DK;
    pa.dtype = std::is_same<InT, __nv_bfloat16>::value ? RDN_BF16 : RDN_F32;
    pa.eps = p.qk_eps;
    pa.x[0] = p.qraw;
    pa.x[1] = p.kraw;
    pa.y[0] = const_cast<void *>(p.q);
    pa.y[1] = const_cast<void *>(p.k);
    if ((e = launch_prologue(pa, false, s)) != cudaSuccess) return e;
  }
  auto prep = chunk_prep_kernel<DK, RDNV, InT>;
  constexpr int smem = (int)sizeof(float) * PrepSm<DK>::FLOATS;
  if ((e = cudaFuncSetAttribute(prep, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess)
    return e;
  RDN_LAUNCH("chunk_prep", s, prep<<<(unsigned)p.nrec, kThreads, smem, s>>>(p));
  return cudaGetLastError();
}

struct RunPrep {
  const FwdParams &p;
  cudaStream_t s;
  template <int DK, bool RDNV, typename InT>
  cudaError_t run() const { return launch_prep_t<DK, RDNV, InT>(p, s); }
};
struct RunScan {
  const FwdParams &p;
  cudaStream_t s;
  template <int DK, bool RDNV, typename InT>
  cudaError_t run() const { return launch_scan<DK, RDNV, InT>(p, s); }
};

struct RunRecompute {
  const FwdParams &p;
  cudaStream_t s;
  template <int DK, bool RDNV, typename InT>
  cudaError_t run() const {
    return launch_scan_t<DK, RDNV, InT, DK == 64 ? 16 : 32, DK == 64 ? 128 : 256, true>(p, s);
  }
};

}  // namespace

cudaError_t launch_recompute(const FwdParams &p, int DK, bool rdnv, bool bf16, cudaStream_t s) {
  return simt_dispatch(DK, rdnv, bf16, RunRecompute{p, s});
}

cudaError_t launch_prep(const FwdParams &p, int DK, bool rdnv, bool bf16, cudaStream_t s) {
  if (fwd_uses_tc(DK, bf16)) return launch_prep_tc(p, !rdnv, s);
  return simt_dispatch(DK, rdnv, bf16, RunPrep{p, s});
}

cudaError_t launch_fwd_parts(const FwdParams &p, int DK, bool rdnv, bool bf16, cudaStream_t s) {
  const cudaError_t e = launch_prep(p, DK, rdnv, bf16, s);
  if (e != cudaSuccess) return e;
  if (fwd_uses_tc(DK, bf16)) return launch_fwd_tc(p, rdnv, s);
  return simt_dispatch(DK, rdnv, bf16, RunScan{p, s});
}

// Block-wide inclusive scan of one value per thread (blockDim.x = 1024).
template <typename Op>
__device__ long long block_incl_scan(long long x, Op op, long long *wsum) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x = op(x, y);
  }
  if (lane == 31) wsum[wid] = x;
  __syncthreads();
  if (wid == 0) {
    long long w = wsum[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w = op(w, y);
    }
    wsum[lane] = w;
  }
  __syncthreads();
  if (wid > 0) x = op(x, wsum[wid - 1]);
  __syncthreads();  // (wsum is reused by the next call)
  return x;
}

// The packed-sequence table FwdParams::seq from cu_seqlens[0 .. N]: first
// tokens are the running maximum of the entries clamped into [0, T] (with
// entry 0 read as 0 and entry N as T, so the table always covers [0, T) in
// order), first chunks the exclusive prefix sum of ceil(len_s / 64).  One CTA.
__global__ void __launch_bounds__(1024) seq_table_kernel(const int *__restrict__ cu, int N, int T,
                                                         int H, ScanCost cost, int nsm,
                                                         long long *__restrict__ seq) {
  __shared__ long long wsum[32];
  __shared__ long long carry;
  __shared__ int ncs[kOrdered];  // the sequences' chunks
  __shared__ unsigned keys[kOrdered];
  const int tid = threadIdx.x;
  if (tid == 0) carry = 0;
  __syncthreads();
  auto mx = [](long long a, long long b) { return a > b ? a : b; };
  auto add = [](long long a, long long b) { return a + b; };
  for (int base = 0; base <= N; base += 1024) {
    const int s = base + tid;
    long long x = 0;
    if (s <= N) x = s == 0 ? 0 : s == N ? T : min(max(cu[s], 0), T);
    x = mx(block_incl_scan(x, mx, wsum), carry);
    if (s <= N) seq[2 * s] = x;
    if (tid == 1023) carry = x;  // (padding reads 0 and leaves the maximum alone)
    __syncthreads();
  }
  if (tid == 0) carry = 0;
  __syncthreads();  // (also orders the token offsets before they are read back)
  for (int base = 0; base <= N; base += 1024) {
    const int s = base + tid;
    const long long nc = s < N ? (seq[2 * s + 2] - seq[2 * s] + C - 1) / C : 0;
    const long long incl = block_incl_scan(nc, add, wsum) + carry;
    if (s <= N) seq[2 * s + 1] = incl - nc;  // entry N: the total
    if (s < min(N, kOrdered)) ncs[s] = (int)nc;
    if (tid == 1023) carry = incl;
    __syncthreads();
  }
  // longest first, equal ones as they come (more than kOrdered sequences: all as they
  // come): few by counting those ahead of each, more by a bitonic sort of (chunks,
  // index) keys in registers, 1024 of them in 55 steps of which 15 go through shared
  // memory.  The kernel takes 9 us by the one and 10 by the other at 80 sequences, 15
  // and 12 at 500, 37 and 13 at 1000.
  int *upper = reinterpret_cast<int *>(seq) + 3;  // of the k-th chunk number: upper[4 k]
  if (N > kOrdered) {  // (entry N's stays 0: no pairs)
    for (int s = tid; s < N; s += 1024) upper[4 * s] = s;
    return;
  }
  if (N <= 256) {
    if (tid >= N) return;
    const int mine = ncs[tid];
    int rank = 0;
    for (int u = 0; u < N; ++u) rank += ncs[u] > mine || (ncs[u] == mine && u < tid);
    upper[4 * rank] = tid;
    if (rank == 0) upper[4 * N] = pairs_for(cost, mine, N, carry, H, nsm);
    return;
  }
  static_assert(kOrdered == 1024, "11 bits of a key");  // (chunks: at most 2^24 tokens / 64)
  unsigned key = tid < N ? (unsigned)ncs[tid] << 11 | (unsigned)(kOrdered - tid) : 0u;
  for (int k = 2; k / 2 < N; k *= 2) {
    for (int d = k / 2; d > 0; d /= 2) {
      unsigned other;
      if (d < 32) {
        other = __shfl_xor_sync(0xffffffffu, key, d);
      } else {
        __syncthreads();  // (the last step's keys have been read)
        keys[tid] = key;
        __syncthreads();
        other = keys[tid ^ d];
      }
      // descending runs where tid & k is 0
      const bool larger = ((tid & d) == 0) == ((tid & k) == 0);
      if ((key < other) == larger) key = other;
    }
  }
  if (tid < N) upper[4 * tid] = kOrdered - (int)(key & 2047u);
  if (tid == 0) upper[4 * N] = pairs_for(cost, key >> 11, N, carry, H, nsm);
}

cudaError_t launch_seq_table(const rdn_fwd_args &a, int variant, bool states, long long *seq,
                             cudaStream_t s) {
  int nsm = 0;
  const cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  RDN_LAUNCH("seq_table", s,
             seq_table_kernel<<<1, 1024, 0, s>>>(a.cu_seqlens, a.num_seqs, a.T, a.H,
                                                 scan_cost(variant == 1, states), nsm, seq));
  return cudaGetLastError();
}

FwdPlan plan_fwd(const rdn_fwd_args &a, int variant) {
  FwdPlan pl;
  pl.NC = (a.T + C - 1) / C;
  pl.prep_bytes = sizeof(float) * (size_t)kRecFloats;
  const size_t nrec = (size_t)call_records(a);
  // per-chunk records, the saved intermediates if asked for, the normalised
  // q, k (RDN_FLAG_QK_NORM), the packed-sequence table, then a 256-byte tail
  pl.total_bytes = pl.prep_bytes * nrec + seq_table_bytes(a) + 256;
  if (a.flags & RDN_FLAG_SAVE_FOR_BWD)
    pl.total_bytes += saved_layout(a).bytes;
  pl.total_bytes += qk_norm_bytes(a);  // (after those: qk_norm_offset)
  return pl;
}

cudaError_t launch_fwd(const rdn_fwd_args &a, int variant, cudaStream_t s) {
  const size_t sbytes = sizeof(float) * (size_t)call_seqs(a) * a.H * a.Dk * a.Dv;
  if (a.T == 0) {  // no tokens: the final states are the initial ones
    cudaError_t e = cudaSuccess;
    if (a.ST) e = a.S0 ? cudaMemcpyAsync(a.ST, a.S0, sbytes, cudaMemcpyDeviceToDevice, s)
                       : cudaMemsetAsync(a.ST, 0, sbytes, s);
    if (e == cudaSuccess && a.RT)
      e = a.R0 ? cudaMemcpyAsync(a.RT, a.R0, sbytes, cudaMemcpyDeviceToDevice, s)
               : cudaMemsetAsync(a.RT, 0, sbytes, s);
    return e;
  }
  FwdParams p = make_fwd_params(a);
  p.ws = (float *)a.workspace;
  const size_t total = plan_fwd(a, variant).total_bytes;
  p.err = status_word();
  p.inject = fault_injection() == 3 ? 1 : 0;
  if (a.cu_seqlens) {
    long long *seq = (long long *)((char *)a.workspace + total - 256 - seq_table_bytes(a));
    const cudaError_t e = launch_seq_table(a, variant, a.S_chunks != nullptr, seq, s);
    if (e != cudaSuccess) return e;
    p.seq = seq;
  }
  if (a.flags & RDN_FLAG_SAVE_FOR_BWD) {
    const SavedLayout l = saved_layout(a);
    p.sv_E = (uint8_t *)a.workspace + l.e;
    p.sv_E2 = (uint8_t *)a.workspace + l.e2;
    p.sv_mask = (unsigned long long *)((char *)a.workspace + l.mask);
  }
  if (p.qk_norm) set_qk_norm_copies(p, a, (char *)a.workspace + qk_norm_offset(a));
  return launch_fwd_parts(p, a.Dk, variant == 1, a.dtype == RDN_BF16, s);
}

}  // namespace rdn
