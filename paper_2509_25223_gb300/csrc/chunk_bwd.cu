// chunk_bwd.cu -- backward of the chunkwise RLA / RDN forward (fp32 SIMT:
// fp32 inputs and d = 64), and the dispatcher of both backward paths.
//
// Reverse mode of the chunk algebra in chunk_fwd.cu (the paper gives no
// backward; this is the adjoint of the forward as computed).  Per chunk,
// given the carried dS, dR (gradients w.r.t. the chunk-end states) and dO:
//
//   auxiliary pass  dOa = diag(gam) dO;  dgam += rowsum(dO * Oa)
//                   dM2 = incl(dOa E2^T);  dE2 = M2^T dOa + diag(wR) K dR
//                   RDN: dX2 = Tg^T dE2, dAg = -strict(dX2 E2^T), dRv = dX2,
//                        dKR = -diag(Gam) dX2;   RLA: dRv = dE2
//                   dR0 = Gam_C dR + K^T dKR + Q^T diag(Gam) dOa
//   clip            dVr = dRv * [|v - P| <= c],  dP = -dVr
//   base pass       dMq = strict(dO E^T);  dAp = strict(dP E^T)
//                   dE = Mq^T dO + Ap^T dP + diag(wS) K dS
//                   RDN: dX = Tb^T dE, dAb = -strict(dX E^T), dV = dVr + dX,
//                        dKS = diag(Gprev) dP - diag(Gam) dX;   RLA: dV = dVr + dE
//                   dS0 = Gam_C dS + K^T dKS + Q^T diag(Gam) dO
//   dK, dQ collect the state products (E dS^T, dKS S0^T, ...); the C x C
//   gradients dAp, dMq, dM2, dAb, dAg and the per-row factors then give
//   d(KK^T), d(QK^T), dbeta, dgamma and the gradient of the in-chunk
//   cumulative log-decay, whose reverse cumulative sum is dg.
//
// Kernel bwd_chain: one CTA per (sequence, head, slice of value columns),
// chunks in reverse: only what the carried dS, dR need, from the forward's
// residual mask (E, E2 and the mask are kept by the forward, or remade by
// chunk_recompute); it keeps dX2, dX, dVr and the chunk-end dS, dR of every
// chunk in the workspace.
// Kernel bwd_post: one CTA per chunk, every product over the value columns
// that no other chunk waits for, and the fold into dq, dk, dg, dbeta, dgamma.
// Its sums over the value columns stay inside one CTA, so nothing is added
// atomically and equal calls give equal bits.
#include "chunk_common.cuh"
#include "simt.cuh"
#include "status.cuh"

namespace rdn {
namespace {

struct BwdParams {
  FwdParams f;  // forward inputs; f.ws = prep records; f.sv_* = E, E2, mask
  const void *dO;
  const float *dST, *dRT;
  const float *Sc, *Rc;  // chunk-start states [record][DK][DV]
  void *dq, *dk, *dv;
  float *dg, *dbeta, *dgamma, *dS0, *dR0;
  // per chunk, bwd_chain to bwd_post: dX2, dVr, dX [record][t][DV] (dX2 with
  // the auxiliary delta rule, dX with the base one) and the gradients w.r.t.
  // the chunk-end states [record][DK][DV]
  float *dX2, *dVr, *dX, *gS, *gR;
  // dv is dO's buffer: bwd_post, which still reads dO, writes it (then dX is kept
  // with either base pass)
  bool dv_late;
  // RDN_FLAG_QK_NORM with bf16 inputs: dq, dk (w.r.t. the normalised q, k)
  // stored here in fp32 for the normalisation's backward; else NULL
  float *gq32, *gk32;
};

// N consecutive elements of a token row as fp32 / from fp32
template <typename InT, int N>
__device__ __forceinline__ void ld_row(const InT *p, float (&v)[N]) {
  if constexpr (sizeof(InT) == 4) {
    simt::ldv<N>((const float *)p, v);
  } else {
#pragma unroll
    for (int j = 0; j < N; j += 2) {
      const uint32_t w = *reinterpret_cast<const uint32_t *>(p + j);
      v[j] = __uint_as_float(w << 16);
      v[j + 1] = __uint_as_float(w & 0xFFFF0000u);
    }
  }
}
template <typename InT, int N>
__device__ __forceinline__ void st_row(InT *p, const float (&v)[N]) {
  if constexpr (sizeof(InT) == 4) {
    simt::stv<N>((float *)p, v);
  } else {
#pragma unroll
    for (int j = 0; j < N; j += 2)
      *reinterpret_cast<__nv_bfloat162 *>(p + j) = __floats2bfloat162_rn(v[j], v[j + 1]);
  }
}

// ---------------------------------------------------------------- kernel 1
// Thread (warp w, lane (lm, ln)) owns rows 2 r0, 2 r0 + 1 (r0 = LM w + lm) and
// columns TN ln .. + TN of every 64-row product: the transposed chunk
// matrices are then read with contiguous rows (M^T's column pair is one
// 8-byte load).  Five phases a chunk: K dS, K dR, M2^T dOa, Mq^T dO | dX2 |
// Ap^T dVr and dR's update | dX | dS's update.  A transposed triangular
// product starts at its warp's first row.  Bound by the FMA pipe and the
// phases' latencies: B = 4, H = 16, T = 2048,
// d = 64 in 0.42 ms, B = 2, H = 8, T = 1000, d = 128 fp32 in 0.19 ms.
template <int DK, int DVS, int NT>
struct ChainSm {  // float offsets
  static constexpr int LDK = DK + 4;
  static constexpr int K = 0, Q = K + C * LDK, MAT = Q + C * LDK;  // MAT: 3 slots [C][C]
  static constexpr int S = MAT + 3 * C * C, R = S + DK * DVS, DO = R + DK * DVS;
  static constexpr int DOA = DO + C * DVS, T1 = DOA + C * DVS, T2 = T1 + C * DVS, T3 = T2 + C * DVS;
  static constexpr int VEC = T3 + C * DVS, FLOATS = VEC + 6 * C;
};

template <int DK, bool RDNV, typename InT, int DVS, int NT>
__global__ void __launch_bounds__(NT, NT == 128 ? 2 : 1) bwd_chain_kernel(BwdParams p) {
  using namespace simt;
  using SM = ChainSm<DK, DVS, NT>;
  constexpr int DV = DK, LDK = SM::LDK;
  constexpr int TN = 32 * DVS / NT, LN = DVS / TN, LM = 32 / LN, TMU = DK / 32;
  static_assert(LM * (NT / 32) == 32, "row pairs of 32");
  extern __shared__ __align__(16) float sm[];
  float *Ks = sm + SM::K, *Qs = sm + SM::Q, *Ss = sm + SM::S, *Rs = sm + SM::R;
  float *DO = sm + SM::DO, *DOA = sm + SM::DOA, *T1 = sm + SM::T1, *T2 = sm + SM::T2;
  float *T3 = sm + SM::T3, *vec = sm + SM::VEC;
  float *mat[3] = {sm + SM::MAT, sm + SM::MAT + C * C, sm + SM::MAT + 2 * C * C};

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int lm, ln;
  lane_mn<LN>(lane, lm, ln);
  const int r0 = LM * warp + lm, n0 = TN * ln;
  const int kw = 2 * LM * warp;  // the warp's first row
  const int H = p.f.H, sq = seq_at(p.f, blockIdx.x / H), h = blockIdx.x % H;
  const SeqSpan sp = seq_span(p.f, sq, h);
  const int j0 = blockIdx.y * DVS;
  const bool dec_res = p.f.mods & RDN_FLAG_DECAYED_RESIDUAL;
  const bool plain = p.f.mods & RDN_FLAG_PLAIN_COMBINE;
  const bool tnh = p.f.mods & RDN_FLAG_TANH_RESIDUAL;
  const bool stl = p.f.mods & RDN_FLAG_STATELESS_AUX;
  const bool rdn_aux = RDNV && !stl;  // the auxiliary pass runs the delta rule

  const size_t sbase = ((size_t)sq * H + h) * DK * DV;
  for (int e = tid; e < DK * DVS / 4; e += NT) {
    const size_t off = sbase + (size_t)(e / (DVS / 4)) * DV + j0 + 4 * (e % (DVS / 4));
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4 *>(Ss + 4 * e) = p.dST ? *reinterpret_cast<const float4 *>(p.dST + off) : z;
    *reinterpret_cast<float4 *>(Rs + 4 * e) = p.dRT ? *reinterpret_cast<const float4 *>(p.dRT + off) : z;
  }

  RowTile<InT, DK, NT> kt, qt;
  constexpr int VU = 6 * C / NT + (6 * C % NT != 0);
  float vr[VU], dor[2][TN], gmr[2], mkr[2][TN];  // mkr: the residual map's derivative
  auto fetch = [&](int c) {  // chunk c's K, Q, dO, gates and mask
    const int n = min(C, sp.len - c * C);
    const size_t row = (size_t)(sp.tok0 + c * C) * H + h;
    kt.fetch((const InT *)p.f.k + row * DK, (size_t)H * DK, n);
    qt.fetch((const InT *)p.f.q + row * DK, (size_t)H * DK, n);
    const float *rec = p.f.ws + (size_t)(sp.rbase + c) * kRecFloats;
#pragma unroll
    for (int u = 0; u < VU; ++u) {
      const int e = tid + u * NT;
      vr[u] = e <= V_GAMC ? rec[OFF_VEC + e] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int t = 2 * r0 + i;
#pragma unroll
      for (int j = 0; j < TN; ++j) dor[i][j] = 0.f;
      gmr[i] = 0.f;
      if (t < n) {
        ld_row<InT, TN>((const InT *)p.dO + (row + (size_t)t * H) * DV + j0 + n0, dor[i]);
        gmr[i] = plain ? 1.f : p.f.gamma[row + (size_t)t * H];
      }
      const size_t m = ((size_t)(sp.rbase + c) * C + t) * DV + j0 + n0;
      if (tnh) {
        ldv<TN>((const float *)p.f.sv_mask + m, mkr[i]);
      } else {
        const uint32_t b = ((const uint8_t *)p.f.sv_mask)[m >> 3] >> (n0 & 7);
#pragma unroll
        for (int j = 0; j < TN; ++j) mkr[i][j] = (b >> j) & 1 ? 1.f : 0.f;
      }
    }
  };
  auto mats = [&](int c) { return p.f.ws + (size_t)(sp.rbase + c) * kRecFloats; };
  const int last = sp.nc - 1;
  if (last >= 0) {
    fetch(last);
    cp_mat<NT>(mat[0], C, mats(last) + OFF_M2);
    cp_mat<NT>(mat[1], C, mats(last) + OFF_MQ);
    if (rdn_aux) cp_mat<NT>(mat[2], C, mats(last) + OFF_TG);
    cp_commit();
  }

  for (int c = last; c >= 0; --c) {
    const int n = min(C, sp.len - c * C);
    const size_t rec = (size_t)(sp.rbase + c);
    kt.put(Ks, LDK, 1.f);
    qt.put(Qs, LDK, p.f.scale);
#pragma unroll
    for (int u = 0; u < VU; ++u)
      if (tid + u * NT < 6 * C) vec[tid + u * NT] = vr[u];
    float dO[2][TN], mk[2][TN], gm[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float d[TN];
      gm[i] = gmr[i];
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        dO[i][j] = dor[i][j];
        mk[i][j] = mkr[i][j];
        d[j] = gm[i] * dO[i][j];
      }
      stv<TN>(DO + (2 * r0 + i) * DVS + n0, dO[i]);
      stv<TN>(DOA + (2 * r0 + i) * DVS + n0, d);
    }
    wait_groups<0>();  // M2, Mq, T_gamma
    __syncthreads();
    const float *Gam = vec + V_GAM, *Gprev = vec + V_GPREV, *wS = vec + V_WS, *wR = vec + V_WR;
    const float GamC = vec[V_GAMC];
    {  // the chunk-end gradients
      float *gs = p.gS + rec * DK * DV + j0, *gr = p.gR + rec * DK * DV + j0;
      for (int e = tid; e < DK * DVS / 4; e += NT) {
        const size_t off = (size_t)(e / (DVS / 4)) * DV + 4 * (e % (DVS / 4));
        *reinterpret_cast<float4 *>(gs + off) = *reinterpret_cast<const float4 *>(Ss + 4 * e);
        *reinterpret_cast<float4 *>(gr + off) = *reinterpret_cast<const float4 *>(Rs + 4 * e);
      }
    }
    // ---- K dS, K dR, M2^T dOa, Mq^T dO; dE2
    float kd[2][TN], x[2][TN], de[2][TN];
    {
      float kr[2][TN];
      zero(kd);
      zero(kr);
      zero(x);
      zero(de);
      mm_ak2<2, TN, 3, 3>(Ks + 2 * r0 * LDK, LDK, Ss + n0, Rs + n0, DVS, DK, kd, kr);
      mm_am<2, TN>(mat[0] + kw * C + 2 * r0, C, DOA + kw * DVS + n0, DVS, C - kw, x);
      mm_am<2, TN>(mat[1] + kw * C + 2 * r0, C, DO + kw * DVS + n0, DVS, C - kw, de);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = 2 * r0 + i;
#pragma unroll
        for (int j = 0; j < TN; ++j) x[i][j] += wR[t] * kr[i][j];
        if (rdn_aux) stv<TN>(T1 + t * DVS + n0, x[i]);
      }
    }
    __syncthreads();
    cp_mat<NT>(mat[0], C, mats(c) + OFF_AP);
    cp_commit();
    if (RDNV) cp_mat<NT>(mat[1], C, mats(c) + OFF_TB);
    cp_commit();
    // ---- dX2 = T_gamma^T dE2; dVr; dKR = -Gam dX2; dQR = Gam dOa
    if (rdn_aux) {
      zero(x);
      mm_am<2, TN>(mat[2] + kw * C + 2 * r0, C, T1 + kw * DVS + n0, DVS, C - kw, x);
    }
    float dvr[2][TN];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int t = 2 * r0 + i;
      const size_t off = (rec * C + t) * DV + j0 + n0;
      float a[TN], b[TN];
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        dvr[i][j] = x[i][j] * mk[i][j];
        a[j] = -Gam[t] * x[i][j];
        b[j] = Gam[t] * (gm[i] * dO[i][j]);
      }
      if (rdn_aux) {
        stv<TN>(p.dX2 + off, x[i]);
        stv<TN>(T2 + t * DVS + n0, a);
      }
      stv<TN>(p.dVr + off, dvr[i]);
      stv<TN>(T3 + t * DVS + n0, dvr[i]);
      stv<TN>(DOA + t * DVS + n0, b);
    }
    wait_groups<1>();  // Ap
    __syncthreads();
    if (c > 0 && rdn_aux) cp_mat<NT>(mat[2], C, mats(c - 1) + OFF_TG);
    cp_commit();
    // ---- dE = Mq^T dO - Ap^T dVr + wS K dS; dR = Gam_C dR + Q^T dQR + K^T dKR
    {
      zero(x);
      mm_am<2, TN>(mat[0] + kw * C + 2 * r0, C, T3 + kw * DVS + n0, DVS, C - kw, x);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = 2 * r0 + i;
#pragma unroll
        for (int j = 0; j < TN; ++j) x[i][j] = de[i][j] - x[i][j] + wS[t] * kd[i][j];
        if (RDNV) stv<TN>(T1 + t * DVS + n0, x[i]);
      }
      const int m0 = TMU * r0;
      float u[TMU][TN];
      zero(u);
      mm_am<TMU, TN>(Qs + m0, LDK, DOA + n0, DVS, C, u);
      if (rdn_aux) mm_am<TMU, TN>(Ks + m0, LDK, T2 + n0, DVS, C, u);
#pragma unroll
      for (int i = 0; i < TMU; ++i) {
        float s[TN];
        ldv<TN>(Rs + (m0 + i) * DVS + n0, s);
#pragma unroll
        for (int j = 0; j < TN; ++j) s[j] = stl ? 0.f : GamC * s[j] + u[i][j];
        stv<TN>(Rs + (m0 + i) * DVS + n0, s);
      }
    }
    wait_groups<1>();  // T_beta
    __syncthreads();
    if (c > 0) cp_mat<NT>(mat[0], C, mats(c - 1) + OFF_M2);
    cp_commit();
    // ---- dX = T_beta^T dE; dV = dVr + dX; dKS = -Gprev dVr - Gam dX; dQS = Gam dO
    if (RDNV) {
      zero(x);
      mm_am<2, TN>(mat[1] + kw * C + 2 * r0, C, T1 + kw * DVS + n0, DVS, C - kw, x);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int t = 2 * r0 + i;
      const float gp = dec_res ? Gam[t] : Gprev[t], gq = plain ? Gprev[t] : Gam[t];
      float a[TN], b[TN], v[TN];
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        v[j] = dvr[i][j] + x[i][j];
        a[j] = -gp * dvr[i][j] - (RDNV ? Gam[t] * x[i][j] : 0.f);
        b[j] = gq * dO[i][j];
      }
      if (RDNV || p.dv_late) stv<TN>(p.dX + (rec * C + t) * DV + j0 + n0, x[i]);
      if (t < n && !p.dv_late)
        st_row<InT, TN>((InT *)p.dv + ((size_t)(sp.tok0 + c * C + t) * H + h) * DV + j0 + n0, v);
      stv<TN>(T2 + t * DVS + n0, a);
      stv<TN>(DO + t * DVS + n0, b);
    }
    __syncthreads();
    if (c > 0) {
      cp_mat<NT>(mat[1], C, mats(c - 1) + OFF_MQ);
      fetch(c - 1);
    }
    cp_commit();
    {  // ---- dS = Gam_C dS + K^T dKS + Q^T dQS
      const int m0 = TMU * r0;
      float u[TMU][TN];
      zero(u);
      mm_am<TMU, TN>(Ks + m0, LDK, T2 + n0, DVS, C, u);
      mm_am<TMU, TN>(Qs + m0, LDK, DO + n0, DVS, C, u);
#pragma unroll
      for (int i = 0; i < TMU; ++i) {
        float s[TN];
        ldv<TN>(Ss + (m0 + i) * DVS + n0, s);
#pragma unroll
        for (int j = 0; j < TN; ++j) s[j] = GamC * s[j] + u[i][j];
        stv<TN>(Ss + (m0 + i) * DVS + n0, s);
      }
    }
    __syncthreads();
  }
  __syncthreads();
  for (int e = tid; e < DK * DVS / 4; e += NT) {
    const size_t off = sbase + (size_t)(e / (DVS / 4)) * DV + j0 + 4 * (e % (DVS / 4));
    if (p.dS0) *reinterpret_cast<float4 *>(p.dS0 + off) = *reinterpret_cast<const float4 *>(Ss + 4 * e);
    if (p.dR0) *reinterpret_cast<float4 *>(p.dR0 + off) = *reinterpret_cast<const float4 *>(Rs + 4 * e);
  }
}

// ---------------------------------------------------------------- kernel 2
// One CTA of 256 threads per chunk.  Thread (ty, tx) owns rows 4 ty .. 4 ty + 3
// and columns tx + 16 j of every product, so a row's sums are shuffles among
// 16 lanes of a warp.  Every value-dimension product is A B^T with
// both operands' rows contiguous (mm_nt); the value dimension is walked in
// slices of JS columns, the next slice's tiles arriving by cp.async while the
// current one is used: first the auxiliary pass (dO, E2, dX2 against R0, dR and
// E2), then the base pass (dO, E, dVr, dX against S0, dS and E).
// The per-row gate sums need no read-outs K S0, Q R0, ...: a row's
// sum_j dKS KS is its k's product with the row of dKS S0^T, which dK takes
// anyway.  kk, qk and the C x C gradients stay in shared memory at the
// positions their thread owns.  Bound by the FMA pipe (two FMAs an
// instruction): the same calls in 0.57 and 0.27 ms.  One kernel that walked
// the chunks with every product, adding its column slices' shares atomically,
// and a finishing pass took 6.19 and 1.85 ms for what the chain and this do in
// 0.99 and 0.46.
constexpr int kPostThreads = 256;
template <int DK>
struct PostSm {  // float offsets
  static constexpr int JS = 2048 / DK, LDJ = JS + 4, LDK = DK + 4, LDC = C + 4;
  static constexpr int STG = (4 * C + 2 * DK) * LDJ;  // a slice's tiles
  static constexpr int K = 0, Q = K + C * LDK, KK = Q + C * LDK, QK = KK + C * LDC;
  static constexpr int DKK = QK + C * LDC, DQK = DKK + C * LDC, ST = DQK + C * LDC;
  static constexpr int VEC = ST + 2 * STG, FLOATS = VEC + 15 * C;
  static_assert(FLOATS * 4 <= 232448, "one CTA's shared memory");
};

template <int DK, bool RDNV, typename InT>
__global__ void __launch_bounds__(kPostThreads, 1) bwd_post_kernel(BwdParams p) {
  using namespace simt;
  using SM = PostSm<DK>;
  constexpr int DV = DK, JS = SM::JS, LDJ = SM::LDJ, LDK = SM::LDK, LDC = SM::LDC;
  constexpr int NH = DK / 64, NSL = DV / JS, NT = kPostThreads;
  extern __shared__ __align__(16) float sm[];
  float *Ks = sm + SM::K, *Qs = sm + SM::Q, *KK = sm + SM::KK, *QK = sm + SM::QK;
  float *DKK = sm + SM::DKK, *DQK = sm + SM::DQK;
  Cum &cum = *reinterpret_cast<Cum *>(sm + SM::VEC);
  float *bet = sm + SM::VEC + 4 * C, *gam = bet + C, *Gam = gam + C, *Gprev = Gam + C;
  float *wS = Gprev + C, *wR = wS + C, *dcum = wR + C, *dcprev = dcum + C, *dout = dcprev + C;
  float *dwS = dout + C, *dwR = dwS + C;

  const long long chunk = blockIdx.x;
  if (chunk >= total_records(p.f)) return;  // (packed sequences: the grid is a bound)
  const int H = p.f.H;
  int sq, h, c;
  rec_decode(p.f, chunk, sq, h, c);
  const SeqSpan sp = seq_span(p.f, sq, h);
  const int n = min(C, sp.len - c * C);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = lane >> 1, ty = 2 * warp + (lane & 1);
  const bool dec_res = p.f.mods & RDN_FLAG_DECAYED_RESIDUAL;
  const bool plain = p.f.mods & RDN_FLAG_PLAIN_COMBINE;
  const bool stl = p.f.mods & RDN_FLAG_STATELESS_AUX;
  const bool rdn_aux = RDNV && !stl;
  const size_t row0 = (size_t)(sp.tok0 + c * C) * H + h;
  const size_t toff = (size_t)chunk * C * DV, soff = (size_t)chunk * DK * DV;

  // tiles of a slice: dO, then three [C] tiles and two [DK] tiles
  auto tile = [&](int s, int i) {
    return sm + SM::ST + (s & 1) * SM::STG + (i < 4 ? i * C : 4 * C + (i - 4) * DK) * LDJ;
  };
  RowTile<InT, JS, NT> dot;
  auto issue = [&](int s) {
    const bool base = s >= NSL;
    const int j = (s % NSL) * JS;
    dot.fetch((const InT *)p.dO + row0 * DV + j, (size_t)H * DV, n);
    const float *src[3] = {base ? (const float *)p.f.sv_E : (const float *)p.f.sv_E2,
                           base ? (RDNV ? p.dX : nullptr) : (rdn_aux ? p.dX2 : nullptr),
                           base ? p.dVr : nullptr};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (!src[i]) continue;
      float *d = tile(s, 1 + i);
      for (int e = tid; e < C * JS / 4; e += NT)
        cp16(d + (e / (JS / 4)) * LDJ + 4 * (e % (JS / 4)),
             src[i] + toff + (size_t)(e / (JS / 4)) * DV + j + 4 * (e % (JS / 4)));
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float *g = base ? (i ? p.gS : p.Sc) : (i ? p.gR : p.Rc);
      float *d = tile(s, 4 + i);
      for (int e = tid; e < DK * JS / 4; e += NT)
        cp16(d + (e / (JS / 4)) * LDJ + 4 * (e % (JS / 4)),
             g + soff + (size_t)(e / (JS / 4)) * DV + j + 4 * (e % (JS / 4)));
    }
    cp_commit();
  };

  issue(0);
  {
    RowTile<InT, DK, NT> kt, qt;
    kt.fetch((const InT *)p.f.k + row0 * DK, (size_t)H * DK, n);
    qt.fetch((const InT *)p.f.q + row0 * DK, (size_t)H * DK, n);
    if (warp == 0) {
      float g2[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int t = lane + 32 * u;
        const bool ok = t < n;
        const size_t go = row0 + (size_t)(ok ? t : 0) * H;
        g2[u] = ok ? p.f.g[go] : 0.f;
        bet[t] = ok ? p.f.beta[go] : 0.f;
        gam[t] = ok ? p.f.gamma[go] : 0.f;
      }
      cum64(g2[0], g2[1], cum);
    } else if (warp < 3) {
      const float *rec = p.f.ws + (size_t)chunk * kRecFloats + OFF_VEC;
      const int t = tid - 32;
      Gam[t] = rec[V_GAM + t];
      Gprev[t] = rec[V_GPREV + t];
      wS[t] = rec[V_WS + t];
      wR[t] = rec[V_WR + t];
    }
    kt.put(Ks, LDK, 1.f);
    qt.put(Qs, LDK, p.f.scale);
    dot.put(tile(0, 0), LDJ, 1.f);
  }
  wait_groups<0>();
  __syncthreads();
  {
    float a[4][4];
    mm_nt<4, 4, DK>(Ks + 4 * ty * LDK, LDK, Ks + tx * LDK, 16 * LDK, a);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) KK[(4 * ty + i) * LDC + tx + 16 * j] = a[i][j];
    mm_nt<4, 4, DK>(Qs + 4 * ty * LDK, LDK, Ks + tx * LDK, 16 * LDK, a);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) QK[(4 * ty + i) * LDC + tx + 16 * j] = a[i][j];
  }

  float dk[4][4 * NH], dq[4][4 * NH];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4 * NH; ++j) dk[i][j] = dq[i][j] = 0.f;
  // per-row partial sums over this thread's columns: gradients w.r.t. the
  // cumulative decay to t and to t - 1, dgamma of the read-out, dwS, dwR;
  // per-column sums over its rows: decay, dbeta, dgamma; <dS, S0> + <dR, R0>
  float pc[4] = {0.f, 0.f, 0.f, 0.f}, pp[4] = {0.f, 0.f, 0.f, 0.f}, po[4] = {0.f, 0.f, 0.f, 0.f};
  float ps[4] = {0.f, 0.f, 0.f, 0.f}, pr[4] = {0.f, 0.f, 0.f, 0.f};
  float cg[4] = {0.f, 0.f, 0.f, 0.f}, cb[4] = {0.f, 0.f, 0.f, 0.f}, cm[4] = {0.f, 0.f, 0.f, 0.f};
  float dgc = 0.f;

  // acc_t += f_t (X St^T)_t over the slice, and s_t += (rows_t . (X St^T)_t)
  auto state_mm = [&](const float *X, const float *St, const float *rows, const float (&f)[4],
                      float (&acc)[4][4 * NH], float (&s)[4]) {
#pragma unroll
    for (int hb = 0; hb < NH; ++hb) {
      float a[4][4];
      mm_nt<4, 4, JS>(X + 4 * ty * LDJ, LDJ, St + (64 * hb + tx) * LDJ, 16 * LDJ, a);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          s[i] = fmaf(rows[(4 * ty + i) * LDK + 64 * hb + tx + 16 * j], a[i][j], s[i]);
          acc[i][4 * hb + j] = fmaf(f[i], a[i][j], acc[i][4 * hb + j]);
        }
    }
  };
  auto add_nt = [&](const float *X, const float *Y, float (&g)[4][4]) {
    float a[4][4];
    mm_nt<4, 4, JS>(X + 4 * ty * LDJ, LDJ, Y + tx * LDJ, 16 * LDJ, a);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) g[i][j] += a[i][j];
  };
  auto state_dot = [&](const float *A, const float *B) {
    for (int e = tid; e < DK * JS / 4; e += NT) {
      const int o = (e / (JS / 4)) * LDJ + 4 * (e % (JS / 4));
      float a[4], b[4];
      ldv<4>(A + o, a);
      ldv<4>(B + o, b);
#pragma unroll
      for (int i = 0; i < 4; ++i) dgc = fmaf(a[i], b[i], dgc);
    }
  };

  {  // ---- the auxiliary pass
    float g1[4][4], g2[4][4], s1[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
    zero(g1);
    zero(g2);
    float fq[4], fk[4], fr[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = 4 * ty + i;
      fq[i] = plain ? Gam[t] : gam[t] * Gam[t];
      fk[i] = -Gam[t];
      fr[i] = wR[t];
    }
    for (int s = 0; s < NSL; ++s) {
      issue(s + 1);
      const float *dO = tile(s, 0), *e2 = tile(s, 1), *x2 = tile(s, 2), *r0 = tile(s, 4), *dr = tile(s, 5);
      if (!stl) {
        state_mm(dO, r0, Qs, fq, dq, s1);
        state_dot(dr, r0);
      }
      state_mm(e2, dr, Ks, fr, dk, pr);
      add_nt(dO, e2, g1);
      if (rdn_aux) {
        state_mm(x2, r0, Ks, fk, dk, s2);
        add_nt(x2, e2, g2);
      }
      dot.put(tile(s + 1, 0), LDJ, 1.f);
      wait_groups<0>();
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = 4 * ty + i;
      pc[i] = fq[i] * s1[i] - Gam[t] * s2[i];
      if (!plain) po[i] = Gam[t] * s1[i];
      if (stl) pr[i] = 0.f;  // (wR is then a constant)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int u = tx + 16 * j;
        float dkk = 0.f, dqk = 0.f;
        if (u <= t) {
          const float dec = expf(cum.to(t, u));
          const float kk = KK[t * LDC + u], qk = QK[t * LDC + u], gu = gam[u];
          const float dm = plain ? g1[i][j] : gam[t] * g1[i][j];  // dM2
          if (stl) {  // M2 = diag(QK): no decay, no rate
            if (u == t) {
              dqk = dm;
              if (!plain) po[i] = fmaf(qk, g1[i][j], po[i]);
            }
          } else {
            const float m = dec * qk;
            if (!plain) po[i] = fmaf(m * gu, g1[i][j], po[i]);
            const float G = dm * m * gu;
            pc[i] += G;
            cg[j] += G;
            cm[j] = fmaf(dm, m, cm[j]);
            dqk = dm * dec * gu;
            if (rdn_aux && u < t) {  // A_gamma
              const float da = -g2[i][j], Gg = da * dec * gu * kk;
              pc[i] += Gg;
              cg[j] += Gg;
              cm[j] = fmaf(da * dec, kk, cm[j]);
              dkk = da * dec * gu;
            }
          }
        }
        DKK[t * LDC + u] = dkk;
        DQK[t * LDC + u] = dqk;
      }
    }
  }
  {  // ---- the base pass
    float g3[4][4], g4[4][4], g5[4][4];
    float s4[4] = {0.f, 0.f, 0.f, 0.f}, s5[4] = {0.f, 0.f, 0.f, 0.f}, s6[4] = {0.f, 0.f, 0.f, 0.f};
    zero(g3);
    zero(g4);
    zero(g5);
    float fq[4], fp[4], fk[4], fs[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = 4 * ty + i;
      fq[i] = plain ? Gprev[t] : Gam[t];
      fp[i] = dec_res ? -Gam[t] : -Gprev[t];
      fk[i] = -Gam[t];
      fs[i] = wS[t];
    }
    for (int s = NSL; s < 2 * NSL; ++s) {
      if (s + 1 < 2 * NSL) issue(s + 1);
      const float *dO = tile(s, 0), *e = tile(s, 1), *dx = tile(s, 2), *dvr = tile(s, 3);
      const float *s0 = tile(s, 4), *ds = tile(s, 5);
      state_mm(dO, s0, Qs, fq, dq, s4);
      state_mm(dvr, s0, Ks, fp, dk, s5);
      if (RDNV) state_mm(dx, s0, Ks, fk, dk, s6);
      state_mm(e, ds, Ks, fs, dk, ps);
      state_dot(ds, s0);
      add_nt(dO, e, g3);
      add_nt(dvr, e, g4);
      if (RDNV) add_nt(dx, e, g5);
      if (s + 1 < 2 * NSL) {
        dot.put(tile(s + 1, 0), LDJ, 1.f);
        wait_groups<0>();
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = 4 * ty + i;
      (plain ? pp : pc)[i] += fq[i] * s4[i];
      (dec_res ? pc : pp)[i] += fp[i] * s5[i];
      if (RDNV) pc[i] += fk[i] * s6[i];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int u = tx + 16 * j;
        if (u < t) {
          const float dec = expf(cum.to(t, u)), decp = expf(cum.before(t, u));
          const float kk = KK[t * LDC + u], qk = QK[t * LDC + u], bu = bet[u];
          float dkk = DKK[t * LDC + u];
          {  // Ap: previous-token decay (decayed residual: to t)
            const float dA = dec_res ? dec : decp, dm = -g4[i][j], G = dm * dA * bu * kk;
            (dec_res ? pc : pp)[i] += G;
            cg[j] += G;
            cb[j] = fmaf(dm * dA, kk, cb[j]);
            dkk = fmaf(dm * dA, bu, dkk);
          }
          {  // Mq (plain combine: decay to t - 1)
            const float dA = plain ? decp : dec, dm = g3[i][j], G = dm * dA * bu * qk;
            (plain ? pp : pc)[i] += G;
            cg[j] += G;
            cb[j] = fmaf(dm * dA, qk, cb[j]);
            DQK[t * LDC + u] += dm * dA * bu;
          }
          if (RDNV) {  // A_beta
            const float da = -g5[i][j], Gb = da * dec * bu * kk;
            pc[i] += Gb;
            cg[j] += Gb;
            cb[j] = fmaf(da * dec, kk, cb[j]);
            dkk = fmaf(da * dec, bu, dkk);
          }
          // both halves of the symmetric d(KK^T) (its diagonal is zero)
          DKK[t * LDC + u] = dkk;
          DKK[u * LDC + t] = dkk;
        }
      }
    }
  }
  if (p.dv_late)  // (every dO of this chunk has been read)
    for (int e = tid; e < n * DV / 4; e += NT) {
      const int t = e / (DV / 4), j = 4 * (e % (DV / 4));
      float v[4], x[4];
      ldv<4>(p.dVr + toff + t * DV + j, v);
      ldv<4>(p.dX + toff + t * DV + j, x);
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] += x[i];
      st_row<InT, 4>((InT *)p.dv + (row0 + (size_t)t * H) * DV + j, v);
    }
  // ---- row sums over a row's 16 lanes, column sums over the block
  float *colp = sm + SM::ST;  // [8 warps][3][C], then the warps' dgc
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int o = 16; o > 1; o >>= 1) {
      pc[i] += __shfl_xor_sync(0xffffffffu, pc[i], o);
      pp[i] += __shfl_xor_sync(0xffffffffu, pp[i], o);
      po[i] += __shfl_xor_sync(0xffffffffu, po[i], o);
      ps[i] += __shfl_xor_sync(0xffffffffu, ps[i], o);
      pr[i] += __shfl_xor_sync(0xffffffffu, pr[i], o);
    }
    if (tx == 0) {
      const int t = 4 * ty + i;
      dcum[t] = pc[i];
      dcprev[t] = pp[i];
      dout[t] = po[i];
      dwS[t] = ps[i];
      dwR[t] = pr[i];
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    cg[j] += __shfl_xor_sync(0xffffffffu, cg[j], 1);
    cb[j] += __shfl_xor_sync(0xffffffffu, cb[j], 1);
    cm[j] += __shfl_xor_sync(0xffffffffu, cm[j], 1);
    if ((lane & 1) == 0) {
      colp[(warp * 3 + 0) * C + tx + 16 * j] = cg[j];
      colp[(warp * 3 + 1) * C + tx + 16 * j] = cb[j];
      colp[(warp * 3 + 2) * C + tx + 16 * j] = cm[j];
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) dgc += __shfl_xor_sync(0xffffffffu, dgc, o);
  if (lane == 0) colp[24 * C + warp] = dgc;
  __syncthreads();
  if (warp == 0) {  // the gates' gradients, lane l for tokens l and 32 + l
    float a[2], b[2], dg2 = 0.f, ends = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) dg2 += colp[24 * C + w];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int t = lane + 32 * u;
      float sg = 0.f, sb = 0.f, sg2 = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        sg += colp[(w * 3 + 0) * C + t];
        sb += colp[(w * 3 + 1) * C + t];
        sg2 += colp[(w * 3 + 2) * C + t];
      }
      const float eC = expf(cum.to(C - 1, t));
      const float we = (dwS[t] * bet[t] + dwR[t] * gam[t]) * eC;
      ends += we;
      a[u] = dcum[t] - sg - we;
      b[u] = dcprev[t];
      if (t < n) {
        const size_t off = row0 + (size_t)t * H;
        p.dbeta[off] = sb + dwS[t] * eC;
        p.dgamma[off] = sg2 + dout[t] + dwR[t] * eC;
      }
    }
    // the chunk-end terms land on the last token (padding has g = 0)
#pragma unroll
    for (int o = 16; o; o >>= 1) ends += __shfl_xor_sync(0xffffffffu, ends, o);
    if (lane == 31) a[1] += ends + dg2 * expf(cum.hi[C - 1]);
    // dg_s = sum_{t >= s} dcum_t + sum_{t > s} dcprev_t: suffix sums
    float x0 = a[0] + b[0], x1 = a[1] + b[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float y0 = __shfl_down_sync(0xffffffffu, x0, o), y1 = __shfl_down_sync(0xffffffffu, x1, o);
      if (lane + o < 32) {
        x0 += y0;
        x1 += y1;
      }
    }
    x0 += __shfl_sync(0xffffffffu, x1, 0);
    if (lane < n) p.dg[row0 + (size_t)lane * H] = x0 - b[0];
    if (lane + 32 < n) p.dg[row0 + (size_t)(lane + 32) * H] = x1 - b[1];
  }
  // ---- dk += (dKK + dKK^T) K + dQK^T Q;  dq += dQK K
#pragma unroll 1
  for (int hb = 0; hb < NH; ++hb) {
    float ak[4][4], aq[4][4];
    zero(ak);
    zero(aq);
#pragma unroll 1
    for (int k = 0; k < C; k += 4) {
      float s[4][4], q4[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        ldv<4>(DKK + (4 * ty + i) * LDC + k, s[i]);
        ldv<4>(DQK + (4 * ty + i) * LDC + k, q4[i]);
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        float m[4];  // row k of dQK: dQK^T's column
        ldv<4>(DQK + (k + kk) * LDC + 4 * ty, m);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int o = (k + kk) * LDK + 64 * hb + tx + 16 * j;
          const float kv = Ks[o], qv = Qs[o];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            ak[i][j] = fmaf(s[i][kk], kv, ak[i][j]);
            ak[i][j] = fmaf(m[i], qv, ak[i][j]);
            aq[i][j] = fmaf(q4[i][kk], kv, aq[i][j]);
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = 4 * ty + i;
      if (t >= n) continue;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const size_t off = (row0 + (size_t)t * H) * DK + 64 * hb + tx + 16 * j;
        const float gk = (NH == 1 || hb == 0 ? dk[i][j] : dk[i][4 * (NH - 1) + j]) + ak[i][j];
        const float gq = p.f.scale * ((NH == 1 || hb == 0 ? dq[i][j] : dq[i][4 * (NH - 1) + j]) + aq[i][j]);
        if (p.gq32) {
          p.gk32[off] = gk;
          p.gq32[off] = gq;
        } else {
          ((InT *)p.dk)[off] = from_f32<InT>(gk);
          ((InT *)p.dq)[off] = from_f32<InT>(gq);
        }
      }
    }
  }
}

template <int DK, bool RDNV, typename InT, int DVS, int NT>
cudaError_t launch_chain_t(const BwdParams &p, cudaStream_t s) {
  auto chain = bwd_chain_kernel<DK, RDNV, InT, DVS, NT>;
  constexpr int smem = (int)sizeof(float) * ChainSm<DK, DVS, NT>::FLOATS;
  const cudaError_t e = cudaFuncSetAttribute(chain, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  RDN_LAUNCH("bwd_chain_f32", s, chain<<<dim3(p.f.nseq * p.f.H, DK / DVS), NT, smem, s>>>(p));
  return cudaGetLastError();
}

struct RunBwd {
  const BwdParams &p;
  cudaStream_t s;
  template <int DK, bool RDNV, typename InT>
  cudaError_t run() const {
    int nsm = 0;
    cudaError_t e = sm_count(&nsm);
    if (e != cudaSuccess) return e;
    const int dvs = scan_columns(DK, (long long)p.f.nseq * p.f.H, nsm);
    if constexpr (DK == 64) {
      e = dvs == 16 ? launch_chain_t<64, RDNV, InT, 16, 128>(p, s)
                    : launch_chain_t<64, RDNV, InT, 8, 128>(p, s);
    } else {
      e = dvs == 32   ? launch_chain_t<128, RDNV, InT, 32, 256>(p, s)
          : dvs == 16 ? launch_chain_t<128, RDNV, InT, 16, 256>(p, s)
                      : launch_chain_t<128, RDNV, InT, 8, 256>(p, s);
    }
    if (e != cudaSuccess) return e;
    auto post = bwd_post_kernel<DK, RDNV, InT>;
    constexpr int smem = (int)sizeof(float) * PostSm<DK>::FLOATS;
    if ((e = cudaFuncSetAttribute(post, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess)
      return e;
    RDN_LAUNCH("bwd_post_f32", s, post<<<(unsigned)p.f.nrec, kPostThreads, smem, s>>>(p));
    return cudaGetLastError();
  }
};

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct BwdLayout {
  size_t prep, chain, saved, states, o, tc, qk, g32, tied, seq, total;
};

// bf16 inputs with d = 128 take the tensor-core backward (RDN, RLA with identity T
// matrices in its records, and every variant flag), all else the fp32 one
bool use_tc_bwd(const rdn_fwd_args &f, int variant) {
  (void)variant;
  return fwd_uses_tc(f.Dk, f.dtype == RDN_BF16);
}

// The forward's per-chunk records are valid input when the caller passes the
// forward's workspace with its chunk-start states (the forward wrote them in
// the format this backward reads: both choose their kernels by fwd_uses_tc).
bool reuse_fwd_records(const rdn_fwd_args &f) { return f.workspace && f.S_chunks; }

// ... and E, E2 and the mask (RDN_FLAG_SAVE_FOR_BWD) with them
bool fwd_saved(const rdn_fwd_args &f) {
  return reuse_fwd_records(f) && (f.flags & RDN_FLAG_SAVE_FOR_BWD);
}

BwdLayout layout(const rdn_bwd_args &a, int variant) {
  const rdn_fwd_args &f = a.fwd;
  const bool tc = use_tc_bwd(f, variant);
  const long long nrec = call_records(f);  // record slots
  BwdLayout l;
  // the forward's records are read from its workspace when it is passed
  l.prep = reuse_fwd_records(f) ? 0 : align256(sizeof(float) * nrec * kRecFloats);
  // what the fp32 chain keeps of each chunk (the tensor-core kernels': l.tc): RDN's
  // dX2, dVr, dX, the chunk-end gradients
  l.chain = tc ? 0 : align256(sizeof(float) * nrec * ((variant ? 3 : 2) * C * f.Dv + 2 * f.Dk * f.Dv));
  // E, E2 and the residual's mask, unless the forward kept them
  l.saved = tc || fwd_saved(f) ? 0 : align256(saved_layout(f).bytes);
  const bool need_states = f.S_chunks == nullptr;
  l.states = need_states ? align256(sizeof(float) * nrec * f.Dk * f.Dv) : 0;  // each of S, R
  const size_t esz = f.dtype == RDN_BF16 ? 2 : 4;
  // (a forward run here writes its o, which nobody reads, where the fp32 chain's
  // first rows go later: a record's 64 rows of Dv floats hold its tokens')
  l.o = need_states && tc ? align256(esz * (size_t)f.B * f.T * f.H * f.Dv) : 0;
  l.tc = tc ? align256(bwd_tc_extra_bytes(nrec, f.flags & RDN_FLAG_TANH_RESIDUAL)) : 0;
  // normalised q, k (RDN_FLAG_QK_NORM), unless the forward's workspace has them
  l.qk = reuse_fwd_records(f) ? 0 : align256(qk_norm_bytes(f));
  // and, with bf16 inputs, dq, dk (w.r.t. the normalised q, k) in fp32 for
  // the normalisation's backward: its projection (dy - y <y, dy>) would
  // otherwise start from bf16-rounded dy
  l.g32 = (f.flags & RDN_FLAG_QK_NORM) && f.dtype == RDN_BF16
              ? align256(2 * sizeof(float) * (size_t)f.B * f.T * f.H * f.Dk)
              : 0;
  l.seq = seq_table_bytes(f);
  // tied gates without a dgamma buffer: the gamma part is made here, then added
  l.tied = (f.flags & RDN_FLAG_TIED_GAMMA) && !a.dgamma
               ? align256(sizeof(float) * (size_t)f.B * f.T * f.H)
               : 0;
  // + the packed-sequence table and a 256-byte tail
  l.total = l.prep + l.chain + l.saved + 2 * l.states + l.o + l.tc + l.qk + l.g32 + l.tied + l.seq + 256;
  return l;
}

}  // namespace

BwdPlan plan_bwd(const rdn_bwd_args &a, int variant) {
  if (a.fwd.T == 0) return BwdPlan{0};
  return BwdPlan{layout(a, variant).total};
}

static __global__ void add_inplace_kernel(float *__restrict__ a, const float *__restrict__ b,
                                          size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    a[i] += b[i];
}

static cudaError_t launch_bwd_impl(const rdn_bwd_args &a, int variant, cudaStream_t s);

cudaError_t launch_bwd(const rdn_bwd_args &a0, int variant, cudaStream_t s) {
  const rdn_fwd_args &f = a0.fwd;
  if (!(f.flags & RDN_FLAG_TIED_GAMMA) || f.T == 0) return launch_bwd_impl(a0, variant, s);
  // tied gates (gamma is beta): the untied gradients, then dbeta += dgamma
  rdn_bwd_args a = a0;
  const BwdLayout l = layout(a0, variant);
  // (after what the untied backward uses: its own plan is l.total - l.tied bytes)
  if (!a.dgamma) a.dgamma = (float *)((char *)a.workspace + l.total - l.tied);
  cudaError_t e = launch_bwd_impl(a, variant, s);
  if (e != cudaSuccess) return e;
  const size_t n = (size_t)f.B * f.T * f.H;
  const unsigned grid = (unsigned)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  RDN_LAUNCH("tied_gate_grad", s, add_inplace_kernel<<<grid, 256, 0, s>>>(a.dbeta, a.dgamma, n));
  return cudaGetLastError();
}

static cudaError_t launch_bwd_impl(const rdn_bwd_args &a, int variant, cudaStream_t s) {
  const rdn_fwd_args &f = a.fwd;
  const size_t sbytes = sizeof(float) * (size_t)call_seqs(f) * f.H * f.Dk * f.Dv;
  if (f.T == 0) {  // no tokens: the initial-state gradients are the upstream ones
    cudaError_t e = cudaSuccess;
    if (a.dS0) e = a.dST ? cudaMemcpyAsync(a.dS0, a.dST, sbytes, cudaMemcpyDeviceToDevice, s)
                         : cudaMemsetAsync(a.dS0, 0, sbytes, s);
    if (e == cudaSuccess && a.dR0)
      e = a.dRT ? cudaMemcpyAsync(a.dR0, a.dRT, sbytes, cudaMemcpyDeviceToDevice, s)
                : cudaMemsetAsync(a.dR0, 0, sbytes, s);
    return e;
  }
  const BwdLayout l = layout(a, variant);
  char *ws = (char *)a.workspace;
  BwdParams p;
  p.f = make_fwd_params(f);
  // fp32 results (RDN_FLAG_F32_OUT in fwd.flags) are the backward's dq, dk, dv;
  // a forward recomputed here keeps its o in fwd.dtype
  const bool grad_f32 = p.f.f32out != 0;
  p.f.f32out = 0;
  p.f.inject = fault_injection() == 4 ? 2 : 0;
  const bool reuse = reuse_fwd_records(f);
  p.f.ws = reuse ? (float *)f.workspace : (float *)ws;
  p.f.err = status_word();
  if (f.cu_seqlens) {  // this call's own copy of the packed-sequence table
    long long *seq = (long long *)(ws + l.total - 256 - l.seq);
    cudaError_t e = launch_seq_table(f, variant, true, seq, s);
    if (e != cudaSuccess) return e;
    p.f.seq = seq;
  }
  if (p.f.qk_norm)  // the normalised q, k: the forward's, or made with this call's records
    set_qk_norm_copies(p.f, f, reuse ? (char *)f.workspace + qk_norm_offset(f)
                                     : ws + l.prep + l.chain + l.saved + 2 * l.states + l.o + l.tc);
  const bool saved = fwd_saved(f);
  if (saved || l.saved) {  // E, E2 and the mask: kept by the forward, or made here
    const SavedLayout sl = saved_layout(f);
    char *base = saved ? (char *)f.workspace : ws + l.prep + l.chain - sl.e;
    p.f.sv_E = (uint8_t *)base + sl.e;
    p.f.sv_E2 = (uint8_t *)base + sl.e2;
    p.f.sv_mask = (unsigned long long *)(base + sl.mask);
  }
  p.f.ST = p.f.RT = nullptr;
  const bool bf = f.dtype == RDN_BF16;
  const bool rdnv = variant == 1;
  const bool tc = use_tc_bwd(f, variant);
  cudaError_t e = cudaSuccess;  // (nothing to launch first when both the states and records are reused)
  if (f.S_chunks == nullptr) {  // recompute the chunk-start states
    p.f.S_chunks = (float *)(ws + l.prep + l.chain + l.saved);
    p.f.R_chunks = (float *)(ws + l.prep + l.chain + l.saved + l.states);
    p.f.o = tc ? ws + l.prep + l.chain + l.saved + 2 * l.states : ws + l.prep;
    e = launch_fwd_parts(p.f, f.Dk, rdnv, bf, s);
  } else if (!reuse) {
    e = launch_prep(p.f, f.Dk, rdnv, bf, s);
  }
  // chunk-start states without the forward's intermediates: remake them chunk
  // by chunk (a forward run above wrote them as it went)
  if (e == cudaSuccess && !tc && f.S_chunks && !saved) e = launch_recompute(p.f, f.Dk, rdnv, bf, s);
  if (e != cudaSuccess) return e;
  p.Sc = p.f.S_chunks;
  p.Rc = p.f.R_chunks;
  p.dX2 = (float *)(ws + l.prep);
  p.dVr = p.dX2 + (rdnv ? (size_t)p.f.nrec * C * f.Dv : 0);
  p.dX = p.dVr + (size_t)p.f.nrec * C * f.Dv;
  p.gS = p.dX + (size_t)p.f.nrec * C * f.Dv;
  p.gR = p.gS + (size_t)p.f.nrec * f.Dk * f.Dv;
  p.dO = a.dO;
  p.dST = a.dST;
  p.dRT = a.dRT;
  p.dq = a.dq;
  p.dk = a.dk;
  p.dv = a.dv;
  p.dv_late = a.dv == a.dO;
  p.dg = a.dg;
  p.dbeta = a.dbeta;
  p.dgamma = a.dgamma;
  p.dS0 = a.dS0;
  p.dR0 = a.dR0;
  p.gq32 = p.gk32 = nullptr;
  if (l.g32) {
    p.gq32 = (float *)(ws + l.prep + l.chain + l.saved + 2 * l.states + l.o + l.tc + l.qk);
    p.gk32 = p.gq32 + (size_t)f.B * f.T * f.H * f.Dk;
  }
  if (tc) {  // (with the normalisation: dq, dk into the fp32 copies, as fp32 results)
    e = launch_bwd_tc(p.f, a.dO, a.dST, a.dRT, p.Sc, p.Rc, p.gq32 ? p.gq32 : a.dq,
                      p.gk32 ? p.gk32 : a.dk, a.dv, a.dg, a.dbeta, a.dgamma, a.dS0, a.dR0,
                      ws + l.prep + l.chain + l.saved + 2 * l.states + l.o, !rdnv, grad_f32,
                      p.gq32 != nullptr, s);
  } else {
    e = simt_dispatch(f.Dk, rdnv, bf, RunBwd{p, s});
  }
  if (e != cudaSuccess || !p.f.qk_norm) return e;
  // dq, dk w.r.t. the caller's x: the normalisation's transposed Jacobian, in place
  rdn_prologue_args pa{};
  pa.rows = (long long)f.B * f.T * f.H;
  pa.D = f.Dk;
  pa.dtype = f.dtype;
  pa.eps = f.qk_eps;
  pa.x[0] = f.q;
  pa.x[1] = f.k;
  pa.dx[0] = a.dq;
  pa.dx[1] = a.dk;
  if (p.gq32) {  // from the fp32 copies
    pa.dy[0] = p.gq32;
    pa.dy[1] = p.gk32;
    return launch_prologue_bwd_f32dy(pa, grad_f32, s);
  }
  pa.dy[0] = a.dq;
  pa.dy[1] = a.dk;
  return launch_prologue(pa, true, s);
}

}  // namespace rdn
