// chunk_common.cuh -- what the chunkwise forward and backward share: the layout
// of the per-chunk records, their parameters, packed sequences, and the rules
// that choose a kernel.
#pragma once
#include "common.cuh"

namespace rdn {

constexpr int C = kChunk;
constexpr int kThreads = 256;

// Per-chunk workspace record written by chunk_prep (floats).
constexpr int kCC = C * C;
constexpr int OFF_TB = 0, OFF_TG = kCC, OFF_AP = 2 * kCC, OFF_MQ = 3 * kCC, OFF_M2 = 4 * kCC;
constexpr int OFF_VEC = 5 * kCC;
// vectors: Gam, Gprev, alpha, wS, wR, then GamC at [5*C]
constexpr int V_GAM = 0, V_GPREV = C, V_ALPHA = 2 * C, V_WS = 3 * C, V_WR = 4 * C, V_GAMC = 5 * C;
constexpr int kRecFloats = OFF_VEC + 6 * C;

// The tensor-core scan reads the same record in a second format: the chunk
// matrices as shared-memory images (bf16 hi + lo parts, K-major, 128-byte
// swizzled), copied to shared memory with bulk copies.  Byte offsets:
//   T_beta  hi | lo  (64 rows each)      [IMG_TB,   IMG_TB + 16 KB)
//   [Ap ; Mq] hi | lo (128 rows each)    [IMG_APMQ, IMG_APMQ + 32 KB)
//   T_gamma hi | lo                      [IMG_TG,   ...)
//   diag(gamma) M2 hi | lo               [IMG_M2,   ...)  (rows t scaled by gamma_t)
//   the gate vectors at the same place as in the fp32 record (OFF_VEC).
constexpr int IMG_TB = 0, IMG_APMQ = 16384, IMG_TG = 49152, IMG_M2 = 65536;
static_assert(IMG_M2 + 16384 == OFF_VEC * 4, "image fills the matrix part of the record");

// T = (I + A)^-1 for a strictly lower 64 x 64 A, by 128 threads (g = thread
// index in the group); W is 32 x 32 scratch (row stride LDW; the block of Tm
// at rows 0..31, columns 32..63 will do, which no stage touches).  The caller synchronises the
// block between the stages (0: diagonal blocks; 1, 2: the 16-row blocks; 3, 4:
// the 32-row block), all groups of the block running the same stage.  The
// 16 x 16 blocks above the diagonal are never written: the caller zeroes them
// once.
template <int LDA, int LDT, int LDW>
__device__ __forceinline__ void inv64_stage(int stage, const float *A, float *Tm, float *W, int g) {
  if (stage == 0) {
    // diagonal 16 x 16 blocks: thread (block, column) forward-substitutes its
    // column, x[r] = delta(r, col) - sum_{m < r} A[r][m] x[m], the terms added
    // in the order of m; the updates of the rows below m are independent, so
    // they are made as soon as x[m] is final (a 16-step chain instead of 120)
    if (g < 64) {
      const int b0 = (g >> 4) * 16, col = g & 15;
      float x[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) x[r] = (r == col) ? 1.f : 0.f;
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        if (m < col) x[m] = 0.f;  // (above the diagonal)
#pragma unroll
        for (int r = m + 1; r < 16; ++r) x[r] = fmaf(-A[(b0 + r) * LDA + b0 + m], x[m], x[r]);
      }
#pragma unroll
      for (int r = 0; r < 16; ++r) Tm[(b0 + r) * LDT + b0 + col] = x[r];
    }
  } else if (stage <= 2) {
    // 16-row blocks (i, j) = (1, 0) and (3, 2): W = A_ij T_jj, then
    // T_ij = -T_ii W; thread (block, row r, columns 4q .. 4q + 3)
    const int bi = 2 * (g >> 6) + 1, bj = bi - 1, r = (g >> 2) & 15, q = g & 3;
    float *w = W + (g >> 6) * 16 * LDW;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    if (stage == 1) {
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const float a = A[(16 * bi + r) * LDA + 16 * bj + k];
        const float4 t = *reinterpret_cast<const float4 *>(Tm + (16 * bj + k) * LDT + 16 * bj + 4 * q);
        acc[0] = fmaf(a, t.x, acc[0]); acc[1] = fmaf(a, t.y, acc[1]);
        acc[2] = fmaf(a, t.z, acc[2]); acc[3] = fmaf(a, t.w, acc[3]);
      }
      *reinterpret_cast<float4 *>(w + r * LDW + 4 * q) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const float a = Tm[(16 * bi + r) * LDT + 16 * bi + k];
        const float4 t = *reinterpret_cast<const float4 *>(w + k * LDW + 4 * q);
        acc[0] = fmaf(a, t.x, acc[0]); acc[1] = fmaf(a, t.y, acc[1]);
        acc[2] = fmaf(a, t.z, acc[2]); acc[3] = fmaf(a, t.w, acc[3]);
      }
      *reinterpret_cast<float4 *>(Tm + (16 * bi + r) * LDT + 16 * bj + 4 * q) =
          make_float4(-acc[0], -acc[1], -acc[2], -acc[3]);
    }
  } else {
    // the 32-row block: W = A[32:64, 0:32] T[0:32, 0:32], then
    // T[32:64, 0:32] = -T[32:64, 32:64] W; thread (rows rp, rp + 16, columns 4q .. 4q + 3)
    const int q = g & 7, rp = g >> 3;
    float a0[4] = {0.f, 0.f, 0.f, 0.f}, a1[4] = {0.f, 0.f, 0.f, 0.f};
    if (stage == 3) {
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        const float x0 = A[(32 + rp) * LDA + k], x1 = A[(48 + rp) * LDA + k];
        const float4 t = *reinterpret_cast<const float4 *>(Tm + k * LDT + 4 * q);
        a0[0] = fmaf(x0, t.x, a0[0]); a0[1] = fmaf(x0, t.y, a0[1]);
        a0[2] = fmaf(x0, t.z, a0[2]); a0[3] = fmaf(x0, t.w, a0[3]);
        a1[0] = fmaf(x1, t.x, a1[0]); a1[1] = fmaf(x1, t.y, a1[1]);
        a1[2] = fmaf(x1, t.z, a1[2]); a1[3] = fmaf(x1, t.w, a1[3]);
      }
      *reinterpret_cast<float4 *>(W + rp * LDW + 4 * q) = make_float4(a0[0], a0[1], a0[2], a0[3]);
      *reinterpret_cast<float4 *>(W + (rp + 16) * LDW + 4 * q) = make_float4(a1[0], a1[1], a1[2], a1[3]);
    } else {
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        const float x0 = Tm[(32 + rp) * LDT + 32 + k], x1 = Tm[(48 + rp) * LDT + 32 + k];
        const float4 t = *reinterpret_cast<const float4 *>(W + k * LDW + 4 * q);
        a0[0] = fmaf(x0, t.x, a0[0]); a0[1] = fmaf(x0, t.y, a0[1]);
        a0[2] = fmaf(x0, t.z, a0[2]); a0[3] = fmaf(x0, t.w, a0[3]);
        a1[0] = fmaf(x1, t.x, a1[0]); a1[1] = fmaf(x1, t.y, a1[1]);
        a1[2] = fmaf(x1, t.z, a1[2]); a1[3] = fmaf(x1, t.w, a1[3]);
      }
      *reinterpret_cast<float4 *>(Tm + (32 + rp) * LDT + 4 * q) =
          make_float4(-a0[0], -a0[1], -a0[2], -a0[3]);
      *reinterpret_cast<float4 *>(Tm + (48 + rp) * LDT + 4 * q) =
          make_float4(-a1[0], -a1[1], -a1[2], -a1[3]);
    }
  }
}

struct FwdParams {
  int B, T, H, NC;
  const void *q, *k, *v;
  const float *g, *beta, *gamma;
  float clip, scale;
  const float *S0, *R0;
  void *o;
  float *ST, *RT, *S_chunks, *R_chunks;
  float *ws;  // NC*B*H records of kRecFloats
  int *err;   // device status word (RDN_ERR_TIMEOUT if a bounded wait gave up) or NULL
  // forward intermediates kept for the backward (RDN_FLAG_SAVE_FOR_BWD) or NULL:
  // E, E2 per chunk as a 32 KB shared-memory image of E^T (rows j, columns t;
  // bf16 hi 16 KB | lo 16 KB, K-major, 128-byte swizzled), the clip mask as
  // [chunk][j] (bit t = |x| <= c)
  uint8_t *sv_E, *sv_E2;
  unsigned long long *sv_mask;
  // Packed variable-length sequences (rdn_fwd_args.cu_seqlens), or NULL for B
  // sequences of T tokens each: for s = 0 .. nseq, {first token, first chunk}
  // of sequence s (entry nseq closes the list: {T, total chunks}).  The upper
  // halves of the chunk numbers hold the sequences from the longest to the
  // shortest and, in entry nseq, whether the sequential tensor-core kernels run
  // on CTA pairs (launch_seq_table).
  const long long *seq;
  int pick;        // of two kernels launched for a packed call, this is the one for single
                   // CTAs (1) or for pairs (2), and the table says which runs; 0: the only one
  int nseq;        // sequences: B, or the number of packed sequences
  long long nrec;  // record slots: B * H * NC, or a bound on H * (total chunks)
  unsigned mods;   // the variant flags (RDN_FLAG_VARIANTS bits of rdn_fwd_args.flags)
  int f32out;      // o stored in fp32 (RDN_FLAG_F32_OUT on the tensor-core forward)
  int inject;      // 1: the tensor-core scan, 2: the backward chain skips its first MMA
                   // completion signal and waits ~5 ms for it (tests)
  // RDN_FLAG_QK_NORM: q and k above are then the normalised copies
  // SiLU(x) / max(||SiLU(x)||, qk_eps), written by the pass that makes the
  // chunk records (launch_t in chunk_fwd.cu), and qraw, kraw the caller's x
  const void *qraw, *kraw;
  float qk_eps;
  int qk_norm;
};

// Where sequence s's tokens and (s, h)'s chunk records are.  Token t of the
// sequence is row (tok0 + t) * H + h of the [tokens][H] inputs; chunk c of
// (s, h) is record rbase + c (also the index of its chunk-start states and
// saved intermediates).  With packed sequences the records of sequence s
// start at (its first chunk) * H, heads one after the other.
struct SeqSpan {
  long long tok0, rbase;
  int len, nc;
};
__host__ __device__ __forceinline__ long long first_chunk(const FwdParams &p, int s) {
  return p.seq[2 * s + 1] & 0xffffffffll;
}
__host__ __device__ __forceinline__ SeqSpan seq_span(const FwdParams &p, int s, int h) {
  SeqSpan q;
  if (p.seq) {
    q.tok0 = p.seq[2 * s];
    q.len = (int)(p.seq[2 * s + 2] - q.tok0);
    q.nc = (q.len + C - 1) / C;
    q.rbase = first_chunk(p, s) * p.H + (long long)h * q.nc;
  } else {
    q.tok0 = (long long)s * p.T;
    q.len = p.T;
    q.nc = p.NC;
    q.rbase = ((long long)s * p.H + h) * p.NC;
  }
  return q;
}
// The k-th sequence to start on: packed sequences from the longest to the
// shortest, since the sequential kernels end with the last chunk of the one
// that ends last.
__device__ __forceinline__ int seq_at(const FwdParams &p, int k) {
  return p.seq ? (int)(p.seq[2 * k + 1] >> 32) : k;
}
// Whether this kernel is the one of a packed call's two that runs.
__device__ __forceinline__ bool picked(const FwdParams &p) {
  return p.pick == 0 || (p.seq[2 * p.nseq + 1] >> 32 != 0) == (p.pick == 2);
}
// chunk records in use (at most nseq * H * NC slots)
__device__ __forceinline__ long long total_records(const FwdParams &p) {
  return p.seq ? first_chunk(p, p.nseq) * p.H : (long long)p.nseq * p.H * p.NC;
}
// record r -> (sequence s, head h, chunk c); r < total_records(p)
__device__ __forceinline__ void rec_decode(const FwdParams &p, long long r, int &s, int &h, int &c) {
  if (!p.seq) {
    if (r <= 0x7fffffffll) {  // (32-bit divisions: a 64-bit one is a long software routine)
      const unsigned ru = (unsigned)r, nc = (unsigned)p.NC, hn = (unsigned)p.H;
      const unsigned bh = ru / nc;
      c = (int)(ru - bh * nc);
      s = (int)(bh / hn);
      h = (int)(bh - (unsigned)s * hn);
      return;
    }
    const long long bh = r / p.NC;
    c = (int)(r - bh * p.NC);
    s = (int)(bh / p.H);
    h = (int)(bh - (long long)s * p.H);
    return;
  }
  int lo = 0, hi = p.nseq - 1;  // the last sequence whose records start at or before r
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first_chunk(p, mid) * p.H <= r) lo = mid; else hi = mid - 1;
  }
  s = lo;
  const int nc = (int)((p.seq[2 * s + 2] - p.seq[2 * s] + C - 1) / C);
  const long long off = r - first_chunk(p, s) * p.H;  // < H * nc
  h = (int)((unsigned)off / (unsigned)nc);
  c = (int)(off - (long long)h * nc);
}

// Where the forward keeps those intermediates: after the nrec record slots.
// With the tanh residual (deriv) the clip mask's place holds the residual
// map's derivative instead: [chunk][j][t] as 16-bit fixed point (grad_q16) on
// the tensor-core path, [chunk][t][j] fp32 on the fp32 path, which keeps every
// intermediate in 32 bits (its E and E2 are [chunk][t][j] fp32, its clip mask
// [chunk][t] rows of Dv bits).
struct SavedLayout {
  size_t e, e2, mask, bytes;  // byte offsets from the workspace base; region size
};
inline size_t mask_bytes_per_chunk(int Dv, bool deriv, bool tc) {
  return deriv ? (size_t)Dv * C * (tc ? 2 : 4) : (size_t)Dv * sizeof(unsigned long long);
}
// Whether a call runs the tensor-core kernels (and its records are
// shared-memory images): bf16 inputs, d = 128, every variant flag, RDN and RLA
// alike.
inline bool fwd_uses_tc(int DK, bool bf16) { return bf16 && DK == 128; }
inline SavedLayout saved_layout(const rdn_fwd_args &a) {
  const size_t nct = (size_t)call_records(a);
  SavedLayout l;
  l.e = nct * sizeof(float) * (size_t)kRecFloats;
  l.e2 = l.e + nct * sizeof(float) * C * a.Dv;
  l.mask = l.e2 + nct * sizeof(float) * C * a.Dv;
  l.bytes = l.mask - l.e + nct * mask_bytes_per_chunk(a.Dv, a.flags & RDN_FLAG_TANH_RESIDUAL,
                                                      fwd_uses_tc(a.Dk, a.dtype == RDN_BF16));
  return l;
}


inline FwdParams make_fwd_params(const rdn_fwd_args &a) {
  FwdParams p;
  p.B = a.B; p.T = a.T; p.H = a.H;
  p.NC = (a.T + C - 1) / C;
  p.q = a.q; p.k = a.k; p.v = a.v;
  p.g = a.g; p.beta = a.beta; p.gamma = a.gamma;
  p.clip = a.clip; p.scale = a.scale;
  p.S0 = a.S0; p.R0 = a.R0;
  p.o = a.o;
  p.ST = a.ST; p.RT = a.RT; p.S_chunks = a.S_chunks; p.R_chunks = a.R_chunks;
  p.ws = nullptr;
  p.err = nullptr;
  p.sv_E = p.sv_E2 = nullptr;
  p.sv_mask = nullptr;
  p.seq = nullptr;  // set by the launcher once the table is in its workspace
  p.pick = 0;
  p.nseq = call_seqs(a);
  p.nrec = call_records(a);
  p.mods = a.flags & RDN_FLAG_VARIANTS;
  p.f32out = (a.flags & RDN_FLAG_F32_OUT) && a.dtype == RDN_BF16;
  p.inject = 0;
  p.qraw = a.q;
  p.kraw = a.k;
  p.qk_eps = a.qk_eps;
  p.qk_norm = (a.flags & RDN_FLAG_QK_NORM) ? 1 : 0;
  return p;
}

// RDN_FLAG_QK_NORM: the normalised q, then k, [tokens][H][Dk] in dtype, at
// qk_norm_offset bytes into the forward's workspace (after the records and
// the saved intermediates) and in the backward's when it makes its own records.
inline size_t qk_norm_bytes(const rdn_fwd_args &a) {
  if (!(a.flags & RDN_FLAG_QK_NORM)) return 0;
  const size_t esz = a.dtype == RDN_BF16 ? 2 : 4;
  return 2 * esz * (size_t)a.B * a.T * a.H * a.Dk;  // (a multiple of 256)
}
inline size_t qk_norm_offset(const rdn_fwd_args &a) {
  const size_t nrec = (size_t)call_records(a);
  size_t off = sizeof(float) * (size_t)kRecFloats * nrec;
  if (a.flags & RDN_FLAG_SAVE_FOR_BWD)
    off += saved_layout(a).bytes;
  return off;
}
// Points p.q, p.k at the normalised copies starting at `base`.
inline void set_qk_norm_copies(FwdParams &p, const rdn_fwd_args &a, char *base) {
  const size_t half = qk_norm_bytes(a) / 2;
  p.q = base;
  p.k = base + half;
}

// Tensor-core scan (fwd_tc.cu): bf16 inputs with d_k = d_v = 128.
cudaError_t launch_fwd_tc(const FwdParams &p, bool rdnv, cudaStream_t s);

// The forward's prep kernel alone (per-chunk records into p.ws, in the format
// that this call's kernels read).
cudaError_t launch_prep(const FwdParams &p, int DK, bool rdnv, bool bf16, cudaStream_t s);

// Tensor-core backward (bwd_tc.cu): recompute, chain and post kernels.
cudaError_t launch_prep_tc(const FwdParams &p, bool rla, cudaStream_t s);
size_t bwd_tc_extra_bytes(long long nrec, bool deriv);  // (deriv: the tanh residual's)
cudaError_t launch_bwd_tc(const FwdParams &f, const void *dO, const float *dST, const float *dRT,
                          const float *Sc, const float *Rc, void *dq, void *dk, void *dv, float *dg,
                          float *dbeta, float *dgamma, float *dS0, float *dR0, char *extra,
                          bool rla, bool grad_f32, bool dqk_f32, cudaStream_t s);

// Launch the forward: prep (per-chunk records into p.ws), then the scan
// (outputs, optional chunk-start states).
cudaError_t launch_fwd_parts(const FwdParams &p, int DK, bool rdnv, bool bf16, cudaStream_t s);

// E, E2 and the residual's mask of every chunk (p.sv_*) from the chunk-start
// states p.S_chunks, p.R_chunks (fp32 path).
cudaError_t launch_recompute(const FwdParams &p, int DK, bool rdnv, bool bf16, cudaStream_t s);

// The current device's SM count.
inline cudaError_t sm_count(int *n) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e != cudaSuccess ? e : cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev);
}

// Whether the forward tensor-core scan gives each (sequence, head) a pair of
// CTAs (fwd_pair.cu) or one: whichever ends first.  What a (sequence, head) costs,
// in 0.1 us, fitted to calls of 4 to 304 heads and 1 to 64 chunks (rdnv: the delta
// rule; states: chunk-start states kept, as for a backward): one CTA `one` and
// `one_chunk` a chunk, a pair `two` and `two_chunk` a chunk, or `two_full` where
// pairs fill the chip and wait for memory.  A pair's chunk is shorter and its
// start longer, so that 16 RDN heads take 18.3 us by one CTA and 20.4 by pairs at
// one chunk, 31.4 and 30.6 at three, 67 and 51 at eight; and pairs need twice the
// SMs: 200 heads of eight chunks take 133 us by one CTA each and 168 by pairs.
struct ScanCost {
  int one, one_chunk, two, two_chunk, two_full;
};
__host__ __device__ inline ScanCost scan_cost(bool rdnv, bool states) {
  if (rdnv) return states ? ScanCost{69, 90, 130, 60, 63} : ScanCost{63, 70, 120, 42, 61};
  return states ? ScanCost{69, 65, 103, 54, 55} : ScanCost{59, 54, 95, 43, 45};
}
// The longest sequence's chain of chunks or the chip's throughput over all `seqs`
// sequences of `chunks` chunks sets the time of either (both sides times nsm).
__host__ __device__ inline bool pairs_for(const ScanCost &c, long long longest, long long seqs,
                                          long long chunks, int H, int nsm) {
  const long long l1 = (c.one + c.one_chunk * longest) * nsm, l2 = (c.two + c.two_chunk * longest) * nsm;
  const long long f1 = (c.one * seqs + c.one_chunk * chunks) * H;
  const long long f2 = (c.two * seqs + c.two_full * chunks) * 2 * H;
  return (l2 > f2 ? l2 : f2) < (l1 > f1 ? l1 : f1);
}
// Where every pair has its two SMs at once the host decides (packed: the lengths
// are on the device, the longest is taken for half of the tokens); where not, equal
// sequences take one CTA each, which needs half the waves at less than twice the time.
inline bool use_pairs(const FwdParams &p, bool rdnv, int nsm) {
  if (2ll * p.nseq * p.H > nsm) return false;
  const ScanCost c = scan_cost(rdnv, p.S_chunks != nullptr);
  if (p.seq) return pairs_for(c, p.nseq > 1 ? (p.NC + 1) / 2 : p.NC, p.nseq, p.NC + p.nseq, p.H, nsm);
  return pairs_for(c, p.NC, p.nseq, (long long)p.nseq * p.NC, p.H, nsm);
}
// ... and packed sequences have both kernels launched and the table say which one
// runs, if pairs can be the choice at all: with one long sequence and the others as
// short as can be, and no more sequences than the table puts in order (kOrdered).
// The other kernel's CTAs return at once, but each takes an SM's shared memory to
// start, 0.64 us a CTA and SM: 2000 sequences of 16 heads 262 us.
constexpr int kOrdered = 1024;  // packed sequences that are put in order of length
inline bool pick_on_device(const FwdParams &p, bool rdnv, int nsm) {
  return p.seq && 2ll * p.nseq * p.H > nsm && p.nseq <= kOrdered &&
         pairs_for(scan_cost(rdnv, p.S_chunks != nullptr), p.NC, p.nseq, p.NC, p.H, nsm);
}

}  // namespace rdn
