// simt.cuh -- register-tiled fp32 products over shared memory for the fp32
// chunk kernels (chunk_fwd.cu, chunk_bwd.cu).
//
// Each thread owns a TM x TN tile of the result and reads both operands as
// 16-byte vectors: 8 shared loads for 64 FMAs of a 4 x 4 tile, against one
// load per FMA operand before, so that the FMA pipe and not the shared-memory
// pipe sets the pace.  Row strides are odd multiples of 4 floats: rows that
// differ by one then start 4 banks apart and the 16-byte loads of 8 lanes fall
// on all 32 banks.
//
// A 16-byte shared load takes 2.25 cycles of the SM where lanes differing in
// lane bit 0, or those differing in bit 1, read the same address, and 4.04
// otherwise, however few addresses there are (measured; 8-byte ones 1.42 and
// 2.07).  So the lanes of a tile are laid out over its rows and columns with
// bit 0 in the one and bit 1 in the other (lane_mn, or a column per lane pair),
// which keeps both operands' loads at the lower cost.
#pragma once
#include "chunk_common.cuh"

namespace rdn {
namespace simt {

// Row lm and column ln of a lane in a warp's 32 / LN x LN lanes (LN 4 or 8):
// columns on lane bits 0, 2 (, 4), rows on the others.
template <int LN>
__device__ __forceinline__ void lane_mn(int lane, int &lm, int &ln) {
  static_assert(LN == 4 || LN == 8, "lanes across");
  ln = (lane & 1) | ((lane >> 1) & 2);
  if (LN == 8) {
    ln |= (lane >> 2) & 4;
    lm = ((lane >> 1) & 1) | ((lane >> 2) & 2);
  } else {
    lm = ((lane >> 1) & 1) | ((lane >> 2) & 6);
  }
}
// v = p[0 .. N), N in {1, 2, 4}, p aligned to N floats
template <int N>
__device__ __forceinline__ void ldv(const float *p, float (&v)[N]) {
  if constexpr (N == 4) {
    const float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  } else if constexpr (N == 2) {
    const float2 a = *reinterpret_cast<const float2 *>(p);
    v[0] = a.x; v[1] = a.y;
  } else {
    v[0] = p[0];
  }
}
template <int N>
__device__ __forceinline__ void stv(float *p, const float (&v)[N]) {
  if constexpr (N == 4) *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else if constexpr (N == 2) *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
  else p[0] = v[0];
}
template <int TM, int TN>
__device__ __forceinline__ void zero(float (&a)[TM][TN]) {
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) a[i][j] = 0.f;
}

// Two packed fp32 FMAs (one instruction): d += a * b per half.  It leaves the
// FMA rate as it is and halves its issue slots, which the loads need.
struct f2 {
  unsigned long long v;
};
__device__ __forceinline__ void fma2(f2 &d, f2 a, f2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d.v) : "l"(a.v), "l"(b.v));
}
__device__ __forceinline__ float sum2(f2 x) {
  return __uint_as_float((uint32_t)x.v) + __uint_as_float((uint32_t)(x.v >> 32));
}

// acc[i][j] = sum over k in [0, K) of A_i[k] B_j[k] for rows A_i = A + i * lda,
// B_j = B + j * ldb (both contiguous in k, 16-byte aligned, K a multiple of
// 4): even and odd k are summed apart, two FMAs an instruction.
template <int TM, int TN, int K>
__device__ __forceinline__ void mm_nt(const float *A, int lda, const float *B, int ldb,
                                      float (&acc)[TM][TN]) {
  f2 s[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) s[i][j].v = 0ull;
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    f2 a[TM][2];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(A + i * lda + k);
      a[i][0].v = x.x;
      a[i][1].v = x.y;
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(B + j * ldb + k);
      const f2 b0{x.x}, b1{x.y};
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        fma2(s[i][j], a[i][0], b0);
        fma2(s[i][j], a[i][1], b1);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = sum2(s[i][j]);
}

// acc[i][j] += sum over k in [k0, k1) of A_i[k] B[k][j], rows A_i = A + i * a_step
// contiguous in k (16-byte loads of 4 k), B rows TN wide ldb apart; only the
// rows i whose bit is set in MASK (multiples of 4 for k0, k1).
template <int TM, int TN, int MASK>
__device__ __forceinline__ void mm_ak(const float *A, int a_step, const float *B, int ldb, int k0,
                                      int k1, float (&acc)[TM][TN]) {
#pragma unroll 4
  for (int k = k0; k < k1; k += 4) {
    float a[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
      if ((MASK >> i) & 1) ldv<4>(A + i * a_step + k, a[i]);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float b[TN];
      ldv<TN>(B + (k + kk) * ldb, b);
#pragma unroll
      for (int i = 0; i < TM; ++i)
        if ((MASK >> i) & 1)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i][kk], b[j], acc[i][j]);
    }
  }
}
// ... and with a second B of its own row mask, sharing the loads of A
template <int TM, int TN, int MASK, int MASK2>
__device__ __forceinline__ void mm_ak2(const float *A, int a_step, const float *B, const float *B2,
                                       int ldb, int K, float (&acc)[TM][TN], float (&acc2)[TM][TN]) {
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    float a[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
      if (((MASK | MASK2) >> i) & 1) ldv<4>(A + i * a_step + k, a[i]);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float b[TN], b2[TN];
      ldv<TN>(B + (k + kk) * ldb, b);
      ldv<TN>(B2 + (k + kk) * ldb, b2);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        if ((MASK >> i) & 1)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i][kk], b[j], acc[i][j]);
        if ((MASK2 >> i) & 1)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc2[i][j] = fmaf(a[i][kk], b2[j], acc2[i][j]);
      }
    }
  }
}
// acc[i][j] += sum over k in [0, K) of A[k][i] B[k][j]: A's rows are k, its TM
// columns contiguous.
template <int TM, int TN>
__device__ __forceinline__ void mm_am(const float *A, int lda, const float *B, int ldb, int K,
                                      float (&acc)[TM][TN]) {
#pragma unroll 8
  for (int k = 0; k < K; ++k) {
    float a[TM], b[TN];
    ldv<TM>(A + k * lda, a);
    ldv<TN>(B + k * ldb, b);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
  }
}

// 16-byte asynchronous copies global -> shared in groups: wait_groups<N>
// returns once all but the newest N committed groups of this thread are done.
__device__ __forceinline__ void cp16(float *dst, const float *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void wait_groups() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// a 64 x 64 chunk matrix of a record into rows of ld floats
template <int NT>
__device__ __forceinline__ void cp_mat(float *dst, int ld, const float *src) {
#pragma unroll
  for (int u = 0; u < C * C / 4 / NT; ++u) {
    const int e = threadIdx.x + u * NT;
    cp16(dst + (e >> 4) * ld + 4 * (e & 15), src + 4 * e);
  }
}

// A tile of 64 token rows x COLS columns of a token-major tensor, fetched into
// registers by NT threads (16-byte loads, zero past the n valid rows) and put
// into shared memory as fp32 later: the loads are in flight over the work in
// between.
template <typename InT, int COLS, int NT>
struct RowTile {
  static constexpr int VEC = 16 / (int)sizeof(InT), CPR = COLS / VEC;  // elements, chunks per row
  static constexpr int TOTAL = C * CPR, U = (TOTAL + NT - 1) / NT;
  uint4 raw[U];
  __device__ __forceinline__ void fetch(const InT *base, size_t row_stride, int n) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = threadIdx.x + u * NT, t = e / CPR, c = e % CPR;
      raw[u] = make_uint4(0u, 0u, 0u, 0u);
      if (t < n) raw[u] = *reinterpret_cast<const uint4 *>(base + (size_t)t * row_stride + c * VEC);
    }
  }
  __device__ __forceinline__ void put(float *dst, int ld, float scale) const {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = threadIdx.x + u * NT, t = e / CPR, c = e % CPR;
      if (TOTAL % NT != 0 && e >= TOTAL) break;
      float *d = dst + t * ld + c * VEC;
      const uint32_t w[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
      if constexpr (VEC == 4) {
        *reinterpret_cast<float4 *>(d) =
            make_float4(scale * __uint_as_float(w[0]), scale * __uint_as_float(w[1]),
                        scale * __uint_as_float(w[2]), scale * __uint_as_float(w[3]));
      } else {  // (a bf16 is the upper half of its fp32)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<float4 *>(d + 4 * h) =
              make_float4(scale * __uint_as_float(w[2 * h] << 16),
                          scale * __uint_as_float(w[2 * h] & 0xFFFF0000u),
                          scale * __uint_as_float(w[2 * h + 1] << 16),
                          scale * __uint_as_float(w[2 * h + 1] & 0xFFFF0000u));
      }
    }
  }
};

// In-chunk cumulative log-decay, kept as an unevaluated sum hi + lo of two
// floats: the decays between tokens are exponentials of differences of sums
// that reach -60 and more, where one float's rounding alone (2e-6) would be
// the largest error of the whole chunk.
struct Cum {
  float hi[C], lo[C];        // sum of g up to and with token t
  float phi[C], plo[C];      // sum before it
  __device__ __forceinline__ float to(int t, int i) const {  // sum over (i, t]
    return (hi[t] - hi[i]) + (lo[t] - lo[i]);
  }
  __device__ __forceinline__ float before(int t, int i) const {  // sum over (i, t - 1]
    return (phi[t] - hi[i]) + (plo[t] - lo[i]);
  }
};
// by one full warp: lane l owns tokens l and 32 + l, ga, gb their log-decays
__device__ __forceinline__ void cum64(float ga, float gb, Cum &c) {
  const int lane = threadIdx.x & 31;
  double a = ga, b = gb;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double ua = __shfl_up_sync(0xffffffffu, a, d), ub = __shfl_up_sync(0xffffffffu, b, d);
    if (lane >= d) {
      a += ua;
      b += ub;
    }
  }
  const double top = __shfl_sync(0xffffffffu, a, 31);
  b += top;
  const double pa = __shfl_up_sync(0xffffffffu, a, 1), pb = __shfl_up_sync(0xffffffffu, b, 1);
  const double v[4] = {a, b, lane ? pa : 0.0, lane ? pb : top};
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float hi = (float)v[u], lo = (float)(v[u] - (double)hi);
    const int t = lane + 32 * (u & 1);
    (u < 2 ? c.hi : c.phi)[t] = hi;
    (u < 2 ? c.lo : c.plo)[t] = isfinite(hi) ? lo : 0.f;
  }
}

}  // namespace simt

// fn.run<DK, RDNV, InT>() for the call's head size, variant and input type
// (bf16 inputs with d = 128 run the tensor-core kernels instead)
template <typename F>
cudaError_t simt_dispatch(int DK, bool rdnv, bool bf16, const F &fn) {
  if (DK == 128) return rdnv ? fn.template run<128, true, float>() : fn.template run<128, false, float>();
  if (bf16) return rdnv ? fn.template run<64, true, __nv_bfloat16>() : fn.template run<64, false, __nv_bfloat16>();
  return rdnv ? fn.template run<64, true, float>() : fn.template run<64, false, float>();
}
// Value columns per CTA of the sequential kernels (forward scan, backward
// chain): fewer columns make a chunk shorter but repeat the reads of K, Q and
// the chunk matrices, and more CTAs may need another wave.  A chunk's cost in us
// by the forward's measurements: d = 128 (one CTA per SM) 16.7, 11.2 and 9.2 for
// 32, 16 and 8 columns; d = 64 with two CTAs on every SM 12.5 and 9.0 for 16 and
// 8, with one 8.3 and 6.1.  The chain's stand in the same relation (17.1, 12.0,
// 10.0; 13.3, 9.5; 8.7, 7.1): timed at every width for 27 numbers of heads from 2
// to 304 in each of d = 128, d = 64, d = 64 bf16 and RLA, the width chosen was the
// chain's best in all of them and the scan's in all but one (77 heads of d = 64,
// 207 us for 193).
inline int scan_columns(int DK, long long heads, int nsm) {
  static const int cols[3] = {32, 16, 8}, cost128[3] = {167, 112, 92}, two64[3] = {0, 125, 90},
                   one64[3] = {0, 83, 61};
  int best = 0;
  long long least = 0;
  for (int i = DK == 64; i < 3; ++i) {
    const long long ctas = heads * (DK / cols[i]);
    long long t;
    if (DK == 64) {
      const long long rest = ctas % (2 * nsm);
      t = ctas / (2 * nsm) * two64[i] + (rest > nsm ? two64[i] : rest ? one64[i] : 0);
    } else {
      t = (ctas + nsm - 1) / nsm * cost128[i];
    }
    if (!best || t < least) {
      best = cols[i];
      least = t;
    }
  }
  return best;
}
}  // namespace rdn
