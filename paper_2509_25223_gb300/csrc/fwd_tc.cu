// fwd_tc.cu -- tensor-core (tcgen05 / TMEM) scan of the chunkwise RLA / RDN
// forward, bf16 inputs, d_k = d_v = 128, one CTA per (sequence, head).
//
// Same chunk algebra as chunk_fwd.cu (see its header), computed in the
// transposed orientation so that every product has the value dimension
// d_v = 128 as its M dimension: TMEM lane j holds value column j.  The 16
// element-wise warps form 4 groups of 128 threads; thread j of group g owns value
// column j for the token columns t in [16g, 16g + 16) of the chunk (and the
// state columns [16g, 16g + 16) and [64 + 16g, 80 + 16g)), so that the four
// warps sharing a TMEM lane quadrant hide one another's latencies.  Per chunk of 64
// tokens, with KQ = [K ; Q] (128 x d_k, exact bf16, unscaled):
//
//   MMA1  D1   = S^T  KQ^T          -> [KS | QS]                  (N=128, K=128)
//   MMA5  D3   = R^T  KQ^T          -> [KR | QR] (chunk-start R, behind MMA1)
//         X    = V - Gam*KS         (= V - alpha * Gprev*KS); QS rescaled in TMEM
//                                      to Gam*scale*QS
//   MMA2  E^T  = X^T  T_beta^T      (over KS; Gprev*KS back in its place after)
//   MMA3  D1  += E^T  [Ap ; Mq]^T   -> [P | Ob]                   (N=128, K=64)
//   MMA4  S   += (wS E)^T K         onto S scaled by Gam_C in TMEM while MMA1
//                                      ran: S_C = Gam_C S + U       (N=128, K=64)
//         r    = clip(V - P)        (Section 3.3; kept in registers)
//         X2   = r - Gam*KR
//   MMA6  E2^T = X2^T T_gamma^T
//   MMA8  R   += (wR E2)^T K        onto R scaled by Gam_C during MMA1: R_C
//   MMA7  D1[:, Ob half] += E2^T (diag(gamma) M2)^T
//         o    = D1[:, Ob half] + gamma * Gam*scale*QR   (= Ob + gamma * Oa)
//
// RLA skips MMA2 and MMA6 (E = V, E2 = r).  X, E, wS E and their auxiliary
// counterparts (magnitude ~ |v|) enter the MMAs as bf16 hi + lo pairs, which
// keeps their rounding well below the state's own scale; so does S in MMA1
// (hi + lo copies); R and the chunk's K, Q are single bf16 (K, Q exactly).
// The states S, R live in TMEM in fp32 for the whole sequence; their bf16
// copies (the A operands of MMA1 and MMA5) are rewritten in shared memory
// after each update.  The state-independent chunk matrices (T_beta, T_gamma, Ap,
// Mq, diag(gamma) M2) come from chunk_prep's records as bf16 hi + lo
// shared-memory images; they are streamed into two slots by bulk copies (slot
// A: T_beta then T_gamma; slot B: [Ap;Mq] then M2) and enter the MMAs as three
// products (hi*hi + hi*lo + lo*hi).
//
// The products are issued by a warp of their own and the copies by another: an
// issuing thread is held for most of its products' time (54 cycles a 128 x 64 x
// 16 product, 70 a 128 x 128 x 16 one, which the operands' shared-memory reads
// set), and as one of the element-wise warps it held up all the others.  What
// the chain of dependent steps does not wait for runs behind it: MMA5 behind
// MMA1, MMA4 behind MMA3 with S's copies made during MMA6, MMA7 behind MMA8
// while R's copy is made, and o is stored during the next chunk's MMA3.  Every
// wait is bounded: a thread whose wait gave up sets the CTA's flag, which all
// read after the next chunk's first barrier.
//
// Measured (128 heads; before, with every product and copy issued by an
// element-wise thread): T = 2048 240 us (293), 7.5 us a chunk; T = 4096 saving
// for the backward 592 us (685), 9.2 us a chunk, of which a CTA moves 390 KB from
// and to HBM (5.4 TB/s of the 6.9 a copy reaches).
//
// TMEM (512 columns): [0,128) S   [128,256) R   [256,384) D1   [384,512) D3
// (D1 holds KS|QS, then E | Ob, Gprev KS + Ap E = P | Ob, then E2 | Ob + gamma
// M2 E2; D3 KR | QR, then (wR E2)^T as MMA8's operand | QR).
#include <cuda.h>
#include <cudaTypedefs.h>

#include "fwd_tc.cuh"

namespace rdn {
namespace {

using namespace fwdtc;

// shared-memory carve-up (bytes from the 1024-aligned dynamic base)
constexpr uint32_t SM_SA = 0;          // S^T bf16, 128 x 128, two 64-col blocks
constexpr uint32_t SM_RA = 32768;      // R^T bf16
constexpr uint32_t SM_KQ = 65536;      // [K ; Q] unscaled, 128 rows x 128, two 64-col blocks
                                       // (K rows also serve as the MN-major B of the updates)
constexpr uint32_t SM_V = 98304;       // V, 64 rows t x 128 columns j, two 8 KB blocks; then the
                                       // previous chunk's o on its way out
constexpr uint32_t SM_SLOTA = 114688;  // T_beta then T_gamma image (hi | lo), 16 KB
constexpr uint32_t SM_SLOTB = 131072;  // [Ap;Mq] then M2 image (hi | lo), 32 KB
// value-like operands are split into bf16 hi + lo parts (two MMAs each):
constexpr uint32_t SM_XE = 163840;     // X^T then E^T (X2^T then E2^T), hi part, 128 x 64
constexpr uint32_t SM_XE_LO = 180224;  //   lo part
constexpr uint32_t SM_W = 196608;      // (wS E)^T hi | lo; from MMA4 to the next MMA1 S - bf16(S)
constexpr uint32_t SM_W_LO = 212992;
// two chunks' gates, fp32: Gam, Gprev, wS, wR, gamma (64 each), GamC
constexpr uint32_t SM_VEC = 229376;
constexpr int kVec = 324;
// mbarriers: chain, slot A, slot B, drain, tiles, then one phase a chunk: MMA2,
// MMA3, MMA4, MMA6, MMA7, MMA8, E's image copied, E2's
constexpr uint32_t SM_BAR = SM_VEC + 2 * kVec * 4;
constexpr int kBars = 13;
constexpr uint32_t SM_SLOT = SM_BAR + 8 * kBars;
constexpr uint32_t SM_FLAG = SM_SLOT + 4;
constexpr size_t kTcSmem = SM_FLAG + 4;
static_assert(kTcSmem <= 232448, "shared memory");

constexpr int kScanThreads = kTcThreads + 64;      // and the issuing and the copying warp
constexpr int kOneMore = kTcThreads + 32;
// named barriers on which the element-wise warps hand operands to the issuing
// warp (X, X2; E, E2 to the copying warp too) and results to the copying warp (O)
constexpr int kBarX = 1, kBarE = 2, kBarX2 = 3, kBarE2 = 4, kBarO = 5, kBarW = 6;

constexpr uint32_t T_S = 0, T_R = 128, T_D1 = 256, T_X = 384;  // T_X: D3

// kGeneric: the variant flags (FwdParams::mods) are read; the method's
// instances have them folded away
template <bool RDNV, bool kGeneric>
__global__ void __launch_bounds__(kScanThreads, 1)
    fwd_tc_kernel(FwdParams p, const __grid_constant__ FwdMaps maps) {
  extern __shared__ __align__(1024) uint8_t sm[];
  const uint32_t sbase = smem_u32(sm);
  if (!picked(p)) return;
  if (sbase & 1023u) {  // the swizzled tiles need a 1024-byte aligned base
    if (threadIdx.x == 0 && p.err) atomicExch(p.err, RDN_ERR_CUDA);
    return;
  }
  uint64_t *bar = reinterpret_cast<uint64_t *>(sm + SM_BAR);
  uint64_t *barA = bar + 1, *barB = bar + 2;  // slot A / slot B bulk copies
  uint64_t *barD = bar + 3;  // the drain after a wait that gave up
  uint64_t *barE = bar + 4;  // a whole chunk's V, K, Q tiles by tensor-map copies
  uint64_t *barM2 = bar + 5, *barM3 = bar + 6, *barM4 = bar + 7, *barM6 = bar + 8, *barM7 = bar + 9,
           *barM8 = bar + 10, *barI = bar + 11, *barJ = bar + 12;
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + SM_SLOT);
  volatile int *flag = reinterpret_cast<volatile int *>(sm + SM_FLAG);

  const int tid = threadIdx.x, warp = tid >> 5;
  const int j = tid & 127;       // value column == TMEM lane
  const int g16 = (warp >> 2) * 16;  // this thread's token (and state) columns start
  const int sq = seq_at(p, blockIdx.x / p.H), h = blockIdx.x % p.H;
  const SeqSpan sp = seq_span(p, sq, h);  // this (sequence, head)'s tokens and records
  const long long tok0 = sp.tok0;
  const int T = sp.len, H = p.H, NC = sp.nc;
  const __nv_bfloat16 *q = (const __nv_bfloat16 *)p.q;
  const __nv_bfloat16 *k = (const __nv_bfloat16 *)p.k;
  const __nv_bfloat16 *v = (const __nv_bfloat16 *)p.v;
  const float clip = p.clip;
  const bool dec_res = kGeneric && (p.mods & RDN_FLAG_DECAYED_RESIDUAL);
  const bool plain = kGeneric && (p.mods & RDN_FLAG_PLAIN_COMBINE);  // o = S_{t-1} q + R_t q
  // the log-cosh residual r = c tanh(x / c); the backward then reads the
  // derivative 1 - (r / c)^2 of each element (16-bit fixed point) where the
  // clip mask goes
  const bool tnh = kGeneric && (p.mods & RDN_FLAG_TANH_RESIDUAL);
  // the stateless correction R_t = r_t k_t^T: no read-out of the carried R
  // (X2 = r, no gamma Gam Q R term in o), R not carried over a chunk (scaled
  // by 0); the records hold the identity T_gamma, diag(gamma qk) and the
  // one-hot wR that make the rest of the pass compute it
  const bool stl = kGeneric && (p.mods & RDN_FLAG_STATELESS_AUX);
  const size_t st_base = ((size_t)sq * p.H + h) * D * D;

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
  const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
  // the waits on the MMAs: normally about a second; a test (p.inject) skips the
  // first phase's completion signal and waits about 5 ms for it instead
  const long long limit = p.inject == 1 ? 10000000ll : 2000000000ll;
  // Chunks between the first and the last are whole: with tensor maps the
  // copying warp brings their tiles by tiled bulk copies.  The first chunk and
  // the last one, which may be ragged, come by cp.async with zero fill.
  auto by_tma = [&](int cc) { return maps.ok && cc > 0 && cc < NC - 1; };
  // whether chunk c's o leaves as two tensor-map tiles (bf16 results, whole chunk)
  auto o_tiles = [&](int c) { return maps.o_ok && T - c * 64 >= 64; };

  if (warp == kTcThreads / 32) {
    // =============================================== the issuing warp (lane 0)
    bool one = (tid & 31) == 0;
    bool skip_commit = p.inject == 1;
    const uint32_t i64 = idesc_bf16(128, 64), i128 = idesc_bf16(128, 128);
    // wait for a copy by the copying warp; when it gave up, nothing more is issued
    // or completed (no barrier is armed again before its phase is complete)
    auto wait_copy = [&](uint64_t *b, uint32_t ph) {
      if (mbar_wait(b, ph)) return true;
      *flag = 1;
      return one = false;
    };
    bool alive = true;
    for (int c = 0; c < NC; ++c) {
      __syncthreads();
      fence_after_sync();
      if (*flag) {
        alive = false;
        break;
      }
      if (one) {  // MMA1 (S as hi + lo), MMA5 behind it (RLA reads only Q R)
        mma_tile(tm + T_D1, sbase + SM_SA, 16384, sbase + SM_KQ, 16384, 8, i128, false);
        mma_tile(tm + T_D1, sbase + SM_W, SM_W_LO - SM_W, sbase + SM_KQ, 16384, 8, i128, true);
        if (!skip_commit) mma_commit(bar);
        skip_commit = false;
        if (RDNV)
          mma_tile(tm + T_X, sbase + SM_RA, 16384, sbase + SM_KQ, 16384, 8, i128, false);
        else
          mma_tile(tm + T_X + 64, sbase + SM_RA, 16384, sbase + SM_KQ + 8192, 16384, 8, i64, false);
      }
      __syncwarp();
      if (RDNV) {
        bar_sync(kBarX, kOneMore);
        fence_after_sync();
        if (one && wait_copy(barA, 0)) {  // MMA2: E^T = X^T T_beta^T into D1[0,64) (over KS)
          mma_split3(tm + T_D1, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTA,
                     sbase + SM_SLOTA + 8192, i64, false);
          mma_commit(bar);
          mma_commit(barM2);
        }
        __syncwarp();
      }
      bar_sync(kBarE, kScanThreads);
      fence_after_sync();
      if (one && wait_copy(barB, 0)) {  // MMA3: D1 += E^T [Ap;Mq]^T; MMA4: S += (wS E)^T K
        mma_split3(tm + T_D1, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTB,
                   sbase + SM_SLOTB + 16384, i128, true);
        mma_commit(bar);
        mma_commit(barM3);
        mma_tile_kmn(tm + T_S, sbase + SM_W, 0, sbase + SM_KQ, 16384, 4, i128, true);
        mma_tile_kmn(tm + T_S, sbase + SM_W_LO, 0, sbase + SM_KQ, 16384, 4, i128, true);
        mma_commit(barM4);
      }
      __syncwarp();
      if (RDNV) {
        bar_sync(kBarX2, kOneMore);
        fence_after_sync();
        if (one && wait_copy(barA, 1)) {  // MMA6: E2^T = X2^T T_gamma^T (into D1[0,64))
          mma_split3(tm + T_D1, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTA,
                     sbase + SM_SLOTA + 8192, i64, false);
          mma_commit(bar);
          mma_commit(barM6);
        }
        __syncwarp();
      }
      bar_sync(kBarE2, kScanThreads);
      fence_after_sync();
      if (one) {  // MMA8: R += (wR E2)^T K (hi, then lo); MMA7 behind it
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          mma_bf16_ta(tm + T_R, tm + T_X + 8 * kk, sdesc_sw128_mn(sbase + SM_KQ + (kk & 3) * 2048, 16384),
                      i128 | kBMajorMN, 1u);
        mma_commit(bar);
        mma_commit(barM8);
        if (wait_copy(barB, 1)) {  // the image is diag(gamma) M2: its product lands on Ob
          mma_split3(tm + T_D1 + 64, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTB,
                     sbase + SM_SLOTB + 8192, i64, true);
          mma_commit(barM7);
        }
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
  if (warp == kTcThreads / 32 + 1) {
    // =============================================== the copying warp
    const bool one = (tid & 31) == 0;
    const int ln = tid & 31;
    uint32_t armA = 0, armB = 0, armE = 0;  // copies armed on the slots' and the tiles' barriers
    auto rec_of = [&](int c) {
      return reinterpret_cast<const uint8_t *>(p.ws + (size_t)(sp.rbase + c) * kRecFloats);
    };
    auto load_a = [&](const uint8_t *src) {
      ++armA;
      mbar_expect_tx(barA, 16384);
      bulk_g2s(sm + SM_SLOTA, src, 16384, barA);
    };
    auto load_b = [&](const uint8_t *src, uint32_t bytes) {
      ++armB;
      mbar_expect_tx(barB, bytes);
      bulk_g2s(sm + SM_SLOTB, src, bytes, barB);
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
      const uint8_t *r = rec_of(c);
      static_assert((kRecFloats * 4) % 16 == 0 && kRecFloats * 4 > 65536, "record");
      prefetch_l2_bulk(r, 65536);
      prefetch_l2_bulk(r + 65536, kRecFloats * 4 - 65536);
      if (!maps.ok) return;
      const int row = (int)(tok0 + (long long)c * 64);
      for (int kb = 0; kb < 2; ++kb) {
        tma_prefetch_3d(maps.v, 64 * kb, h, row);
        tma_prefetch_3d(maps.k, 64 * kb, h, row);
        tma_prefetch_3d(maps.q, 64 * kb, h, row);
      }
    };
    // chunk c's o, staged by the element-wise warps
    auto send = [&](int c) {
      if (one && o_tiles(c)) {
        for (int kb = 0; kb < 2; ++kb)
          tma_store_3d(maps.o, 64 * kb, h, (int)(tok0 + (long long)c * 64), sm + SM_V + 8192 * kb);
        bulk_commit();
      }
    };
    auto image = [&](uint8_t *dst, int c) {  // the E^T / E2^T image (hi | lo) for the backward
      static_assert(SM_XE_LO == SM_XE + 16384, "contiguous");
      bulk_s2g(dst + (size_t)(sp.rbase + c) * 32768, sm + SM_XE, 32768);
      bulk_commit();
    };
    if (NC > 0) {
      if (one) {
        if (RDNV) load_a(rec_of(0) + IMG_TB);
        load_b(rec_of(0) + IMG_APMQ, 32768);
      }
      load_gates(0);
      put_gates(0);
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
    for (int c = 0; c < NC; ++c) {
      const bool more = c + 1 < NC;
      const bool tma_next = more && by_tma(c + 1);
      const uint32_t ph = (uint32_t)c & 1u;
      if (by_tma(c) && one) await(barE, (armE - 1) & 1u);
      __syncwarp();
      __syncthreads();
      if (*flag) {
        alive = false;
        break;
      }
      if (more) load_gates(c + 1);
      if (one) {
        if (p.sv_E2 && c > 0) {
          bulk_wait_read();
          mbar_arrive(barJ);  // X may come over the chunk before's E2
        }
        if (more) prefetch_chunk(c + 1);
        if (RDNV) {
          await(barM2, ph);
          if (good) load_a(rec_of(c) + IMG_TG);
        }
      }
      __syncwarp();
      if (more) put_gates(c + 1);  // (its set was last read for chunk c - 1)
      bar_sync(kBarE, kScanThreads);
      if (one && p.sv_E) {
        image(p.sv_E, c);
        bulk_wait_read();
        mbar_arrive(barI);  // X2 may come over E
      }
      __syncwarp();
      bar_sync(kBarO, kOneMore);
      if (c > 0) send(c - 1);
      if (one) {
        bulk_wait_read();
        if (good && tma_next) {
          const int row = (int)(tok0 + (long long)(c + 1) * 64);
          ++armE;
          mbar_expect_tx(barE, 49152);
          for (int kb = 0; kb < 2; ++kb) tma_load_3d(sm + SM_V + kb * 8192, maps.v, 64 * kb, h, row, barE);
        }
      }
      __syncwarp();
      if (more && !by_tma(c + 1)) bar_arrive(kBarW, kOneMore);  // (V's place is free)
      if (one) {
        await(barM3, ph);
        if (good) load_b(rec_of(c) + IMG_M2, 16384);
        if (RDNV) {
          await(barM6, ph);
          if (good && more) load_a(rec_of(c + 1) + IMG_TB);
        }
      }
      __syncwarp();
      bar_sync(kBarE2, kScanThreads);
      if (one) {
        await(barM8, ph);
        if (good && tma_next) {  // K, Q are done with
          const int row = (int)(tok0 + (long long)(c + 1) * 64);
          for (int kb = 0; kb < 2; ++kb) {
            tma_load_3d(sm + SM_KQ + kb * 16384, maps.k, 64 * kb, h, row, barE);
            tma_load_3d(sm + SM_KQ + kb * 16384 + 8192, maps.q, 64 * kb, h, row, barE);
          }
        }
        if (p.sv_E2) image(p.sv_E2, c);  // (behind what the next chunk waits for)
        if (more) {
          await(barM7, ph);
          if (good) load_b(rec_of(c + 1) + IMG_APMQ, 32768);
        }
      }
      __syncwarp();
    }
    if (alive && NC > 0) {
      bar_sync(kBarO, kOneMore);
      send(NC - 1);
    }
    if (one) bulk_wait_all();
    __syncthreads();
    if ((!alive || *flag) && one) {  // every copy armed has landed, bounded
      if (armA) mbar_wait(barA, (armA - 1) & 1u);
      if (armB) mbar_wait(barB, (armB - 1) & 1u);
      if (armE) mbar_wait(barE, (armE - 1) & 1u);
    }
    __syncwarp();
    fence_before_sync();
    __syncthreads();
    return;
  }

  // ================================================= the 16 element-wise warps
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
  // chunk tiles (rows t, exact bf16, zero past the sequence end), asynchronous
  auto fetch = [&](int c) {
    const int t0 = c * 64, n = min(64, T - t0);
    for (int e = tid; e < 64 * 16; e += kTcThreads) {
      const int t = e >> 4, ch = e & 15;
      const bool vld = t < n;
      const size_t off = ((size_t)(tok0 + t0 + (vld ? t : 0)) * H + h) * D + ch * 8;
      const int blk = ch >> 3, cc = (ch & 7) * 8;
      cp_async16(sm + SM_V + blk * 8192 + sw128(t, cc), v + off, vld);
      cp_async16(sm + SM_KQ + blk * 16384 + sw128(t, cc), k + off, vld);
      cp_async16(sm + SM_KQ + blk * 16384 + sw128(64 + t, cc), q + off, vld);
    }
  };
  if (NC > 0) fetch(0);

  // S's bf16 copy and lo part (s - bf16(s)), 16 columns: the read-outs K S, Q S
  // use S to ~16 bits.  RLA's state is not contracted by a delta term and its
  // prediction S k is a large sum the residual v - S k cancels against; RDN's
  // single-bf16 read-outs put the output error of the long-context workload
  // (T = 16384) at the 2e-2 RMS bound.
  auto put_s = [&](int c0, const float (&s)[16]) {
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      hi[i] = pack_bf16(s[2 * i], s[2 * i + 1]);
      lo[i] = pack_bf16(s[2 * i] - __uint_as_float(hi[i] << 16),
                        s[2 * i + 1] - __uint_as_float(hi[i] & 0xFFFF0000u));
    }
    const uint32_t blk = (uint32_t)(c0 >> 6) * 16384u;
    static_assert(SM_W_LO - SM_W == 16384, "the lo part's second key block");
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint32_t at = blk + sw128(j, (c0 & 63) + 8 * u);
      *reinterpret_cast<uint4 *>(sm + SM_SA + at) =
          make_uint4(hi[4 * u], hi[4 * u + 1], hi[4 * u + 2], hi[4 * u + 3]);
      *reinterpret_cast<uint4 *>(sm + SM_W + at) =
          make_uint4(lo[4 * u], lo[4 * u + 1], lo[4 * u + 2], lo[4 * u + 3]);
    }
  };
  // initial states -> TMEM (fp32) and bf16 A operands
  for (int c0 = g16; c0 < D; c0 += 64) {
    float s[16], r[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      s[i] = p.S0 ? p.S0[st_base + (size_t)(c0 + i) * D + j] : 0.f;
      r[i] = p.R0 ? p.R0[st_base + (size_t)(c0 + i) * D + j] : 0.f;
    }
    tmem_st16x2(tm + lane + T_S + c0, s, tm + lane + T_R + c0, r);
    put_s(c0, s);
    st_row16(sm + SM_RA, 16384, j, c0, r);
    if (p.S_chunks && NC > 0) {  // the first chunk's start states, for the backward
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        p.S_chunks[(size_t)sp.rbase * D * D + (size_t)(c0 + i) * D + j] = s[i];
        p.R_chunks[(size_t)sp.rbase * D * D + (size_t)(c0 + i) * D + j] = r[i];
      }
    }
  }
  // a state's TMEM copy times the chunk's total decay, in place (its updates
  // accumulate onto it); this thread's columns.  The values it reads are the
  // chunk-start state; R's goes to `start` ([i][j], fp32; NULL = not kept) here,
  // while MMA1 runs (S's in copy_s: half the stores at each place).
  auto scale_state = [&](uint32_t col, float f, float *start) {
    float x[16], y[16];
    tmem_ld16x2(tm + lane + col + g16, x, tm + lane + col + g16 + 64, y);
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
    tmem_st16x2(tm + lane + col + g16, x, tm + lane + col + g16 + 64, y);
  };
  // S (= Gam_C S + U, complete in TMEM) -> its copies (W has been read)
  auto copy_s = [&](int c) {
    warp_wait(barM4, (uint32_t)c & 1u);
    fence_after_sync();
    float s0[16], s1[16];
    tmem_ld16x2(tm + lane + T_S + g16, s0, tm + lane + T_S + g16 + 64, s1);
    put_s(g16, s0);
    put_s(g16 + 64, s1);
    if (p.S_chunks && c + 1 < NC) {  // the next chunk's start state, for the backward
      float *start = p.S_chunks + (size_t)(sp.rbase + c + 1) * D * D;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        start[(size_t)(g16 + i) * D + j] = s0[i];
        start[(size_t)(g16 + 64 + i) * D + j] = s1[i];
      }
    }
  };
  uint32_t ow[8];  // the previous chunk's o at this thread's column, pairs of tokens
  // o into V's place as the tiles that leave (every V of this chunk has been read)
  auto stage_o = [&](int c) {
    if (o_tiles(c)) {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        *reinterpret_cast<unsigned short *>(sm + SM_V + (j >> 6) * 8192 + sw128(g16 + i, j & 63)) =
            (unsigned short)(i & 1 ? ow[i >> 1] >> 16 : ow[i >> 1]);
    }
  };

  bool alive = true;
  for (int c = 0; c < NC && alive; ++c) {
    const size_t ci = (size_t)(sp.rbase + c);  // chunk index of the saved intermediates
    const bool more = c + 1 < NC;
    if (!by_tma(c)) cp_async_wait_all();
    fence_async_smem();
    fence_before_sync();
    __syncthreads();  // (with the copying warp, which has waited for the tiles)
    fence_after_sync();
    if (*flag) {
      alive = false;
      break;
    }
    const float *Gam = reinterpret_cast<const float *>(sm + SM_VEC) + kVec * (c & 1);
    const float *Gprev = Gam + 64, *wS = Gam + 128, *wR = Gam + 192, *gamv = Gam + 256;
    {
      const float GamC = Gam[320];
      scale_state(T_S, GamC, nullptr);
      scale_state(T_R, stl ? 0.f : GamC, p.S_chunks && c > 0 ? p.R_chunks + ci * D * D : nullptr);
    }
    wait_chain();
    if (p.sv_E2 && c > 0) warp_wait(barJ, (uint32_t)(c - 1) & 1u);  // (its image has left XE)
    // ---- X = V - Gam KS (= V - alpha Gprev KS); P accumulates onto Gprev KS (kept in
    // registers while MMA2 overwrites it), Ob onto Gam scale QS
    float gks[16], vv[16];
    {
      float x[16], gm[16];
      tmem_ld16(tm + lane + T_D1 + g16, gks);
      lds16(Gam + g16, gm);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        vv[i] = __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(
            sm + SM_V + (j >> 6) * 8192 + sw128(g16 + i, j & 63)));
        x[i] = vv[i] - gm[i] * gks[i];
      }
      if (RDNV) {
        st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, x);
        publish(kBarX, kOneMore);
      }
      lds16(dec_res ? Gam + g16 : Gprev + g16, gm);  // (decayed residual: P = a S_{t-1} k)
#pragma unroll
      for (int i = 0; i < 16; ++i) gks[i] *= gm[i];
    }
    if (RDNV) wait_chain();
    // ---- E, wS E
    {
      float e[16], w[16], x[16];
      tmem_ld16x2(tm + lane + T_D1 + g16, e, tm + lane + T_D1 + 64 + g16, x);
      lds16(plain ? Gprev + g16 : Gam + g16, w);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        x[i] *= w[i] * p.scale;
        if (!RDNV) e[i] = vv[i];
      }
      tmem_st16x2(tm + lane + T_D1 + g16, gks, tm + lane + T_D1 + 64 + g16, x);
      lds16(wS + g16, w);
#pragma unroll
      for (int i = 0; i < 16; ++i) w[i] *= e[i];
      st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, e);
      st_row16_split(sm + SM_W, sm + SM_W_LO, j, g16, w);
    }
    publish(kBarE, kScanThreads);
    if (RDNV) {  // (MMA2 was waited for: every warp has read its V)
      if (c > 0) stage_o(c - 1);
      publish(kBarO, kOneMore);
    }
    wait_chain();
    if (!RDNV) {
      if (c > 0) stage_o(c - 1);
      publish(kBarO, kOneMore);
    }
    // ---- r = clip(V - P);  X2 = r - Gam KR
    float r[16];
    {
      float pp[16];
      tmem_ld16(tm + lane + T_D1 + g16, pp);
      if (!tnh && !p.sv_mask) {
#pragma unroll
        for (int i = 0; i < 16; ++i) r[i] = clampf(vv[i] - pp[i], clip);
      } else if (!tnh) {
        unsigned msk = 0u;  // bit i: |x| <= c at t = g16 + i (the clip passes the gradient)
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float x = vv[i] - pp[i];
          if (fabsf(x) <= clip) msk |= 1u << i;
          r[i] = clampf(x, clip);
        }
        // bits [g16, g16 + 16) of the column's 64-bit mask word (little-endian)
        reinterpret_cast<uint16_t *>(p.sv_mask + ci * D + j)[g16 >> 4] = (uint16_t)msk;
      } else {
        uint32_t dg[8];  // the derivative at t = g16 .. g16 + 15, pairs of 16-bit words
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
    }
    if (p.sv_E) warp_wait(barI, (uint32_t)c & 1u);  // (E's image has left XE)
    if (RDNV) {
      {
        float x[16], gm[16];
        tmem_ld16(tm + lane + T_X + g16, x);
        lds16(Gam + g16, gm);
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = stl ? r[i] : r[i] - gm[i] * x[i];
        st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, x);
      }
      publish(kBarX2, kOneMore);
      copy_s(c);
      wait_chain();
      tmem_ld16(tm + lane + T_D1 + g16, r);  // E2
    }
    // ---- E2, wR E2
    {
      float w[16];
      uint32_t hi[8], lo[8];
      lds16(wR + g16, w);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        split_pack_bf16(w[2 * i] * r[2 * i], w[2 * i + 1] * r[2 * i + 1], hi[i], lo[i]);
      tmem_st8x2(tm + lane + T_X + g16 / 2, hi, tm + lane + T_X + 32 + g16 / 2, lo);
      st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, r);
    }
    publish(kBarE2, kScanThreads);
    if (!RDNV) copy_s(c);
    wait_chain();
    {  // R (= Gam_C R + U2) -> its copy
      float r0[16], r1[16];
      tmem_ld16x2(tm + lane + T_R + g16, r0, tm + lane + T_R + g16 + 64, r1);
      st_row16(sm + SM_RA, 16384, j, g16, r0);
      st_row16(sm + SM_RA, 16384, j, g16 + 64, r1);
    }
    warp_wait(barM7, (uint32_t)c & 1u);
    fence_after_sync();
    if (more && !by_tma(c + 1)) {  // (K, Q and V's place are free)
      bar_sync(kBarW, kOneMore);
      fetch(c + 1);
    }
    {  // o = (Ob + diag(gamma) M2 E2) + gamma * Gam QR
      const int t0 = c * 64, n = min(64, T - t0);
      float ob[16], oa[16], gm[16], gv[16];
      tmem_ld16x2(tm + lane + T_D1 + 64 + g16, ob, tm + lane + T_X + 64 + g16, oa);
      lds16(Gam + g16, gm);
      lds16(gamv + g16, gv);
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (!stl) ob[i] = fmaf((plain ? 1.f : gv[i]) * gm[i] * p.scale, oa[i], ob[i]);
      if (o_tiles(c)) {
#pragma unroll
        for (int i = 0; i < 8; ++i) ow[i] = pack_bf16(ob[2 * i], ob[2 * i + 1]);
      } else {  // fp32 results, the ragged last chunk
        const size_t row = ((size_t)(tok0 + t0 + g16) * H + h) * D + j;
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (g16 + i < n) {
            if (p.f32out) ((float *)p.o)[row + (size_t)i * H * D] = ob[i];
            else ((__nv_bfloat16 *)p.o)[row + (size_t)i * H * D] = __float2bfloat16_rn(ob[i]);
          }
      }
    }
  }

  if (alive && NC > 0) {
    stage_o(NC - 1);
    publish(kBarO, kOneMore);
  }
  __syncthreads();
  if (*flag) alive = false;
  if (alive) {  // final states
    for (int c0 = g16; c0 < D; c0 += 64) {
      float s[16], r[16];
      tmem_ld16x2(tm + lane + T_S + c0, s, tm + lane + T_R + c0, r);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        if (p.ST) p.ST[st_base + (size_t)(c0 + i) * D + j] = s[i];
        if (p.RT) p.RT[st_base + (size_t)(c0 + i) * D + j] = r[i];
      }
    }
  }
  cp_async_wait_all();
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tm, 512);
}

}  // namespace

namespace {
// the driver's tensor-map encoder, looked up once through the runtime (no
// link against the driver library)
PFN_cuTensorMapEncodeTiled_v12000 tile_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  }();
  return fn;
}
}  // namespace

bool make_tile_map(void *map128, const void *base, int D, int H, long long rows) {
  static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
  const auto enc = tile_map_encoder();
  if (!enc || !base || rows < 1) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)H, (cuuint64_t)rows};
  const cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)H * D * 2};  // bytes, dims 1, 2
  const cuuint32_t box[3] = {64, 1, 64};
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(reinterpret_cast<CUtensorMap *>(map128), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
             const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t launch_fwd_tc(const FwdParams &p, bool rdnv, cudaStream_t s) {
  fwdtc::FwdMaps maps;
  const long long rows = (long long)p.B * p.T;
  maps.ok = make_tile_map(maps.v, p.v, D, p.H, rows) && make_tile_map(maps.k, p.k, D, p.H, rows) &&
            make_tile_map(maps.q, p.q, D, p.H, rows);
  int nsm = 0;
  cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  FwdParams one = p;
  const bool both = pick_on_device(p, rdnv, nsm);
  maps.o_ok = !p.f32out && make_tile_map(maps.o, p.o, D, p.H, rows);
  if (both || use_pairs(p, rdnv, nsm)) {
    FwdParams two = p;
    two.pick = both ? 2 : 0;
    if ((e = launch_fwd_pair(two, maps, rdnv, s)) != cudaSuccess || !both) return e;
    one.pick = 1;
  }
  const bool generic = p.mods != 0;
  auto kern = rdnv ? (generic ? fwd_tc_kernel<true, true> : fwd_tc_kernel<true, false>)
                   : (generic ? fwd_tc_kernel<false, true> : fwd_tc_kernel<false, false>);
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem);
  if (e != cudaSuccess) return e;
  RDN_LAUNCH("fwd_tc_scan", s, kern<<<p.nseq * p.H, kScanThreads, kTcSmem, s>>>(one, maps));
  return cudaGetLastError();
}

}  // namespace rdn
