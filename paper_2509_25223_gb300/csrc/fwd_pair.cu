// fwd_pair.cu -- the tensor-core forward scan of fwd_tc.cu over a pair of CTAs
// (a cluster of two SMs) per (sequence, head), for calls whose sequences are
// too few to fill the chip.
//
// The scan is a chain of dependent phases per chunk, so a single sequence is
// bound by their latencies and not by any pipe.  The base recurrence never
// reads the auxiliary one: CTA 0 carries S, forms E, the clipped residual r
// and the base output Ob, and sends r and Ob (32 fp32 values a thread, the
// same thread mapping on both sides) into CTA 1's shared memory; CTA 1 carries
// R and finishes the output, one chunk behind.  Products and arithmetic are
// those of fwd_tc.cu, in the same order: the results are the same bits.
//
// Within a CTA only the carried state is a chain (operand names as there):
//
//   CTA 0:  K S  ->  X  ->  MMA2 E   ->  wS E   ->  MMA4 S  ->  S's copies
//   CTA 1:  K R  ->  X2 ->  MMA6 E2  ->  wR E2  ->  MMA8 R  ->  R's copy
//
// and what hangs off it is issued behind it on the tensor pipe and finished
// under a later phase: MMA3 [P | Ob] and MMA7 behind MMA4 and MMA8 on a barrier
// of their own, their read-outs (r and Ob handed over; o stored) under the next
// chunk's first product, whose accumulators are a second set of TMEM columns.
// The products are issued by a warp of their own and the copies by another: an
// issuing thread is held for most of its products' time (54 cycles a 128 x 64 x
// 16 product, 70 a 128 x 128 x 16 one, which the operands' shared-memory reads
// set); as one of the 16 element-wise warps it held up all the others, and
// issuing the copies as well it delayed the next chunk's K and Q by 800 cycles.
//
// The hand-over is one 64 KB buffer in CTA 1, filled by bulk copies of each
// warp's part from CTA 0's shared memory, with a pair of mbarriers: `full` in
// CTA 1 (the copies' bytes), `empty` in CTA 0 (one arrival per warp of CTA 1
// once it holds the values in registers; CTA 0 then also reuses what it copied
// from).  Every wait is bounded: a thread whose wait gave up sets the CTA's
// flag, which all read after the next chunk's first barrier; a CTA that gave up
// stops, its partner's waits then run out too, and the two meet at the
// cluster's barrier before either releases its shared memory.
#include "fwd_tc.cuh"

namespace rdn {
namespace {

using namespace fwdtc;

// shared memory (bytes from the 1024-aligned base); both CTAs:
constexpr uint32_t SM_ST = 0;        // the carried state's bf16 copy, two 64-column blocks
constexpr uint32_t SM_KQ = 32768;    // [K ; Q], 128 rows x 128
constexpr uint32_t SM_XE = 65536;    // X^T then E^T (X2^T then E2^T), hi | lo
constexpr uint32_t SM_XE_LO = 81920;
constexpr uint32_t SM_OUT = 98304;   // CTA 0: Ob, fp32, being handed over; CTA 1: o's rows
constexpr uint32_t SM_SLOTA = 131072;  // T_beta / T_gamma image (hi | lo)
constexpr uint32_t SM_SLOTB = 147456;  // [Ap ; Mq] image, 32 KB / M2 image, 16 KB
// CTA 0: r, fp32, being handed over (32 KB), V;  CTA 1: the hand-over buffer (r | Ob)
constexpr uint32_t SM_RES = 180224, SM_V = 212992;
constexpr uint32_t SM_X = 163840;
// two chunks' gates, fp32: Gam, Gprev / gamma, wS / wR (64 each), GamC
constexpr uint32_t SM_VEC = 229376;
constexpr int kVec = 196;
constexpr uint32_t SM_BAR = SM_VEC + 2 * kVec * 4;
// mbarriers: chain, slot A, slot B, drain, tiles, hand-over, side, MMA2 / 6, MMA4 / 8, image
constexpr uint32_t SM_SLOT = SM_BAR + 80;
constexpr uint32_t SM_FLAG = SM_SLOT + 4;
constexpr size_t kPairSmem = SM_FLAG + 4;
static_assert(SM_X + 65536 == SM_VEC && SM_V + 16384 == SM_VEC, "carve-up");
static_assert(kPairSmem <= 232448, "shared memory");

constexpr int kPairThreads = kTcThreads + 64;  // and the issuing and the copying warp
constexpr int kHandThreads = kTcThreads + 32;  // the element-wise warps and one of the two
// named barriers on which the element-wise warps hand operands to the issuing
// warp (X, E) and results to the copying warp (O), one among themselves, and one
// on which both wait before the last chunk's results (Z).  No barrier may be
// arrived at again before all its threads have joined the time before: within the
// loop the chunk's first barrier, which every warp joins, keeps two uses apart;
// behind it nothing does, so that the last use of O waits on Z, which the copying
// warp joins once it has left O.
constexpr int kBarX = 1, kBarE = 2, kBarO = 3, kBarW = 4, kBarZ = 5;

// TMEM columns: the state; CTA 0: KS | QS, then E | Ob, then P | Ob, two sets by
// the chunk's parity, then as A operands S's lo part and (wS E)^T (hi | lo), so
// that their shared memory can hold what is being handed over; CTA 1: KR | QR,
// two sets, where (wR E2)^T takes KR's place, and E2 | Ob
constexpr uint32_t T_ST = 0, T_PAR = 128, T_D1 = 384, T_SLO = 384, T_W = 448;

template <bool RDNV, bool kGeneric>
__global__ void __launch_bounds__(kPairThreads, 1)
    fwd_pair_kernel(FwdParams p, const __grid_constant__ FwdMaps maps) {
  extern __shared__ __align__(1024) uint8_t sm[];
  const uint32_t sbase = smem_u32(sm);
  if (!picked(p)) return;
  if (sbase & 1023u) {  // (the same in both CTAs)
    if (threadIdx.x == 0 && p.err) atomicExch(p.err, RDN_ERR_CUDA);
    return;
  }
  uint64_t *bar = reinterpret_cast<uint64_t *>(sm + SM_BAR);
  uint64_t *barA = bar + 1, *barB = bar + 2, *barD = bar + 3, *barE = bar + 4;
  uint64_t *barX = bar + 5;  // CTA 1: full; CTA 0: empty
  uint64_t *barN = bar + 6;  // the products issued behind the chain's
  uint64_t *barM2 = bar + 7, *barM4 = bar + 8;  // MMA2 / 6 and MMA4 / 8, for the copying warp
  uint64_t *barJ = bar + 9;  // E's image has left
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + SM_SLOT);
  volatile int *flag = reinterpret_cast<volatile int *>(sm + SM_FLAG);

  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t rank = cluster_rank();
  const bool base = rank == 0;     // CTA 0: S; CTA 1: R
  const int j = tid & 127;         // value column == TMEM lane
  const int g16 = (warp >> 2) * 16;  // this thread's token (and state) columns start
  const int sq = seq_at(p, (blockIdx.x >> 1) / p.H), h = (blockIdx.x >> 1) % p.H;
  const SeqSpan sp = seq_span(p, sq, h);
  const long long tok0 = sp.tok0;
  const int T = sp.len, H = p.H, NC = sp.nc;
  const __nv_bfloat16 *q = (const __nv_bfloat16 *)p.q;
  const __nv_bfloat16 *k = (const __nv_bfloat16 *)p.k;
  const __nv_bfloat16 *v = (const __nv_bfloat16 *)p.v;
  const float clip = p.clip;
  // (the variants: fwd_tc.cu)
  const bool dec_res = kGeneric && (p.mods & RDN_FLAG_DECAYED_RESIDUAL);
  const bool plain = kGeneric && (p.mods & RDN_FLAG_PLAIN_COMBINE);
  const bool tnh = kGeneric && (p.mods & RDN_FLAG_TANH_RESIDUAL);
  const bool stl = kGeneric && (p.mods & RDN_FLAG_STATELESS_AUX);
  const size_t st_base = ((size_t)sq * p.H + h) * D * D;
  uint8_t *keep = base ? p.sv_E : p.sv_E2;  // E's images (hi | lo) for the backward

  if (tid == 0) {
    for (int b = 0; b < 5; ++b) mbar_init(bar + b, 1);
    mbar_init(barX, base ? kTcThreads / 32 : 1);
    mbar_init(barN, 1);
    mbar_init(barM2, 1);
    mbar_init(barM4, 1);
    mbar_init(barJ, 1);
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
  const long long limit = p.inject == 1 ? 10000000ll : 2000000000ll;
  const uint32_t peer_bar = map_rank(barX, rank ^ 1u);
  const uint32_t peer_x = map_rank(sm + SM_X, 1u);
  uint32_t phase = 0;  // chain phases waited for (parity)
  // a warp's wait: one lane polls (512 polling threads take shared-memory
  // bandwidth from the products' operands)
  auto warp_wait = [&](uint64_t *b, uint32_t parity) {
    if ((tid & 31) == 0 && !mbar_wait(b, parity, limit)) *flag = 1;
    __syncwarp();
  };
  auto wait_chain = [&] {
    warp_wait(bar, phase);
    phase ^= 1u;
    fence_after_sync();
  };
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
  // (CTA 1) whether chunk c's o leaves as two tensor-map tiles (whole chunks of
  // bf16 results; a row-by-row copy of 64 rows holds its source for 4k cycles)
  auto o_tiles = [&](int c) { return maps.o_ok && T - c * 64 >= 64; };
  auto by_tma = [&](int cc) { return maps.ok && cc > 0 && cc < NC - 1; };
  if (warp == kTcThreads / 32) {
    // =============================================== the issuing warp (lane 0)
    bool one = (tid & 31) == 0;
    bool skip_commit = p.inject == 1 && base;
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
      const uint32_t d1 = T_PAR + 128u * (c & 1), tw = base ? T_W : d1;
      __syncthreads();
      fence_after_sync();
      if (*flag) {
        alive = false;
        break;
      }
      if (one) {  // the state's read-outs [K ; Q] S (S as hi + lo) / [K ; Q] R (RLA: Q R)
        if (base) {
          mma_tile(tm + d1, sbase + SM_ST, 16384, sbase + SM_KQ, 16384, 8, i128, false);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_bf16_ta(tm + d1, tm + T_SLO + 8 * kk,
                        sdesc_sw128(sbase + SM_KQ + (kk >> 2) * 16384 + (kk & 3) * 32), i128, 1u);
        } else if (RDNV) {
          mma_tile(tm + d1, sbase + SM_ST, 16384, sbase + SM_KQ, 16384, 8, i128, false);
        } else {
          mma_tile(tm + d1 + 64, sbase + SM_ST, 16384, sbase + SM_KQ + 8192, 16384, 8, i64, false);
        }
        if (RDNV || base) {
          if (!skip_commit) mma_commit(bar);
          skip_commit = false;
        }
      }
      __syncwarp();
      if (RDNV) {  // MMA2: E^T = X^T T_beta^T / MMA6: E2^T = X2^T T_gamma^T
        bar_sync(kBarX, kHandThreads);
        fence_after_sync();
        if (one && wait_copy(barA, (uint32_t)c & 1u)) {
          mma_split3(tm + (base ? d1 : T_D1), sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTA,
                     sbase + SM_SLOTA + 8192, i64, false);
          mma_commit(bar);
          mma_commit(barM2);
        }
        __syncwarp();
      }
      bar_sync(kBarE, kHandThreads);
      fence_after_sync();
      if (one) {
        // MMA4: S += (wS E)^T K / MMA8: R += (wR E2)^T K (hi, then lo); behind it
        // MMA3: D1 += E^T [Ap;Mq]^T / MMA7: Ob += E2^T (gamma M2)^T
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          mma_bf16_ta(tm + T_ST, tm + tw + 8 * kk, sdesc_sw128_mn(sbase + SM_KQ + (kk & 3) * 2048, 16384),
                      i128 | kBMajorMN, 1u);
        mma_commit(bar);
        mma_commit(barM4);
        if (wait_copy(barB, (uint32_t)c & 1u)) {
          if (base)
            mma_split3(tm + d1, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTB,
                       sbase + SM_SLOTB + 16384, i128, true);
          else
            mma_split3(tm + T_D1 + 64, sbase + SM_XE, sbase + SM_XE_LO, sbase + SM_SLOTB,
                       sbase + SM_SLOTB + 8192, i64, true);
          mma_commit(barN);
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
    cluster_sync();
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
    auto load_a = [&](int c) {  // T_beta / T_gamma
      ++armA;
      mbar_expect_tx(barA, 16384);
      bulk_g2s(sm + SM_SLOTA, rec_of(c) + (base ? IMG_TB : IMG_TG), 16384, barA);
    };
    auto load_b = [&](int c) {  // [Ap ; Mq] / M2
      const uint32_t bytes = base ? 32768u : 16384u;
      ++armB;
      mbar_expect_tx(barB, bytes);
      bulk_g2s(sm + SM_SLOTB, rec_of(c) + (base ? IMG_APMQ : IMG_M2), bytes, barB);
    };
    auto arm_tiles = [&] {
      ++armE;
      mbar_expect_tx(barE, base ? 49152u : 32768u);
    };
    auto load_v = [&](int c) {
      const int row = (int)(tok0 + (long long)c * 64);
      for (int kb = 0; kb < 2; ++kb) tma_load_3d(sm + SM_V + kb * 8192, maps.v, 64 * kb, h, row, barE);
    };
    auto load_kq = [&](int c) {
      const int row = (int)(tok0 + (long long)c * 64);
      for (int kb = 0; kb < 2; ++kb) {
        tma_load_3d(sm + SM_KQ + kb * 16384, maps.k, 64 * kb, h, row, barE);
        tma_load_3d(sm + SM_KQ + kb * 16384 + 8192, maps.q, 64 * kb, h, row, barE);
      }
    };
    // a chunk's gates, lane l those of tokens l and l + 32: loaded a chunk ahead,
    // written to their set once nothing reads it any more
    float g0[2], g1[2], g2[2], gc = 0.f;
    auto load_gates = [&](int c) {
      const float *rc = p.ws + (size_t)(sp.rbase + c) * kRecFloats + OFF_VEC;
      const int t0 = c * 64, n = min(64, T - t0);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int t = ln + 32 * u;
        g0[u] = rc[V_GAM + t];
        g1[u] = base ? rc[V_GPREV + t] : t < n ? p.gamma[(size_t)(tok0 + t0 + t) * H + h] : 0.f;
        g2[u] = rc[(base ? V_WS : V_WR) + t];
      }
      gc = rc[V_GAMC];
    };
    auto put_gates = [&](int c) {
      float *v = reinterpret_cast<float *>(sm + SM_VEC) + kVec * (c & 1);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int t = ln + 32 * u;
        v[t] = g0[u];
        v[64 + t] = g1[u];
        v[128 + t] = g2[u];
      }
      if (ln == 0) v[192] = gc;
    };
    // L2 prefetch of what this CTA reads of a chunk
    auto prefetch_chunk = [&](int c) {
      const uint8_t *r = rec_of(c);
      prefetch_l2_bulk(r + (base ? IMG_TB : IMG_TG), base ? 49152 : 32768);
      static_assert(IMG_APMQ == IMG_TB + 16384 && IMG_M2 == IMG_TG + 16384, "contiguous images");
      prefetch_l2_bulk(r + OFF_VEC * 4, (kRecFloats - OFF_VEC) * 4);
      if (!maps.ok) return;
      const int row = (int)(tok0 + (long long)c * 64);
      for (int kb = 0; kb < 2; ++kb) {
        tma_prefetch_3d(maps.k, 64 * kb, h, row);
        tma_prefetch_3d(maps.q, 64 * kb, h, row);
        if (base) tma_prefetch_3d(maps.v, 64 * kb, h, row);
      }
    };
    // CTA 0: chunk c's r and Ob, staged by the element-wise warps -> CTA 1;
    // CTA 1: chunk c's o rows -> global memory
    uint32_t handed = 0;
    auto send = [&](int c) {
      bar_sync(kBarO, kHandThreads);
      if (base) {
        if (one) {
          bulk_s2s(peer_x, sm + SM_RES, 32768, peer_bar);
          bulk_s2s(peer_x + 32768, sm + SM_OUT, 32768, peer_bar);
        }
        ++handed;
        return;
      }
      const int t0 = c * 64, n = min(64, T - t0);
      if (o_tiles(c)) {
        if (one) {
          for (int kb = 0; kb < 2; ++kb)
            tma_store_3d(maps.o, 64 * kb, h, (int)(tok0 + t0), sm + SM_OUT + 8192 * kb);
          bulk_commit();
        }
        return;
      }
      const uint32_t bytes = p.f32out ? 512u : 256u;
      for (int t = ln; t < n; t += 32)
        bulk_s2g((uint8_t *)p.o + ((size_t)(tok0 + t0 + t) * H + h) * bytes, sm + SM_OUT + t * bytes, bytes);
      bulk_commit();
    };
    if (NC > 0) {
      if (one) {
        if (RDNV) load_a(0);
        load_b(0);
      }
      load_gates(0);
      put_gates(0);
    }
    bool alive = true, good = true;  // good: (lane 0) no wait of this warp gave up
    // (a wait that gave up leaves its phase incomplete, which takes no further
    // arrival: nothing is armed after it)
    auto await = [&](bool done) {
      if (!done) {
        good = false;
        *flag = 1;
      }
    };
    for (int c = 0; c < NC; ++c) {
      const bool more = c + 1 < NC;
      const bool tma_next = more && by_tma(c + 1);
      if (by_tma(c) && one) await(mbar_wait(barE, (armE - 1) & 1u));
      // o of the chunk before has left its staging; E's image, which went out
      // behind it (lane 0), is waited for past the barrier
      if (one && keep && c > 0) bulk_wait_read_all_but_last();
      else bulk_wait_read();
      __syncwarp();
      __syncthreads();
      if (*flag) {
        alive = false;
        break;
      }
      if (more) load_gates(c + 1);
      if (one) {
        if (keep && c > 0) {
          bulk_wait_read();
          mbar_arrive(barJ);
        }
        if (more) prefetch_chunk(c + 1);
        if (c > 0) {  // slot B: free once chunk c - 1's product with it is complete
          await(mbar_wait(barN, (uint32_t)(c - 1) & 1u, limit));
          if (good) load_b(c);
        }
      }
      __syncwarp();
      if (c > 0) send(c - 1);
      if (RDNV) {
        if (one) {
          await(mbar_wait(barM2, (uint32_t)c & 1u, limit));
          if (good && more) load_a(c + 1);
          if (good && base && tma_next) {  // (every V of this chunk has been read)
            arm_tiles();
            load_v(c + 1);
          }
        }
        __syncwarp();
        if (more) put_gates(c + 1);  // (CTA 1: chunk c - 1's are read before MMA6)
      }
      if (one) {
        await(mbar_wait(barM4, (uint32_t)c & 1u, limit));
        if (good && tma_next) {  // K, Q are done with
          if (!RDNV || !base) arm_tiles();
          if (!RDNV && base) load_v(c + 1);
          load_kq(c + 1);
        }
        if (keep) {
          static_assert(SM_XE_LO == SM_XE + 16384, "contiguous");
          bulk_s2g(keep + (size_t)(sp.rbase + c) * 32768, sm + SM_XE, 32768);
          bulk_commit();
        }
        // the copies of chunk c - 1 have left what chunk c's are staged in next
        if (base && c > 0) await(mbar_wait_cluster(barX, (uint32_t)(c - 1) & 1u, limit));
      }
      __syncwarp();
      if (!RDNV && more) put_gates(c + 1);
    }
    if (alive && NC > 0) {
      bulk_wait_read();  // (what the last chunk's results are staged in is free)
      __syncwarp();
      bar_sync(kBarZ, kHandThreads);
      send(NC - 1);
    }
    bulk_wait_all();
    __syncthreads();
    if ((!alive || *flag) && one) {  // every copy armed has landed, bounded
      if (armA) mbar_wait(barA, (armA - 1) & 1u);
      if (armB) mbar_wait(barB, (armB - 1) & 1u);
      if (armE) mbar_wait(barE, (armE - 1) & 1u);
      if (handed) mbar_wait_cluster(barX, (handed - 1) & 1u, limit);  // (those into CTA 1)
    }
    __syncwarp();
    fence_before_sync();
    __syncthreads();
    cluster_sync();
    return;
  }

  // ================================================= the 16 element-wise warps
  if (NC > 0) {
    if (base) fetch_v(0);
    fetch_kq(0);
  }

  // a state's bf16 copy, and CTA 0's also its lo part (s - bf16(s)), 16 columns
  auto put_state = [&](int c0, const float (&s)[16]) {
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      hi[i] = pack_bf16(s[2 * i], s[2 * i + 1]);
      lo[i] = pack_bf16(s[2 * i] - __uint_as_float(hi[i] << 16),
                        s[2 * i + 1] - __uint_as_float(hi[i] & 0xFFFF0000u));
    }
    const uint32_t blk = (uint32_t)(c0 >> 6) * 16384u;
#pragma unroll
    for (int u = 0; u < 2; ++u)
      *reinterpret_cast<uint4 *>(sm + SM_ST + blk + sw128(j, (c0 & 63) + 8 * u)) =
          make_uint4(hi[4 * u], hi[4 * u + 1], hi[4 * u + 2], hi[4 * u + 3]);
    if (base) tmem_st8(tm + lane + T_SLO + c0 / 2, lo);
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

  // hand this warp's shared-memory writes and TMEM accesses to the issuing or
  // the copying warp
  auto publish = [&](int id) {
    fence_async_smem();
    fence_before_sync();
    bar_arrive(id, kHandThreads);
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
  float vv[16];         // CTA 0: this thread's V entries of the last chunk begun
  // CTA 0: chunk c's P | Ob are complete: r = clip(V - P); r and Ob -> CTA 1.
  // (The copies of chunk c - 1 have left their places: the copying warp saw
  // `empty` before this chunk's first barrier.)
  auto hand_over = [&](int c) {
    const size_t ci = (size_t)(sp.rbase + c);
    const uint32_t d1 = T_PAR + 128u * (c & 1);
    warp_wait(barN, (uint32_t)c & 1u);
    fence_after_sync();
    float pp[16], ob[16];
    tmem_ld16x2(tm + lane + d1 + g16, pp, tm + lane + d1 + 64 + g16, ob);
    if (!tnh && !p.sv_mask) {
#pragma unroll
      for (int i = 0; i < 16; ++i) pp[i] = clampf(vv[i] - pp[i], clip);
    } else if (!tnh) {
      unsigned msk = 0u;  // bit i: |x| <= c at t = g16 + i
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float x = vv[i] - pp[i];
        if (fabsf(x) <= clip) msk |= 1u << i;
        pp[i] = clampf(x, clip);
      }
      reinterpret_cast<uint16_t *>(p.sv_mask + ci * D + j)[g16 >> 4] = (uint16_t)msk;
    } else {
      uint32_t dg[8];
#pragma unroll
      for (int i = 0; i < 16; i += 2) {
        const float x0 = vv[i] - pp[i], x1 = vv[i + 1] - pp[i + 1];
        pp[i] = resid_map(x0, clip, true);
        pp[i + 1] = resid_map(x1, clip, true);
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
    float4 *xr = reinterpret_cast<float4 *>(sm + SM_RES + 2048 * warp) + (tid & 31);
    float4 *xo = reinterpret_cast<float4 *>(sm + SM_OUT + 2048 * warp) + (tid & 31);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      xr[32 * i] = make_float4(pp[4 * i], pp[4 * i + 1], pp[4 * i + 2], pp[4 * i + 3]);
      xo[32 * i] = make_float4(ob[4 * i], ob[4 * i + 1], ob[4 * i + 2], ob[4 * i + 3]);
    }
    publish(kBarO);
  };
  // CTA 1: chunk c's Ob + gamma M2 E2 is complete: o = that + gamma Gam QR,
  // staged as tiles or rows [t][j] (2-byte stores of them straight to
  // global memory took 2.9k cycles a chunk)
  auto finish_o = [&](int c) {
    const float *Gam = reinterpret_cast<const float *>(sm + SM_VEC) + kVec * (c & 1), *gamv = Gam + 64;
    warp_wait(barN, (uint32_t)c & 1u);
    fence_after_sync();
    float ob[16], oa[16], gm[16], gv[16];
    tmem_ld16x2(tm + lane + T_D1 + 64 + g16, ob, tm + lane + T_PAR + 128u * (c & 1) + 64 + g16, oa);
    lds16(Gam + g16, gm);
    lds16(gamv + g16, gv);
    const bool tiles = o_tiles(c);
    __nv_bfloat16 *stg = reinterpret_cast<__nv_bfloat16 *>(sm + SM_OUT) + g16 * D + j;
    float *stg32 = reinterpret_cast<float *>(sm + SM_OUT) + g16 * D + j;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float gg = plain ? 1.f : gv[i];
      const float ov = stl ? ob[i] : fmaf(gg * gm[i] * p.scale, oa[i], ob[i]);
      if (tiles)
        *reinterpret_cast<__nv_bfloat16 *>(sm + SM_OUT + (j >> 6) * 8192 + sw128(g16 + i, j & 63)) =
            __float2bfloat16_rn(ov);
      else if (p.f32out) stg32[i * D] = ov;
      else stg[i * D] = __float2bfloat16_rn(ov);
    }
    publish(kBarO);
  };
  // (wS E)^T / (wR E2)^T as an A operand in TMEM
  auto put_w = [&](uint32_t col, const float (&w)[16]) {
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) split_pack_bf16(w[2 * i], w[2 * i + 1], hi[i], lo[i]);
    tmem_st8x2(tm + lane + col + g16 / 2, hi, tm + lane + col + 32 + g16 / 2, lo);
  };
  // CTA 1: this warp has used what it read of the hand-over buffer (r and ob: the
  // arrival orders nothing, the uses before it do)
  auto taken = [&](bool got) {
    __syncwarp();
    if (got && (tid & 31) == 0) mbar_arrive_remote_relaxed(peer_bar);
    __syncwarp();  // (TMEM accesses follow, which take whole warps)
  };

  bool alive = true;
  for (int c = 0; c < NC && alive; ++c) {
    const size_t ci = (size_t)(sp.rbase + c);  // chunk index of the saved intermediates
    const bool more = c + 1 < NC;
    if (!by_tma(c)) cp_async_wait_all();
    float *start = (chunks && c > 0) ? chunks + ci * D * D : nullptr;
    fence_async_smem();
    fence_before_sync();
    __syncthreads();  // (with the copying warp, which has waited for the tiles)
    fence_after_sync();
    if (*flag) {
      alive = false;
      break;
    }
    const float *Gam = reinterpret_cast<const float *>(sm + SM_VEC) + kVec * (c & 1);
    const float *Gp = Gam + 64, *ww = Gam + 128;
    const float GamC = Gam[192];
    const uint32_t d1 = T_PAR + 128u * (c & 1);
    if (base) {
      if (c > 0) hand_over(c - 1);
      if (!RDNV) scale_state(GamC, start);
      wait_chain();
      if (keep && c > 0) warp_wait(barJ, (uint32_t)(c - 1) & 1u);  // (E's image has left XE)
      float gks[16];
      {
        float x[16], gm[16];
        tmem_ld16(tm + lane + d1 + g16, gks);
        lds16(Gam + g16, gm);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          vv[i] = __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(
              sm + SM_V + (j >> 6) * 8192 + sw128(g16 + i, j & 63)));
          x[i] = vv[i] - gm[i] * gks[i];
        }
        if (RDNV) st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, x);
        lds16(dec_res ? Gam + g16 : Gp + g16, gm);
#pragma unroll
        for (int i = 0; i < 16; ++i) gks[i] *= gm[i];
      }
      if (RDNV) {
        publish(kBarX);
        scale_state(GamC, start);  // (the read-outs use the state's bf16 copies)
        wait_chain();
      }
      {  // E, wS E; P and Ob accumulate onto Gprev KS and Gam scale QS
        float e[16], w[16], x[16];
        tmem_ld16x2(tm + lane + d1 + g16, e, tm + lane + d1 + 64 + g16, x);
        lds16(plain ? Gp + g16 : Gam + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          x[i] *= w[i] * p.scale;
          if (!RDNV) e[i] = vv[i];
        }
        tmem_st16x2(tm + lane + d1 + g16, gks, tm + lane + d1 + 64 + g16, x);
        lds16(ww + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] *= e[i];
        put_w(T_W, w);
        st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, e);
      }
    } else {
      if (c > 0) finish_o(c - 1);
      if (RDNV) wait_chain();
      else scale_state(stl ? 0.f : GamC, start);
      bool got = true;  // (lane 0)
      if ((tid & 31) == 0 && !mbar_wait_cluster(barX, (uint32_t)c & 1u, limit)) {
        got = false;
        *flag = 1;
      }
      __syncwarp();
      if (keep && c > 0) warp_wait(barJ, (uint32_t)(c - 1) & 1u);  // (E2's image has left XE)
      float r[16], ob[16];
      {
        const float4 *x = reinterpret_cast<const float4 *>(sm + SM_X + 2048 * warp) + (tid & 31);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 a = x[32 * i], b = x[2048 + 32 * i];
          r[4 * i] = a.x; r[4 * i + 1] = a.y; r[4 * i + 2] = a.z; r[4 * i + 3] = a.w;
          ob[4 * i] = b.x; ob[4 * i + 1] = b.y; ob[4 * i + 2] = b.z; ob[4 * i + 3] = b.w;
        }
        // (a phase that has not completed takes no further arrival)
        if (got && tid == 0 && more) mbar_expect_tx(barX, 65536);
        __syncwarp();
      }
      if (RDNV) {  // ---- X2 = r - Gam KR;  MMA6: E2^T = X2^T T_gamma^T
        {
          float x[16], gm[16];
          tmem_ld16(tm + lane + d1 + g16, x);
          lds16(Gam + g16, gm);
#pragma unroll
          for (int i = 0; i < 16; ++i) x[i] = stl ? r[i] : r[i] - gm[i] * x[i];
          st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, x);
        }
        publish(kBarX);
        tmem_st16(tm + lane + T_D1 + 64 + g16, ob);
        taken(got);
        scale_state(stl ? 0.f : GamC, start);
        wait_chain();
      } else {
        tmem_st16(tm + lane + T_D1 + 64 + g16, ob);
      }
      {
        float e[16], w[16];
        if (RDNV) {
          tmem_ld16(tm + lane + T_D1 + g16, e);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) e[i] = r[i];
        }
        lds16(ww + g16, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] *= e[i];
        put_w(d1, w);
        st_row16_split(sm + SM_XE, sm + SM_XE_LO, j, g16, e);
        if (!RDNV) taken(got);  // (r was used only here)
      }
    }
    publish(kBarE);
    // the updated state -> its bf16 copies; K, Q are done with
    wait_chain();
    if (more && !by_tma(c + 1)) {  // (every thread is past its reads of V)
      bar_sync(kBarW, kTcThreads);
      if (base) fetch_v(c + 1);
      fetch_kq(c + 1);
    }
    {
      float s0[16], s1[16];
      tmem_ld16x2(tm + lane + T_ST + g16, s0, tm + lane + T_ST + g16 + 64, s1);
      put_state(g16, s0);
      put_state(g16 + 64, s1);
    }
  }

  if (alive && NC > 0) {  // the last chunk's read-outs
    bar_sync(kBarZ, kHandThreads);  // (the chunk before's have left)
    if (base) {
      hand_over(NC - 1);
      // until CTA 1 holds them
      if (tid == 0 && !mbar_wait_cluster(barX, (uint32_t)(NC - 1) & 1u, limit)) *flag = 1;
      __syncwarp();
    } else {
      finish_o(NC - 1);
    }
  }
  __syncthreads();
  if (*flag) alive = false;
  if (alive) {  // final state
    float *fin = base ? p.ST : p.RT;
    for (int c0 = g16; c0 < D && fin; c0 += 64) {
      float s[16];
      tmem_ld16(tm + lane + T_ST + c0, s);
#pragma unroll
      for (int i = 0; i < 16; ++i) fin[st_base + (size_t)(c0 + i) * D + j] = s[i];
    }
  }
  cp_async_wait_all();
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
  cfg.blockDim = dim3(kPairThreads);
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
