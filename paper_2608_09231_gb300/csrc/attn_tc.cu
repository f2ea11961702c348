// Joint attention on the 5th-generation tensor cores (head_dim 128, 16-bit operands).
//
// One CTA owns two 128-row query tiles (A and B) of one head and walks the keys in
// tiles of 128:
//   warp 0       TMA producer: both Q tiles once, then K and V^T tiles into 2-stage rings of
//                their own
//   warp 1       MMA issuer, ping-pong between the tiles:
//                  S_A,0  S_B,0 | PV_A,j  S_A,j+1 | PV_B,j  S_B,j+1 | ...
//                so the tensor core computes one tile's products while the other tile's
//                softmax runs
//   warps 4..7   softmax of tile A, warps 8..11 softmax of tile B: thread = query row; S
//                row read from TMEM into registers in one round trip, P = exp2(s - m)
//                packed to 16 bits and written back into TMEM over the S columns.
// Bound: tensor core and softmax in turn (a key tile's 32 MMAs are 2,048 cycles).  K is free
// again after the scores, V only after the PV product: with K and V in one ring stage, the
// next K was requested when the last PV ended and awaited one product later, less than the
// latency of 64 KB from L2.  Rings of their own give each load a key tile's time.  The
// softmax groups hold a whole S row, so they take the issuing warps' registers.
// Measured, one ring and 200 registers for all against this: 4608 tokens x 24 heads 204 -> 172
// us (1517 TFLOP/s; rings alone 180), 7145 x 24 487 -> 421, 16,384 x 40 3450 -> 3176.  Slower:
// an issuing warp for each query tile (212, 521, 3884: both softmaxes then run at the same
// time and the tensor core idles).  No gain: PV issued in two halves as P arrives.
// The PV product takes P straight from TMEM as its A operand, so P never touches
// shared memory; shared memory only feeds Q, K and V^T.  O stays in TMEM for the whole
// key loop.  The running max only moves (and O is rescaled in TMEM) when a tile's max
// exceeds it by more than 8 in log2 units, so P <= 2^8; the final division by the row
// sum uses the same max, which makes the result the exact softmax up to rounding.
// V arrives transposed per head ([head][dh][token]) from the QKV projection's epilogue,
// which makes it a K-major B operand.
// Operands are bf16 or fp16 (F16): q, k, v and P all of that type (an MMA's A and B share
// one type).  The sampling path uses fp16: its 11-bit significand rounds q and k, whose
// errors the softmax exponent amplifies, eight times more finely than bf16, and P stays
// within fp16's range because the lazy maximum bounds it by 2^8.
#include <cmath>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"

namespace bag {

namespace {
constexpr int AT_M = 128, AT_N = 128, AT_D = 128;
constexpr int AT_CHUNK = 128 * 64 * 2;  // 128 rows x 64 bf16 = one 128-byte-swizzle column
constexpr int AT_TILE = 2 * AT_CHUNK;   // 128 x 128 bf16
constexpr int AT_STAGES = 2;            // of the K ring and of the V ring
constexpr int AT_OFF_Q = 0;             // Q_A, Q_B
constexpr int AT_OFF_K = 2 * AT_TILE;
constexpr int AT_OFF_V = AT_OFF_K + AT_STAGES * AT_TILE;
constexpr int AT_OFF_BAR = AT_OFF_V + AT_STAGES * AT_TILE;
constexpr int AT_SMEM = AT_OFF_BAR + 256 + 1024;
constexpr int AT_TMEM_COLS = 512;  // S_A [0,128) S_B [128,256) O_A [256,384) O_B [384,512)
constexpr int AT_THREADS = 384;
// registers a thread: 168 at launch (65,536 / 384); the issuing warps' group gives up 96 and
// the two softmax groups take 48 each: 128 * 72 + 256 * 216 = 384 * 168.  How much moves matters
// little: 72 / 216, 88 / 208 and 104 / 200 take 170, 170 and 172 us (4608 tokens x 24 heads), 408,
// 420 and 406 (7145 x 24), 3289, 3290 and 3373 (16,384 x 40), with 236, 208 and 28 bytes of spill
// loads reported by ptxas; without setmaxnreg 4608 x 24 takes 176.
constexpr int AT_REGS_ISSUE = 72, AT_REGS_SOFTMAX = 216;
constexpr int AT_OLD = 36;         // floats a row in the output transpose
// exchange of partial outputs (C > 1), over the Q, K and V tiles: 2 * AT_M rows of AT_D
// floats (4 more a row against bank conflicts), then (maximum, sum) of each
constexpr int AT_XLD = AT_D + 4;
constexpr int AT_OFF_ML = 2 * AT_M * AT_XLD * 4;
static_assert(AT_OFF_ML + 2 * AT_M * 8 <= AT_OFF_BAR, "the exchange fits the operand tiles");

struct AttnTcParams {
  int nq, nk;
  void* o;
  long ldo;
  void* o2;     // rows >= o_split are written to o2 (same row index and stride)
  int o_split;
  // branch blockIdx.z: q / k row offsets, V^T row offset (per branch block), outputs
  int br_q_rows, br_k_rows, br_v_rows;
  void* o_b1;
  void* o2_b1;
  float scale_log2;
  int pairs;    // query tile pairs of a head
  int whole;    // C > 1: units (pair, head) with a CTA of their own; the others take a cluster
  const DevState* st;
  int flag_want;
  int* err;
};

BAG_DEV float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Three-input maximum and packed two-lane fp32 FMA / add (one instruction each for two
// elements of the S row, halving the softmax's issue slots for these steps).
BAG_DEV float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
BAG_DEV void fma2(float& d0, float& d1, float a0, float a1, float b, float c) {
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %4};\n\tmov.b64 rc, {%5, %5};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b), "f"(c));
}
BAG_DEV void add2(float& d0, float& d1, float a0, float a1) {
  asm("{\n\t.reg .b64 ra, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rd, {%0, %1};\n\t"
      "add.rn.f32x2 rd, rd, ra;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "+f"(d0), "+f"(d1)
      : "f"(a0), "f"(a1));
}

// 32 consecutive 32-bit TMEM columns of this thread's lane, without the wait (the caller
// issues tcgen05.wait::ld once for several loads)
BAG_DEV void tmem_ld32_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
      "[%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
}

BAG_DEV void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 16 consecutive 32-bit TMEM columns of this thread's lane
BAG_DEV void tmem_st16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
      "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]),
      "r"(v[15])
      : "memory");
}

// D (TMEM) += A (TMEM, 16-bit elements packed two per column) * B (shared memory)
BAG_DEV void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
}  // namespace

// C > 1: clusters of C CTAs.  The first p.whole units (query tile pair, head) have a CTA each,
// as with C = 1; every later unit is shared by a cluster, each CTA walking its part of the
// key tiles.  Rank r then collects 2 * AT_M / C rows of every CTA's unnormalised output,
// maximum and sum through distributed shared memory and merges them in rank order.  Used
// where whole units would leave a wave mostly idle (attention_split).
// ROWS (C = 1): the output leaves from registers, a row a lane.  With few rows there are few
// stores to gather, and the way through shared memory is four more steps at the end of a short
// call: 64 queries x 64 keys x 2 heads 8.9 against 7.9 us a call, 64 x 64 x 40 9.1 against 8.8,
// 128 x 128 x 16 8.8 against 8.5, 128 x 128 x 40 9.1 against 9.4, 256 x 256 x 24 10.9 against 13.0
// (attention_rows).  A kernel of its own: as a branch it made 7145 x 24 1.7 % slower.
template <bool F16, int C, bool ROWS = false>
__global__ void __launch_bounds__(AT_THREADS, 1)
    attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV, const AttnTcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sQ = smem + AT_OFF_Q;
  uint8_t* sK = smem + AT_OFF_K;
  uint8_t* sV = smem + AT_OFF_V;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + AT_OFF_BAR);
  uint64_t* q_full = bars + 0;
  uint64_t* k_full = bars + 1;    // [2]
  uint64_t* k_empty = bars + 3;   // [2]
  uint64_t* v_full = bars + 5;    // [2]
  uint64_t* v_empty = bars + 7;   // [2]
  uint64_t* s_full = bars + 9;    // [2] per query tile
  uint64_t* p_full = bars + 11;   // [2]
  uint64_t* o_done = bars + 13;   // [2]
  uint64_t* drain = bars + 15;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 16);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int rank = C > 1 ? (int)cluster_ctarank() : 0;
  const bool split = C > 1 && (int)blockIdx.x >= p.whole;  // uniform over a cluster
  int head = blockIdx.y, pair = blockIdx.x;
  if constexpr (C > 1) {  // units along x
    const int unit = split ? p.whole + ((int)blockIdx.x - p.whole) / C : (int)blockIdx.x;
    head = unit / p.pairs;
    pair = unit % p.pairs;
  }
  const int q0 = pair * 2 * AT_M;
  const int br = blockIdx.z;  // guidance branch (0 unless two branches share the launch)
  const int qr0 = q0 + br * p.br_q_rows, kr0 = br * p.br_k_rows, vr0 = br * p.br_v_rows;
  const int nkt = (p.nk + AT_N - 1) / AT_N;
  const int j0 = split ? rank * nkt / C : 0;                     // this CTA's first key tile
  const int nkb = (split ? (rank + 1) * nkt / C : nkt) - j0;      // and how many (>= 1)

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(k_full + i, 1);
      mbar_init(k_empty + i, 1);
      mbar_init(v_full + i, 1);
      mbar_init(v_empty + i, 1);
      mbar_init(s_full + i, 1);
      mbar_init(p_full + i, 4);  // one arrival per softmax warp of the tile
      mbar_init(o_done + i, 1);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  grid_dep_sync();
  if (epi_skip(p.st, p.flag_want)) return;
  __syncwarp();
  if (warp == 1) {
    tmem_alloc(tmem_slot, AT_TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(AT_REGS_ISSUE));
    if (warp == 0 && lane == 0) {
      // ---------------- TMA producer ----------------
      mbar_arrive_expect_tx(q_full, 2 * AT_TILE);
      for (int x = 0; x < 2; ++x) {
        tma_load_2d(sQ + x * AT_TILE, &tmQ, head * AT_D, qr0 + x * AT_M, q_full);
        tma_load_2d(sQ + x * AT_TILE + AT_CHUNK, &tmQ, head * AT_D + 64, qr0 + x * AT_M, q_full);
      }
      int kj = 0, vj = 0;  // tiles issued
      for (int j = 0; j < nkb; ++j) {
        const int s = j % AT_STAGES;
        const uint32_t ph = ((j / AT_STAGES) & 1) ^ 1;
        if (!mbar_wait(k_empty + s, ph, abort_flag)) break;
        uint8_t* k = sK + s * AT_TILE;
        mbar_arrive_expect_tx(k_full + s, AT_TILE);
        tma_load_2d(k, &tmK, head * AT_D, kr0 + (j0 + j) * AT_N, k_full + s);
        tma_load_2d(k + AT_CHUNK, &tmK, head * AT_D + 64, kr0 + (j0 + j) * AT_N, k_full + s);
        ++kj;
        if (!mbar_wait(v_empty + s, ph, abort_flag)) break;
        uint8_t* v = sV + s * AT_TILE;
        mbar_arrive_expect_tx(v_full + s, AT_TILE);
        tma_load_2d(v, &tmV, (j0 + j) * AT_N, vr0 + head * AT_D, v_full + s);
        tma_load_2d(v + AT_CHUNK, &tmV, (j0 + j) * AT_N + 64, vr0 + head * AT_D, v_full + s);
        ++vj;
      }
      if (vj < nkb) {
        // wait (bounded) for copies still in flight before the CTA may exit
        const uint64_t t0 = global_ns();
        auto landed = [&](uint64_t* bar, uint32_t ph) {
          while (!mbar_try_wait(bar, ph) && global_ns() - t0 < kWaitLimitNs) {
          }
        };
        landed(q_full, 0);
        for (int j = max(0, kj - AT_STAGES); j < kj; ++j) landed(k_full + j % AT_STAGES, (j / AT_STAGES) & 1);
        for (int j = max(0, vj - AT_STAGES); j < vj; ++j) landed(v_full + j % AT_STAGES, (j / AT_STAGES) & 1);
      }
    } else if (warp == 1) {
      // ---------------- MMA issuer (converged warp, one elected lane issues) ----------------
      constexpr uint32_t idesc = F16 ? idesc_f16_f32(AT_M, AT_N) : idesc_bf16_f32(AT_M, AT_N);
      const uint32_t q_addr = smem_u32(sQ), k_addr = smem_u32(sK), v_addr = smem_u32(sV);
      // K step kk of a tile: 64-column chunk kk / 4, 32 bytes per step inside it (16-byte units)
      auto koff = [](int kk) { return (uint64_t)(((kk >> 2) * AT_CHUNK + (kk & 3) * 32) >> 4); };
      // S of query tile x and key tile j; release: the tile's K is no longer needed
      auto issue_s = [&](int x, int j, bool release) {
        const uint64_t qd = sw128_desc(q_addr + x * AT_TILE);
        const uint64_t kd = sw128_desc(k_addr + (j % AT_STAGES) * AT_TILE);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < AT_D / 16; ++kk)
            mma_bf16(tmem + x * 128, qd + koff(kk), kd + koff(kk), idesc, kk > 0 ? 1u : 0u);
          mma_commit(s_full + x);
          if (release) mma_commit(k_empty + j % AT_STAGES);
        }
        __syncwarp();
      };
      // commit: a barrier to signal once these products are done (null: none)
      auto issue_pv = [&](int x, int j, uint64_t* commit) {
        const uint64_t vd = sw128_desc(v_addr + (j % AT_STAGES) * AT_TILE);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < AT_N / 16; ++kk)
            mma_bf16_ts(tmem + 256 + x * 128, tmem + x * 128 + kk * 8, vd + koff(kk), idesc,
                        (j > 0 || kk > 0) ? 1u : 0u);
          if (commit) mma_commit(commit);
        }
        __syncwarp();
      };
      auto wait = [&](uint64_t* bar, uint32_t ph) {
        const bool w = mbar_wait_warp(bar, ph, abort_flag);
        tc_fence_after();
        return w;
      };
      bool ok = wait(q_full, 0) && wait(k_full, 0);
      if (ok) {
        issue_s(0, 0, false);
        issue_s(1, 0, true);
      }
      for (int j = 0; j < nkb && ok; ++j) {
        const int s = j % AT_STAGES, s1 = (j + 1) % AT_STAGES;
        const bool more = j + 1 < nkb;
        ok = wait(v_full + s, (j / AT_STAGES) & 1);
        for (int x = 0; x < 2 && ok; ++x) {
          // PV_j of this tile, then its S_{j+1} into the columns P_j came from (in issue order)
          if (!(ok = wait(p_full + x, j & 1))) break;
          issue_pv(x, j, x ? v_empty + s : (more ? nullptr : o_done + 0));
          if (more) {
            if (x == 0 && !(ok = wait(k_full + s1, ((j + 1) / AT_STAGES) & 1))) break;
            issue_s(x, j + 1, x == 1);
          } else if (x == 1) {
            if (elect_one()) mma_commit(o_done + 1);
            __syncwarp();
          }
        }
      }
      if (elect_one()) {
        mma_commit(drain);
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(drain, 0) && global_ns() - t0 < kWaitLimitNs) {
        }
      }
    }
    __syncwarp();
    if (split) {  // the two barriers of the exchange
      cluster_sync_all();
      cluster_sync_all();
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(AT_REGS_SOFTMAX));
    // ---------------- softmax warpgroups (warps 4..7: tile A, 8..11: tile B) ----------------
    const int x = (warp - 4) >> 2;
    const int quad = warp & 3;
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    const uint32_t s_addr = tmem + lane_base + x * 128;
    const uint32_t o_addr = tmem + lane_base + 256 + x * 128;
    float m_use = -INFINITY, l = 0.f;
    bool ok = true;
    for (int j = 0; j < nkb; ++j) {
      const bool w = mbar_wait(s_full + x, j & 1, abort_flag);
      if (!__all_sync(0xffffffffu, w)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const int kvalid = p.nk - (j0 + j) * AT_N;  // keys of this tile that exist (< 128 only at the end)
      // the whole S row in registers: four loads, one wait
      uint32_t r[AT_N];
#pragma unroll
      for (int c = 0; c < AT_N / 32; ++c) tmem_ld32_nowait(s_addr + c * 32, r + c * 32);
      tmem_ld_wait();
      if (kvalid < AT_N) {
#pragma unroll
        for (int i = 0; i < AT_N; ++i)
          if (i >= kvalid) r[i] = __float_as_uint(-INFINITY);
      }
      // row maximum: four independent chains of three-input maxima
      float mq[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) mq[u] = fmaxf(__uint_as_float(r[2 * u]), __uint_as_float(r[2 * u + 1]));
#pragma unroll
      for (int i = 8; i < AT_N; i += 8)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          mq[u] = max3(mq[u], __uint_as_float(r[i + 2 * u]), __uint_as_float(r[i + 2 * u + 1]));
      const float mx = fmaxf(fmaxf(mq[0], mq[1]), fmaxf(mq[2], mq[3]));
      const float mx2 = mx * p.scale_log2;
      float alpha = 1.f;
      if (mx2 > m_use + 8.f) {
        alpha = ex2(m_use - mx2);
        m_use = mx2;
        l *= alpha;
      }
      // a tile of nothing but -inf scores before any other weighs nothing
      const float neg_m = m_use == -INFINITY ? 0.f : -m_use;
      // P = exp2(s * scale - m) (masked keys give exp2(-inf) = 0), packed 16-bit pairs
      // written over the S columns already read
      float ls0 = 0.f, ls1 = 0.f;
#pragma unroll
      for (int c = 0; c < AT_N / 32; ++c) {
        uint32_t pk[16];
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          float x0, x1;
          fma2(x0, x1, __uint_as_float(r[c * 32 + i]), __uint_as_float(r[c * 32 + i + 1]),
               p.scale_log2, neg_m);
          const float a0 = ex2(x0), a1 = ex2(x1);
          add2(ls0, ls1, a0, a1);
          pk[i / 2] = F16 ? pack_f16x2(a0, a1) : pack_bf16x2(a0, a1);
        }
        tmem_st16(s_addr + c * 16, pk);
      }
      l += ls0 + ls1;
      // O_x holds PV of every earlier key tile (the S of this tile was issued after it);
      // rescale it before this tile's PV is issued
      if (j > 0 && __any_sync(0xffffffffu, alpha != 1.f)) {
#pragma unroll 1
        for (int c = 0; c < AT_D / 32; ++c) {
          float o[32];
          tmem_ld32(o_addr + c * 32, o);
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] *= alpha;
          tmem_st32(o_addr + c * 32, o);
        }
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full + x);
    }
    if (ok) ok = __all_sync(0xffffffffu, mbar_wait(o_done + x, 0, abort_flag));
    tc_fence_after();
    if (split) {
      constexpr int RPO = 2 * AT_M / C;  // rows a rank merges
      __syncwarp();
      cluster_sync_all();  // every CTA's products are done: the operand tiles are free
      if (ok) {
        const int R = x * AT_M + quad * 32 + lane;
        const int at = rank * RPO + R % RPO;
        const uint32_t dst = mapa_shared(smem_u32(smem), (uint32_t)(R / RPO));
#pragma unroll 1
        for (int c = 0; c < AT_D; c += 32) {
          float o[32];
          tmem_ld32(o_addr + c, o);
#pragma unroll
          for (int i = 0; i < 32; i += 4)
            st_cluster4(dst + (uint32_t)(at * AT_XLD + c + i) * 4, o[i], o[i + 1], o[i + 2], o[i + 3]);
        }
        st_cluster2(dst + AT_OFF_ML + (uint32_t)at * 8, m_use, l);
      }
      __syncwarp();
      cluster_sync_all();  // every part has arrived; no access to another CTA follows
      const float* part = reinterpret_cast<const float*>(smem);
      const float2* ml = reinterpret_cast<const float2*>(smem + AT_OFF_ML);
      void* o1 = br ? p.o_b1 : p.o;
      void* o2 = br ? p.o2_b1 : p.o2;
#pragma unroll 2
      for (int lr = warp - 4; lr < RPO; lr += 8) {  // a warp a row, four columns a lane
        float2 f[C];
        float m = -INFINITY, den = 0.f;
#pragma unroll
        for (int s = 0; s < C; ++s) {
          f[s] = ml[s * RPO + lr];
          m = fmaxf(m, f[s].x);
        }
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < C; ++s) {
          const float w = f[s].x == -INFINITY ? 0.f : ex2(f[s].x - m);
          const float4 o = *reinterpret_cast<const float4*>(part + (s * RPO + lr) * AT_XLD + lane * 4);
          den += w * f[s].y;
          acc.x += w * o.x;
          acc.y += w * o.y;
          acc.z += w * o.z;
          acc.w += w * o.w;
        }
        const float inv = 1.f / den;
        const int q = q0 + rank * RPO + lr;
        if (q < p.nq) {
          uint2 u;
          u.x = pack_bf16x2(acc.x * inv, acc.y * inv);
          u.y = pack_bf16x2(acc.z * inv, acc.w * inv);
          *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(o2 && q >= p.o_split ? o2 : o1) +
                                    (long)q * p.ldo + head * AT_D + lane * 4) = u;
        }
      }
    } else if (ROWS) {
      if (ok) {
        const float inv = 1.f / l;
        const int q = q0 + x * AT_M + quad * 32 + lane;
        void* o1 = br ? p.o_b1 : p.o;
        void* o2 = br ? p.o2_b1 : p.o2;
        void* ob = o2 && q >= p.o_split ? o2 : o1;
#pragma unroll 1
        for (int c = 0; c < AT_D; c += 32) {
          float o[32];
          tmem_ld32(o_addr + c, o);
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] *= inv;
          if (q < p.nq) store_vals<32>(ob, (long)q * p.ldo + head * AT_D + c, o, kStoreBF16);
        }
      }
    } else if (ok) {
      const float inv = 1.f / l;
      // through shared memory (this tile's Q, which no product reads any more): four lanes
      // hold 32 consecutive columns of a row, so a store covers eight rows' 64-byte runs
      float* buf = reinterpret_cast<float*>(sQ + x * AT_TILE) + quad * 32 * AT_OLD;
      const int r = lane >> 2, c8 = (lane & 3) * 8;
      const int qw = q0 + x * AT_M + quad * 32 + r;
      void* o1 = br ? p.o_b1 : p.o;
      void* o2 = br ? p.o2_b1 : p.o2;
#pragma unroll 1
      for (int c = 0; c < AT_D; c += 32) {
        float o[32];
        tmem_ld32(o_addr + c, o);
#pragma unroll
        for (int i = 0; i < 32; i += 4)
          *reinterpret_cast<float4*>(buf + lane * AT_OLD + i) =
              make_float4(o[i] * inv, o[i + 1] * inv, o[i + 2] * inv, o[i + 3] * inv);
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int q = qw + 8 * u;
          float v[8];
          ld_chunk<8>(buf + (8 * u + r) * AT_OLD + c8, v);
          if (q < p.nq)
            store_vals<8>(o2 && q >= p.o_split ? o2 : o1, (long)q * p.ldo + head * AT_D + c + c8, v, kStoreBF16);
        }
        __syncwarp();
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag && p.err) atomicOr(p.err, 1);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, AT_TMEM_COLS);
  }
}

static int g_sms = 1;

cudaError_t attention_tc_init() {
  const void* kernels[] = {(const void*)attn_tc_kernel<false, 1>, (const void*)attn_tc_kernel<false, 2>,
                           (const void*)attn_tc_kernel<false, 4>, (const void*)attn_tc_kernel<true, 1>,
                           (const void*)attn_tc_kernel<true, 2>,  (const void*)attn_tc_kernel<true, 4>,
                           (const void*)attn_tc_kernel<false, 1, true>, (const void*)attn_tc_kernel<true, 1, true>};
  cudaError_t r = cudaSuccess;
  for (const void* k : kernels)
    if (r == cudaSuccess) r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, AT_SMEM);
  int dev = 0;
  if (r == cudaSuccess) r = cudaGetDevice(&dev);
  if (r == cudaSuccess) r = cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
  return r;
}

// CTAs per cluster and the units that keep a CTA of their own, for `units` (query tile pair,
// head) of one guidance branch and `nkt` key tiles: a launch of fewer units than SMs shares
// each unit among 2 or 4 CTAs; a longer one shares the units of its last wave where they
// leave at least half of the SMs idle.  A key tile takes about 1.45 us and sharing about 7 us
// (cluster launch, two barriers, the exchange), hence the least numbers of key tiles.  Planned
// from one branch's units, so that guided and unguided samples give the same bits.
// Measured: 7145 tokens x 24 heads (672 units on 152 SMs, the last 64 shared) 432 -> 399 us;
// 1536 x 4 heads 25.6 -> 19.9 us, 3000 x 2 42.9 -> 25.2, 5000 x 8 122 -> 101; with 4 key tiles
// (455 x 4), shared by four, 13.9 -> 16.9 us.
static int attention_split(int units, int nkt, int* whole) {
  *whole = units;
  if (units < g_sms) {
    // clusters of four reach 144 of 152 SMs
    const int c = units * 4 <= g_sms - g_sms / 16 && nkt >= 12 ? 4 : (units * 2 <= g_sms && nkt >= 16 ? 2 : 1);
    if (c > 1) *whole = 0;
    return c;
  }
  const int rest = units % g_sms;
  if (rest == 0 || rest * 2 > g_sms || nkt < 16 || (units - rest) % 2) return 1;
  *whole = units - rest;
  return 2;
}

// Whether an unshared launch writes its output a row a lane (see attn_tc_kernel).
static bool attention_rows(int nq, int heads) { return nq <= AT_M && (long)nq * heads <= 2560; }

int attention_tc_supported(const AttnArgs& a) {
  if (!a.bf16 || a.dh != AT_D || a.v_mode != 1) return 0;
  if (a.ldq % 8 || a.ldk % 8 || a.vpad % 8 || a.ldo % 8) return 0;
  if ((reinterpret_cast<uintptr_t>(a.q) | reinterpret_cast<uintptr_t>(a.k) |
       reinterpret_cast<uintptr_t>(a.v) | reinterpret_cast<uintptr_t>(a.o)) & 15)
    return 0;
  return a.nq > 0 && a.nk > 0 && a.vpad >= a.nk;
}

cudaError_t attention_tc(const AttnArgs& a, int* err, cudaStream_t s) {
  CUtensorMap tq, tk, tv;
  const uint64_t width = (uint64_t)a.heads * AT_D;
  const int nbr = a.nbr > 1 ? 2 : 1;
  // with two branches the maps span both (the rows past a branch's last query or key are
  // never stored, resp. masked, and its V^T block is zero beyond nk up to vpad)
  const uint64_t qrows = nbr > 1 ? (uint64_t)a.br_q_rows + a.nq : (uint64_t)a.nq;
  const uint64_t krows = nbr > 1 ? (uint64_t)a.br_k_rows + a.nk : (uint64_t)a.nk;
  if (encode_tmap_2d_bf16(&tq, a.q, width, qrows, (uint64_t)a.ldq * 2, 64, AT_M) ||
      encode_tmap_2d_bf16(&tk, a.k, width, krows, (uint64_t)a.ldk * 2, 64, AT_N) ||
      encode_tmap_2d_bf16(&tv, a.v, (uint64_t)a.nk, width * nbr, (uint64_t)a.vpad * 2, 64, AT_D))
    return cudaErrorInvalidValue;
  AttnTcParams p;
  p.nq = a.nq;
  p.nk = a.nk;
  p.o = a.o;
  p.ldo = a.ldo;
  p.o2 = a.o2;
  p.o_split = a.o_split;
  p.br_q_rows = nbr > 1 ? (int)a.br_q_rows : 0;
  p.br_k_rows = nbr > 1 ? (int)a.br_k_rows : 0;
  p.br_v_rows = nbr > 1 ? (int)width : 0;
  p.o_b1 = a.o_b1;
  p.o2_b1 = a.o2_b1;
  p.scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)AT_D));
  p.st = a.st;
  p.flag_want = a.flag_want;
  p.err = err;
  p.pairs = (a.nq + 2 * AT_M - 1) / (2 * AT_M);
  const int units = p.pairs * a.heads;
  const int c = attention_split(units, (a.nk + AT_N - 1) / AT_N, &p.whole);
  const dim3 grid = c > 1 ? dim3((unsigned)(p.whole + (units - p.whole) * c), 1, nbr) : dim3(p.pairs, a.heads, nbr);
  auto launch = [&](auto kernel) {
    launch_cluster(kernel, c > 1 ? (unsigned)c : 0u, grid, AT_THREADS, AT_SMEM, s, tq, tk, tv, p);
  };
  const bool rows = c == 1 && attention_rows(a.nq, a.heads);
  if (rows)
    a.f16 ? launch(attn_tc_kernel<true, 1, true>) : launch(attn_tc_kernel<false, 1, true>);
  else if (a.f16)
    c == 4 ? launch(attn_tc_kernel<true, 4>)
           : (c == 2 ? launch(attn_tc_kernel<true, 2>) : launch(attn_tc_kernel<true, 1>));
  else
    c == 4 ? launch(attn_tc_kernel<false, 4>)
           : (c == 2 ? launch(attn_tc_kernel<false, 2>) : launch(attn_tc_kernel<false, 1>));
  return cudaGetLastError();
}

}  // namespace bag
