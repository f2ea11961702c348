// Projections of the DiT block: C[M,N] = A[M,K] W[N,K]^T with a fused epilogue.
//
// bf16 operands run on the 5th-generation tensor cores: warp-specialised kernels with one TMA
// producer warp, one MMA-issuing warp and four or eight epilogue warps.  Operand tiles (64
// columns wide, 128-byte swizzle) stream through a multi-stage shared-memory ring guarded by
// mbarriers; tcgen05.mma accumulates fp32 tiles in tensor memory.  Three of them: CTA pairs
// with 256 x 256 tiles, and single CTAs with 128 x 128 or 128 x 64 tiles (both persistent,
// accumulators double-buffered so that the epilogue of one tile overlaps the main loop of the
// next), and clusters that split K where there are few tiles.  fp32 operands (the fp32
// configuration, which must hold 1e-4 relative parity) use a CUDA-core kernel with the same
// epilogue.
#include <algorithm>
#include <cstdio>
#include <mutex>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"

namespace bag {

// ---------------------------------------------------------------------------
// TMA descriptor encoding through the driver entry point
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

int encode_tmap_2d_bf16(CUtensorMap* map, const void* base, uint64_t inner, uint64_t outer,
                        uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return -1;
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {row_stride_bytes};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims,
                  strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : (int)r;
}

static int num_sms() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 148;
  }
  return n;
}

// ---------------------------------------------------------------------------
// CUDA-core GEMM (fp32 or bf16 operands, fp32 accumulation)
// ---------------------------------------------------------------------------
// One CTA computes a 32 x 32 tile; its eight warps split every 64-wide K slice (8 columns
// each), so that each warp holds the whole tile (4 x 8 per lane) and the partial tiles are
// summed in warp order at the end.  Bound: latency.  The fp32 backbones are small (a few
// hundred rows, K up to a few thousand), so a launch has few output tiles and a long K
// chain; small tiles put a CTA on most SMs, the split shortens the chain eightfold, and a
// four-stage cp.async ring covers the L2 latency.  Rows are 68 floats apart in shared
// memory (eight rows x 16 bytes hit all 32 banks).
// Measured against 64 x 64 tiles with one K chain per CTA, scalar loads and no prefetch
// (profiled launches): 288 x 256 x 1280 158 -> 21 us, 288 x 1792 x 256 37 -> 22 us.
// bf16 operands (cross-checks of the tensor-core kernels) are fetched a slice ahead into
// registers: loaded and stored in one go they took 988 us for 2048 x 2048 x 2048 (64 x 64 tiles
// 753), now 507, unaligned 649; 1024 x 1024 x 1024 151 (131), now 76; 4096 x 4096 x 512 1047 (701),
// now 605, unaligned 756.
constexpr int SG_T = 32, SG_BK = 64, SG_LD = SG_BK + 4, SG_STAGES = 4, SG_WARPS = 8;
constexpr int SG_TILE = SG_T * SG_LD;  // floats of one operand's tile in one stage
constexpr int SG_SMEM = SG_STAGES * 2 * SG_TILE * 4;
static_assert(SG_SMEM >= SG_WARPS * SG_T * SG_T * 4, "the partial tiles reuse the ring");

BAG_DEV void cp_async16(float* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}

// Rows r0 .. r0 + 31 of P (columns k0 .. k0 + 63) into shared memory, zeros outside, copied
// asynchronously: fp32 rows of 16-byte aligned float4 groups (K a multiple of 4).
BAG_DEV void sg_load_async(float* dst, const float* __restrict__ P, long ld, int r0, int rows, int k0, int K) {
#pragma unroll
  for (int i = threadIdx.x; i < SG_T * SG_BK / 4; i += SG_WARPS * 32) {
    const int r = i / (SG_BK / 4), c = (i % (SG_BK / 4)) * 4;
    const bool ok = r0 + r < rows && k0 + c < K;
    cp_async16(dst + r * SG_LD + c, ok ? P + (long)(r0 + r) * ld + k0 + c : P, ok);
  }
}

// The same slice of a bf16 operand, which has to be converted, in two steps with the products
// of a slice in between: into registers (eight values a thread), then into shared memory.
// VEC: one 16-byte load (K and ld multiples of 8, P 16-byte aligned); else eight single ones.
static_assert(SG_T * SG_BK == 8 * SG_WARPS * 32, "eight values of an operand's slice a thread");
template <bool VEC>
BAG_DEV uint4 sg_fetch(const __nv_bfloat16* __restrict__ P, long ld, int r0, int rows, int k0, int K) {
  const int r = r0 + threadIdx.x / (SG_BK / 8), c = k0 + threadIdx.x % (SG_BK / 8) * 8;
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  const unsigned short* p = reinterpret_cast<const unsigned short*>(P) + (long)r * ld + c;
  if (r < rows && c < K) {
    if constexpr (VEC) {
      v = __ldg(reinterpret_cast<const uint4*>(p));
    } else {
      uint32_t x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = c + u < K ? __ldg(p + u) : 0u;
      v = make_uint4(x[0] | x[1] << 16, x[2] | x[3] << 16, x[4] | x[5] << 16, x[6] | x[7] << 16);
    }
  }
  return v;
}
BAG_DEV void sg_put(float* dst, uint4 v) {
  float4* d = reinterpret_cast<float4*>(dst + threadIdx.x / (SG_BK / 8) * SG_LD + threadIdx.x % (SG_BK / 8) * 8);
  auto pair = [](uint32_t a, uint32_t b) {
    return make_float4(__uint_as_float(a << 16), __uint_as_float(a & 0xffff0000u), __uint_as_float(b << 16),
                       __uint_as_float(b & 0xffff0000u));
  };
  d[0] = pair(v.x, v.y);
  d[1] = pair(v.z, v.w);
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(SG_WARPS * 32) gemm_simt_kernel(const T* __restrict__ A, long lda,
                                                                  const T* __restrict__ W, long ldw,
                                                                  int M, int N, int K, const Epi e) {
  grid_dep_sync();
  if (epi_skip(e.st, e.flag_want)) return;
  epi_bump(e);
  const int t = epi_step(e);
  extern __shared__ __align__(16) float sg[];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int ty = lane / 4, tx = lane % 4;  // rows ty + 8 i, columns tx + 4 j of the tile
  const int num_n = (N + SG_T - 1) / SG_T;
  const int m0 = blockIdx.x / num_n * SG_T, n0 = blockIdx.x % num_n * SG_T;
  const int nk = (K + SG_BK - 1) / SG_BK;
  [[maybe_unused]] uint4 fa, fw;  // bf16: the slice after the last one in the ring
  [[maybe_unused]] auto fetch = [&](int kb) {
    if constexpr (sizeof(T) == 2) {
      if (kb < nk) {
        fa = sg_fetch<VEC>(A, lda, m0, M, kb * SG_BK, K);
        fw = sg_fetch<VEC>(W, ldw, n0, N, kb * SG_BK, K);
      }
    }
  };
  auto load = [&](int kb) {
    float* d = sg + (kb % SG_STAGES) * 2 * SG_TILE;
    if constexpr (sizeof(T) == 2) {
      if (kb < nk) {
        sg_put(d, fa);
        sg_put(d + SG_TILE, fw);
      }
      fetch(kb + 1);
    } else {
      if (kb < nk) {
        sg_load_async(d, A, lda, m0, M, kb * SG_BK, K);
        sg_load_async(d + SG_TILE, W, ldw, n0, N, kb * SG_BK, K);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  };
  float acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  fetch(0);
  for (int kb = 0; kb < SG_STAGES - 1; ++kb) load(kb);
  for (int kb = 0; kb < nk; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(SG_STAGES - 2) : "memory");
    __syncthreads();  // slice kb has landed for all threads; slice kb - 1 is consumed
    load(kb + SG_STAGES - 1);
    const float* sa = sg + (kb % SG_STAGES) * 2 * SG_TILE + warp * 8;
    const float* sw = sa + SG_TILE;
#pragma unroll
    for (int k = 0; k < 8; k += 4) {
      float4 a[4], w[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(sa + (ty + 8 * i) * SG_LD + k);
#pragma unroll
      for (int j = 0; j < 8; ++j) w[j] = *reinterpret_cast<const float4*>(sw + (tx + 4 * j) * SG_LD + k);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          acc[i][j] += a[i].x * w[j].x;
          acc[i][j] += a[i].y * w[j].y;
          acc[i][j] += a[i].z * w[j].z;
          acc[i][j] += a[i].w * w[j].w;
        }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) sg[(warp * SG_T + ty + 8 * i) * SG_T + tx + 4 * j] = acc[i][j];
  __syncthreads();
  const int r = threadIdx.x / 8, c = (threadIdx.x % 8) * 4;
  float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int w = 0; w < SG_WARPS; ++w) {
    const float4 p = *reinterpret_cast<const float4*>(sg + (w * SG_T + r) * SG_T + c);
    v[0] += p.x;
    v[1] += p.y;
    v[2] += p.z;
    v[3] += p.w;
  }
  // N is a multiple of 4, so a column group is inside or outside as a whole
  if (m0 + r < M && n0 + c < N) epi_apply<4>(e, t, m0 + r, n0 + c, v);
}

// ---------------------------------------------------------------------------
// tcgen05 GEMM
// ---------------------------------------------------------------------------
constexpr int TC_BM = 128, TC_BK = 64;

// Tile order within one problem: groups of G row tiles, each group visiting every
// column tile with the row tile varying fastest.  A wave of tiles then shares at most G
// row tiles of A (which stay in L2 while the group walks the columns) instead of
// streaming all of A once per column tile; G comes from the L2 share one group's rows
// may take (tile_group_rows).
BAG_DEV void raster(int l, int num_m, int num_n, int G, int& mt, int& nt) {
  const int per_group = G * num_n;
  const int g = l / per_group;
  const int idx = l - g * per_group;
  const int gm = min(G, num_m - g * G);
  mt = g * G + idx % gm;
  nt = idx / gm;
}

#ifndef BAG_TILE_GROUP_L2_MB
#define BAG_TILE_GROUP_L2_MB 40
#endif
// Row tiles per group: as many BM-row slices of A (K bf16 columns, twice as many for a
// split A) as fit in the L2 share, at least 1, at most all of them.
static int tile_group_rows(int M, int BM, int K, int a_split) {
  const int num_m = (M + BM - 1) / BM;
  if (num_m <= 0) return 1;
  const double slice = (double)BM * K * 2.0 * (a_split ? 2 : 1);
  const int g = (int)((double)BAG_TILE_GROUP_L2_MB * 1048576.0 / slice);
  return std::max(1, std::min(num_m, g));
}

// Per epilogue warp: a shared-memory tile for transposing 32 x 32 accumulators (V: rows of
// 33 words; fp32 rows: 36 words, so that 16-byte accesses are aligned and conflict-free).
constexpr int kF32Ld = 36;
constexpr int kVtScratchFloats = 32 * kF32Ld;

BAG_DEV uint16_t to16(float x, bool f16) {
  return f16 ? __half_as_ushort(__float2half_rn(x)) : __bfloat16_as_ushort(__float2bfloat16_rn(x));
}
BAG_DEV uint32_t pack16x2(float a, float b, bool f16) { return f16 ? pack_f16x2(a, b) : pack_bf16x2(a, b); }

// V columns of a QKV projection with 16-bit (bf16 or fp16) storage, stored transposed per head
// (vt[(head * dh + e) * vpad + token]): the warp's 32 rows x 32 columns.  Whole blocks of one
// branch whose token offset is 16-byte aligned pass through shared memory (rows of 33 words)
// so that four lanes hold 32 consecutive tokens of a column and a warp store covers eight
// columns' 64-byte runs; the others (a ragged text length, the last rows) store from
// registers, lane = token, 64 bytes of one column at a time.
BAG_DEV void store_vt_warp(const Epi& e, int row, int col, float* v, float* sbuf) {
  const int lane = threadIdx.x & 31;
  const int row0 = row - lane;
  const bool f16 = e.qkv_type == kStoreF16;
  const int cc = col + e.col_base - 2 * e.d;  // column within V
  uint16_t* vbase = reinterpret_cast<uint16_t*>(e.v);
  const bool br1 = e.br_rows > 0 && row0 >= e.br_rows;
  const bool one_branch = e.br_rows == 0 || br1 || row0 + 31 < e.br_rows;
  const long jr0 = row0 - (br1 ? e.br_rows : 0) + e.row_off;
  uint16_t* dst = vbase + (br1 ? e.br_vt : 0) + (long)cc * e.vpad + jr0;
  if (row0 + 31 < e.M && one_branch && (reinterpret_cast<uintptr_t>(dst) & 15) == 0 && e.vpad % 8 == 0) {
#pragma unroll
    for (int j = 0; j < 32; ++j) sbuf[lane * 33 + j] = v[j];
    __syncwarp();
    const int r = lane >> 2, c = (lane & 3) * 8;  // column r of each group of eight, tokens c .. c + 7
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int cl = p * 8 + r;
      const float b = e.bias ? __ldg(e.bias + col + cl) : 0.f;
      float x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = sbuf[(c + k) * 33 + cl] + b;
      uint4 w;
      w.x = pack16x2(x[0], x[1], f16);
      w.y = pack16x2(x[2], x[3], f16);
      w.z = pack16x2(x[4], x[5], f16);
      w.w = pack16x2(x[6], x[7], f16);
      *reinterpret_cast<uint4*>(dst + (long)cl * e.vpad + c) = w;
    }
    __syncwarp();  // the tile may be overwritten
    return;
  }
  if (row >= e.M) return;
  epi_add_bias<32>(e, col, v);
  const bool b1 = e.br_rows > 0 && row >= e.br_rows;
  uint16_t* d = vbase + (b1 ? e.br_vt : 0) + (long)cc * e.vpad + row - (b1 ? e.br_rows : 0) + e.row_off;
#pragma unroll
  for (int j = 0; j < 32; ++j) d[(long)j * e.vpad] = to16(v[j], f16);
}

// Whether an epilogue reads or writes fp32 rows that store_f32_warp can take 16 bytes at a time.
static __host__ __device__ __forceinline__ bool f32_rows(const Epi& e) {
  uintptr_t p = reinterpret_cast<uintptr_t>(e.bias);
  long ld;
  if ((e.kind == EPI_STORE || e.kind == EPI_GELU) && e.out_bf16 == kStoreF32) {
    p |= reinterpret_cast<uintptr_t>(e.out);
    ld = e.ldo;
  } else if (e.kind == EPI_GATED_RES || e.kind == EPI_RES_ADD) {
    p |= reinterpret_cast<uintptr_t>(e.resid);
    ld = e.ldr;
    if (e.kind == EPI_GATED_RES) {
      p |= reinterpret_cast<uintptr_t>(e.gate);
      if (e.br_rows > 0) p |= reinterpret_cast<uintptr_t>(e.gate_u);
      ld |= e.gate_step;
    }
  } else {
    return false;
  }
  return (p & 15) == 0 && ld % 4 == 0;
}

// 32 rows x 32 columns of fp32 output (or of an fp32 residual update), one warp: the
// accumulators pass through shared memory so that eight lanes hold 32 consecutive columns of
// a row.  A warp access then covers four whole 128-byte lines, where a lane that keeps its
// own row touches 32 lines with 16 bytes each, and bias and gate are read once for eight
// rows.  The same sums and products element by element as epi_apply.
// Measured, row per lane against this: 1373 x 12288 x 3072 fp32 store 76.6 -> 69.3 us, with GELU
// 89.5 -> 73.8; 4608 x 12288 x 3072 209 -> 186 us; 4096 x 3072 x 128 39 -> 29 us; gated residual
// 4608 x 3072 x 15360 256 -> 240 us.
BAG_DEV void store_f32_warp(const Epi& e, int t, int row0, int col0, const float* v, float* buf) {
  const int lane = threadIdx.x & 31, r = lane >> 3, c = (lane & 7) * 4;
#pragma unroll
  for (int j = 0; j < 32; j += 4)
    *reinterpret_cast<float4*>(buf + lane * kF32Ld + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const float4 b = e.bias ? __ldg(reinterpret_cast<const float4*>(e.bias + col0 + c)) : zero;
  __syncwarp();
  float4 a[8];
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    a[p] = *reinterpret_cast<const float4*>(buf + (p * 4 + r) * kF32Ld + c);
    a[p].x += b.x;
    a[p].y += b.y;
    a[p].z += b.z;
    a[p].w += b.w;
  }
  __syncwarp();  // the tile may be overwritten
  const int row = row0 + r;
  if (e.kind == EPI_STORE || e.kind == EPI_GELU) {
    float* o = reinterpret_cast<float*>(e.out) + (long)row * e.ldo + col0 + c;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      if (row + 4 * p >= e.M) break;
      if (e.kind == EPI_GELU)
        a[p] = make_float4(gelu_tanh(a[p].x), gelu_tanh(a[p].y), gelu_tanh(a[p].z), gelu_tanh(a[p].w));
      *reinterpret_cast<float4*>(o + (long)(4 * p) * e.ldo) = a[p];
    }
    return;
  }
  float* o = e.resid + (long)row * e.ldr + col0 + c;
  float4 h[8];
#pragma unroll
  for (int p = 0; p < 8; ++p)
    h[p] = row + 4 * p < e.M ? *reinterpret_cast<const float4*>(o + (long)(4 * p) * e.ldr) : zero;
  float4 g0 = make_float4(1.f, 1.f, 1.f, 1.f), g1 = g0;
  if (e.kind == EPI_GATED_RES) {
    const long at = (long)t * e.gate_step + col0 + c;
    g0 = __ldg(reinterpret_cast<const float4*>(e.gate + at));
    g1 = e.br_rows > 0 ? __ldg(reinterpret_cast<const float4*>(e.gate_u + at)) : g0;
  }
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    if (row + 4 * p >= e.M) break;
    const float4 g = e.br_rows > 0 && row + 4 * p >= e.br_rows ? g1 : g0;
    h[p].x += g.x * a[p].x;
    h[p].y += g.y * a[p].y;
    h[p].z += g.z * a[p].z;
    h[p].w += g.w * a[p].w;
    *reinterpret_cast<float4*>(o + (long)(4 * p) * e.ldr) = h[p];
  }
}

// Whether store_16_warp takes an epilogue's 16-bit outputs (V goes to store_vt_warp).
static __host__ __device__ __forceinline__ bool rows16(const Epi& e) {
  uintptr_t p = reinterpret_cast<uintptr_t>(e.bias);
  long ld;
  if (e.kind == EPI_STORE || e.kind == EPI_GELU) {
    if (e.out_bf16 == kStoreF32) return false;
    p |= reinterpret_cast<uintptr_t>(e.out);
    ld = e.ldo;
  } else if (e.kind == EPI_QKV) {
    if (e.v_mode != 1 || e.qkv_type == kStoreF32 || !e.act_bf16) return false;
    p |= reinterpret_cast<uintptr_t>(e.q) | reinterpret_cast<uintptr_t>(e.k) | reinterpret_cast<uintptr_t>(e.mlp) |
         reinterpret_cast<uintptr_t>(e.rope) | reinterpret_cast<uintptr_t>(e.qn_q) |
         reinterpret_cast<uintptr_t>(e.qn_k);
    ld = e.ldqk | e.ldm;
  } else {
    return false;
  }
  return (p & 15) == 0 && ld % 8 == 0;
}

// 32 rows x 32 columns of 16-bit output, one warp, through shared memory as in
// store_f32_warp: four lanes hold 32 consecutive columns of a row, so that a warp access
// covers eight rows' 64-byte runs (and eight rows' rotation table entries, 128 bytes each).
// rs: 1 / RMS of this lane's row (QK-norm).  The same operations element by element as
// epi_apply.  Loads inside each row's branch instead of up front cost one L2 round trip per
// row (910 x 3584 x 512 with QK-norm 30 -> 37 us).
// Measured, row per lane against this (with store_vt_warp): 4608 x 21504 x 3072, QKV with
// rotation and GELU, 365 -> 331 us; 910 x 1536 x 512 unchanged.
BAG_DEV void store_16_warp(const Epi& e, int row0, int col0, const float* v, float* buf, float rs) {
  const int lane = threadIdx.x & 31, r = lane >> 2, c = (lane & 3) * 8;
#pragma unroll
  for (int j = 0; j < 32; j += 4)
    *reinterpret_cast<float4*>(buf + lane * kF32Ld + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
  float b[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) b[j] = 0.f;
  if (e.bias) ld_chunk<8>(e.bias + col0 + c, b);
  void* base = e.out;
  long ld = e.ldo;
  int type = e.out_bf16, cc = col0 + c, region = 3;
  bool gelu = e.kind == EPI_GELU;
  if (e.kind == EPI_QKV) {
    const int lc = col0 + e.col_base;
    region = min(lc / e.d, 3);
    cc = lc - region * e.d + c;
    gelu = region == 3;
    base = region == 0 ? e.q : (region == 1 ? e.k : e.mlp);
    ld = region < 2 ? e.ldqk : e.ldm;
    type = region < 2 ? e.qkv_type : kStoreBF16;
  }
  // every row's operands before any row's arithmetic: four rows a lane, one round trip
  const int row = row0 + r;
  int orow[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) orow[p] = row + 8 * p;
  float4 q[8];  // rotation: (cos, sin) pairs of columns c .. c + 7
  const bool rot = region < 2 && e.rope;
  if (region < 2) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int at = min(row + 8 * p, e.M - 1);
      const bool br1 = e.br_rows > 0 && at >= e.br_rows;     // unconditional branch
      const int jr = at - (br1 ? e.br_rows : 0) + e.row_off;  // joint-sequence row
      orow[p] = jr + (br1 ? (int)e.br_qk : 0);
      if (rot) {
        const float4* cs = reinterpret_cast<const float4*>(e.rope + (long)jr * (e.dh / 2) + cc % e.dh / 2);
        q[2 * p] = __ldg(cs);
        q[2 * p + 1] = __ldg(cs + 1);
      }
    }
  }
  __syncwarp();
  float a[32];
#pragma unroll
  for (int p = 0; p < 4; ++p) ld_chunk<8>(buf + (p * 8 + r) * kF32Ld + c, a + 8 * p);
  __syncwarp();  // the tile may be overwritten
#pragma unroll
  for (int j = 0; j < 32; ++j) a[j] += b[j & 7];
  if (gelu) {
#pragma unroll
    for (int j = 0; j < 32; ++j) a[j] = gelu_tanh_fast(a[j]);
  } else if (region < 2) {
    if (e.qn_q) {
      float w[8];
      ld_chunk<8>((region == 0 ? e.qn_q : e.qn_k) + cc % e.dh, w);
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float rr = __shfl_sync(0xffffffffu, rs, p * 8 + r);
#pragma unroll
        for (int j = 0; j < 8; ++j) a[8 * p + j] = a[8 * p + j] * rr * w[j];
      }
    }
    if (rot) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        float* y = a + 4 * u;
        const float x0 = y[0], x1 = y[1], x2 = y[2], x3 = y[3];
        y[0] = x0 * q[u].x - x1 * q[u].y;
        y[1] = x0 * q[u].y + x1 * q[u].x;
        y[2] = x2 * q[u].z - x3 * q[u].w;
        y[3] = x2 * q[u].w + x3 * q[u].z;
      }
    }
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
    if (row + 8 * p < e.M) store_vals<8>(base, (long)orow[p] * ld + cc, a + 8 * p, type);
}

// Epilogue classes.  A kernel is compiled for one class, so that it carries the registers and
// instructions of its own epilogue only: with all of them in one kernel every small change to
// one spilled another's registers.
//   EP_F32  fp32 rows (f32_rows): stores, GELU, residual updates (146 registers)
//   EP_16   16-bit outputs (rows16) without QK-norm (168)
//   EP_16N  16-bit outputs with QK-norm (168)
//   EP_ANY  everything without QK-norm, also rows that are not 16-byte aligned, and launches of
//           two problems whose classes differ (226)
// Measured, one class against four: small guided sample 1727 -> 1634 us, 50 steps of a FLUX
// block 14.00 -> 13.80 ms, double block 915 -> 896 us.
enum { EP_ANY = 0, EP_F32 = 1, EP_16 = 2, EP_16N = 3 };
static int epi_class(const Epi& e) { return f32_rows(e) ? EP_F32 : (rows16(e) ? (e.qn_q ? EP_16N : EP_16) : EP_ANY); }

// One thread's row of a BN-column accumulator in TMEM (lane base already in tb) through
// the epilogue, columns col0 .. col0 + BN - 1.  vt_buf: this warp's transpose tile.
template <int BN, int EP>
BAG_DEV void drain_accumulator(const Epi& e, int t, int row, int col0, uint32_t tb, float* vt_buf) {
  const int row0 = row - (int)(threadIdx.x & 31);
  const bool vt_warp = EP != EP_F32 && e.kind == EPI_QKV && e.v_mode == 1 && e.qkv_type != kStoreF32;
  const bool f32 = EP == EP_F32 || (EP == EP_ANY && f32_rows(e));
  const bool h16 = EP == EP_16 || EP == EP_16N || (EP == EP_ANY && rows16(e));
  auto chunk = [&](int c, float rs) {  // 32 columns; the branches are warp-uniform
    float v[32];
    tmem_ld32(tb + (uint32_t)c, v);
    const int col = col0 + c;
    if (f32)
      store_f32_warp(e, t, row0, col, v, vt_buf);
    else if (vt_warp && col < e.N && (col + e.col_base) / e.d == 2)
      store_vt_warp(e, row, col, v, vt_buf);
    else if (h16)
      store_16_warp(e, row0, col, v, vt_buf, rs);
    else
      epi_apply<32>(e, t, row, col, v);
  };
  if constexpr (EP != EP_16N) {
#pragma unroll 1
    for (int c = 0; c < BN; c += 32) chunk(c, 1.f);
  } else {
    // QK-norm: the tile holds whole heads (BN a multiple of dh, checked at launch); a first pass
    // over each q / k head takes its sum of squares (bias included), the second applies the
    // epilogue with 1 / RMS.  The TMEM loads are warp-wide, so every lane takes them whatever
    // its row.
#pragma unroll 1
    for (int h0 = 0; h0 < BN; h0 += e.dh) {
      const int col = col0 + h0;
      float rs = 1.f;
      if ((col + e.col_base) / e.d < 2 && col < e.N) {
        float ss = 0.f;
#pragma unroll 1
        for (int c = 0; c < e.dh; c += 32) {
          float v[32];
          tmem_ld32(tb + (uint32_t)(h0 + c), v);
          epi_add_bias<32>(e, col + c, v);
#pragma unroll
          for (int j = 0; j < 32; ++j) ss = fmaf(v[j], v[j], ss);
        }
        rs = rsqrtf(ss / (float)e.dh + 1e-6f);
      }
#pragma unroll 1
      for (int c = 0; c < e.dh; c += 32) chunk(h0 + c, rs);
    }
  }
}

// Epilogue warps: a launch on this kernel has a tile or two per SM, so its drain is hidden
// behind little; eight warps (two to each lane quarter, half the columns each) halve it, where
// the class leaves them the registers.  Small guided sample 1667 -> 1648 us, small Wan-shaped
// sample 1115 -> 1098 us.
template <int BN, int EP>
struct TcCfg {
  static constexpr int WARPS = EP == EP_F32 || EP == EP_16 ? 8 : 4;
  static constexpr int THREADS = 64 + 32 * WARPS;
  static constexpr int STAGES = (BN == 128 ? 6 : 8) - (WARPS == 8);
  static constexpr int A_BYTES = TC_BM * TC_BK * 2;
  static constexpr int B_BYTES = BN * TC_BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int TMEM_COLS = 2 * BN;
  static constexpr int SMEM = STAGES * STAGE_BYTES + 1024 + 256 + WARPS * kVtScratchFloats * 4;
};

template <int BN, int EP>
__global__ void __launch_bounds__(TcCfg<BN, EP>::THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmB0,
                   const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                   const __grid_constant__ Epi e0, const __grid_constant__ Epi e1, int M0, int M1,
                   int N, int K, int a_split, int g0, int g1, int* err) {
  grid_dep_sync();
  // Two independent problems with the same N and K may share one launch (problem 1 has
  // M1 rows, possibly 0): their tiles form one list, problem 0's first, so a small
  // problem fills the SMs the large one leaves idle in its last wave.
  using C = TcCfg<BN, EP>;
  if (epi_skip(e0.st, e0.flag_want)) return;
  epi_bump(e0);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + C::STAGES * C::A_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::STAGES * C::STAGE_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* tfull = empty + C::STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  float* vt_scratch = reinterpret_cast<float*>(smem + C::STAGES * C::STAGE_BYTES + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int num_m0 = (M0 + TC_BM - 1) / TC_BM, num_m1 = (M1 + TC_BM - 1) / TC_BM, num_n = N / BN;
  const int tiles0 = num_m0 * num_n;
  auto decode = [&](int tile, int& pb, int& mt, int& nt) {
    if (tile < tiles0) {
      pb = 0;
      raster(tile, num_m0, num_n, g0, mt, nt);
    } else {
      pb = 1;
      raster(tile - tiles0, num_m1, num_n, g1, mt, nt);
    }
  };
  // a_split: A holds [hi | lo] bf16 halves of an fp32 activation ([M, 2K]); the K loop
  // runs twice as long, feeding each W chunk once with hi and once with lo, so the
  // product is accurate to fp32 accumulation while W is streamed once.
  const int tiles = tiles0 + num_m1 * num_n, kit = (a_split ? 2 : 1) * (K / TC_BK);
  const int t = epi_step(e0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tfull + 1, 1);
    mbar_init(tempty, C::WARPS);  // one arrival per epilogue warp
    mbar_init(tempty + 1, C::WARPS);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmA0);
    tma_prefetch_desc(&tmB0);
    if (M1 > 0) {
      tma_prefetch_desc(&tmA1);
      tma_prefetch_desc(&tmB1);
    }
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      int s = 0;
      uint32_t ph = 0;
      long issued = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        int pb, mt, nt;
        decode(tile, pb, mt, nt);
        const CUtensorMap* tmA = pb ? &tmA1 : &tmA0;
        const CUtensorMap* tmB = pb ? &tmB1 : &tmB0;
        for (int kb = 0; kb < kit; ++kb) {
          if (!mbar_wait(empty + s, ph ^ 1, abort_flag)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(full + s, C::STAGE_BYTES);
          const int ka = a_split ? (kb & 1) * K + (kb >> 1) * TC_BK : kb * TC_BK;
          const int kw = a_split ? (kb >> 1) * TC_BK : kb * TC_BK;
          tma_load_2d(sA + s * C::A_BYTES, tmA, ka, mt * TC_BM, full + s);
          tma_load_2d(sB + s * C::B_BYTES, tmB, kw, nt * BN, full + s);
          ++issued;
          if (++s == C::STAGES) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok) {
        // drain: wait (bounded) for the copies this thread may still have in flight
        const uint64_t t0 = global_ns();
        for (int i = 0; i < C::STAGES && i < issued; ++i) {
          if (--s < 0) {
            s = C::STAGES - 1;
            ph ^= 1;
          }
          while (!mbar_try_wait(full + s, ph) && global_ns() - t0 < kWaitLimitNs) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (converged warp, one elected lane issues) ----------------
    constexpr uint32_t idesc = idesc_bf16_f32(TC_BM, BN);
    const uint32_t a_base = smem_u32(sA), b_base = smem_u32(sB);
    int s = 0;
    uint32_t ph = 0;
    int acc = 0;
    uint32_t aph = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
      if (!mbar_wait_warp(tempty + acc, aph ^ 1, abort_flag)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t dt = tmem_base + (uint32_t)(acc * BN);
      for (int kb = 0; kb < kit; ++kb) {
        if (!mbar_wait_warp(full + s, ph, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t ad = sw128_desc(a_base + s * C::A_BYTES);
        const uint64_t bd = sw128_desc(b_base + s * C::B_BYTES);
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < TC_BK / 16; ++k)  // 32 bytes along K: two 16-byte units
            mma_bf16(dt, ad + 2 * k, bd + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          mma_commit(empty + s);
        }
        __syncwarp();
        if (++s == C::STAGES) {
          s = 0;
          ph ^= 1;
        }
      }
      if (!ok) break;
      if (elect_one()) mma_commit(tfull + acc);
      __syncwarp();
      acc ^= 1;
      if (acc == 0) aph ^= 1;
    }
    // make sure every issued MMA has finished before TMEM is released
    if (elect_one()) {
      mma_commit(drain);
      const uint64_t t0 = global_ns();
      while (!mbar_try_wait(drain, 0) && global_ns() - t0 < kWaitLimitNs) {
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue (each four warps cover TMEM lane quarters 2,3,0,1) ----------------
    constexpr int W = BN * 4 / C::WARPS;
    const int q = warp & 3, c0 = (warp - 2) / 4 * W;
    int acc = 0;
    uint32_t aph = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      int pb, mt, nt;
      decode(tile, pb, mt, nt);
      const Epi& e = pb ? e1 : e0;
      bool ok = mbar_wait(tfull + acc, aph, abort_flag);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const int row = mt * TC_BM + q * 32 + lane;
      const uint32_t tb = tmem_base + (uint32_t)(acc * BN + c0) + ((uint32_t)(q * 32) << 16);
      drain_accumulator<W, EP>(e, t, row, nt * BN + c0, tb, vt_scratch + (warp - 2) * kVtScratchFloats);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty + acc);
      acc ^= 1;
      if (acc == 0) aph ^= 1;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag && err) atomicOr(err, 1);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

// Class of a launch of one or two problems.
static int launch_class(const Epi& e0, int M1, const Epi& e1) {
  return M1 <= 0 || epi_class(e0) == epi_class(e1) ? epi_class(e0) : EP_ANY;
}

template <int BN>
static cudaError_t launch_tc(const void* A0, long lda0, const void* W0, long ldw0, int M0,
                             const Epi& e0, const void* A1, long lda1, const void* W1, long ldw1,
                             int M1, const Epi& e1, int N, int K, int* err, cudaStream_t s,
                             int a_split) {
  const uint64_t ka = (uint64_t)K * (a_split ? 2 : 1);
  CUtensorMap ta0, tb0, ta1, tb1;
  if (encode_tmap_2d_bf16(&ta0, A0, ka, (uint64_t)M0, (uint64_t)lda0 * 2, TC_BK, TC_BM) ||
      encode_tmap_2d_bf16(&tb0, W0, (uint64_t)K, (uint64_t)N, (uint64_t)ldw0 * 2, TC_BK, BN))
    return cudaErrorInvalidValue;
  if (M1 > 0) {
    if (encode_tmap_2d_bf16(&ta1, A1, ka, (uint64_t)M1, (uint64_t)lda1 * 2, TC_BK, TC_BM) ||
        encode_tmap_2d_bf16(&tb1, W1, (uint64_t)K, (uint64_t)N, (uint64_t)ldw1 * 2, TC_BK, BN))
      return cudaErrorInvalidValue;
  } else {
    ta1 = ta0;
    tb1 = tb0;
  }
  const int tiles = ((M0 + TC_BM - 1) / TC_BM + (M1 + TC_BM - 1) / TC_BM) * (N / BN);
  const int grid = std::min(tiles, num_sms());
  auto launch = [&](auto kernel, int threads, int smem) {
    launch_kernel(kernel, grid, threads, smem, s, ta0, tb0, ta1, tb1, e0, e1, M0, M1, N, K, a_split,
                  tile_group_rows(M0, TC_BM, K, a_split), tile_group_rows(M1, TC_BM, K, a_split), err);
  };
  const int ep = launch_class(e0, M1, e1);
  if (ep == EP_F32)
    launch(gemm_tc_kernel<BN, EP_F32>, TcCfg<BN, EP_F32>::THREADS, TcCfg<BN, EP_F32>::SMEM);
  else if (ep == EP_16)
    launch(gemm_tc_kernel<BN, EP_16>, TcCfg<BN, EP_16>::THREADS, TcCfg<BN, EP_16>::SMEM);
  else if (ep == EP_16N) {
    if constexpr (BN == 128)
      launch(gemm_tc_kernel<BN, EP_16N>, TcCfg<BN, EP_16N>::THREADS, TcCfg<BN, EP_16N>::SMEM);
    else
      return cudaErrorNotSupported;  // whole heads of 128 in a tile
  } else
    launch(gemm_tc_kernel<BN, EP_ANY>, TcCfg<BN, EP_ANY>::THREADS, TcCfg<BN, EP_ANY>::SMEM);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Split-K GEMM: a cluster of S CTAs computes one 128 x 64 tile, each CTA a contiguous
// share of the K blocks.  The CTAs then exchange accumulator rows through distributed
// shared memory (rank o receives rows [o, o + 1) * 128 / S of every CTA), sum them in rank
// order and apply the epilogue to their rows, so the result is deterministic.
// Bound: latency.  A launch with few tiles leaves most SMs idle while each busy one takes
// its operands at one SM's L2 rate (24 KB a K block, measured about 0.28 us); the split
// divides that chain by S.  Epilogues that need whole heads or 32 x 32 blocks (EPI_QKV)
// stay on the unsplit kernels.
// Measured (profiled launches): 4096 x 64 x 3072 30.7 -> 16.3 us, 910 x 512 x 2560 19.0 -> 16.2,
// 390 x 512 x 1536 16.1 -> 12.1, 378 x 64 x 512 17.2 -> 11.4.
// ---------------------------------------------------------------------------
constexpr int SK_BN = 64, SK_STAGES = 3, SK_LD = SK_BN + 4;
constexpr int SK_A_BYTES = TC_BM * TC_BK * 2, SK_B_BYTES = SK_BN * TC_BK * 2;
constexpr int SK_STAGE_BYTES = SK_A_BYTES + SK_B_BYTES;
constexpr int SK_RECV_BYTES = TC_BM * SK_LD * 4;  // S slots of 128 / S rows
constexpr int SK_SMEM = SK_STAGES * SK_STAGE_BYTES + SK_RECV_BYTES + 1024 + 256;

template <int S>
__global__ void __launch_bounds__(192)
    gemm_splitk_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmB0,
                       const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                       const __grid_constant__ Epi e0, const __grid_constant__ Epi e1, int M0, int M1,
                       int N, int K, int a_split, int* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + SK_STAGES * SK_A_BYTES;
  float* recv = reinterpret_cast<float*>(smem + SK_STAGES * SK_STAGE_BYTES);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + SK_STAGES * SK_STAGE_BYTES + SK_RECV_BYTES);
  uint64_t* empty = full + SK_STAGES;
  uint64_t* tfull = empty + SK_STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int rank = (int)cluster_ctarank();
  const int num_n = N / SK_BN, tiles0 = (M0 + TC_BM - 1) / TC_BM * num_n;
  int tile = blockIdx.x / S;
  const bool pb = tile >= tiles0;  // problem 1's tiles follow problem 0's
  if (pb) tile -= tiles0;
  const int mt = tile / num_n, nt = tile % num_n;
  const CUtensorMap* tmA = pb ? &tmA1 : &tmA0;
  const CUtensorMap* tmB = pb ? &tmB1 : &tmB0;
  const Epi& e = pb ? e1 : e0;
  const int kit = (a_split ? 2 : 1) * (K / TC_BK);
  const int kb0 = rank * kit / S, kb1 = (rank + 1) * kit / S;

  if (threadIdx.x == 0) {
    for (int s = 0; s < SK_STAGES; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    mbar_init(tfull, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(tmA);
    tma_prefetch_desc(tmB);
  }
  grid_dep_sync();
  // every CTA of a cluster sees the same flag, so they leave together
  if (epi_skip(e0.st, e0.flag_want)) return;
  epi_bump(e0);
  const int t = epi_step(e0);
  __syncwarp();
  if (warp == 1) {
    tmem_alloc(tmem_slot, SK_BN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();  // barriers initialised, tensor memory allocated, every CTA running
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      int s = 0;
      uint32_t ph = 0;
      int issued = 0;
      bool ok = true;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait(empty + s, ph ^ 1, abort_flag)) {
          ok = false;
          break;
        }
        mbar_arrive_expect_tx(full + s, SK_STAGE_BYTES);
        const int ka = a_split ? (kb & 1) * K + (kb >> 1) * TC_BK : kb * TC_BK;
        const int kw = a_split ? (kb >> 1) * TC_BK : kb * TC_BK;
        tma_load_2d(sA + s * SK_A_BYTES, tmA, ka, mt * TC_BM, full + s);
        tma_load_2d(sB + s * SK_B_BYTES, tmB, kw, nt * SK_BN, full + s);
        ++issued;
        if (++s == SK_STAGES) {
          s = 0;
          ph ^= 1;
        }
      }
      if (!ok) {
        // drain: wait (bounded) for the copies this thread may still have in flight
        const uint64_t t0 = global_ns();
        for (int i = 0; i < SK_STAGES && i < issued; ++i) {
          if (--s < 0) {
            s = SK_STAGES - 1;
            ph ^= 1;
          }
          while (!mbar_try_wait(full + s, ph) && global_ns() - t0 < kWaitLimitNs) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (converged warp, one elected lane issues) ----------------
    constexpr uint32_t idesc = idesc_bf16_f32(TC_BM, SK_BN);
    const uint32_t a_base = smem_u32(sA), b_base = smem_u32(sB);
    int s = 0;
    uint32_t ph = 0;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!mbar_wait_warp(full + s, ph, abort_flag)) break;
      tc_fence_after();
      const uint64_t ad = sw128_desc(a_base + s * SK_A_BYTES);
      const uint64_t bd = sw128_desc(b_base + s * SK_B_BYTES);
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < TC_BK / 16; ++k)
          mma_bf16(tmem_base, ad + 2 * k, bd + 2 * k, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
        mma_commit(empty + s);
      }
      __syncwarp();
      if (++s == SK_STAGES) {
        s = 0;
        ph ^= 1;
      }
    }
    // all MMAs issued so far (whatever happened above) finish before tfull completes, and
    // the bounded wait keeps tensor memory until then
    if (elect_one()) {
      mma_commit(tfull);
      const uint64_t t0 = global_ns();
      while (!mbar_try_wait(tfull, 0) && global_ns() - t0 < kWaitLimitNs) {
      }
    }
    __syncwarp();
  } else {
    // ---------------- exchange: each warp's 32 accumulator rows to their owners ----------------
    const int q = warp & 3;
    const bool ok = mbar_wait(tfull, 0, abort_flag);
    if (__all_sync(0xffffffffu, ok)) {
      tc_fence_after();
      constexpr int RPO = TC_BM / S;  // rows per owner
      const int r = q * 32 + lane;
      const uint32_t dst = mapa_shared(smem_u32(recv), (uint32_t)(r / RPO)) +
                           (uint32_t)((rank * RPO + r % RPO) * SK_LD * 4);
      const uint32_t tb = tmem_base + ((uint32_t)(q * 32) << 16);
#pragma unroll
      for (int c = 0; c < SK_BN; c += 32) {
        float v[32];
        tmem_ld32(tb + (uint32_t)c, v);
#pragma unroll
        for (int j = 0; j < 32; j += 4) st_cluster4(dst + (uint32_t)(c + j) * 4, v[j], v[j + 1], v[j + 2], v[j + 3]);
      }
    }
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();  // every CTA's rows have arrived; no access to another CTA follows
  if (warp >= 2 && !*abort_flag) {
    constexpr int RPO = TC_BM / S, NV = SK_BN / S;  // 128 threads: S per row, NV columns each
    const int i = threadIdx.x - 64, lr = i / S, c = (i % S) * NV;
    float v[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = 0.f;
#pragma unroll
    for (int p = 0; p < S; ++p) {
      float w[NV];
      ld_chunk<NV>(recv + (p * RPO + lr) * SK_LD + c, w);
#pragma unroll
      for (int j = 0; j < NV; ++j) v[j] += w[j];
    }
    epi_apply<NV>(e, t, mt * TC_BM + rank * RPO + lr, nt * SK_BN + c, v);
  }
  if (threadIdx.x == 0 && *abort_flag && err) atomicOr(err, 1);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, SK_BN);
  }
}

// CTAs per tile for a launch of `tiles` 128 x 64 tiles and `kit` K blocks: the largest
// split, up to 4, that keeps the launch within one CTA per SM (clusters of eight leave 32 of
// the 152 SMs without a place; up to two CTAs an SM made the small guided sample 1592 -> 1663
// us); 1: the unsplit kernels.  A guided launch may hold twice the planned tiles; two CTAs fit
// on an SM.
// From SK_MIN_KB K blocks on.  As single calls, unsplit against split (us): 32 x 1024 x 256, two
// CTAs, 6.2 against 7.9; 32 x 1024 x 448 7.0 against 8.5; eight blocks, 300 x 512 x 512, four
// CTAs, 8.2 against 8.5 and with GELU 8.7 in both; 300 x 512 x 1024 9.8 against 9.0; two CTAs,
// 1000 x 512 x 1024, 10.0 against 9.8.  In the samples, where programmatic launch hides the
// cluster's start, eight blocks already gain (small Wan-shaped sample 1113 -> 1037 us, small
// guided one 1630 -> 1600).
constexpr int SK_MIN_KB = 8;
static int splitk_ctas(int tiles, int kit, int ns) {
  if (kit < SK_MIN_KB) return 1;
  for (int s = 4; s > 1; s /= 2)
    if (tiles * s <= ns) return s;
  return 1;
}

static cudaError_t launch_splitk(int S, const void* A0, long lda0, const void* W0, long ldw0, int M0,
                                 const Epi& e0, const void* A1, long lda1, const void* W1, long ldw1,
                                 int M1, const Epi& e1, int N, int K, int* err, cudaStream_t s,
                                 int a_split) {
  const uint64_t ka = (uint64_t)K * (a_split ? 2 : 1);
  CUtensorMap ta0, tb0, ta1, tb1;
  if (encode_tmap_2d_bf16(&ta0, A0, ka, (uint64_t)M0, (uint64_t)lda0 * 2, TC_BK, TC_BM) ||
      encode_tmap_2d_bf16(&tb0, W0, (uint64_t)K, (uint64_t)N, (uint64_t)ldw0 * 2, TC_BK, SK_BN))
    return cudaErrorInvalidValue;
  if (M1 > 0) {
    if (encode_tmap_2d_bf16(&ta1, A1, ka, (uint64_t)M1, (uint64_t)lda1 * 2, TC_BK, TC_BM) ||
        encode_tmap_2d_bf16(&tb1, W1, (uint64_t)K, (uint64_t)N, (uint64_t)ldw1 * 2, TC_BK, SK_BN))
      return cudaErrorInvalidValue;
  } else {
    ta1 = ta0;
    tb1 = tb0;
  }
  const int tiles = ((M0 + TC_BM - 1) / TC_BM + (M1 + TC_BM - 1) / TC_BM) * (N / SK_BN);
  auto launch = [&](auto kernel) {
    launch_cluster(kernel, (unsigned)S, (unsigned)(tiles * S), 192, SK_SMEM, s, ta0, tb0, ta1, tb1, e0, e1, M0, M1,
                   N, K, a_split, err);
  };
  S == 4 ? launch(gemm_splitk_kernel<4>) : launch(gemm_splitk_kernel<2>);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// CTA-pair GEMM: clusters of two CTAs compute 256 x 256 tiles with cta_group::2 MMAs
// (M = 256, N = 256, K = 16 per instruction).  Each CTA stages its own 128 rows of A
// and 128 rows of W per k-block (32 KB instead of the single-CTA 128 x 256 tile's
// 48 KB), so every SM moves a third less shared-memory operand data per MMA cycle, the
// limit of the single-CTA kernel.  Roles as in gemm_tc_kernel: warp 0 of each CTA loads
// its halves (completion signalled on the even CTA's barrier), warp 1 of the even CTA
// issues the MMAs and multicasts their completion to both CTAs, warps 2..5 of each CTA
// (2..9 for fp32 rows with few K blocks) drain its 128 accumulator rows.
// ---------------------------------------------------------------------------
constexpr int PR_BM = 256, PR_BN = 256;
constexpr int PR_HALF_BYTES = 128 * TC_BK * 2;  // one CTA's A or W half-tile per k-block
constexpr int PR_STAGE_BYTES = 2 * PR_HALF_BYTES;
constexpr int PR_TMEM_COLS = 2 * PR_BN;         // double-buffered accumulator
// WARPS epilogue warps.  Four drain a tile while the next one is multiplied; with few K blocks
// the drain is the longer part, and eight (two to each lane quarter, half the columns each)
// halve it, at the price of a stage of the ring.
template <int WARPS>
struct PrCfg {
  static constexpr int STAGES = WARPS == 8 ? 5 : 6;
  static constexpr int THREADS = 64 + 32 * WARPS;
  static constexpr int SMEM = STAGES * PR_STAGE_BYTES + 1024 + 256 + WARPS * kVtScratchFloats * 4;
};

template <int EP, int EW>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PrCfg<EW>::THREADS, 1)
    gemm_pair_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmB0,
                     const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                     const __grid_constant__ Epi e0, const __grid_constant__ Epi e1, int M0, int M1,
                     int N, int K, int a_split, int g0, int g1, int* err) {
  constexpr int STAGES = PrCfg<EW>::STAGES;
  grid_dep_sync();
  // both CTAs of a pair see the same flag, so they leave together
  if (epi_skip(e0.st, e0.flag_want)) return;
  epi_bump(e0);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * PR_HALF_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * PR_STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  float* vt_scratch = reinterpret_cast<float*>(smem + STAGES * PR_STAGE_BYTES + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int num_m0 = (M0 + PR_BM - 1) / PR_BM, num_m1 = (M1 + PR_BM - 1) / PR_BM, num_n = N / PR_BN;
  const int tiles0 = num_m0 * num_n;
  auto decode = [&](int tile, int& pb, int& mt, int& nt) {
    if (tile < tiles0) {
      pb = 0;
      raster(tile, num_m0, num_n, g0, mt, nt);
    } else {
      pb = 1;
      raster(tile - tiles0, num_m1, num_n, g1, mt, nt);
    }
  };
  const int tiles = tiles0 + num_m1 * num_n, kit = (a_split ? 2 : 1) * (K / TC_BK);
  const int t = epi_step(e0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full + s, 1);   // even CTA: its producer's expect_tx; both CTAs' bytes
      mbar_init(empty + s, 1);  // both CTAs: one multicast commit per consumed stage
    }
    mbar_init(tfull, 1);
    mbar_init(tfull + 1, 1);
    mbar_init(tempty, 2 * EW);     // even CTA: every epilogue warp of both CTAs
    mbar_init(tempty + 1, 2 * EW);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmA0);
    tma_prefetch_desc(&tmB0);
    if (M1 > 0) {
      tma_prefetch_desc(&tmA1);
      tma_prefetch_desc(&tmB1);
    }
  }
  __syncwarp();
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, PR_TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();  // barriers of both CTAs initialised, tensor memory allocated
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer (both CTAs: their own halves) ----------------
      int s = 0;
      uint32_t ph = 0;
      long issued = 0;
      bool ok = true;
      for (int tile = pair; tile < tiles && ok; tile += npairs) {
        int pb, mt, nt;
        decode(tile, pb, mt, nt);
        const CUtensorMap* tmA = pb ? &tmA1 : &tmA0;
        const CUtensorMap* tmB = pb ? &tmB1 : &tmB0;
        for (int kb = 0; kb < kit; ++kb) {
          if (!mbar_wait(empty + s, ph ^ 1, abort_flag)) {
            ok = false;
            break;
          }
          if (rank == 0) mbar_arrive_expect_tx(full + s, 2 * PR_STAGE_BYTES);
          const uint32_t fb = mapa_shared(smem_u32(full + s), 0);
          const int ka = a_split ? (kb & 1) * K + (kb >> 1) * TC_BK : kb * TC_BK;
          const int kw = a_split ? (kb >> 1) * TC_BK : kb * TC_BK;
          tma_load_2d_pair(sA + s * PR_HALF_BYTES, tmA, ka, mt * PR_BM + (int)rank * 128, fb);
          tma_load_2d_pair(sB + s * PR_HALF_BYTES, tmB, kw, nt * PR_BN + (int)rank * 128, fb);
          ++issued;
          if (++s == STAGES) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok && rank == 0) {
        // drain (bounded): both CTAs' copies in flight complete on this CTA's barriers
        const uint64_t t0 = global_ns();
        for (int i = 0; i < STAGES && i < issued; ++i) {
          if (--s < 0) {
            s = STAGES - 1;
            ph ^= 1;
          }
          while (!mbar_try_wait(full + s, ph) && global_ns() - t0 < kWaitLimitNs) {
          }
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // -------- MMA issuer (even CTA; converged warp, one elected lane issues) --------
      constexpr uint32_t idesc = idesc_bf16_f32(PR_BM, PR_BN);
      const uint32_t a_base = smem_u32(sA), b_base = smem_u32(sB);
      int s = 0;
      uint32_t ph = 0;
      int acc = 0;
      uint32_t aph = 0;
      bool ok = true;
      for (int tile = pair; tile < tiles && ok; tile += npairs) {
        if (!mbar_wait_warp(tempty + acc, aph ^ 1, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t dt = tmem_base + (uint32_t)(acc * PR_BN);
        for (int kb = 0; kb < kit; ++kb) {
          if (!mbar_wait_warp(full + s, ph, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t ad = sw128_desc(a_base + s * PR_HALF_BYTES);
          const uint64_t bd = sw128_desc(b_base + s * PR_HALF_BYTES);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k)  // 32 bytes along K: two 16-byte units
              mma_bf16_pair(dt, ad + 2 * k, bd + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
            mma_commit_pair(empty + s, 3);
          }
          __syncwarp();
          if (++s == STAGES) {
            s = 0;
            ph ^= 1;
          }
        }
        if (!ok) break;
        if (elect_one()) mma_commit_pair(tfull + acc, 3);
        __syncwarp();
        acc ^= 1;
        if (acc == 0) aph ^= 1;
      }
      // every issued MMA has finished before tensor memory is released
      if (elect_one()) {
        mma_commit_pair(drain, 1);
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(drain, 0) && global_ns() - t0 < kWaitLimitNs) {
        }
      }
      __syncwarp();
    }
  } else {
    // ---------------- epilogue (both CTAs: their 128 rows of each tile) ----------------
    // (eight warps: two to each lane quarter, half the columns each)
    constexpr int W = PR_BN * 4 / EW;
    const int q = warp & 3, c0 = (warp - 2) / 4 * W;
    int acc = 0;
    uint32_t aph = 0;
    const uint32_t te_remote = mapa_shared(smem_u32(tempty), 0);
    for (int tile = pair; tile < tiles; tile += npairs) {
      int pb, mt, nt;
      decode(tile, pb, mt, nt);
      const Epi& e = pb ? e1 : e0;
      bool ok = mbar_wait(tfull + acc, aph, abort_flag);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const int row = mt * PR_BM + (int)rank * 128 + q * 32 + lane;
      const uint32_t tb = tmem_base + (uint32_t)(acc * PR_BN + c0) + ((uint32_t)(q * 32) << 16);
      drain_accumulator<W, EP>(e, t, row, nt * PR_BN + c0, tb, vt_scratch + (warp - 2) * kVtScratchFloats);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0)
          mbar_arrive(tempty + acc);
        else
          mbar_arrive_remote(te_remote + (uint32_t)(acc * sizeof(uint64_t)));
      }
      acc ^= 1;
      if (acc == 0) aph ^= 1;
    }
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();  // no CTA of the pair still uses the pair's tensor memory
  if (threadIdx.x == 0 && *abort_flag && err) atomicOr(err, 1);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, PR_TMEM_COLS);
  }
}

// Tiles of the pair kernel for a launch of one or two problems; it is used when N is a
// multiple of 256 and there are at least as many 256 x 256 tiles as CTA pairs.
static int pair_tiles(int M0, int M1, int N) {
  return ((M0 + PR_BM - 1) / PR_BM + (M1 + PR_BM - 1) / PR_BM) * (N / PR_BN);
}

static cudaError_t launch_pair(const void* A0, long lda0, const void* W0, long ldw0, int M0,
                               const Epi& e0, const void* A1, long lda1, const void* W1, long ldw1,
                               int M1, const Epi& e1, int N, int K, int* err, cudaStream_t s,
                               int a_split) {
  const uint64_t ka = (uint64_t)K * (a_split ? 2 : 1);
  CUtensorMap ta0, tb0, ta1, tb1;
  if (encode_tmap_2d_bf16(&ta0, A0, ka, (uint64_t)M0, (uint64_t)lda0 * 2, TC_BK, 128) ||
      encode_tmap_2d_bf16(&tb0, W0, (uint64_t)K, (uint64_t)N, (uint64_t)ldw0 * 2, TC_BK, 128))
    return cudaErrorInvalidValue;
  if (M1 > 0) {
    if (encode_tmap_2d_bf16(&ta1, A1, ka, (uint64_t)M1, (uint64_t)lda1 * 2, TC_BK, 128) ||
        encode_tmap_2d_bf16(&tb1, W1, (uint64_t)K, (uint64_t)N, (uint64_t)ldw1 * 2, TC_BK, 128))
      return cudaErrorInvalidValue;
  } else {
    ta1 = ta0;
    tb1 = tb0;
  }
  const int pairs = std::min(pair_tiles(M0, M1, N), num_sms() / 2);
  auto launch = [&](auto kernel, int threads, int smem) {
    launch_kernel(kernel, 2 * pairs, threads, smem, s, ta0, tb0, ta1, tb1, e0, e1, M0, M1, N, K, a_split,
                  tile_group_rows(M0, PR_BM, K, a_split), tile_group_rows(M1, PR_BM, K, a_split), err);
  };
  const int ep = launch_class(e0, M1, e1);
  // fp32 rows with at most 16 K blocks take eight epilogue warps: 4096 x 3072 x 128 27.2 -> 22.5
  // us as a profiled launch, 1373 x 12288 x 3072 with GELU 74.8 -> 75.8
  using P4 = PrCfg<4>;
  using P8 = PrCfg<8>;
  if (ep == EP_F32 && (a_split ? 2 : 1) * (K / TC_BK) <= 16)
    launch(gemm_pair_kernel<EP_F32, 8>, P8::THREADS, P8::SMEM);
  else if (ep == EP_F32)
    launch(gemm_pair_kernel<EP_F32, 4>, P4::THREADS, P4::SMEM);
  else if (ep == EP_16)
    launch(gemm_pair_kernel<EP_16, 4>, P4::THREADS, P4::SMEM);
  else if (ep == EP_16N)
    launch(gemm_pair_kernel<EP_16N, 4>, P4::THREADS, P4::SMEM);
  else
    launch(gemm_pair_kernel<EP_ANY, 4>, P4::THREADS, P4::SMEM);
  return cudaGetLastError();
}

int gemm_uses_pair(int M0, int M1, int N) {
  return N % PR_BN == 0 && num_sms() >= 2 && pair_tiles(M0, M1, N) >= num_sms() / 2;
}

cudaError_t attention_tc_init();

cudaError_t kernels_init() {
  cudaError_t r = cudaSuccess;
  auto smem = [&](auto kernel, int bytes) {
    if (r == cudaSuccess) r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  smem(gemm_tc_kernel<128, EP_ANY>, TcCfg<128, EP_ANY>::SMEM);
  smem(gemm_tc_kernel<128, EP_F32>, TcCfg<128, EP_F32>::SMEM);
  smem(gemm_tc_kernel<128, EP_16>, TcCfg<128, EP_16>::SMEM);
  smem(gemm_tc_kernel<128, EP_16N>, TcCfg<128, EP_16N>::SMEM);
  smem(gemm_tc_kernel<64, EP_ANY>, TcCfg<64, EP_ANY>::SMEM);
  smem(gemm_tc_kernel<64, EP_F32>, TcCfg<64, EP_F32>::SMEM);
  smem(gemm_tc_kernel<64, EP_16>, TcCfg<64, EP_16>::SMEM);
  smem(gemm_pair_kernel<EP_ANY, 4>, PrCfg<4>::SMEM);
  smem(gemm_pair_kernel<EP_F32, 4>, PrCfg<4>::SMEM);
  smem(gemm_pair_kernel<EP_F32, 8>, PrCfg<8>::SMEM);
  smem(gemm_pair_kernel<EP_16, 4>, PrCfg<4>::SMEM);
  smem(gemm_pair_kernel<EP_16N, 4>, PrCfg<4>::SMEM);
  smem(gemm_splitk_kernel<2>, SK_SMEM);
  smem(gemm_splitk_kernel<4>, SK_SMEM);
  smem(gemm_simt_kernel<float, true>, SG_SMEM);
  smem(gemm_simt_kernel<__nv_bfloat16, true>, SG_SMEM);
  smem(gemm_simt_kernel<__nv_bfloat16, false>, SG_SMEM);
  if (r == cudaSuccess) r = attention_tc_init();
  num_sms();
  return r;
}

int gemm_tc_supported(int M, int N, int K, long lda, long ldw) {
  if (M <= 0 || K <= 0 || K % TC_BK != 0 || N % 64 != 0) return 0;
  if (lda % 8 != 0 || ldw % 8 != 0) return 0;
  return get_encode_fn() != nullptr;
}

// tensor-core launch of one or two problems (M1 = 0: one); picks the widest tile that
// still gives every SM at least one tile
static cudaError_t gemm_tc2(const void* A0, long lda0, const void* W0, long ldw0, int M0,
                            const Epi& e0, const void* A1, long lda1, const void* W1, long ldw1,
                            int M1, const Epi& e1, int N, int K, int* err, cudaStream_t s,
                            int a_split) {
  const uintptr_t ptrs = reinterpret_cast<uintptr_t>(A0) | reinterpret_cast<uintptr_t>(W0) |
                         (M1 > 0 ? (reinterpret_cast<uintptr_t>(A1) | reinterpret_cast<uintptr_t>(W1)) : 0);
  if ((ptrs & 15) || !gemm_tc_supported(M0, N, K, lda0, ldw0) ||
      (M1 > 0 && !gemm_tc_supported(M1, N, K, lda1, ldw1)))
    return cudaErrorNotSupported;
  if (a_split && (lda0 < 2L * K || (M1 > 0 && lda1 < 2L * K))) return cudaErrorInvalidValue;
  const int ns = num_sms();
  const int mt = (M0 + TC_BM - 1) / TC_BM + (M1 + TC_BM - 1) / TC_BM;
  // QK-norm epilogues need whole heads in a tile (bf16 backbones have heads of 128) and 16-byte
  // aligned 16-bit operands (the contexts' buffers)
  const bool qkn = e0.qn_q || (M1 > 0 && e1.qn_q);
  if (qkn && (e0.dh != 128 || (M1 > 0 && e1.dh != 128) || launch_class(e0, M1, e1) != EP_16N))
    return cudaErrorNotSupported;
  if (e0.kind != EPI_QKV && (M1 <= 0 || e1.kind != EPI_QKV)) {
    const int mtp = e0.plan_rows > 0 ? (e0.plan_rows + TC_BM - 1) / TC_BM : mt;
    const int split = splitk_ctas(mtp * (N / SK_BN), (a_split ? 2 : 1) * (K / TC_BK), ns);
    if (split > 1)
      return launch_splitk(split, A0, lda0, W0, ldw0, M0, e0, A1, lda1, W1, ldw1, M1 > 0 ? M1 : 0, e1, N, K, err,
                           s, a_split);
  }
  if (gemm_uses_pair(M0, M1 > 0 ? M1 : 0, N))
    return launch_pair(A0, lda0, W0, ldw0, M0, e0, A1, lda1, W1, ldw1, M1 > 0 ? M1 : 0, e1, N, K, err, s,
                       a_split);
  if (N % 128 == 0 && (mt * (N / 128) >= ns || qkn))
    return launch_tc<128>(A0, lda0, W0, ldw0, M0, e0, A1, lda1, W1, ldw1, M1, e1, N, K, err, s, a_split);
  if (qkn) return cudaErrorNotSupported;
  return launch_tc<64>(A0, lda0, W0, ldw0, M0, e0, A1, lda1, W1, ldw1, M1, e1, N, K, err, s, a_split);
}

cudaError_t gemm2(const void* A0, long lda0, const void* W0, long ldw0, int M0, const Epi& epi0,
                  const void* A1, long lda1, const void* W1, long ldw1, int M1, const Epi& epi1,
                  int N, int K, int* err, cudaStream_t s) {
  if (N <= 0 || (M0 <= 0 && M1 <= 0)) return cudaSuccess;
  Epi e0 = epi0, e1 = epi1;
  e0.M = M0;
  e0.N = N;
  e1.M = M1;
  e1.N = N;
  if (M0 <= 0) return gemm_tc2(A1, lda1, W1, ldw1, M1, e1, nullptr, 0, nullptr, 0, 0, e1, N, K, err, s, 0);
  return gemm_tc2(A0, lda0, W0, ldw0, M0, e0, A1, lda1, W1, ldw1, M1 > 0 ? M1 : 0, e1, N, K, err, s, 0);
}

cudaError_t gemm(const void* A, long lda, const void* W, long ldw, int M, int N, int K,
                 int in_bf16, const Epi& epi_in, int* err, cudaStream_t s, int force_simt,
                 int a_split) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  Epi e = epi_in;
  e.M = M;
  e.N = N;
  if (in_bf16 && !force_simt) {
    // bf16 operands always take the tensor-core path; a shape or pointer it cannot
    // tile is an error, never a silent switch to the CUDA-core kernel
    return gemm_tc2(A, lda, W, ldw, M, e, nullptr, 0, nullptr, 0, 0, e, N, K, err, s, a_split);
  }
  if (a_split) return cudaErrorInvalidValue;
  // transposed V and QK-norm are epilogues of the tensor-core kernels
  if (e.kind == EPI_QKV && (e.v_mode != 0 || e.qn_q)) return cudaErrorNotSupported;
  if (N % 4 != 0) return cudaErrorInvalidValue;
  const long tiles = (long)((N + SG_T - 1) / SG_T) * ((M + SG_T - 1) / SG_T);
  if (tiles > 0x7fffffffL) return cudaErrorInvalidValue;
  const uintptr_t ptrs = reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(W);
  if (in_bf16) {
    const bool vec = K % 8 == 0 && lda % 8 == 0 && ldw % 8 == 0 && (ptrs & 15) == 0;
    launch_kernel(vec ? gemm_simt_kernel<__nv_bfloat16, true> : gemm_simt_kernel<__nv_bfloat16, false>,
                  (unsigned)tiles, SG_WARPS * 32, SG_SMEM, s, reinterpret_cast<const __nv_bfloat16*>(A), lda,
                  reinterpret_cast<const __nv_bfloat16*>(W), ldw, M, N, K, e);
  } else {
    // the fp32 backbones' operands: rows of whole float4 groups
    if (K % 4 || lda % 4 || ldw % 4 || (ptrs & 15)) return cudaErrorNotSupported;
    launch_kernel(gemm_simt_kernel<float, true>, (unsigned)tiles, SG_WARPS * 32, SG_SMEM, s,
                  reinterpret_cast<const float*>(A), lda, reinterpret_cast<const float*>(W), ldw, M, N, K, e);
  }
  return cudaGetLastError();
}

}  // namespace bag
