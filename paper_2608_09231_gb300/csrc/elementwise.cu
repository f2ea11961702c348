// Memory-bound kernels of the cached denoising step and the on-device gate.
//
//  * ln_mod: row LayerNorm + adaLN modulation (1 + scale) * LN(x) + shift, optionally
//    fused with the trajectory signal (per-row partial sums of |m_t - m_last| and
//    |m_last|, the relative-L1 drift of the first block's modulated input).
//  * gate_step: one CTA; reduces the signal partials in a fixed order, forms the gate
//    inputs, evaluates the 3->16->1 gate in fp32 with every product and sum rounded
//    separately, applies Algorithm 2's two forced rules, updates the counters and the
//    step log, and hands the decision to a CUDA-graph conditional node.
//    The final layer's ln_mod also keeps the residual cache: R = h_out - h_in on a full
//    step, h_out = h_in + R on a reused one (plain residual reuse).
//  * stream_init: the residual stream a full step starts from.
//  * small helpers: sinusoidal timestep features, seeded fills.
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"

namespace bag {

// ---------------------------------------------------------------------------
// LayerNorm + modulation (+ signal)
// ---------------------------------------------------------------------------
// Block-wide sum through a shared array that this CTA uses for nothing else: one barrier
// (no barrier is needed before the writes, since no earlier reduction reads the array).
template <int TH>
BAG_DEV float block_sum_fresh(float v, float* red) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  float s = 0.f;
#pragma unroll
  for (int w = 0; w < TH / 32; ++w) s += red[w];
  return s;
}

// Four block-wide sums at once, through an array used for nothing else.
template <int TH>
BAG_DEV float4 block_sum4_fresh(float4 v, float4* red) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
    v.z += __shfl_xor_sync(0xffffffffu, v.z, off);
    v.w += __shfl_xor_sync(0xffffffffu, v.w, off);
  }
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int w = 0; w < TH / 32; ++w) {
    s.x += red[w].x;
    s.y += red[w].y;
    s.z += red[w].z;
    s.w += red[w].w;
  }
  return s;
}

BAG_DEV void load4(const void* p, long off, int bf16, float* r) {
  if (bf16) {
    const uint2 u = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(p) + off);
    const __nv_bfloat162 r01 = *reinterpret_cast<const __nv_bfloat162*>(&u.x);
    const __nv_bfloat162 r23 = *reinterpret_cast<const __nv_bfloat162*>(&u.y);
    r[0] = __low2float(r01);
    r[1] = __high2float(r01);
    r[2] = __low2float(r23);
    r[3] = __high2float(r23);
  } else {
    const float4 r4 = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p) + off);
    r[0] = r4.x;
    r[1] = r4.y;
    r[2] = r4.z;
    r[3] = r4.w;
  }
}

// Four floats of a row that this SM reads once: they take no L1 lines from the modulation
// vectors, which every row reads.  Kept for 50 steps of a FLUX block, 13.51 -> 13.39 ms.  Single
// launches on the device, plain loads against these: 4608 x 3072 over rotating buffers 17.7 ->
// 17.1 us but 12.8 -> 14.1 on one buffer, whose rows are in L2; 4608 x 5120 27.0 -> 25.6 and 27.3
// -> 23.1; 32,760 x 5120 148 -> 149.
BAG_DEV float4 ld_once(const float4* p) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}

// Bulk prefetch of `bytes` (a multiple of 16, 16-byte aligned) into L2.
BAG_DEV void l2_prefetch(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(p)), "r"(bytes)
               : "memory");
}

// Four consecutive elements (16-bit or fp32) copied bit for bit.
BAG_DEV void copy4(void* dst, const void* src, long off, int bf16) {
  if (bf16)
    *(reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(dst) + off)) =
        *(reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(src) + off));
  else
    *(reinterpret_cast<float4*>(reinterpret_cast<float*>(dst) + off)) =
        *(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(src) + off));
}

// One CTA of TH threads per row, VPT float4 per thread (cols <= TH * 4 * VPT): the row stays
// in registers, and the register limit (MINB CTAs per SM) keeps many rows in flight; the
// kernel is bound by the latency of its phases (load, two reductions, store), not by a pipe.
// LN_SIGNAL: with the trajectory signal.
// LN_CACHE: the final layer's pass also keeps the residual cache (see LnArgs).  As passes of
// their own, the cache update or the reuse (12 bytes an element each) and this pass took
// 26 + 20 us on 4096 x 3072 (profiled launches), together they take 29 us; and the patch
// embedding, which no longer writes the stream's copy on every step, 60 -> 39 us.
// Threads, measured: 128 with six float4 each are best for plain rows up to 3072 columns
// (4608 x 3072 from L2 16.2 -> 14.5 us with 48 registers instead of the signal's 64; 256 threads
// 18.4); the passes with more operands per column and wider rows want more threads with fewer
// columns (128 -> 256 threads: signal of 4096 x 3072 34.9 -> 30.6 us and final layer 29 -> 27 us
// as profiled launches, 32,760 x 5120 188 -> 149 us, 6.75 TB/s).
enum { LN_PLAIN = 0, LN_SIGNAL = 1, LN_CACHE = 2 };
constexpr int LN_MAX_COLS = 6144;
template <int TH, int VPT, int MINB, int MODE>
__global__ void __launch_bounds__(TH, MINB) ln_mod_kernel(const LnArgs a) {
  grid_dep_sync();
  if (epi_skip(a.st, a.flag_want)) return;
  // one shared array per reduction of the row, so that each takes a single barrier
  __shared__ float red_mean[TH / 32], red_var[TH / 32];
  const int row = blockIdx.x;
  if (row >= a.rows) return;
  if (threadIdx.x == 0 && a.prefetch_rows > 0 && row + a.prefetch_rows < a.rows) {
    // one bulk L2 prefetch per input row that a CTA of a later wave will read, so that
    // its loads find the row in L2 (row strides are multiples of 16 bytes)
    const long pr = (long)row + a.prefetch_rows;
    l2_prefetch(a.x + pr * a.ldx, (uint32_t)a.cols * 4u);
    if constexpr (MODE == LN_SIGNAL) {
      const uint32_t rb = (uint32_t)a.cols * (a.y_bf16 ? 2u : 4u);
      const long off = pr * a.ldy * (a.y_bf16 ? 2 : 4);
      l2_prefetch(reinterpret_cast<const char*>(a.sig_ref2) + off, rb);
      l2_prefetch(reinterpret_cast<const char*>(a.sig_ref) + off, rb);
    }
  }
  const int t = a.st ? a.st->t : 0;
  const float* x = a.x + (long)row * a.ldx;
  const int nv = a.cols / 4;
  float4 v[VPT];
  float s = 0.f;
  if constexpr (MODE == LN_CACHE) {
    const bool second = row >= a.split;
    const long crow = (long)(second ? row - a.split : row) * a.ldx;
    const float4* hin = reinterpret_cast<const float4*>(a.cache_in + crow);
    float4* R = reinterpret_cast<float4*>((second ? a.cache_r2 : a.cache_r) + crow);
    const bool full = a.st->flag != 0;
    const float4* src = full ? reinterpret_cast<const float4*>(x) : R;
    float4 h[VPT];
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      const int c = threadIdx.x + i * TH;
      if (c < nv) {
        v[i] = ld_once(src + c);
        h[i] = ld_once(hin + c);
      }
    }
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      const int c = threadIdx.x + i * TH;
      if (c < nv) {
        if (full)
          R[c] = make_float4(v[i].x - h[i].x, v[i].y - h[i].y, v[i].z - h[i].z, v[i].w - h[i].w);
        else
          v[i] = make_float4(h[i].x + v[i].x, h[i].y + v[i].y, h[i].z + v[i].z, h[i].w + v[i].w);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int c = threadIdx.x + i * TH;
    if (c < nv) {
      if constexpr (MODE != LN_CACHE) v[i] = ld_once(reinterpret_cast<const float4*>(x) + c);
      s += (v[i].x + v[i].y) + (v[i].z + v[i].w);
    }
  }
  float mean = 0.f, rstd = 1.f;  // identity: y = x
  if (!a.identity) {
    mean = block_sum_fresh<TH>(s, red_mean) / (float)a.cols;
    float q = 0.f;
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      const int c = threadIdx.x + i * TH;
      if (c < nv) {
        const float dx = v[i].x - mean, dy = v[i].y - mean, dz = v[i].z - mean, dw = v[i].w - mean;
        q += (dx * dx + dy * dy) + (dz * dz + dw * dw);
      }
    }
    rstd = rsqrtf(block_sum_fresh<TH>(q, red_var) / (float)a.cols + 1e-6f);
  }
  // the previous step was fully computed: its observable (ref2) is the new reference
  [[maybe_unused]] const bool refresh = MODE == LN_SIGNAL && a.sig_ref_w && a.st && a.st->t > 0 && a.st->t_last == a.st->t - 1;
  const float* sh;
  const float* sc;
  if (row < a.split) {
    sh = a.shift_a;
    sc = a.scale_a;
  } else if (a.split2 <= 0 || row < a.split2) {
    sh = a.shift_b;
    sc = a.scale_b;
  } else if (row < a.split3) {
    sh = a.shift_c;
    sc = a.scale_c;
  } else {
    sh = a.shift_d;
    sc = a.scale_d;
  }
  if (sh) sh += (long)t * a.mod_step;
  if (sc) sc += (long)t * a.mod_step;
  [[maybe_unused]] float sig_num = 0.f, sig_den = 0.f, sig_num2 = 0.f, sig_den2 = 0.f;
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int c = threadIdx.x + i * TH;
    if (c < nv) {
      float y[4] = {(v[i].x - mean) * rstd, (v[i].y - mean) * rstd, (v[i].z - mean) * rstd,
                    (v[i].w - mean) * rstd};
      if (sc) {
        const float4 s4 = reinterpret_cast<const float4*>(sc)[c];
        y[0] *= 1.f + s4.x;
        y[1] *= 1.f + s4.y;
        y[2] *= 1.f + s4.z;
        y[3] *= 1.f + s4.w;
      }
      if (sh) {
        const float4 h4 = reinterpret_cast<const float4*>(sh)[c];
        y[0] += h4.x;
        y[1] += h4.y;
        y[2] += h4.z;
        y[3] += h4.w;
      }
      const long off = (long)row * a.ldy + 4 * c;
      if constexpr (MODE == LN_SIGNAL) {
        // both references are read before y is stored: sig_ref2 may be the y buffer
        // itself (the previous step's observable, replaced by this step's)
        float r[4], r2[4], yy[4];
        load4(a.sig_ref2, off, a.y_bf16, r2);
        if (refresh) {
          copy4(a.sig_ref_w, a.sig_ref2, off, a.y_bf16);
#pragma unroll
          for (int j = 0; j < 4; ++j) r[j] = r2[j];
        } else {
          load4(a.sig_ref, off, a.y_bf16, r);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          yy[j] = a.y_bf16 ? bf16_round(y[j]) : y[j];
          sig_num += fabsf(yy[j] - r[j]);
          sig_den += fabsf(r[j]);
          sig_num2 += fabsf(yy[j] - r2[j]);
          sig_den2 += fabsf(r2[j]);
        }
      }
      if (a.y_bf16) {
        uint2 u;
        u.x = pack_bf16x2(y[0], y[1]);
        u.y = pack_bf16x2(y[2], y[3]);
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.y) + off) = u;
      } else {
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(a.y) + off) =
            make_float4(y[0], y[1], y[2], y[3]);
      }
    }
  }
  if constexpr (MODE == LN_SIGNAL) {
    __shared__ float4 red4[TH / 32];
    const float4 t4 = block_sum4_fresh<TH>(make_float4(sig_num, sig_den, sig_num2, sig_den2), red4);
    if (threadIdx.x == 0) reinterpret_cast<float4*>(a.sig_partial)[row] = t4;
  }
}

int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// Launch of one row per CTA.  The signal pass reads two reference tensors last touched a step
// earlier (in HBM): each CTA prefetches into L2 the rows a CTA one wave later will read
// (distance = the CTAs resident on the GPU; bulk copies need 16-byte aligned rows).  The
// stack's LN-mods read rows the producing GEMM has just written (mostly still in L2):
// measured slower with the prefetch, so they take none.
template <int TH, int VPT, int MINB, int MODE>
static cudaError_t launch_ln(LnArgs a, cudaStream_t s) {
  const bool aligned = ((a.ldx * 4) % 16 == 0) && ((a.cols * 4) % 16 == 0) &&
                       (a.ldy * (a.y_bf16 ? 2 : 4)) % 16 == 0;
  a.prefetch_rows = (MODE == LN_SIGNAL && aligned) ? sm_count() * MINB : 0;
  return launch_kernel(ln_mod_kernel<TH, VPT, MINB, MODE>, a.rows, TH, 0, s, a);
}

cudaError_t ln_mod(const LnArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  if (a.cols % 4 != 0 || a.cols > LN_MAX_COLS) return cudaErrorInvalidValue;
  auto launch = [&](auto mode) {
    constexpr int M = decltype(mode)::value;
    if (a.cols > 5120) return launch_ln<256, 6, 4, M>(a, s);
    if (a.cols > 3072) return launch_ln<256, 5, 5, M>(a, s);
    if constexpr (M == LN_PLAIN)
      return launch_ln<128, 6, 10, M>(a, s);
    else
      return launch_ln<256, 3, M == LN_SIGNAL ? 7 : 6, M>(a, s);
  };
  const cudaError_t r = a.sig_on ? launch(std::integral_constant<int, LN_SIGNAL>{})
                                 : (a.cache_in ? launch(std::integral_constant<int, LN_CACHE>{})
                                               : launch(std::integral_constant<int, LN_PLAIN>{}));
  const cudaError_t last = cudaGetLastError();  // also taken off the thread, or the next check reports it again
  return r == cudaSuccess ? last : r;
}

// ---------------------------------------------------------------------------
// standalone relative L1
// ---------------------------------------------------------------------------
// This lane's share of sum|a - b| and sum|b| of one row: lanes of `width` take 16-byte
// groups in turn (VEC: rows of whole 16-byte groups), or single elements.
template <typename T, bool VEC>
BAG_DEV float2 rel_l1_row(const T* __restrict__ a, const T* __restrict__ b, long cols, int lane, int width) {
  float n[2] = {0.f, 0.f}, d[2] = {0.f, 0.f};  // two chains each
  auto add = [&](int k, float x, float y) {
    n[k] += fabsf(x - y);
    d[k] += fabsf(y);
  };
  if constexpr (VEC) {
    constexpr int E = 16 / sizeof(T);
    const uint4* a4 = reinterpret_cast<const uint4*>(a);
    const uint4* b4 = reinterpret_cast<const uint4*>(b);
#pragma unroll 4
    for (long c = lane; c < cols / E; c += width) {
      const uint4 x = __ldg(a4 + c), y = __ldg(b4 + c);
      const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if constexpr (sizeof(T) == 2) {  // bf16: the upper half of an fp32
          add(0, __uint_as_float(xs[j] << 16), __uint_as_float(ys[j] << 16));
          add(1, __uint_as_float(xs[j] & 0xffff0000u), __uint_as_float(ys[j] & 0xffff0000u));
        } else {
          add(j & 1, __uint_as_float(xs[j]), __uint_as_float(ys[j]));
        }
      }
    }
  } else {
#pragma unroll 4
    for (long c = lane; c < cols; c += width) {
      if constexpr (sizeof(T) == 2)
        add(0, __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(a)[c]),
            __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(b)[c]));
      else
        add(0, a[c], b[c]);
    }
  }
  return make_float2(n[0] + n[1], d[0] + d[1]);
}

BAG_DEV float2 warp_sum2(float2 v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
  }
  return v;
}

// Row partials go to the caller's scratch, which is aligned for floats only.
BAG_DEV void rel_l1_partial(float* partial, long row, float2 s) {
  partial[2 * row] = s.x;
  partial[2 * row + 1] = s.y;
}

BAG_DEV void rel_l1_store(float* out, float2 s) {
  out[0] = __fdiv_rn(s.x, s.y);
  out[1] = s.x;
  out[2] = s.y;
}

// Row partials, WPR warps of a 128-thread CTA per row.  Bound: HBM, 2 * rows * cols
// elements.  One warp per row needs no barrier and keeps eight 16-byte loads a lane in
// flight; with few rows four warps share one, so that the SMs are filled.
// Measured with the sum over rows (in a graph, warm L2), against a CTA a row with 2-byte loads
// and one warp summing the rows: 4096 x 3072 bf16 17.1 -> 6.3 us, 32,760 x 5120 bf16 238 -> 99
// us (6.76 TB/s), 1024 x 1024 fp32 5.5 -> 3.6 us.
constexpr int RL_THREADS = 128;
template <typename T, bool VEC, int WPR>
__global__ void __launch_bounds__(RL_THREADS) rel_l1_kernel(const T* a, const T* b, long rows, long cols,
                                                            float* partial) {
  grid_dep_sync();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if constexpr (WPR == 1) {
    const long row = (long)blockIdx.x * (RL_THREADS / 32) + warp;
    if (row >= rows) return;
    const float2 s = warp_sum2(rel_l1_row<T, VEC>(a + row * cols, b + row * cols, cols, lane, 32));
    if (lane == 0) rel_l1_partial(partial, row, s);
  } else {
    __shared__ float2 red[RL_THREADS / 32];
    const long row = blockIdx.x;
    const float2 s =
        warp_sum2(rel_l1_row<T, VEC>(a + row * cols, b + row * cols, cols, (int)threadIdx.x, RL_THREADS));
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      float2 t = red[0];
#pragma unroll
      for (int w = 1; w < RL_THREADS / 32; ++w) {
        t.x += red[w].x;
        t.y += red[w].y;
      }
      rel_l1_partial(partial, row, t);
    }
  }
}

// out[0] = sum(num) / sum(den), out[1] = sum(num), out[2] = sum(den) over the per-row
// partials, summed in a fixed order by one CTA.
constexpr int RF_THREADS = 1024;
__global__ void __launch_bounds__(RF_THREADS) rel_l1_finalize_kernel(const float* partial, long rows, float* out) {
  grid_dep_sync();
  __shared__ float2 red[RF_THREADS / 32];
  float2 s = make_float2(0.f, 0.f);
#pragma unroll 4
  for (long r = threadIdx.x; r < rows; r += RF_THREADS) {
    s.x += partial[2 * r];
    s.y += partial[2 * r + 1];
  }
  s = warp_sum2(s);
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x >= 32) return;
  s = warp_sum2(red[threadIdx.x]);
  if (threadIdx.x == 0) rel_l1_store(out, s);
}

// Small inputs in one launch: a cluster of eight CTAs, a warp per row, the CTAs' sums
// exchanged through distributed shared memory and added in a fixed tree (one after another the
// relative error over 80 seeds was 60e-9 at 256 x 256 fp32, 46e-9 before; 48e-9 now).  It saves a call one
// of its two launches, which are most of a small call's time; the rule is for the time of calls
// in a loop.  One launch against two, us a call (and on the device, in a graph): 1 x 1024 fp32
// 4.1 (2.8) against 5.1 (2.8), 64 x 512 fp32 4.1 (2.8) against 5.2 (2.9), 128 x 512 bf16 4.1 (2.8)
// against 5.0 (2.8), 256 x 256 fp32 4.9 (2.9) against 5.2 (2.9).  Past each limit it loses: more
// rows than warps, 512 x 128 fp32 6.0 against 5.2; wider rows, which one warp walks alone, 16 x
// 2048 fp32 6.1 against 5.1, 1 x 65,536 fp32 49 against 25, unaligned 64 x 255 6.1 against 5.0;
// more bytes, 256 x 512 fp32 5.1 (3.3) against 5.1 (2.9).
constexpr int RC_CTAS = 8, RC_THREADS = 1024;
constexpr int RC_ROWS = RC_CTAS * RC_THREADS / 32;
constexpr long RC_BYTES = 512l << 10;  // of both inputs
// Widest row: four loads a lane (16-byte groups, or elements).
template <typename T, bool VEC>
constexpr long rc_cols() {
  return 4 * 32 * (VEC ? 16 / (long)sizeof(T) : 1);
}
template <typename T, bool VEC>
__global__ void __cluster_dims__(RC_CTAS, 1, 1) __launch_bounds__(RC_THREADS)
    rel_l1_cluster_kernel(const T* a, const T* b, long rows, long cols, float* partial, float* out) {
  // rank 0's shared memory may be written once rank 0 is known to run: arrive here, wait before
  // the store, so that the rows in between hide the barrier
  cluster_arrive();
  grid_dep_sync();
  __shared__ float2 red[RC_THREADS / 32];
  __shared__ __align__(8) float2 total[RC_CTAS];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t rank = cluster_ctarank();
  float2 s = make_float2(0.f, 0.f);
  const long row = warp * RC_CTAS + (int)rank;
  if (row < rows) {
    s = warp_sum2(rel_l1_row<T, VEC>(a + row * cols, b + row * cols, cols, lane, 32));
    if (lane == 0) rel_l1_partial(partial, row, s);
  }
  if (lane == 0) red[warp] = s;
  __syncthreads();
  cluster_wait();
  if (warp == 0) {
    s = warp_sum2(lane < RC_THREADS / 32 ? red[lane] : make_float2(0.f, 0.f));
    if (lane == 0)
      st_cluster2(mapa_shared(smem_u32(total + rank), 0), s.x, s.y);
  }
  __syncwarp();
  cluster_sync_all();  // the sums have arrived; no access to another CTA follows
  if (rank == 0 && warp == 0) {
    s = warp_sum2(lane < RC_CTAS ? total[lane] : make_float2(0.f, 0.f));
    if (lane == 0) rel_l1_store(out, s);
  }
}

cudaError_t rel_l1(const void* a, const void* b, int bf16, long rows, long cols, float* scratch, float* out, int pdl,
                   cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  const int es = bf16 ? 2 : 4;
  const bool vec =
      cols * es % 16 == 0 && ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
  auto run = [&](auto t, auto v) -> cudaError_t {
    using T = decltype(t);
    constexpr bool V = decltype(v)::value;
    const T* ta = static_cast<const T*>(a);
    const T* tb = static_cast<const T*>(b);
    if (rows <= RC_ROWS && cols <= rc_cols<T, V>() && rows * cols * 2 * es <= RC_BYTES)
      return launch_kernel(rel_l1_cluster_kernel<T, V>, RC_CTAS, RC_THREADS, 0, s, ta, tb, rows, cols, scratch, out);
    // from eight rows an SM on, a warp a row
    cudaError_t r;
    if (rows >= (long)sm_count() * 8)
      r = launch_kernel(rel_l1_kernel<T, V, 1>, (unsigned)((rows + 3) / 4), RL_THREADS, 0, s, ta, tb, rows, cols,
                        scratch);
    else
      r = launch_kernel(rel_l1_kernel<T, V, 4>, (unsigned)rows, RL_THREADS, 0, s, ta, tb, rows, cols, scratch);
    if (r != cudaSuccess) return r;
    g_pdl = pdl != 0;  // the second kernel is resident and waiting when the first completes
    r = launch_kernel(rel_l1_finalize_kernel, 1, RF_THREADS, 0, s, scratch, rows, out);
    g_pdl = false;
    return r;
  };
  cudaError_t r;
  if (bf16)
    r = vec ? run(uint16_t{}, std::true_type{}) : run(uint16_t{}, std::false_type{});
  else
    r = vec ? run(float{}, std::true_type{}) : run(float{}, std::false_type{});
  const cudaError_t last = cudaGetLastError();
  return r == cudaSuccess ? last : r;
}

// ---------------------------------------------------------------------------
// gate + pacing (one CTA)
// ---------------------------------------------------------------------------
// Gate parameters: every layer's W [out][in] (row-major) then b, in evaluation order,
// from offset 0; z-score mean at kGateMu, standard deviation at kGateSd (3 or 6 used).
//   kind 0 (3 inputs): 3 -> 16 -> 1
//   kind 1 (6 inputs): 6 -> 8 -> 8 -> 32 -> 1
//   kind 2 (6 inputs): [budget 3 -> 8 -> 8 | trajectory 3 -> 8 -> 8] -> 16 -> 32 -> 1
// Every hidden layer is followed by ReLU.  Each output of a dense layer is summed by one
// lane in a fixed order (bias first, then inputs in index order, every product and sum
// rounded on its own) so the logit is reproducible bit for bit by any IEEE fp32
// evaluation in the same order; the outputs of a layer are independent of one another
// and run on the lanes of one warp.
//
// The kernel is pure latency: it sits between the signal pass and the decision, and
// nothing overlaps it.  128 threads (512 from 1024 rows on) sum the row partials, and the
// parameters are in shared memory before the predecessor finishes.  One warp that walked
// the rows alone, its first lane reading the parameters from global memory one dependent
// sum after another, took 10.6 us (3-input gate, 4096 rows), 15.3 us (WAN6, 390 rows),
// 73.7 us (WAN6, 32,760 rows) per launch in a chain; this takes 3.8, 3.3 and 12.9 us.
constexpr int GATE_THREADS = 512;

// Output `lane` (< out) of a layer at p with inputs x (shared memory); its W and b in p.
BAG_DEV float dense_lane(const float* p, int out, int in, const float* x, int lane, bool relu) {
  float h = p[out * in + lane];
  for (int i = 0; i < in; ++i) h = __fadd_rn(h, __fmul_rn(p[lane * in + i], x[i]));
  return relu && !(h > 0.f) ? 0.f : h;
}

__global__ void __launch_bounds__(GATE_THREADS)
    gate_kernel(DevState* st, const float* partial, int rows, const float* gp, int kind, float thr, int T,
                int B, int policy, const uint8_t* pmask, float delta, float* log,
                cudaGraphConditionalHandle handle, int use_cond) {
  __shared__ float gs[kGateFloats];
  __shared__ float4 red[GATE_THREADS / 32];
  __shared__ float xs[6], la[32], lb[32];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  // the gate's parameters are written by no kernel of a step: read ahead of the wait
  const int np = kind == 0 ? 81 : (kind == 1 ? 449 : 785);
  for (int i = threadIdx.x; i < np; i += blockDim.x) gs[i] = gp[i];
  if (threadIdx.x < kGateFloats - kGateMu) gs[kGateMu + threadIdx.x] = gp[kGateMu + threadIdx.x];
  grid_dep_sync();
  const int t = st->t, c = st->c, t_last = st->t_last;
  // sums over rows: thread k takes rows k, k + blockDim, ...; then a fixed tree of lanes and warps
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (t > 0) {
    const float4* p4 = reinterpret_cast<const float4*>(partial);
#pragma unroll 4
    for (int r = threadIdx.x; r < rows; r += blockDim.x) {
      const float4 v = p4[r];
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    }
  }
  auto warp_sum = [](float4 v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
      v.z += __shfl_xor_sync(0xffffffffu, v.z, off);
      v.w += __shfl_xor_sync(0xffffffffu, v.w, off);
    }
    return v;
  };
  s = warp_sum(s);
  if (lane == 0) red[warp] = s;
  __syncthreads();
  if (warp != 0) return;
  s = warp_sum(lane < blockDim.x / 32 ? red[lane] : make_float4(0.f, 0.f, 0.f, 0.f));
  const float num = s.x, den = s.y, num2 = s.z, den2 = s.w;
  float* L = log + (long)t * kLogFloats;
  int m = 1, gbit = 1;
  float z = 0.f, f0 = 0.f, f1 = 0.f, drift = 0.f, step = 0.f;
  float sb[3] = {0.f, 0.f, 0.f};
  if (t > 0) {  // uniform over the warp
    f0 = __fdiv_rn((float)(B - c), (float)B);
    f1 = __fdiv_rn((float)(T - t), (float)T);
    drift = __fdiv_rn(num, den);
    step = __fdiv_rn(num2, den2);
    sb[0] = __fdiv_rn((float)B, (float)T);
    sb[1] = f0;
    sb[2] = __fdiv_rn((float)(B - c), (float)(T - t));
    const int nin = kind == 0 ? 3 : 6;
    if (lane < nin) {
      float f;
      if (kind == 0)
        f = lane == 0 ? f0 : (lane == 1 ? f1 : drift);
      else
        f = lane < 3 ? sb[lane] : (lane == 3 ? (float)(t - t_last) : (lane == 4 ? drift : step));
      xs[lane] = __fdiv_rn(__fsub_rn(f, gs[kGateMu + lane]), gs[kGateSd + lane]);
    }
    __syncwarp();
    const float* last;  // the output layer's parameters and inputs
    const float* hin;
    int nh;
    if (kind == 0) {
      if (lane < 16) la[lane] = dense_lane(gs, 16, 3, xs, lane, true);
      last = gs + 16 * 3 + 16;
      hin = la;
      nh = 16;
    } else if (kind == 1) {
      if (lane < 8) la[lane] = dense_lane(gs, 8, 6, xs, lane, true);
      __syncwarp();
      if (lane < 8) lb[lane] = dense_lane(gs + 56, 8, 8, la, lane, true);
      __syncwarp();
      la[lane] = dense_lane(gs + 56 + 72, 32, 8, lb, lane, true);
      last = gs + 56 + 72 + 288;
      hin = la;
      nh = 32;
    } else {
      // the two branches side by side: lanes 0-7 budget, 8-15 trajectory (each branch's
      // two layers are 32 + 72 parameters)
      const int br = lane / 8;
      if (lane < 16) la[lane] = dense_lane(gs + br * 104, 8, 3, xs + 3 * br, lane % 8, true);
      __syncwarp();
      if (lane < 16) lb[lane] = dense_lane(gs + br * 104 + 32, 8, 8, la + 8 * br, lane % 8, true);
      __syncwarp();
      la[lane] = dense_lane(gs + 208, 32, 16, lb, lane, true);
      last = gs + 208 + 544;
      hin = la;
      nh = 32;
    }
    __syncwarp();
    z = dense_lane(last, 1, nh, hin, 0, false);  // every lane, the same sum
    gbit = z > thr ? 1 : 0;
    if (policy == 0) {  // Algorithm 2
      m = gbit;
      if (B - c >= T - t) m = 1;  // spend the remainder
      if (B - c == 0) m = 0;      // budget exhausted
    } else if (policy == 1) {     // uncached sampling
      m = 1;
    } else if (policy == 4) {     // online threshold on the drift, no budget
      m = drift > delta ? 1 : 0;
    } else {                      // caller-given or static evenly spaced mask
      m = pmask[t] ? 1 : 0;
    }
  }
  if (lane != 0) return;
  if (use_cond) cudaGraphSetConditional(handle, (unsigned)m);
  st->flag = m;
  if (m) {
    st->c = c + 1;
    st->t_last = t;
  }
  float4* L4 = reinterpret_cast<float4*>(L);  // kLogFloats is a multiple of four
  L4[0] = make_float4(f0, f1, drift, z);
  L4[1] = make_float4((float)gbit, (float)m, (float)c, t > 0 ? (float)(t - t_last) : 0.f);
  L4[2] = make_float4(sb[0], sb[1], sb[2], num);
  L4[3] = make_float4(den, step, num2, den2);
}

cudaError_t gate_step(DevState* st, const float* sig_partial, int sig_rows, const float* gate_params,
                      int gate_kind, float thr, int T, int B, int policy, const uint8_t* policy_mask,
                      float delta, float* log, unsigned long long cond_handle, int use_cond,
                      cudaStream_t s) {
  launch_kernel(gate_kernel, 1, sig_rows < 1024 ? 128 : GATE_THREADS, 0, s, st, sig_partial, sig_rows, gate_params, gate_kind, thr, T, B,
                policy, policy_mask, delta, log, (cudaGraphConditionalHandle)cond_handle, use_cond);
  return cudaGetLastError();
}

// out = a + b
__global__ void residual_add_kernel(float4* out, const float4* a, const float4* b, long n4) {
  grid_dep_sync();
  const long stride = (long)gridDim.x * blockDim.x;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
    const float4 x = a[i], y = b[i];
    out[i] = make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w);
  }
}

static int grid_for(long n, int threads) {
  long b = (n + threads - 1) / threads;
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 148;
  }
  long cap = (long)sms * 8;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (int)b;
}

cudaError_t residual_add(float* out, const float* a, const float* b, long n, cudaStream_t s) {
  if (n % 4 != 0) return cudaErrorInvalidValue;
  launch_kernel(residual_add_kernel, grid_for(n / 4, 256), 256, 0, s, reinterpret_cast<float4*>(out),
                reinterpret_cast<const float4*>(a), reinterpret_cast<const float4*>(b), n / 4);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------
// Row-contiguous copies, so each block of the stream is one run of float4 groups (rows are
// multiples of 64 elements).  One launch for all blocks: on small backbones a launch is what
// such a copy costs.
__global__ void stream_init_kernel(const DevState* st, int flag_want, float4* h, const void* txt0,
                                   const void* txt1, int txt_bf16, const float4* h_in, int nb, long nx4, long ni4) {
  grid_dep_sync();
  if (epi_skip(st, flag_want)) return;
  const long n_txt = nb * nx4, n = n_txt + nb * ni4;
  const long stride = (long)gridDim.x * blockDim.x;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    if (i < n_txt) {
      float r[4];
      load4(i < nx4 ? txt0 : txt1, 4 * (i < nx4 ? i : i - nx4), txt_bf16, r);
      h[i] = make_float4(r[0], r[1], r[2], r[3]);
    } else {
      const long k = i - n_txt;
      h[i] = h_in[k < ni4 ? k : k - ni4];
    }
  }
}

cudaError_t stream_init(const DevState* st, int flag_want, float* h, const void* txt0, const void* txt1,
                        int txt_bf16, const float* h_in, int nb, int nx, int ni, int d, cudaStream_t s) {
  if (d % 4 != 0) return cudaErrorInvalidValue;
  const long nx4 = (long)nx * d / 4, ni4 = (long)ni * d / 4;
  launch_kernel(stream_init_kernel, grid_for(nb * (nx4 + ni4), 256), 256, 0, s, st, flag_want,
                reinterpret_cast<float4*>(h), txt0, txt1, txt_bf16, reinterpret_cast<const float4*>(h_in), nb, nx4,
                ni4);
  return cudaGetLastError();
}

// The bounded-wait failure path on purpose: the barrier expects one arrival that never
// comes, mbar_wait gives up after kWaitLimitNs and the error is recorded like any
// kernel's timed-out wait.
__global__ void wait_timeout_kernel(DevState* st) {
  grid_dep_sync();
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x != 0) return;
  abort_flag = 0;
  mbar_init(&bar, 1);
  fence_mbar_init();
  if (!mbar_wait(&bar, 0, &abort_flag)) atomicOr(&st->err, 2);
}

cudaError_t wait_timeout_probe(DevState* st, cudaStream_t s) {
  launch_kernel(wait_timeout_kernel, 1, 32, 0, s, st);
  return cudaGetLastError();
}

// Sinusoidal features of 1000 * sigma_t, sigma_t = 1 - t/T, for every step t < T:
// [cos(1000 sigma_t f_j), sin(1000 sigma_t f_j)], f_j = exp(-ln(10000) j / (dim/2)).
__global__ void sinusoid_kernel(void* out, int out_bf16, const double* sigma, int T, int dim) {
  grid_dep_sync();
  const int t = blockIdx.x, j = threadIdx.x;
  const int half = dim / 2;
  if (t >= T || j >= dim) return;
  const double sig = sigma[t];
  const int jj = j < half ? j : j - half;
  const double f = exp(-log(10000.0) * (double)jj / (double)half);
  const double arg = 1000.0 * sig * f;
  const float v = (float)(j < half ? cos(arg) : sin(arg));
  if (out_bf16)
    reinterpret_cast<__nv_bfloat16*>(out)[(long)t * dim + j] = __float2bfloat16_rn(v);
  else
    reinterpret_cast<float*>(out)[(long)t * dim + j] = v;
}

cudaError_t sinusoid_all(void* out, int out_bf16, const double* sigma, int T, int dim, cudaStream_t s) {
  launch_kernel(sinusoid_kernel, T, dim, 0, s, out, out_bf16, sigma, T, dim);
  return cudaGetLastError();
}

// Wan: per-block modulation = shared projection of the time embedding + block table.
// shared8d: [T][8d] (6d shared block modulation, then 2d final-layer modulation);
// mod_all:  [T][nblocks*6d + 2d].
__global__ void expand_wan_kernel(float* mod_all, const float* shared8d, const float* tables,
                                  int T, int nblocks, int d) {
  grid_dep_sync();
  const long per = (long)nblocks * 6 * d + 2 * d;
  const long n = (long)T * per;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const long t = i / per, j = i % per;
    const float* sh = shared8d + t * 8 * d;
    if (j < (long)nblocks * 6 * d) {
      const long b = j / (6 * d), c = j % (6 * d);
      mod_all[i] = sh[c] + tables[b * 6 * d + c];
    } else {
      mod_all[i] = sh[6 * d + (j - (long)nblocks * 6 * d)];
    }
  }
}

cudaError_t expand_wan_mod(float* mod_all, const float* shared8d, const float* tables, int T,
                           int nblocks, int d, cudaStream_t s) {
  launch_kernel(expand_wan_kernel, grid_for((long)T * nblocks * 6 * d, 256), 256, 0, s, mod_all,
                shared8d, tables, T, nblocks, d);
  return cudaGetLastError();
}

__global__ void split_bf16_kernel(__nv_bfloat16* dst, const float* src, long rows, long cols) {
  grid_dep_sync();
  const long n = rows * cols;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const long r = i / cols, c = i % cols;
    const float x = src[i];
    const __nv_bfloat16 hi = __float2bfloat16_rn(x);
    dst[r * 2 * cols + c] = hi;
    dst[r * 2 * cols + cols + c] = __float2bfloat16_rn(x - __bfloat162float(hi));
  }
}

cudaError_t split_bf16(__nv_bfloat16* dst, const float* src, long rows, long cols, cudaStream_t s) {
  if (rows * cols <= 0) return cudaSuccess;
  launch_kernel(split_bf16_kernel, grid_for(rows * cols, 256), 256, 0, s, dst, src, rows, cols);
  return cudaGetLastError();
}

__global__ void to_bf16_kernel(__nv_bfloat16* dst, const float* src, long n) {
  grid_dep_sync();
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    dst[i] = __float2bfloat16_rn(src[i]);
}

cudaError_t to_bf16(__nv_bfloat16* dst, const float* src, long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  launch_kernel(to_bf16_kernel, grid_for(n, 256), 256, 0, s, dst, src, n);
  return cudaGetLastError();
}

// Seeded fill: SplitMix64 stream (state s + (i+1) * golden, finalised by mix), the four
// 16-bit chunks summed and centred (Irwin-Hall(4)), scaled by c32 in fp32, plus an
// fp32 offset when it is nonzero.
BAG_DEV uint64_t sm64_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void fill_synth_kernel(void* dst, long n, uint64_t start, float offset, float c32, int bf16) {
  grid_dep_sync();
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const uint64_t u = sm64_mix(start + (uint64_t)(i + 1) * 0x9E3779B97F4A7C15ull);
    const long q = (long)(u & 0xFFFF) + (long)((u >> 16) & 0xFFFF) + (long)((u >> 32) & 0xFFFF) +
                   (long)(u >> 48) - 131070;
    float v = __fmul_rn((float)q, c32);
    if (offset != 0.f) v = __fadd_rn(offset, v);
    if (bf16)
      reinterpret_cast<__nv_bfloat16*>(dst)[i] = __float2bfloat16_rn(v);
    else
      reinterpret_cast<float*>(dst)[i] = v;
  }
}

cudaError_t fill_synth(void* dst, long n, uint64_t start, float offset, float c32, int bf16,
                       cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  launch_kernel(fill_synth_kernel, grid_for(n, 256), 256, 0, s, dst, n, start, offset, c32, bf16);
  return cudaGetLastError();
}

}  // namespace bag
