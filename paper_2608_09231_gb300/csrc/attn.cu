// Joint attention softmax(q k^T / sqrt(dh)) v per head, flash-style (online softmax,
// O(N) memory).  This file holds the CUDA-core kernel used for the fp32
// configuration and for shapes the tensor-core kernel does not tile; the tcgen05
// kernel lives in attn_tc.cu.
#include <cmath>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"

namespace bag {

template <typename T>
BAG_DEV float ldv(const void* p, long i) {
  if constexpr (sizeof(T) == 2)
    return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[i]);
  else
    return reinterpret_cast<const float*>(p)[i];
}

// N consecutive elements (2 or 4).  VEC: one load (fp32 rows of the contexts are 16-byte
// aligned; bf16 rows 8-byte); else one each.  bf16 with one load per element, against one per
// four: 1024 tokens x 8 heads of 64 330 -> 145 us, 2048 x 8 of 128 2272 -> 871 (keys and values
// staged in shared memory for sixteen queries: 203 and 1887); transposed V 525 -> 195 (313).
template <typename T, bool VEC, int N>
BAG_DEV void ldvn(const void* p, long i, float* v) {
  if constexpr (VEC && sizeof(T) == 2) {
    uint32_t w[N / 2];
    if constexpr (N == 4) {
      const uint2 u = *reinterpret_cast<const uint2*>(reinterpret_cast<const T*>(p) + i);
      w[0] = u.x;
      w[1] = u.y;
    } else {
      w[0] = *reinterpret_cast<const uint32_t*>(reinterpret_cast<const T*>(p) + i);
    }
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      v[2 * k] = __uint_as_float(w[k] << 16);
      v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
  } else if constexpr (VEC && N == 4) {
    const float4 f = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p) + i);
    v[0] = f.x;
    v[1] = f.y;
    v[2] = f.z;
    v[3] = f.w;
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = ldv<T>(p, i + k);
  }
}

// CTA = eight queries of one head; its warps take the key tiles (32 keys) in turn, each with
// its own running maximum, sum and output for all eight queries, merged in warp order at the
// end.  Scores: lane = key, which reads its own K row four elements at a time
// against the queries broadcast from shared memory (8 x 4 products per K load); the
// weights pass through shared memory so that the output has lane = head dimensions and
// reads V rows coalesced.  Bound: latency (the fp32 backbones have a few hundred tokens);
// few queries per CTA and the keys split over warps keep every SM busy with a short chain.
// Measured against sixteen queries per CTA whose four warps walked all keys one barrier
// after another (profiled launches, heads of 64): 288 tokens x 4 heads 41 us, 17.9 with eight
// warps, which leave the ninth tile for a second round, 13.7 with twelve; 512 x 4 69 us, 26 and
// 36; 1024 x 16 366 us, 286 and 352.  Twelve warps win only where they take all tiles in one
// round and every CTA has an SM to itself: 384 x 2 (96 CTAs) 15.2 us against 18.6 with eight,
// but 320 x 4 (160 CTAs) 22.8 against 21.8, 288 x 6 23.8 against 21.9, and with two rounds in
// both 512 x 2 21.9 against 19.8.  Heads of 128 take eight (the outputs to merge take 4 KB a warp).
constexpr int SA_Q = 8, SA_KT = 32;

template <typename T, int DH, int SA_WARPS, bool VEC = true>
__global__ void __launch_bounds__(SA_WARPS * 32) attn_simt_kernel(const AttnArgs a) {
  grid_dep_sync();
  if (epi_skip(a.st, a.flag_want)) return;
  constexpr int R = DH / 32;  // head dimensions per lane: lane * R .. lane * R + R - 1
  __shared__ __align__(16) float Qs[SA_Q][DH];
  // a warp's weights of one key tile, and at the end its outputs, share its part of Os
  __shared__ __align__(16) float Os[SA_WARPS][SA_Q][DH];
  __shared__ float ms[SA_WARPS][SA_Q], ls[SA_WARPS][SA_Q];
  const int head = blockIdx.y, q0 = blockIdx.x * SA_Q;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  float(*Ps)[SA_KT] = reinterpret_cast<float(*)[SA_KT]>(Os[warp]);
  const float scale = rsqrtf((float)DH);
  for (int i = threadIdx.x; i < SA_Q * DH; i += blockDim.x) {
    const int r = i / DH, c = i % DH, q = q0 + r;
    Qs[r][c] = q < a.nq ? ldv<T>(a.q, (long)q * a.ldq + head * DH + c) * scale : 0.f;
  }
  __syncthreads();
  float m[SA_Q], l[SA_Q], o[SA_Q][R];  // l: this lane's keys only
#pragma unroll
  for (int i = 0; i < SA_Q; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) o[i][r] = 0.f;
  }
  for (int kb = warp * SA_KT; kb < a.nk; kb += SA_WARPS * SA_KT) {
    const bool valid = kb + lane < a.nk;
    const long krow = (long)(valid ? kb + lane : a.nk - 1) * a.ldk + head * DH;
    float s[SA_Q];
#pragma unroll
    for (int i = 0; i < SA_Q; ++i) s[i] = 0.f;
#pragma unroll 8
    for (int c = 0; c < DH; c += 4) {
      float k4[4];
      ldvn<T, VEC, 4>(a.k, krow + c, k4);
#pragma unroll
      for (int i = 0; i < SA_Q; ++i) {
        const float4 q4 = *reinterpret_cast<const float4*>(&Qs[i][c]);
        s[i] += q4.x * k4[0];
        s[i] += q4.y * k4[1];
        s[i] += q4.z * k4[2];
        s[i] += q4.w * k4[3];
      }
    }
    __syncwarp();  // every lane has read the previous tile's weights
#pragma unroll
    for (int i = 0; i < SA_Q; ++i) {
      const float si = valid ? s[i] : -INFINITY;
      float mx = si;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      const float mn = fmaxf(m[i], mx);
      // scores that all underflowed to -inf weigh nothing unless every warp's did
      const float base = mn == -INFINITY ? 0.f : mn;
      const float p = expf(si - base);  // 0 past the last key
      const float corr = expf(m[i] - base);
      Ps[i][lane] = p;
      l[i] = l[i] * corr + p;
#pragma unroll
      for (int r = 0; r < R; ++r) o[i][r] *= corr;
      m[i] = mn;
    }
    __syncwarp();
    const int nkt = min(SA_KT, a.nk - kb);
#pragma unroll 2
    for (int j = 0; j < nkt; j += 4) {
      float v[4][R];  // past the last key weight and value are zero (a zero weight times an infinity is not)
      if (a.v_mode == 0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool in = kb + j + u < a.nk;
          ldvn<T, VEC, R>(a.v, (long)min(kb + j + u, a.nk - 1) * a.ldv + head * DH + lane * R, v[u]);
#pragma unroll
          for (int r = 0; r < R; ++r) v[u][r] = in ? v[u][r] : 0.f;
        }
      } else {
        // four keys of a column: in bounds also at the end (vpad is a multiple of 8)
#pragma unroll
        for (int r = 0; r < R; ++r) {
          float x[4];
          ldvn<T, VEC, 4>(a.v, (long)(head * DH + lane * R + r) * a.vpad + kb + j, x);
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u][r] = kb + j + u < a.nk ? x[u] : 0.f;
        }
      }
#pragma unroll
      for (int i = 0; i < SA_Q; ++i) {
        const float4 p4 = *reinterpret_cast<const float4*>(&Ps[i][j]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          o[i][r] += p4.x * v[0][r];
          o[i][r] += p4.y * v[1][r];
          o[i][r] += p4.z * v[2][r];
          o[i][r] += p4.w * v[3][r];
        }
      }
    }
  }
  __syncwarp();  // every lane has read the last tile's weights
#pragma unroll
  for (int i = 0; i < SA_Q; ++i) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);
    if (lane == 0) {
      ms[warp][i] = m[i];
      ls[warp][i] = l[i];
    }
#pragma unroll
    for (int r = 0; r < R; ++r) Os[warp][i][lane * R + r] = o[i][r];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < SA_Q * DH; i += blockDim.x) {
    const int r = i / DH, c = i % DH, q = q0 + r;
    if (q >= a.nq) continue;
    float mx = ms[0][r];  // warp 0 always has a key tile
#pragma unroll
    for (int w = 1; w < SA_WARPS; ++w) mx = fmaxf(mx, ms[w][r]);
    float num = 0.f, den = 0.f;
#pragma unroll
    for (int w = 0; w < SA_WARPS; ++w) {
      const float f = expf(ms[w][r] - mx);  // 0 for a warp without keys
      num += f * Os[w][r][c];
      den += f * ls[w][r];
    }
    const float val = num / den;
    const long idx = (long)q * a.ldo + head * DH + c;
    void* ob = (a.o2 && q >= a.o_split) ? a.o2 : a.o;
    if (a.bf16)
      reinterpret_cast<__nv_bfloat16*>(ob)[idx] = __float2bfloat16_rn(val);
    else
      reinterpret_cast<float*>(ob)[idx] = val;
  }
}

cudaError_t attention_tc(const AttnArgs& a, int* err, cudaStream_t s);

cudaError_t attention(const AttnArgs& a, int* err, cudaStream_t s, int force_simt) {
  if (a.nq <= 0) return cudaSuccess;
  // bf16 attention runs on the tensor cores; a call the tensor-core kernel cannot take
  // (head_dim != 128, V not transposed, unaligned operands) is refused rather than sent
  // to the CUDA-core kernel, which serves fp32 backbones and explicit cross-checks only
  if (a.bf16 && !force_simt) {
    if (!attention_tc_supported(a)) return cudaErrorNotSupported;
    return attention_tc(a, err, s);
  }
  if (a.f16 || a.nbr > 1) return cudaErrorNotSupported;  // tensor-core kernel only
  dim3 grid((a.nq + SA_Q - 1) / SA_Q, a.heads);
  auto launch = [&](auto kernel, int warps) { launch_kernel(kernel, grid, warps * 32, 0, s, a); };
  const bool one_round = a.nk > 8 * SA_KT && a.nk <= 12 * SA_KT && (long)grid.x * grid.y <= sm_count();
  const bool vec = ((reinterpret_cast<uintptr_t>(a.k) | reinterpret_cast<uintptr_t>(a.v)) & 7) == 0 &&
                   a.ldk % 4 == 0 && (a.v_mode ? a.vpad : a.ldv) % 4 == 0;  // bf16 rows
  using B = __nv_bfloat16;
  if (a.dh == 64 && one_round)
    !a.bf16 ? launch(attn_simt_kernel<float, 64, 12>, 12)
            : (vec ? launch(attn_simt_kernel<B, 64, 12>, 12) : launch(attn_simt_kernel<B, 64, 12, false>, 12));
  else if (a.dh == 64)
    !a.bf16 ? launch(attn_simt_kernel<float, 64, 8>, 8)
            : (vec ? launch(attn_simt_kernel<B, 64, 8>, 8) : launch(attn_simt_kernel<B, 64, 8, false>, 8));
  else if (a.dh == 128)
    !a.bf16 ? launch(attn_simt_kernel<float, 128, 8>, 8)
            : (vec ? launch(attn_simt_kernel<B, 128, 8>, 8) : launch(attn_simt_kernel<B, 128, 8, false>, 8));
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

}  // namespace bag
