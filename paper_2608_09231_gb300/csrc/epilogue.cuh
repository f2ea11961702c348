// Fused GEMM epilogues: every projection of the DiT block finishes here, so that no
// separate elementwise pass re-reads its output.
//   QKV (+ RoPE on q and k, V written transposed per head for the attention kernel's
//   K-major B operand) and the GELU'd MLP half of a single-stream block's linear1,
//   gated residual h += g * y (out-projection, linear2, MLP down), plain/GELU/SiLU
//   stores, and the flow-matching Euler update x += (sigma_{t+1} - sigma_t) v.
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace bag {

BAG_DEV int epi_step(const Epi& e) { return e.st ? e.st->t : 0; }

// The first kernel of a step advances the step index (no kernel before it in the step
// reads it, and this kernel does not).
BAG_DEV void epi_bump(const Epi& e) {
  if (e.bump && blockIdx.x == 0 && threadIdx.x == 0) e.bump->t += 1;
}

// Early exit for kernels captured on one side of the full/reuse branch.
BAG_DEV bool epi_skip(const DevState* st, int flag_want) {
  return st != nullptr && flag_want >= 0 && st->flag != flag_want;
}

// type: kStoreF32, kStoreBF16 or kStoreF16
template <int NV>
BAG_DEV void store_vals(void* base, long idx, const float* v, int type) {
  if (type == kStoreF16) {
    __half* p = reinterpret_cast<__half*>(base) + idx;
    if constexpr (NV % 8 == 0) {
      if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
        for (int j = 0; j < NV; j += 8) {
          uint4 u;
          u.x = pack_f16x2(v[j], v[j + 1]);
          u.y = pack_f16x2(v[j + 2], v[j + 3]);
          u.z = pack_f16x2(v[j + 4], v[j + 5]);
          u.w = pack_f16x2(v[j + 6], v[j + 7]);
          *reinterpret_cast<uint4*>(p + j) = u;
        }
        return;
      }
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) p[j] = __float2half_rn(v[j]);
  } else if (type == kStoreBF16) {
    __nv_bfloat16* p = reinterpret_cast<__nv_bfloat16*>(base) + idx;
    if constexpr (NV % 8 == 0) {
      if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
        for (int j = 0; j < NV; j += 8) {
          uint4 u;
          u.x = pack_bf16x2(v[j], v[j + 1]);
          u.y = pack_bf16x2(v[j + 2], v[j + 3]);
          u.z = pack_bf16x2(v[j + 4], v[j + 5]);
          u.w = pack_bf16x2(v[j + 6], v[j + 7]);
          *reinterpret_cast<uint4*>(p + j) = u;
        }
        return;
      }
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) p[j] = __float2bfloat16_rn(v[j]);
  } else {
    float* p = reinterpret_cast<float*>(base) + idx;
    if constexpr (NV % 4 == 0) {
      if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
        for (int j = 0; j < NV; j += 4)
          *reinterpret_cast<float4*>(p + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        return;
      }
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) p[j] = v[j];
  }
}

// NV consecutive fp32 values from a 16-byte aligned address.
template <int NV>
BAG_DEV void ld_chunk(const float* p, float* v) {
#pragma unroll
  for (int j = 0; j < NV; j += 4) {
    const float4 f = *reinterpret_cast<const float4*>(p + j);
    v[j] = f.x;
    v[j + 1] = f.y;
    v[j + 2] = f.z;
    v[j + 3] = f.w;
  }
}

// Apply the epilogue to NV consecutive accumulators v[0..NV) of output row `row`,
// columns [col0, col0 + NV).  NV is even and col0 is a multiple of NV; the chunk never
// straddles a q/k/v/mlp boundary (those are multiples of 64 columns).
// Bias of the output columns col0 .. col0 + NV - 1 (16-byte loads when aligned).
template <int NV>
BAG_DEV void epi_add_bias(const Epi& e, int col0, float* v) {
  if (e.bias) {
    if (NV % 4 == 0 && (reinterpret_cast<uintptr_t>(e.bias + col0) & 15) == 0) {
      const float4* b4 = reinterpret_cast<const float4*>(e.bias + col0);
#pragma unroll
      for (int j = 0; j < NV; j += 4) {
        const float4 b = __ldg(b4 + j / 4);
        v[j] += b.x;
        v[j + 1] += b.y;
        v[j + 2] += b.z;
        v[j + 3] += b.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < NV; ++j) v[j] += __ldg(e.bias + col0 + j);
    }
  }
}

// EPI_QKV q / k columns: the rotation of joint-sequence row jr; cc is the column within the
// region.  (Per-head RMSNorm is applied in store_16_warp alone.)
template <int NV>
BAG_DEV void epi_rotate(const Epi& e, int jr, int cc, float* v) {
  if (e.rope) {
    const int e0 = cc % e.dh;
    const float2* cs = e.rope + (long)jr * (e.dh / 2) + e0 / 2;
    if constexpr (NV % 4 == 0) {
      // two (cos, sin) pairs per 16-byte load (the table row offset is a multiple of
      // NV / 2 pairs, so 16-byte aligned)
      const float4* cs4 = reinterpret_cast<const float4*>(cs);
#pragma unroll
      for (int p = 0; p < NV / 4; ++p) {
        const float4 r = __ldg(cs4 + p);
        const float x0 = v[4 * p], x1 = v[4 * p + 1], x2 = v[4 * p + 2], x3 = v[4 * p + 3];
        v[4 * p] = x0 * r.x - x1 * r.y;
        v[4 * p + 1] = x0 * r.y + x1 * r.x;
        v[4 * p + 2] = x2 * r.z - x3 * r.w;
        v[4 * p + 3] = x2 * r.w + x3 * r.z;
      }
    } else {
#pragma unroll
      for (int p = 0; p < NV / 2; ++p) {
        const float2 r = __ldg(cs + p);
        const float x0 = v[2 * p], x1 = v[2 * p + 1];
        v[2 * p] = x0 * r.x - x1 * r.y;
        v[2 * p + 1] = x0 * r.y + x1 * r.x;
      }
    }
  }
}

template <int NV>
BAG_DEV void epi_apply(const Epi& e, int t, int row, int col0, float* v) {
  if (row >= e.M || col0 >= e.N) return;
  epi_add_bias<NV>(e, col0, v);
  switch (e.kind) {
    case EPI_STORE:
      store_vals<NV>(e.out, (long)row * e.ldo + col0, v, e.out_bf16);
      break;
    case EPI_GELU:
      if (e.out_bf16) {
#pragma unroll
        for (int j = 0; j < NV; ++j) v[j] = gelu_tanh_fast(v[j]);
      } else {
#pragma unroll
        for (int j = 0; j < NV; ++j) v[j] = gelu_tanh(v[j]);
      }
      store_vals<NV>(e.out, (long)row * e.ldo + col0, v, e.out_bf16);
      break;
    case EPI_SILU:
#pragma unroll
      for (int j = 0; j < NV; ++j) v[j] = silu(v[j]);
      store_vals<NV>(e.out, (long)row * e.ldo + col0, v, e.out_bf16);
      break;
    case EPI_QKV: {
      const int lc = col0 + e.col_base;
      const int region = lc / e.d;
      if (region >= 3) {
#pragma unroll
        for (int j = 0; j < NV; ++j) v[j] = e.act_bf16 ? gelu_tanh_fast(v[j]) : gelu_tanh(v[j]);
        store_vals<NV>(e.mlp, (long)row * e.ldm + (lc - 3 * e.d), v, e.act_bf16);
        break;
      }
      const bool br1 = e.br_rows > 0 && row >= e.br_rows;       // unconditional branch
      const int jr = row - (br1 ? e.br_rows : 0) + e.row_off;  // joint-sequence row
      const long qr = jr + (br1 ? e.br_qk : 0);                // q / k / v buffer row
      const int cc = lc - region * e.d;
      if (region < 2) epi_rotate<NV>(e, jr, cc, v);
      if (region == 0) {
        store_vals<NV>(e.q, qr * e.ldqk + cc, v, e.qkv_type);
      } else if (region == 1) {
        store_vals<NV>(e.k, qr * e.ldqk + cc, v, e.qkv_type);
      } else {  // (transposed V goes through store_vt_warp)
        store_vals<NV>(e.v, qr * e.ldqk + cc, v, e.qkv_type);
      }
      break;
    }
    case EPI_GATED_RES: {
      const float* g = (e.br_rows > 0 && row >= e.br_rows ? e.gate_u : e.gate) + (long)t * e.gate_step + col0;
      float* r = e.resid + (long)row * e.ldr + col0;
      if (NV % 4 == 0 && ((reinterpret_cast<uintptr_t>(g) | reinterpret_cast<uintptr_t>(r)) & 15) == 0) {
#pragma unroll
        for (int j = 0; j < NV; j += 4) {
          const float4 g4 = __ldg(reinterpret_cast<const float4*>(g + j));
          float4 h = *reinterpret_cast<float4*>(r + j);
          h.x += g4.x * v[j];
          h.y += g4.y * v[j + 1];
          h.z += g4.z * v[j + 2];
          h.w += g4.w * v[j + 3];
          *reinterpret_cast<float4*>(r + j) = h;
        }
      } else {
#pragma unroll
        for (int j = 0; j < NV; ++j) r[j] += __ldg(g + j) * v[j];
      }
      break;
    }
    case EPI_RES_ADD: {
      float* r = e.resid + (long)row * e.ldr + col0;
#pragma unroll
      for (int j = 0; j < NV; ++j) r[j] += v[j];
      break;
    }
    case EPI_EULER: {
      // The sampler's buffers are 16-byte aligned with rows of 64 elements.  Every operand of
      // a chunk is read before anything is stored: loads and stores that alternate element by
      // element serialise one memory round trip each (a UniPC update of 390 x 64 elements
      // took 87 us that way with its product, 16 us now).
      constexpr int CH = NV % 8 == 0 ? 8 : 4;
      static_assert(NV % CH == 0, "whole float4 groups");
      const long idx0 = (long)row * e.ldx + col0;
      const float ds = e.dsig[t];
      float k[kUniCoefs];
      if (e.uni_coef) {
#pragma unroll
        for (int i = 0; i < kUniCoefs; ++i) k[i] = __ldg(e.uni_coef + (long)t * kUniCoefs + i);
      }
#pragma unroll
      for (int j0 = 0; j0 < NV; j0 += CH) {
        const long idx = idx0 + j0;
        float x[CH], nx[CH], vc[CH], w[CH];
        ld_chunk<CH>(e.x + idx, x);
#pragma unroll
        for (int j = 0; j < CH; ++j) w[j] = v[j0 + j];
        if (e.vcond) {  // classifier-free guidance: v_u + g (v_c - v_u)
          ld_chunk<CH>(e.vcond + idx, vc);
#pragma unroll
          for (int j = 0; j < CH; ++j) w[j] = w[j] + e.guidance * (vc[j] - w[j]);
        }
        if (e.uni_coef) {
          // UniPC: m_i = x_i - sigma_i v; corrected x_i^c (a combination of x_i, the previous
          // corrected sample and m_{i-1}, m_{i-2}, m_i); x_{i+1} from x_i^c, m_i, m_{i-1}.
          // Terms whose weight is zero are not read (uniform across the grid).
          float* mcur = ((t & 1) ? e.uni_m1 : e.uni_m0) + idx;         // holds m_{i-2}; receives m_i
          const float* mprev = ((t & 1) ? e.uni_m0 : e.uni_m1) + idx;  // m_{i-1}
          const bool use_last = k[UC_CLAST] != 0.f, use_m2 = k[UC_CM2] != 0.f;
          const bool use_m1 = k[UC_CM1] != 0.f || k[UC_DM1] != 0.f;
          float m[CH], xc[CH], xl[CH], m1[CH], m2[CH];
          if (use_last) ld_chunk<CH>(e.uni_xl + idx, xl);
          if (use_m1) ld_chunk<CH>(mprev, m1);
          if (use_m2) ld_chunk<CH>(mcur, m2);
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            m[j] = x[j] - k[UC_SIG] * w[j];
            xc[j] = k[UC_CX] * x[j] + k[UC_CMT] * m[j];
            if (!use_m1) m1[j] = 0.f;
            if (use_last) xc[j] += k[UC_CLAST] * xl[j];
            if (use_m1) xc[j] += k[UC_CM1] * m1[j];
            if (use_m2) xc[j] += k[UC_CM2] * m2[j];
            nx[j] = k[UC_DX] * xc[j] + k[UC_DM0] * m[j] + k[UC_DM1] * m1[j];
          }
          store_vals<CH>(e.uni_xl, idx, xc, kStoreF32);
          store_vals<CH>(mcur, 0, m, kStoreF32);
        } else {
#pragma unroll
          for (int j = 0; j < CH; ++j) nx[j] = x[j] + ds * w[j];
        }
        store_vals<CH>(e.x, idx, nx, kStoreF32);
        if (e.xb) {
          // next step's patch-embedding operand: bf16 hi | lo halves of the new latent
          float lo[CH];
#pragma unroll
          for (int j = 0; j < CH; ++j) lo[j] = nx[j] - bf16_round(nx[j]);
          const long hi = (long)row * 2 * e.ldx + col0 + j0;
          store_vals<CH>(e.xb, hi, nx, kStoreBF16);
          store_vals<CH>(e.xb, hi + e.ldx, lo, kStoreBF16);
        }
      }
      break;
    }
    case EPI_VEC: {
#pragma unroll
      for (int j = 0; j < NV; ++j) v[j] += (e.addend ? e.addend[col0 + j] : 0.f);
      store_vals<NV>(e.out, (long)row * e.ldo + col0, v, 0);
#pragma unroll
      for (int j = 0; j < NV; ++j) v[j] = silu(v[j]);
      store_vals<NV>(e.out2, (long)row * e.ldo2 + col0, v, e.out2_bf16);
      break;
    }
    default:
      break;
  }
}

}  // namespace bag
