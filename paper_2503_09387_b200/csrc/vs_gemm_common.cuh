// What the two kernels of the linear layers (vs_gemm_tcgen05.cu, vs_gemm_pair.cu) share: barriers, descriptors, tensor-memory
// loads, and the finishing of an output row -- bias, RoPE, norm scale, SwiGLU, residual, rounding and the stores.
#pragma once
#include "vs_common.cuh"
#include "vs_ptx.cuh"

namespace vs {
namespace gemm {

constexpr int kStageABytes = GEMM_BLOCK_M * GEMM_BLOCK_K * 2;   // 16 KiB
constexpr int kMaxDynSmem = 227 * 1024;

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void tcgen05_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tcgen05_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor, K-major operand, 128-byte swizzle: rows of 128 bytes,
// 8-row groups 1024 bytes apart (stride byte offset), descriptor version 1, layout 2.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);          // start address, 16-byte units
  d |= (uint64_t)1 << 16;                            // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024u >> 4) << 32;                 // stride byte offset
  d |= (uint64_t)1 << 46;                            // descriptor version (Blackwell)
  d |= (uint64_t)2 << 61;                            // SWIZZLE_128B
  return d;
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}

// One finishing thread's place in a 128-feature tile: four rotation pairs (features f1 .. f1 + 3 and f2 .. f2 + 3) of one head.
struct Place { int f1, f2, k0, hs; bool on, rotate; };
__device__ __forceinline__ Place place_of(const ProjectionOut& o, int E_out, int m0, int te) {
  Place pl;
  const int half = o.D >> 1, p0 = (te & 15) * 4, hl = p0 / half;      // first of 4 rotation pairs inside the tile, local head
  pl.k0 = p0 - hl * half;
  pl.f1 = hl * o.D + pl.k0; pl.f2 = pl.f1 + half;
  pl.hs = (m0 + pl.f1) / o.D;                                         // head slot: Q heads, then K heads, then V heads
  pl.on = m0 + pl.f2 + 3 < E_out;
  pl.rotate = o.mode < 4 && pl.hs < o.Hq + o.Hkv;
  return pl;
}
__device__ __forceinline__ void bias_of(const ProjectionOut& o, const Place& pl, int m0, float (&bb1)[4], float (&bb2)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) { bb1[i] = 0.f; bb2[i] = 0.f; }
  if (o.bias == nullptr || !pl.on) return;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    bb1[i] = __bfloat162float(o.bias[m0 + pl.f1 + i]);
    bb2[i] = __bfloat162float(o.bias[m0 + pl.f2 + i]);
  }
}

// What a launch does with a finished row, known when the code is compiled: the projection (modes 0 to 3), or mode 4, 5 or 6.  (One
// kernel with all of them: the code of a row is run once or twice a launch, so what lies between its parts is fetched for nothing.)
enum Finish { FIN_PROJECT = 0, FIN_RESIDUAL = 4, FIN_SWIGLU = 5, FIN_LOGITS = 6 };
// What the finishing of a token row reads from global memory, asked for ahead of the arithmetic.
struct FinishIn { float4 ra, rb; uint2 r1, r2; };
template <int kFin>
__device__ __forceinline__ FinishIn finish_in(const ProjectionOut& o, const Place& pl, int E_out, int m0e, int row) {
  FinishIn in;
  in.ra = in.rb = make_float4(1.f, 0.f, 1.f, 0.f);
  in.r1 = in.r2 = make_uint2(0u, 0u);
  if (kFin == FIN_PROJECT && pl.rotate) {
    const float2* rp = o.rope + (size_t)row * (o.D >> 1) + pl.k0;
    in.ra = *reinterpret_cast<const float4*>(rp);
    in.rb = *reinterpret_cast<const float4*>(rp + 2);
  }
  if (kFin == FIN_RESIDUAL && o.lin_res != nullptr) {
    const bf16* rp = o.lin_res + (size_t)row * E_out + m0e + pl.f1;
    in.r1 = *reinterpret_cast<const uint2*>(rp);
    in.r2 = *reinterpret_cast<const uint2*>(rp + (pl.f2 - pl.f1));
  }
  return in;
}

// a1, a2: the summed products of the row's four pairs.  te & 15 == threadIdx.x & 15 within the half warp that shares the row.
template <int kFin>
__device__ __forceinline__ void finish_row(const ProjectionOut& o, const BatchParams& bp, const Place& pl, int E_out, int m0e, int row,
                                           const float4& a1, const float4& a2, float rsc, const float (&bb1)[4], const float (&bb2)[4],
                                           const FinishIn& in, int te) {
  const int f1 = pl.f1, f2 = pl.f2, k0 = pl.k0, hs = pl.hs, D = o.D, half = D >> 1, rps = bp.rows_per_stream;
  float x1[4] = {a1.x, a1.y, a1.z, a1.w}, x2[4] = {a2.x, a2.y, a2.z, a2.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { x1[i] = fmaf(x1[i], rsc, bb1[i]); x2[i] = fmaf(x2[i], rsc, bb2[i]); }
  if (kFin == FIN_PROJECT && pl.rotate) {
    const float cs[4] = {in.ra.x, in.ra.z, in.rb.x, in.rb.z}, sn[4] = {in.ra.y, in.ra.w, in.rb.y, in.rb.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float y1 = x1[i] * cs[i] - x2[i] * sn[i];
      const float y2 = x2[i] * cs[i] + x1[i] * sn[i];
      x1[i] = y1; x2[i] = y2;
    }
  }
  if constexpr (kFin == FIN_SWIGLU) {
    // SwiGLU: features f1.. are gate rows, f2 = f1 + 64.. the matching up rows
    __align__(8) bf16 av[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) av[i] = __float2bfloat16_rn(x1[i] / (1.f + __expf(-x1[i])) * x2[i]);
    bf16* dst = o.lin_out + (size_t)row * (E_out >> 1) + (m0e >> 1) + f1;
    if (VS_STORE_OK(bp, o.lin_out_region, dst, 8)) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(av);
    return;
  }
  if constexpr (kFin == FIN_LOGITS) {
    // plain linear layer, rows kept in fp32 (logits of the vocabulary projection); the buffer is the caller's
    float* fo = static_cast<float*>(o.final_out) + (size_t)row * E_out + m0e;
    *reinterpret_cast<float4*>(fo + f1) = make_float4(x1[0], x1[1], x1[2], x1[3]);
    *reinterpret_cast<float4*>(fo + f2) = make_float4(x2[0], x2[1], x2[2], x2[3]);
    return;
  }
  if constexpr (kFin == FIN_RESIDUAL) {
    // linear layer + residual; the rows as stored (bf16) also give the next RMSNorm its statistics
    const size_t c1 = (size_t)row * E_out + m0e + f1, c2 = (size_t)row * E_out + m0e + f2;
    if (o.lin_res != nullptr) {
      const uint2 r1 = in.r1, r2 = in.r2;
      const float2 a0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r1.x)), a1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r1.y));
      const float2 b0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r2.x)), b1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r2.y));
      x1[0] += a0.x; x1[1] += a0.y; x1[2] += a1.x; x1[3] += a1.y;
      x2[0] += b0.x; x2[1] += b0.y; x2[2] += b1.x; x2[3] += b1.y;
    }
    __align__(8) bf16 s1[4], s2[4];
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s1[i] = __float2bfloat16_rn(x1[i]); s2[i] = __float2bfloat16_rn(x2[i]);
      const float u1 = __bfloat162float(s1[i]), u2 = __bfloat162float(s2[i]);
      ss += u1 * u1 + u2 * u2;
    }
    if (VS_STORE_OK(bp, o.lin_out_region, o.lin_out + c1, 8) && VS_STORE_OK(bp, o.lin_out_region, o.lin_out + c2, 8)) {
      *reinterpret_cast<uint2*>(o.lin_out + c1) = *reinterpret_cast<const uint2*>(s1);
      *reinterpret_cast<uint2*>(o.lin_out + c2) = *reinterpret_cast<const uint2*>(s2);
    }
    if (o.final_out != nullptr) {
      if (o.final_fp32) {
        float* fo = static_cast<float*>(o.final_out);
        *reinterpret_cast<float4*>(fo + c1) = make_float4(__bfloat162float(s1[0]), __bfloat162float(s1[1]), __bfloat162float(s1[2]), __bfloat162float(s1[3]));
        *reinterpret_cast<float4*>(fo + c2) = make_float4(__bfloat162float(s2[0]), __bfloat162float(s2[1]), __bfloat162float(s2[2]), __bfloat162float(s2[3]));
      } else {
        bf16* fo = static_cast<bf16*>(o.final_out);
        *reinterpret_cast<uint2*>(fo + c1) = *reinterpret_cast<const uint2*>(s1);
        *reinterpret_cast<uint2*>(fo + c2) = *reinterpret_cast<const uint2*>(s2);
      }
    }
    if (o.ss_out != nullptr) {
      if (o.next_gain != nullptr) {
        __align__(8) bf16 g1[4], g2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          g1[i] = __float2bfloat16_rn(__bfloat162float(s1[i]) * __bfloat162float(o.next_gain[m0e + f1 + i]));
          g2[i] = __float2bfloat16_rn(__bfloat162float(s2[i]) * __bfloat162float(o.next_gain[m0e + f2 + i]));
        }
        if (VS_STORE_OK(bp, DR_XN, o.xn_out + c1, 8) && VS_STORE_OK(bp, DR_XN, o.xn_out + c2, 8)) {
          *reinterpret_cast<uint2*>(o.xn_out + c1) = *reinterpret_cast<const uint2*>(g1);
          *reinterpret_cast<uint2*>(o.xn_out + c2) = *reinterpret_cast<const uint2*>(g2);
        }
      }
      // the 16 threads that share the row (a half warp) add their parts in a fixed order
      const unsigned hm = 0xFFFFu << (threadIdx.x & 16u);
#pragma unroll
      for (int sh = 8; sh > 0; sh >>= 1) ss += __shfl_xor_sync(hm, ss, sh);
      float* sp = o.ss_out + (size_t)row * o.ss_out_parts + m0e / GEMM_BLOCK_M;
      if ((te & 15) == 0 && VS_STORE_OK(bp, DR_ROW_SS, sp, 4)) *sp = ss;
    }
    return;
  }
  __align__(8) bf16 o1[4], o2[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { o1[i] = __float2bfloat16_rn(x1[i]); o2[i] = __float2bfloat16_rn(x2[i]); }
  const uint2 w1 = *reinterpret_cast<const uint2*>(o1), w2 = *reinterpret_cast<const uint2*>(o2);
  if (hs < o.Hq) {
    // the query never leaves the step, so it is kept as a bf16 pair (hi + lo): the score
    // Q K^T then sees a 16-bit mantissa instead of 8 at the cost of a second MMA
    __align__(8) bf16 l1[4], l2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      l1[i] = __float2bfloat16_rn(x1[i] - __bfloat162float(o1[i]));
      l2[i] = __float2bfloat16_rn(x2[i] - __bfloat162float(o2[i]));
    }
    if (o.q_tiled != nullptr) {
      // straight into the attention kernel's operand layout: one block per (batch entry, 16-token
      // row tile, KV head) holding [hi | lo][128 rows = g * 16 + token][D], rows of 128 bytes per
      // 64 dims with the 16-byte units XOR-ed by the row (the MMA's 128-byte swizzle)
      const int G = o.Hq / o.Hkv;
      const int b = row / rps, tt = row - b * rps;
      const int n_rt = (rps + 15) >> 4;
      const size_t tile = ((size_t)b * n_rt + (size_t)(tt >> 4)) * o.Hkv + (size_t)(hs / G);
      const int r = (hs % G) * 16 + (tt & 15);
      uint8_t* tb = reinterpret_cast<uint8_t*>(o.q_tiled) + tile * (size_t)(2 * 128 * D * 2);
      const int c1 = k0 >> 3, c2 = (k0 + half) >> 3;
      const uint32_t o_1 = (uint32_t)((c1 >> 3) * (128 * 128) + r * 128 + (((c1 & 7) ^ (r & 7)) << 4) + (k0 & 7) * 2);
      const uint32_t o_2 = (uint32_t)((c2 >> 3) * (128 * 128) + r * 128 + (((c2 & 7) ^ (r & 7)) << 4) + (k0 & 7) * 2);
      const uint32_t lo_off = (uint32_t)(128 * D * 2);
      if (VS_STORE_OK(bp, DR_Q_TILED, tb + o_1, 8) && VS_STORE_OK(bp, DR_Q_TILED, tb + lo_off + o_2, 8)) {
        *reinterpret_cast<uint2*>(tb + o_1) = w1;
        *reinterpret_cast<uint2*>(tb + o_2) = w2;
        *reinterpret_cast<uint2*>(tb + lo_off + o_1) = *reinterpret_cast<const uint2*>(l1);
        *reinterpret_cast<uint2*>(tb + lo_off + o_2) = *reinterpret_cast<const uint2*>(l2);
      }
    } else {
      const size_t qo = (size_t)row * o.Hq * D + (size_t)hs * D + k0;
      if (VS_STORE_OK(bp, DR_Q, o.q + qo, 8) && VS_STORE_OK(bp, DR_Q, o.q + qo + half, 8) &&
          VS_STORE_OK(bp, DR_Q_LO, o.q_lo + qo, 8) && VS_STORE_OK(bp, DR_Q_LO, o.q_lo + qo + half, 8)) {
        *reinterpret_cast<uint2*>(o.q + qo) = w1;
        *reinterpret_cast<uint2*>(o.q + qo + half) = w2;
        *reinterpret_cast<uint2*>(o.q_lo + qo) = *reinterpret_cast<const uint2*>(l1);
        *reinterpret_cast<uint2*>(o.q_lo + qo + half) = *reinterpret_cast<const uint2*>(l2);
      }
    }
  } else {
    const bool is_k = hs < o.Hq + o.Hkv;
    const int hkv = is_k ? hs - o.Hq : hs - o.Hq - o.Hkv;
    bf16* f = (is_k ? o.kf : o.vf) + (size_t)row * o.Hkv * D + (size_t)hkv * D + k0;
    if (VS_STORE_OK(bp, is_k ? DR_KF : DR_VF, f, 8) && VS_STORE_OK(bp, is_k ? DR_KF : DR_VF, f + half, 8)) {
      *reinterpret_cast<uint2*>(f) = w1;
      *reinterpret_cast<uint2*>(f + half) = w2;
    }
    const int b = row / rps, tt = row - b * rps;
    const int sid = bp.entry[b].stream_id;
    bf16* dst = nullptr;
    if (o.mode == 0) {
      if (tt == rps - 1 && o.M > 0) {
        const int slot = o.free_slot[sid * o.free_slot_stride];
        dst = (is_k ? o.bank_k : o.bank_v) + (((size_t)sid * o.Hkv + hkv) * o.slots + slot) * D + k0;
      }
    } else if (o.mode != 3) {
      const int tb = (o.mode == 1) ? bp.entry[b].prefix_len : bp.entry[b].text_len;
      dst = (is_k ? o.text_k : o.text_v) + (((size_t)sid * o.Hkv + hkv) * o.text_cap + tb + tt) * D + k0;
    }
    // (the carrier row goes to the bank, text rows to the prefix or the tail)
    const int dreg = (o.mode == 0) ? (is_k ? DR_BANK_K : DR_BANK_V)
                                     : (o.mode == 1 ? (is_k ? DR_PREFIX_K : DR_PREFIX_V) : (is_k ? DR_TAIL_K : DR_TAIL_V));
    if (dst != nullptr && VS_STORE_OK(bp, dreg, dst, 8) && VS_STORE_OK(bp, dreg, dst + half, 8)) {
      *reinterpret_cast<uint2*>(dst) = w1;
      *reinterpret_cast<uint2*>(dst + half) = w2;
    }
  }
}

}  // namespace gemm
}  // namespace vs
