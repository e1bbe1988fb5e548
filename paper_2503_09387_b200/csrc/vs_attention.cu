// Decode attention (Section 3.3, decoding phase; Eq. 1 per head with grouped KV heads): one
// query token per stream attends over [prompt prefix | carrier bank | text of the turn].  No
// visual-token K/V exists at this point -- only carriers.
//
// Bound by reading the stored keys and values once and, for one stream, by the latency of that read
// and of the merges behind it.  One CTA = one key split x one KV head x one stream, 8 warps; all
// query heads of the group (at most 8) are the 8-column operand of mma.sync.m16n8k16, so K and V are
// read once per group, straight from global memory into fragment registers:
//   S^T = K Q^T   (16 keys x 8 heads; a lane's 16 contiguous bytes of a key row feed two MMAs, a
//                  permutation of the dims that K and Q share; Q as its bf16 hi + lo pair)
//   O^T += V^T P^T (16 dims x 8 heads; byte permutes pair the rows of four keys into the A operand, rows
//                  of a tile being dims 8g + j; P, fp32, enters as a bf16 hi + lo pair -- 16 bits of
//                  mantissa -- transposed by movmatrix)
// A warp holds 16 keys (8 KB) of K and V in registers and its next 16 in flight to shared memory, two CTAs fit an SM (64 KB of
// stages and 41 KB each).  A lane copies the pieces that it reads itself, so nobody waits for anybody.  (A tile asked for once the one
// before was multiplied, a round of eight warps took 2.8 us, now 1.5: 16 streams of 1150 keys, projection included, 28.6 against
// 26.6 us.)  Warps merge their (m, l, O)
// through shared memory.  The key splits of one (stream, KV head) are a thread-block cluster (1, 2, 4
// or 8 CTAs): each CTA pushes the slice of its partial rows that a peer finishes into that peer's
// shared memory and arrives at the cluster's hardware barrier; every CTA then combines and stores its
// own slice -- no global scratch, no atomics, no polling; the co-scheduled cluster is what guarantees
// that the barrier completes.
// (One CTA per query head, K and V read once per head: 53 us for 16 streams of 1150 keys.)
#include "vs_common.cuh"
#include "vs_ptx.cuh"

namespace vs {

namespace {

constexpr int kDecThreads = 256;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kTileKeys = 16;
constexpr int kHeads = 8;       // query heads of a KV group, padded
constexpr int kMaxCluster = DEC_SPLIT_MAX;

__device__ __forceinline__ void st_shared_cluster_f4(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void st_shared_cluster_f2(uint32_t addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
constexpr int stage_bytes(int D) { return kDecWarps * kTileKeys * D * 2 * 2; }

template <int D>
__global__ void __launch_bounds__(kDecThreads, 2) decode_attn_kernel(DecodeArgs a, BatchParams bp) {
  constexpr int KC = D / 32;            // 16-byte pieces of a key row per lane (QK)
  constexpr int VC = D / 64;            // 16-byte pieces of a value row per lane (PV)
  constexpr int MT = D / 16;            // 16-dim tiles of O^T
  extern __shared__ __align__(16) uint8_t stage_s[];              // [warp][piece][lane] 16 bytes
  __shared__ __align__(16) uint4 q_s[2][kHeads][D / 8];           // hi, lo; chunk index XOR 4 in odd rows
  __shared__ __align__(16) float st_o[kDecWarps][kHeads][D];      // the warps' unnormalised rows
  __shared__ float2 st_ml[kDecWarps][kHeads];                     // ... with their (max, denominator)
  __shared__ __align__(16) float peer_o[kHeads * D];              // [split][slice]: what the cluster's CTAs leave for this one
  __shared__ float2 peer_ml[kMaxCluster][kHeads];

  // what follows from the parameters alone comes before the wait on the stream's earlier kernels
  const int split = blockIdx.x, hkv = blockIdx.y, b = blockIdx.z;
  const int sid = bp.entry[b].stream_id;
  const int G = a.Hq / a.Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t4 = lane & 3;
  const int count = bp.entry[b].count;
  const bool bank_full = (a.M > 0 && count == a.M);
  // first phase of the cluster's barrier: "this CTA runs", so that nobody writes into the shared memory of a
  // CTA that has not started; everyone arrives here and waits only just before its remote writes
  if (a.nsplit > 1) cluster_arrive_relaxed();

  int P, NB, TL;
  if (a.to_prefix) { P = bp.entry[b].prefix_len + 1; NB = 0; TL = 0; }
  else { P = bp.entry[b].prefix_len; NB = (a.M == 0) ? 0 : (bank_full ? a.M + 1 : count); TL = bp.entry[b].text_len + 1; }
  const int Lv = P + NB + TL;
  const int begin = (int)(((long long)Lv * split) / a.nsplit);
  const int end = (int)(((long long)Lv * (split + 1)) / a.nsplit);
  const int n_tiles = (end - begin + kTileKeys - 1) / kTileKeys;

  const size_t hoff = (size_t)sid * a.Hkv + hkv;
  const size_t o_pre = hoff * a.maxP * D, o_bank = hoff * a.slots * D, o_tail = hoff * a.maxT * D;
  // row v of the key axis, as an element offset, and which of the three stores it lies in
  auto row_of = [&](int v, const bf16* p, const bf16* bk, const bf16* t) {
    return v < P ? p + o_pre + (size_t)v * D : (v < P + NB ? bk + o_bank + (size_t)(v - P) * D : t + o_tail + (size_t)(v - P - NB) * D);
  };
  // Only the step's own token (the last key) was written by the kernel just before this one; every
  // other key, and the bank's metadata, date from earlier steps, whose kernels had completed before
  // that kernel let this one start.  So the first tile of K/V rows is fetched before the wait.
  // The slot being refilled holds no carrier: its key is fetched like any other (the row exists)
  // and masked when the scores are formed.
  const int hole = bank_full ? P + a.meta[sid].free_slot : -1;
  const int own_v = Lv - 1;
  uint4 kr[2][KC], vr[4][VC];
  const int kofs = 4 * (g >> 1) + (g & 1);               // S^T rows g and g + 8 are keys kofs and kofs + 2 of the tile
  // late == false: every key of the tile but the step's own; late == true: the step's own only
  auto load_tile = [&](int v0, bool late) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int v = v0 + kofs + 2 * i;
      if (v < end && ((v == own_v) == late)) {
        const uint4* kp = reinterpret_cast<const uint4*>(row_of(v, a.prefix_k, a.bank_k, a.tail_k));
#pragma unroll
        for (int c = 0; c < KC; ++c) kr[i][c] = kp[t4 + 4 * c];
      } else if (!late) {
#pragma unroll
        for (int c = 0; c < KC; ++c) kr[i][c] = make_uint4(0, 0, 0, 0);
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int v = v0 + 4 * t4 + r;
      if (v < end && ((v == own_v) == late)) {
        const uint4* vp = reinterpret_cast<const uint4*>(row_of(v, a.prefix_v, a.bank_v, a.tail_v));
#pragma unroll
        for (int c = 0; c < VC; ++c) vr[r][c] = vp[g + 8 * c];
      } else if (!late) {
#pragma unroll
        for (int c = 0; c < VC; ++c) vr[r][c] = make_uint4(0, 0, 0, 0);
      }
    }
  };
  if (warp < n_tiles) load_tile(begin + warp * kTileKeys, false);
  // The tile after goes through shared memory, a lane's pieces where this lane will read them: its copies are on their way while this
  // one is multiplied.  Before the wait too, unless the step's own key is in it.
  const uint32_t stage = smem_u32(stage_s) + (uint32_t)(warp * (2 * KC + 4 * VC) * 512 + lane * 16);
  auto fetch_tile = [&](int v0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int v = v0 + kofs + 2 * i;
      const uint4* kp = reinterpret_cast<const uint4*>(row_of(v < end ? v : begin, a.prefix_k, a.bank_k, a.tail_k));
#pragma unroll
      for (int c = 0; c < KC; ++c) cp_async16(stage + (uint32_t)((i * KC + c) * 512), kp + t4 + 4 * c, v < end);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int v = v0 + 4 * t4 + r;
      const uint4* vp = reinterpret_cast<const uint4*>(row_of(v < end ? v : begin, a.prefix_v, a.bank_v, a.tail_v));
#pragma unroll
      for (int c = 0; c < VC; ++c) cp_async16(stage + (uint32_t)((2 * KC + r * VC + c) * 512), vp + g + 8 * c, v < end);
    }
    cp_async_commit();
  };
  auto take_tile = [&]() {
    cp_async_wait<0>();
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int c = 0; c < KC; ++c) kr[i][c] = lds128(stage + (uint32_t)((i * KC + c) * 512));
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < VC; ++c) vr[r][c] = lds128(stage + (uint32_t)((2 * KC + r * VC + c) * 512));
    // The next copies go over these pieces: nothing else orders an asynchronous copy behind loads that have merely been issued.  (16 streams
    // of 1150 keys, projection included: 24.4 us, 25.5 without the fence; with the copies issued after the MMAs instead 27.3.)
    __threadfence_block();
  };
  const bool early = warp + kDecWarps < n_tiles && begin + (warp + kDecWarps + 1) * kTileKeys <= own_v;
  if (early) fetch_tile(begin + (warp + kDecWarps) * kTileKeys);

  VS_STAMP(bp, 5, 0);
  pdl_wait();
  pdl_launch_dependents();
  VS_STAMP(bp, 5, 1);
  // the step's own key and the query are both fresh: their loads go out together
  if (warp < n_tiles) load_tile(begin + warp * kTileKeys, true);
  for (int i = tid; i < 2 * kHeads * (D / 8); i += kDecThreads) {
    const int which = i / (kHeads * (D / 8)), r = i - which * (kHeads * (D / 8)), hd = r / (D / 8), c = r - hd * (D / 8);
    uint4 v = make_uint4(0, 0, 0, 0);
    if (hd < G) v = reinterpret_cast<const uint4*>((which ? a.q_lo : a.q) + ((size_t)b * a.Hq + (size_t)hkv * G + hd) * D)[c];
    q_s[which][hd][c ^ ((hd & 1) << 2)] = v;
  }
  __syncthreads();
  VS_STAMP(bp, 5, 2);

  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};     // heads 2 * t4 and 2 * t4 + 1
  float o[MT][4];
#pragma unroll
  for (int j = 0; j < MT; ++j) { o[j][0] = 0.f; o[j][1] = 0.f; o[j][2] = 0.f; o[j][3] = 0.f; }

  for (int ti = warp; ti < n_tiles; ti += kDecWarps) {
    const int v0 = begin + ti * kTileKeys;
    if (ti != warp) take_tile();
    if (ti + kDecWarps < n_tiles && !(ti == warp && early)) fetch_tile(v0 + kDecWarps * kTileKeys);
    float s[4] = {0.f, 0.f, 0.f, 0.f}, sl[4] = {0.f, 0.f, 0.f, 0.f};   // high and low query halves: two shorter chains
#pragma unroll
    for (int c = 0; c < KC; ++c) {
      const int ch = (t4 + 4 * c) ^ ((g & 1) << 2);
      const uint4 qh = q_s[0][g][ch], ql = q_s[1][g][ch];
      mma_bf16(s, kr[0][c].x, kr[1][c].x, kr[0][c].y, kr[1][c].y, qh.x, qh.y);
      mma_bf16(sl, kr[0][c].x, kr[1][c].x, kr[0][c].y, kr[1][c].y, ql.x, ql.y);
      mma_bf16(s, kr[0][c].z, kr[1][c].z, kr[0][c].w, kr[1][c].w, qh.z, qh.w);
      mma_bf16(sl, kr[0][c].z, kr[1][c].z, kr[0][c].w, kr[1][c].w, ql.z, ql.w);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) s[e] += sl[e];
    const int va = v0 + kofs, vb = va + 2;
    const bool ina = va < end && va != hole, inb = vb < end && vb != hole;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      s[e] = ina ? s[e] * a.scale_log2e : -INFINITY;
      s[2 + e] = inb ? s[2 + e] * a.scale_log2e : -INFINITY;
      float mx = fmaxf(s[e], s[2 + e]);
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
      const float mn = fmaxf(m[e], mx);
      const float mu = (mn == -INFINITY) ? 0.f : mn;          // a tile of masked keys alone
      const float sc = exp2f(m[e] - mu);                      // exp2f(-inf) = 0 on the first keys
      s[e] = exp2f(s[e] - mu);
      s[2 + e] = exp2f(s[2 + e] - mu);
      l[e] = l[e] * sc + (s[e] + s[2 + e]);
      m[e] = mn;
#pragma unroll
      for (int j = 0; j < MT; ++j) { o[j][e] *= sc; o[j][2 + e] *= sc; }
    }
    const uint32_t pa = pack2(s[0], s[1]), pb = pack2(s[2], s[3]);
    const float2 fa = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&pa));
    const float2 fb = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&pb));
    const uint32_t ph0 = transpose_8x8(pa), ph1 = transpose_8x8(pb);
    const uint32_t pl0 = transpose_8x8(pack2(s[0] - fa.x, s[1] - fa.y)), pl1 = transpose_8x8(pack2(s[2] - fb.x, s[3] - fb.y));
#pragma unroll
    for (int j = 0; j < MT; ++j) {
      // tile j: row g = dim 8 g + j, row g + 8 = dim D / 2 + 8 g + j (D = 128) or 8 g + 4 + j (D = 64); k 2 t4, 2 t4 + 1 =
      // keys 4 t4, 4 t4 + 1 of the tile, k 2 t4 + 8, + 9 = keys 4 t4 + 2, + 3
      const int j2 = (D == 128) ? j : j + 4, c2 = (D == 128) ? VC - 1 : 0;
      const uint32_t sel = (j & 1) ? 0x7632u : 0x5410u;
      const uint32_t a0 = __byte_perm(word(vr[0][0], j >> 1), word(vr[1][0], j >> 1), sel);
      const uint32_t a1 = __byte_perm(word(vr[0][c2], j2 >> 1), word(vr[1][c2], j2 >> 1), sel);
      const uint32_t a2 = __byte_perm(word(vr[2][0], j >> 1), word(vr[3][0], j >> 1), sel);
      const uint32_t a3 = __byte_perm(word(vr[2][c2], j2 >> 1), word(vr[3][c2], j2 >> 1), sel);
      mma_bf16(o[j], a0, a1, a2, a3, ph0, ph1);
      mma_bf16(o[j], a0, a1, a2, a3, pl0, pl1);
    }
  }

  VS_STAMP(bp, 5, 3);
  // warps -> CTA (a warp without a tile has nothing to leave)
  const int n_used = min(n_tiles, kDecWarps);
  if (warp < n_used) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) l[e] += __shfl_xor_sync(0xffffffffu, l[e], off);
      if (g == 0) st_ml[warp][2 * t4 + e] = make_float2(m[e], l[e]);
      float4* dst = reinterpret_cast<float4*>(st_o[warp][2 * t4 + e]);
#pragma unroll
      for (int hh = 0; hh < 2; ++hh)
#pragma unroll
        for (int j = 0; j < MT; j += 4)
          dst[merge_unit(2 * t4 + e, (D == 128 ? hh * 16 + j / 4 : hh) + 2 * g)] =
              make_float4(o[j][2 * hh + e], o[j + 1][2 * hh + e], o[j + 2][2 * hh + e], o[j + 3][2 * hh + e]);
    }
  }
  const int nsplit = a.nsplit;
  const int slice = G * D / nsplit;                      // outputs (head, dim) that one CTA of the cluster finishes
  const size_t out_off = ((size_t)b * a.Hq + (size_t)hkv * G) * D;
  // the residual input of what this thread stores: fetched ahead of the barriers
  const int my = nsplit == 1 ? 4 * tid : split * slice + 4 * tid;
  const bool mine = 4 * tid < slice;
  uint2 h_res = make_uint2(0u, 0u);
  if (a.h_out != nullptr && mine) h_res = *reinterpret_cast<const uint2*>(a.h_in + out_off + my);
  __syncthreads();

  auto store_row = [&](float4 v) {
    if (!VS_STORE_OK(bp, a.out_region, static_cast<uint8_t*>(a.out) + (out_off + my) * (a.out_fp32 ? 4 : 2), a.out_fp32 ? 16 : 8)) return;
    if (a.out_fp32) *reinterpret_cast<float4*>(static_cast<float*>(a.out) + out_off + my) = v;
    else *reinterpret_cast<uint2*>(static_cast<bf16*>(a.out) + out_off + my) = make_uint2(pack2(v.x, v.y), pack2(v.z, v.w));
    if (a.h_out != nullptr && VS_STORE_OK(bp, a.h_out_region, a.h_out + out_off + my, 8)) {
      const float2 h0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h_res.x));
      const float2 h1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h_res.y));
      *reinterpret_cast<uint2*>(a.h_out + out_off + my) = make_uint2(pack2(h0.x + v.x, h0.y + v.y), pack2(h1.x + v.z, h1.y + v.w));
    }
  };
  // this CTA's partial of outputs 4 tid .. + 3 (G * D <= 1024 of them), all of one head
  const int idx = 4 * tid, hd = idx / D, dim = idx - hd * D;
  float M = -INFINITY, Lsum = 0.f;
  float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
  if (hd < G) {
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) if (w < n_used) M = fmaxf(M, st_ml[w][hd].x);
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) {
      if (w < n_used) {
        const float2 ml = st_ml[w][hd];
        const float wt = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - M);
        const float4 v = reinterpret_cast<const float4*>(st_o[w][hd])[merge_unit(hd, dim / 4)];
        Lsum = fmaf(ml.y, wt, Lsum);
        O.x = fmaf(v.x, wt, O.x); O.y = fmaf(v.y, wt, O.y); O.z = fmaf(v.z, wt, O.z); O.w = fmaf(v.w, wt, O.w);
      }
    }
  }
  if (nsplit == 1) {
    const float inv = (Lsum > 0.f) ? 1.f / Lsum : 0.f;
    if (mine) store_row(make_float4(O.x * inv, O.y * inv, O.z * inv, O.w * inv));
    VS_STAMP(bp, 5, 15);
    return;
  }

  VS_STAMP(bp, 5, 4);
  cluster_wait_acquire();                           // phase 1 (every CTA of the cluster has started) -- long since complete
  if (hd < G) {
    const int owner = idx / slice;                  // slice is a multiple of 4
    const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(&peer_o[split * slice + idx - owner * slice]));
    st_shared_cluster_f4(map_shared_rank(dst, (uint32_t)owner), O);
    if (dim < 4 * nsplit) {                         // thread dim / 4 of the head tells rank dim / 4 the head's (max, denominator)
      const uint32_t ml = static_cast<uint32_t>(__cvta_generic_to_shared(&peer_ml[split][hd]));
      st_shared_cluster_f2(map_shared_rank(ml, (uint32_t)(dim >> 2)), make_float2(M, Lsum));
    }
  }
  cluster_arrive_release();                         // phase 2: "my partials are in place"
  cluster_wait_acquire();                           // nothing of a peer is read or written from here on
  VS_STAMP(bp, 5, 5);
  if (mine) {
    const int h2 = my / D;
    float Mx = -INFINITY;
    for (int r = 0; r < nsplit; ++r) Mx = fmaxf(Mx, peer_ml[r][h2].x);
    float den = 0.f;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < kMaxCluster; ++r) {
      if (r < nsplit) {
        const float2 ml = peer_ml[r][h2];
        const float wt = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - Mx);
        const float4 p = *reinterpret_cast<const float4*>(&peer_o[r * slice + 4 * tid]);
        den = fmaf(ml.y, wt, den);
        v.x = fmaf(p.x, wt, v.x); v.y = fmaf(p.y, wt, v.y); v.z = fmaf(p.z, wt, v.z); v.w = fmaf(p.w, wt, v.w);
      }
    }
    const float inv = (den > 0.f) ? 1.f / den : 0.f;
    store_row(make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv));
  }
  VS_STAMP(bp, 5, 15);
}

}  // namespace

cudaError_t decode_attention_init() {
  const cudaError_t e = cudaFuncSetAttribute(decode_attn_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, stage_bytes(128));
  return e != cudaSuccess ? e : cudaFuncSetAttribute(decode_attn_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, stage_bytes(64));
}

cudaError_t launch_decode_attention(const DecodeArgs& a, const BatchParams& bp, cudaStream_t st) {
  if (a.nsplit != 1 && a.nsplit != 2 && a.nsplit != 4 && a.nsplit != 8) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.nsplit, a.Hkv, bp.n_active);
  cfg.blockDim = dim3(kDecThreads);
  cfg.dynamicSmemBytes = (size_t)stage_bytes(a.D);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;            // the key splits of a row are one cluster
  attr[1].val.clusterDim.x = a.nsplit; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (a.D == 128) return cudaLaunchKernelEx(&cfg, decode_attn_kernel<128>, a, bp);
  if (a.D == 64) return cudaLaunchKernelEx(&cfg, decode_attn_kernel<64>, a, bp);
  return cudaErrorInvalidValue;
}

}  // namespace vs
