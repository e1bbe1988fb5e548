// A text step of a few token rows (Section 3.3's answer tokens, short questions) through ALL layers in one
// launch, and the language-model head of a few rows: everything such a step does is bound by reading the weight
// matrices once, so one persistent kernel streams them without a break while the rest of the step -- rotation,
// attention over the stored keys, norms, residuals, SwiGLU -- runs beside the stream.
//
// One CTA per SM.  Warp roles:
//   0..7  compute: mma.sync.m16n8k16 on weight tiles in shared memory (weight rows on M, tokens on N), the
//         finishing of tiles, the attention
//   8     weight loader: one thread, tensor copies (TMA) into a ring of 32 KB stages, phase after phase and layer after layer, held back
//         by nothing but the ring (weights are constant): when a phase starts, up to 200 KB per SM of its weights --
//         4.5 us of HBM time -- are there already
//   9     token-row loader: the K slab of the rows that belongs to a stage, as soon as the phase's input is complete
//   10    RMSNorm row scales of a phase from the parts its producer left
// Phases of a layer: QKV -> attention [-> W_o -> gate/up -> W_down].  A phase's input is complete when its counter in
// global memory (L2) says so: CTAs count themselves in after a fence, whoever needs the input polls.
// Every weight phase is a flat list of stages (tile by tile along K) cut into gridDim.x equal runs, so every SM reads the
// same number of bytes whatever the shape (3584 x 18944 is 112 stages of every SM; whole tiles would leave a third of
// the chip idle).  A tile cut by a boundary is summed by the CTA that holds its beginning, which comes to it last; the CTA
// that holds its end comes to it first and leaves the partial sums in global memory.  All sums have a fixed order.
// A tile's 16 rows are 8 rotation pairs of a head (rows g and g + 8 of the MMA: both elements in one thread), or 8 gate and
// 8 up rows; a tile is two such sub-tiles (the slab of the token rows is read for 32 weight rows).
// Attention: a unit = (token row, KV head, share of the keys) per CTA, all query heads of the group as the 8 columns
// of S^T = K Q^T and O^T = V^T P^T (see decode_attn_kernel, whose arithmetic this is); the last unit of a row and head to
// finish combines the shares in order.
// The whole grid is resident (one CTA per SM; that an SM holds one is checked when a handle is made), so every wait ends; all are bounded: on expiry the CTA
// raises its abort flag, every later wait returns at once, copies in flight are awaited (bounded) and the status is set.
// Where this kernel is taken, and what the launches cost there: token_step_pays.  (At the Qwen2-7B shape one row costs 90 us a full
// layer, 92 by launches, where its weights take 71 us of HBM time.  Through the attention layers alone it is 16.5 us a layer against
// 11.4 by the two launches, which is why these still run there.  Stamps of such a layer: 5.4 us from the projection's input being
// known to its last store, about 4 for the attention, the other 7 until counters are seen, twice a layer.)
#include "vs_common.cuh"
#include "vs_ptx.cuh"

namespace vs {

namespace {

constexpr int kCW = 8;                            // compute warps
constexpr int kCT = kCW * 32;
constexpr int kThreads = kCT + 96;
constexpr int kKeysPerTile = 16;
constexpr int kHeads = 8;
constexpr int kMaxStages = 12;
constexpr int kCntStride = 32;                    // counters lie a cache line apart
enum { PH_QKV = 0, PH_ATT, PH_WO, PH_GU, PH_DN, PH_LM };

// Bounded; false (at once) when it expired or another role of the CTA already gave up.  (Out of line, like what else runs
// once a phase: a layer's code has to fit the instruction cache.)
__device__ __noinline__ bool stage_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  uint32_t spins = 0;
  unsigned long long t0 = 0;
  while (!mbar_try_wait(bar, parity)) {
    if (*abort_flag) return false;
    if ((++spins & 255u) == 0u) {
      const unsigned long long now = global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kWaitLimitNs) { *abort_flag = 1; return false; }
    }
  }
  return true;
}
__device__ __forceinline__ bool stage_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_try_wait(bar, parity) || stage_wait_slow(bar, parity, abort_flag);
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) { asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ void add_release(int* p, int v) { asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
// (release and acquire are cumulative: after a barrier of the block, one thread's covers what the others stored or will load)
__device__ __forceinline__ int add_acq_rel(int* p, int v) {
  int r;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(r) : "l"(p), "r"(v) : "memory");
  return r;
}
__device__ __forceinline__ int ld_relaxed(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// until *p >= target (counters only grow during a launch).  Polls with relaxed loads, far apart: an acquiring load invalidates
// the SM's L1, and a loop of them slowed every shared-memory access of the SM down several times.
__device__ __noinline__ bool wait_count(const int* p, int target, volatile int* abort_flag) {
  uint32_t spins = 0;
  unsigned long long t0 = 0;
  while (ld_relaxed(p) < target) {
    __nanosleep(20);
    if (*abort_flag) return false;
    if ((++spins & 63u) == 0u) {
      const unsigned long long now = global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kWaitLimitNs) { *abort_flag = 1; return false; }
    }
  }
  ld_acquire(p);
  return true;
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, int w, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar) : "memory");
}
// this thread's arrival, once the copies it has issued so far have landed
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
// MMA row g of an 8-row group is row pi(g) of the group in memory: the two rows that a quarter warp reads side by side are then
// four apart, where the 128-byte swizzle puts the same 64 bytes of them into different banks
__device__ __forceinline__ int pi(int g) { return (g >> 1) | ((g & 1) << 2); }
__device__ __forceinline__ void compute_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
static_assert(kCT == 256, "the named barrier above counts 256 threads");
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float2 unpack2(uint32_t w) { return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w)); }
__device__ __forceinline__ float ld_bf16_cg(const bf16* p) {
  const unsigned short u = __ldcg(reinterpret_cast<const unsigned short*>(p));
  return __uint_as_float((uint32_t)u << 16);
}

#ifdef VS_TRACE
#define TOK_STAMP(ev, l) do { if (bp.trace != nullptr && (cta == 0 || cta == 100) && lane == 0) { unsigned long long t_; asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t_)); bp.trace[((cta ? 1 : 0) * 32 + (ev)) * 64 + ((l) & 63)] = t_; } } while (0)
#else
#define TOK_STAMP(ev, l)
#endif
// What every role derives in the same way: the run of stages of this CTA in a weight phase.
struct Phase {
  int K, kst, tiles;            // reduction length, stages per tile, tiles
  int s0, s1;                   // this CTA's stages
};
constexpr int KS = 512;                           // K elements of a stage (32 KB of weights)
constexpr int MT = 2;                             // 16-row sub-tiles of a weight tile
__device__ __noinline__ Phase make_phase(const TokArgs& a, int kind, int cta, int ncta) {
  Phase p;
  int rows = 0;
  if (kind == PH_QKV) { rows = (a.Hq + 2 * a.Hkv) * a.D; p.K = a.d; }
  else if (kind == PH_WO) { rows = a.d; p.K = a.d; }
  else if (kind == PH_GU) { rows = 2 * a.d_ff; p.K = a.d; }
  else if (kind == PH_DN) { rows = a.d; p.K = a.d_ff; }
  else { rows = a.vocab; p.K = a.d; }
  p.kst = (p.K + KS - 1) / KS;
  p.tiles = rows / (16 * MT);
  // whole tiles, where that makes the longest run no more than two stages longer than the average: a cut tile costs its
  // owner about 1.5 us at the end of the phase (a flag and a partial sum from another SM)
  const int most = (p.tiles + ncta - 1) / ncta;
  if ((most * p.kst - 2) * ncta <= p.tiles * p.kst) {
    p.s0 = p.tiles * cta / ncta * p.kst;
    p.s1 = p.tiles * (cta + 1) / ncta * p.kst;
    return p;
  }
  const uint32_t total = (uint32_t)(p.tiles * p.kst);              // (the launch checks that total * ncta fits 32 bits)
  p.s0 = (int)(total * (uint32_t)cta / (uint32_t)ncta);
  p.s1 = (int)(total * (uint32_t)(cta + 1) / (uint32_t)ncta);
  return p;
}
// counter of phase `kind` of layer l; 0 is the input's normalisation
__device__ __forceinline__ int* counter(const TokArgs& a, int l, int kind) { return a.counters + (size_t)(1 + l * 5 + kind) * kCntStride; }

// waits until the token rows that phase `kind` of layer l reads are complete
__device__ __noinline__ bool wait_input(const TokArgs& a, int l, int kind, int ncta, volatile int* abort_flag) {
  const int* c; int n;
  if (kind == PH_LM || (kind == PH_QKV && l == 0)) {
    if (kind == PH_QKV && !a.use_rmsnorm) return true;           // the caller's rows
    c = a.counters; n = a.rows;
  }
  else if (kind == PH_QKV) { c = a.full ? counter(a, l - 1, PH_DN) : counter(a, l - 1, PH_ATT); n = a.full ? ncta : a.rows * a.Hkv; }
  else if (kind == PH_WO) { c = counter(a, l, PH_ATT); n = a.rows * a.Hkv; }
  else if (kind == PH_GU) { c = counter(a, l, PH_WO); n = ncta; }
  else { c = counter(a, l, PH_GU); n = ncta; }
  return wait_count(c, n, abort_flag);
}
__device__ __forceinline__ const bf16* layer_input(const TokArgs& a, int l) {
  if (l == 0) return static_cast<const bf16*>(a.hidden);
  return a.full ? a.hbuf[0] : a.hbuf[(l - 1) & 1];
}
// the rows a weight phase multiplies
__device__ __forceinline__ const bf16* phase_rows(const TokArgs& a, int l, int kind) {
  if (kind == PH_QKV) return (a.use_rmsnorm && a.layers[l].gain != nullptr) ? a.xn : layer_input(a, l);
  if (kind == PH_WO) return a.attn_rows;
  if (kind == PH_GU) return (a.use_rmsnorm && a.layers[l].gain2 != nullptr) ? a.xn : a.hbuf[1];
  if (kind == PH_DN) return a.act;
  return a.xn;
}

// What the finishing of an accumulator reads from global memory, asked for before its last stage is multiplied.
struct FinishIn {
  float b1, b2;                  // QKV: bias of the two features; W_o, W_down: the next norm's gain there
  float r1[2], r2[2];            // W_o, W_down: residual of (feature, token)
};
template <int D>
__device__ __forceinline__ FinishIn finish_in(const TokArgs& a, int l, int kind, int mt, int nt, int lane) {
  const int pg = pi(lane >> 2), n0 = nt * 8 + 2 * (lane & 3);
  FinishIn f = {0.f, 0.f, {0.f, 0.f}, {0.f, 0.f}};
  if (kind == PH_QKV) {
    const bf16* bias = a.layers[l].bias;
    const int hs = mt / (D / 16), f1 = hs * D + (mt - hs * (D / 16)) * 8 + pg;
    if (bias != nullptr) { f.b1 = __bfloat162float(bias[f1]); f.b2 = __bfloat162float(bias[f1 + D / 2]); }
  } else if (kind == PH_WO || kind == PH_DN) {
    const bf16* res = kind == PH_WO ? layer_input(a, l) : a.hbuf[1];
    const bf16* gain = kind == PH_WO ? a.layers[l].gain2 : (l + 1 == a.L ? nullptr : a.layers[l + 1].gain);
    const int f1 = mt * 16 + pg;
    if (gain != nullptr) { f.b1 = __bfloat162float(gain[f1]); f.b2 = __bfloat162float(gain[f1 + 8]); }
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (n0 + e < a.rows) { f.r1[e] = ld_bf16_cg(res + (size_t)(n0 + e) * a.d + f1); f.r2[e] = ld_bf16_cg(res + (size_t)(n0 + e) * a.d + f1 + 8); }
  }
  return f;
}

// Finishes one 16 x 8 accumulator: v = (row r, token n0), (row r, n0 + 1), (row r + 8, n0), (row r + 8, n0 + 1) of 16-row
// sub-tile mt, r = pi(lane / 4), n0 = nt * 8 + 2 * (lane % 4).
template <int D, int NT>
__device__ __forceinline__ void finish_item(const TokArgs& a, const BatchParams& bp, int l, int kind, int mt, int nt, float4 v, const FinishIn& in, int lane,
                                            const float2* rope_s, const float* rsc_s, unsigned long long* best_s) {
  constexpr int half = D / 2;
  const int g = lane >> 2, pg = pi(g), n0 = nt * 8 + 2 * (lane & 3), rows = a.rows;
  float x1[2] = {v.x, v.y}, x2[2] = {v.z, v.w};
  if (kind == PH_QKV) {
    const int hs = mt / (D / 16), k0 = (mt - hs * (D / 16)) * 8 + pg;     // head slot (Q heads, K heads, V heads), index inside the half head
    const int rps = bp.rows_per_stream;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int row = n0 + e;
      if (row >= rows) continue;
      const float rsc = a.use_rmsnorm ? rsc_s[row] : 1.f;
      float y1 = fmaf(x1[e], rsc, in.b1), y2 = fmaf(x2[e], rsc, in.b2);
      if (hs < a.Hq + a.Hkv) {
        const float2 cs = rope_s[row * half + k0];
        const float r1 = y1 * cs.x - y2 * cs.y, r2 = y2 * cs.x + y1 * cs.y;
        y1 = r1; y2 = r2;
      }
      const bf16 o1 = __float2bfloat16_rn(y1), o2 = __float2bfloat16_rn(y2);
      if (hs < a.Hq) {
        // the query stays inside the step: kept as a bf16 pair (hi + lo)
        const size_t qo = (size_t)row * a.Hq * D + (size_t)hs * D + k0;
        if (VS_STORE_OK(bp, DR_Q, a.q + qo, 2) && VS_STORE_OK(bp, DR_Q, a.q + qo + half, 2) &&
            VS_STORE_OK(bp, DR_Q_LO, a.q_lo + qo, 2) && VS_STORE_OK(bp, DR_Q_LO, a.q_lo + qo + half, 2)) {
          a.q[qo] = o1; a.q[qo + half] = o2;
          a.q_lo[qo] = __float2bfloat16_rn(y1 - __bfloat162float(o1));
          a.q_lo[qo + half] = __float2bfloat16_rn(y2 - __bfloat162float(o2));
        }
      } else {
        const bool is_k = hs < a.Hq + a.Hkv;
        const int hkv = is_k ? hs - a.Hq : hs - a.Hq - a.Hkv;
        bf16* f = (is_k ? a.kf : a.vf) + ((size_t)row * a.Hkv + hkv) * D + k0;
        if (VS_STORE_OK(bp, is_k ? DR_KF : DR_VF, f, 2) && VS_STORE_OK(bp, is_k ? DR_KF : DR_VF, f + half, 2)) { f[0] = o1; f[half] = o2; }
        const int b = row / rps, tt = row - b * rps, sid = bp.entry[b].stream_id;
        const int tb = a.to_prefix ? bp.entry[b].prefix_len : bp.entry[b].text_len, cap = a.to_prefix ? a.maxP : a.maxT;
        bf16* base = a.to_prefix ? (is_k ? a.prefix_k : a.prefix_v) + (size_t)l * a.ls_prefix : (is_k ? a.tail_k : a.tail_v) + (size_t)l * a.ls_tail;
        bf16* dst = base + (((size_t)sid * a.Hkv + hkv) * cap + tb + tt) * D + k0;
        const int dreg = a.to_prefix ? (is_k ? DR_PREFIX_K : DR_PREFIX_V) : (is_k ? DR_TAIL_K : DR_TAIL_V);
        (void)dreg;
        if (VS_STORE_OK(bp, dreg, dst, 2) && VS_STORE_OK(bp, dreg, dst + half, 2)) { dst[0] = o1; dst[half] = o2; }
      }
    }
  } else if (kind == PH_GU) {
    const int f = mt * 8 + pg;                                           // row g: gate, row g + 8: up
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int row = n0 + e;
      if (row >= rows) continue;
      const float rsc = a.use_rmsnorm ? rsc_s[row] : 1.f;
      const float gt = x1[e] * rsc, up = x2[e] * rsc;
      bf16* dst = a.act + (size_t)row * a.d_ff + f;
      if (VS_STORE_OK(bp, DR_ACT, dst, 2)) *dst = __float2bfloat16_rn(gt / (1.f + __expf(-gt)) * up);
    }
  } else if (kind == PH_LM) {
    const int f1 = mt * 16 + pg;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int row = n0 + e;
      const bool valid = row < rows;
      const float rsc = (a.use_rmsnorm && valid) ? rsc_s[row] : 1.f;
      const float y1 = x1[e] * rsc, y2 = x2[e] * rsc;
      if (valid) { a.logits[(size_t)row * a.vocab + f1] = y1; a.logits[(size_t)row * a.vocab + f1 + 8] = y2; }
      if (a.next_token != nullptr) {
        // (a NaN is never larger; a row without a number above -inf offers nothing)
        unsigned long long k = 0ull;
        if (valid && y1 > -INFINITY) k = argmax_key(y1, f1);
        if (valid && y2 > -INFINITY) { const unsigned long long k2 = argmax_key(y2, f1 + 8); if (k2 > k) k = k2; }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) { const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, k, o); if (k2 > k) k = k2; }
        if (valid && g == 0 && k != 0ull) atomicMax(best_s + row, k);
      }
    }
  } else {
    // linear layer + residual (W_o: + the layer's input, W_down: + h1); the rows as stored give the next norm its statistics
    bf16* out = kind == PH_WO ? a.hbuf[1] : a.hbuf[0];
    const bool last = kind == PH_DN && l + 1 == a.L;
    const bf16* gain = kind == PH_WO ? a.layers[l].gain2 : (last ? nullptr : a.layers[l + 1].gain);
    float* ss = a.ss + (kind == PH_WO ? (size_t)TOK_MAX_ROWS * a.ss_cap : 0);
    const int f1 = mt * 16 + pg, reg = kind == PH_WO ? DR_HBUF1 : DR_HBUF0;
    (void)reg;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int row = n0 + e;
      const bool valid = row < rows;
      float sq = 0.f;
      if (valid) {
        const size_t c1 = (size_t)row * a.d + f1, c2 = c1 + 8;
        const bf16 s1 = __float2bfloat16_rn(x1[e] + in.r1[e]), s2 = __float2bfloat16_rn(x2[e] + in.r2[e]);
        if (VS_STORE_OK(bp, reg, out + c1, 2) && VS_STORE_OK(bp, reg, out + c2, 2)) { out[c1] = s1; out[c2] = s2; }
        const float u1 = __bfloat162float(s1), u2 = __bfloat162float(s2);
        sq = u1 * u1 + u2 * u2;
        if (last) {
          if (a.out_fp32) { static_cast<float*>(a.out)[c1] = u1; static_cast<float*>(a.out)[c2] = u2; }
          else { static_cast<bf16*>(a.out)[c1] = s1; static_cast<bf16*>(a.out)[c2] = s2; }
        }
        if (a.use_rmsnorm && gain != nullptr && VS_STORE_OK(bp, DR_XN, a.xn + c1, 2) && VS_STORE_OK(bp, DR_XN, a.xn + c2, 2)) {
          a.xn[c1] = __float2bfloat16_rn(u1 * in.b1);
          a.xn[c2] = __float2bfloat16_rn(u2 * in.b2);
        }
      }
      if (a.use_rmsnorm && !last) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        float* sp = ss + (size_t)row * a.ss_cap + mt;
        if (valid && g == 0 && VS_STORE_OK(bp, DR_TOK, sp, 4)) *sp = sq;
      }
    }
  }
}

template <int D, int NT>   // head size; 8-token columns
__global__ void __launch_bounds__(kThreads, 1) token_kernel(const __grid_constant__ TokArgs a, const __grid_constant__ BatchParams bp) {
  constexpr int TM = 16 * MT;                     // a stage: 32 weight rows x KS elements, and KS elements of every token row
  constexpr uint32_t kStageW = TM * KS * 2;       // the weights of a stage; behind them the token rows, RS bytes apart (64 more than
  constexpr int RS = KS * 2 + 64;                 // their slab: two neighbouring rows lie in different banks)
  constexpr int ITEMS = MT * NT;                  // 16 x 8 accumulators of a tile
  constexpr int KC = D / 32, VC = D / 64, OT = D / 16;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // carve: ring | union { red [8 warps][ITEMS][32] float4, st_o [8][8][D] float } | rotation table | control
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t ring = smem_u32(smem);
  uint8_t* u_base = smem + a.ring_bytes;
  float4* red = reinterpret_cast<float4*>(u_base);
  float* st_o = reinterpret_cast<float*>(u_base);
  constexpr int kUnion = (kCW * ITEMS * 512 > kCW * kHeads * D * 4) ? kCW * ITEMS * 512 : kCW * kHeads * D * 4;
  float2* rope_s = reinterpret_cast<float2*>(u_base + kUnion);                            // [rows][D / 2]
  uint8_t* ctl = u_base + kUnion + (size_t)NT * 8 * (D / 2) * 8;
  uint4 (*q_s)[kHeads][D / 8] = reinterpret_cast<uint4 (*)[kHeads][D / 8]>(ctl);          // [hi | lo][8][D / 8]
  float2 (*st_ml)[kHeads] = reinterpret_cast<float2 (*)[kHeads]>(ctl + 2 * kHeads * D * 2);
  float* rsc_s = reinterpret_cast<float*>(ctl + 2 * kHeads * D * 2 + kCW * kHeads * 8);   // [16] row scales
  float* sum_s = rsc_s + TOK_MAX_ROWS;                                                   // [8]
  unsigned long long* best_s = reinterpret_cast<unsigned long long*>(sum_s + 8);         // [16] greedy-choice keys
  volatile int* abort_flag = reinterpret_cast<volatile int*>(best_s + TOK_MAX_ROWS);
  int* bcast = const_cast<int*>(abort_flag) + 1;
  const uint32_t bars = smem_u32(best_s + TOK_MAX_ROWS + 2);
  auto full = [&](int s) { return bars + 8u * (uint32_t)s; };                     // the weights' bytes and the 32 lanes that bring the token rows
  auto empty = [&](int s) { return bars + 8u * (uint32_t)(kMaxStages + s); };
  const uint32_t rs_bar = bars + 8u * (uint32_t)(2 * kMaxStages);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cta = blockIdx.x, ncta = gridDim.x;
  const int stages = a.stages, rows = a.rows;
  const uint32_t stage_bytes = (kStageW + (uint32_t)rows * RS + 1023u) & ~1023u;
  if (tid == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(full(s), 33); mbar_init(empty(s), kCW); }
    mbar_init(rs_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (tid < TOK_MAX_ROWS) best_s[tid] = 0ull;
  __syncthreads();
  // Every role walks the phases in order (one loop with the phase as a variable: a copy of the code per phase did not fit
  // the instruction cache).
  const int n_layers = a.vocab > 0 ? 1 : a.L, last_kind = a.vocab > 0 ? PH_LM : (a.full ? PH_DN : PH_ATT);
  auto for_phases = [&](auto f) {
#pragma unroll 1
    for (int l = 0; l < n_layers; ++l)
#pragma unroll 1
      for (int kind = a.vocab > 0 ? PH_LM : PH_QKV; kind <= last_kind; ++kind) f(l, kind);
  };

  if (warp == kCW) {
    // ---- weight loader: one thread, one tensor copy (two for a gate / up pair) a stage ------------------------
    int n = 0, slot = 0;                           // stages issued, the next one's place in the ring
    uint32_t par = 1;                              // ... and the parity its emptying is waited with
    if (lane == 0)
      for_phases([&](int l, int kind) {
        if (kind == PH_ATT) return;
        const Phase p = make_phase(a, kind, cta, ncta);
        const TokLayer* ly = a.layers + l;
        const CUtensorMap* tm = kind == PH_QKV ? &ly->tm_qkv : kind == PH_WO ? &ly->tm_o : kind == PH_GU ? &ly->tm_gate
                              : kind == PH_DN ? &ly->tm_down : a.tm_lm;
        asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory");
        int tile = p.s0 / p.kst, kk = p.s0 - tile * p.kst;
#pragma unroll 1
        for (int s = p.s0; s < p.s1; ++s, ++n) {
          if (!stage_wait(empty(slot), par, abort_flag)) return;
          const uint32_t dst = ring + slot * stage_bytes;
          const int kb = kk * (KS / 64);           // (blocks past the end of a row read as zeros)
          mbar_arrive_expect_tx(full(slot), kStageW);
          if (kind == PH_QKV) {
            const int hs = tile * MT / (D / 16), pb = tile * MT - hs * (D / 16);
            tma_load_4d(dst, tm, 0, pb * 8, 2 * hs, kb, full(slot));
          } else if (kind == PH_GU) {
            tma_load_4d(dst, tm, 0, tile * MT * 8, 0, kb, full(slot));
            tma_load_4d(dst + kStageW / 2, &ly->tm_up, 0, tile * MT * 8, 0, kb, full(slot));
          } else {
            tma_load_4d(dst, tm, 0, tile * TM, 0, kb, full(slot));
          }
          if (++kk == p.kst) { kk = 0; ++tile; }
          if (++slot == stages) { slot = 0; par ^= 1u; }
        }
      });
    pdl_wait();
    if (*abort_flag && lane == 0)                  // let the copies in flight land before the shared memory is given up
      for (int i = max(0, n - stages); i < n; ++i) {
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(full(i % stages), (uint32_t)(i / stages) & 1u)) if (global_ns() - t0 > kWaitLimitNs) break;
      }
  } else if (warp == kCW + 1) {
    // ---- token-row loader: 16 bytes a lane --------------------------------------------------------------
    pdl_wait();
    pdl_launch_dependents();
    int slot = 0;
    uint32_t par = 1;
    for_phases([&](int l, int kind) {
      if (kind == PH_ATT) return;
      const Phase p = make_phase(a, kind, cta, ncta);
      const bf16* x = phase_rows(a, l, kind);
      if (p.s0 < p.s1) {
        if (lane == 0) wait_input(a, l, kind, ncta, abort_flag);
        __syncwarp();
        if (kind == PH_QKV) TOK_STAMP(13, l);
      }
      int kk = p.s0 % p.kst;
#pragma unroll 1
      for (int s = p.s0; s < p.s1; ++s) {
        if (!__all_sync(0xffffffffu, stage_wait(empty(slot), par, abort_flag))) return;
        const uint32_t dst = ring + slot * stage_bytes + kStageW;
        const int k0 = kk * KS;
        static_assert(KS == 512, "two 16-byte pieces of a row's slab a lane");
        const bool in0 = k0 + lane * 8 < p.K, in1 = k0 + 256 + lane * 8 < p.K;
#pragma unroll 1
        for (int r = 0; r < rows; ++r) {
          const bf16* src = x + (size_t)r * p.K + k0 + lane * 8;
          if (in0) cp_async16(dst + (uint32_t)r * RS + lane * 16, src);
          if (in1) cp_async16(dst + (uint32_t)r * RS + 512 + lane * 16, src + 256);
        }
        cp_async_arrive(full(slot));
        if (++kk == p.kst) kk = 0;
        if (++slot == stages) { slot = 0; par ^= 1u; }
      }
    });
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp == kCW + 2) {
    // ---- row scales ------------------------------------------------------------------------------
    pdl_wait();
    pdl_launch_dependents();
    if (a.use_rmsnorm)
      for_phases([&](int l, int kind) {
        if (kind != PH_QKV && kind != PH_GU && kind != PH_LM) return;
        const Phase p = make_phase(a, kind, cta, ncta);
        if (p.s0 >= p.s1) return;
        if (lane == 0) wait_input(a, l, kind, ncta, abort_flag);
        __syncwarp();
        const int parts = (kind == PH_LM || (kind == PH_QKV && l == 0)) ? 1 : (a.full ? a.d / 16 : a.Hkv);
        const float* ss = a.ss + (kind == PH_GU ? (size_t)TOK_MAX_ROWS * a.ss_cap : 0);
        // lanes of a row: as many as it has parts (up to 32), so that few-part rows are summed side by side
        int lpr = 1;
        while (lpr < parts && lpr < 32) lpr <<= 1;
#pragma unroll 1
        for (int r0 = 0; r0 < rows; r0 += 32 / lpr) {
          const int r = r0 + lane / lpr;
          float t = 0.f;
#pragma unroll 1
          for (int i0 = lane & (lpr - 1); i0 < parts; i0 += 8 * lpr) {
            float u[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) u[j] = (r < rows && i0 + j * lpr < parts) ? __ldcg(ss + (size_t)r * a.ss_cap + i0 + j * lpr) : 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) t += u[j];
          }
#pragma unroll 1
          for (int o = lpr >> 1; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
          if ((lane & (lpr - 1)) == 0 && r < rows) rsc_s[r] = rsqrtf(t / (float)a.d + a.eps);
        }
        if (kind == PH_QKV) TOK_STAMP(14, l);
        __syncwarp();
        if (lane == 0) mbar_arrive(rs_bar);
      });
  } else {
    // ---- compute ------------------------------------------------------------------------------------
    const int g = lane >> 2, t4 = lane & 3;
    const int rps = bp.rows_per_stream;
    if (a.vocab == 0)
#pragma unroll 1
      for (int i = tid; i < rows * (D / 2); i += kCT) {
        const int row = i / (D / 2), k = i - row * (D / 2), b = row / rps;
        double sn, cs;
        sincos((double)(bp.entry[b].pos_base + (row - b * rps)) * a.inv_freq[k], &sn, &cs);
        rope_s[i] = make_float2((float)cs, (float)sn);
      }
    pdl_wait();
    pdl_launch_dependents();

    // the input's normalisation: sum of squares of every row, and the row as the first phase reads it
    if (a.use_rmsnorm || a.vocab > 0)
#pragma unroll 1
      for (int r = cta; r < rows; r += ncta) {
        const bf16* gain = a.vocab > 0 ? a.gain_f : a.layers[0].gain;
        float ss = 0.f;
#pragma unroll 2
        for (int c = tid * 2; c < a.d; c += 2 * kCT) {
          uint32_t hv;
          if (a.hidden_fp32) {
            const float2 f = *reinterpret_cast<const float2*>(static_cast<const float*>(a.hidden) + (size_t)r * a.d + c);
            hv = pack2(f.x, f.y);
          } else {
            hv = *reinterpret_cast<const uint32_t*>(static_cast<const bf16*>(a.hidden) + (size_t)r * a.d + c);
          }
          const float2 v = unpack2(hv);
          ss += v.x * v.x + v.y * v.y;
          if (a.use_rmsnorm && gain != nullptr) {
            const float2 gv = unpack2(*reinterpret_cast<const uint32_t*>(gain + c));
            hv = pack2(v.x * gv.x, v.y * gv.y);
          }
          if ((a.vocab > 0 || gain != nullptr) && VS_STORE_OK(bp, DR_XN, a.xn + (size_t)r * a.d + c, 4))
            *reinterpret_cast<uint32_t*>(a.xn + (size_t)r * a.d + c) = hv;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        if (lane == 0) sum_s[warp] = ss;
        compute_bar();
        if (tid == 0) {
          float t = 0.f;
#pragma unroll
          for (int i = 0; i < kCW; ++i) t += sum_s[i];
          float* sp = a.ss + (size_t)r * a.ss_cap;
          if (VS_STORE_OK(bp, DR_TOK, sp, 4)) *sp = t;
          if (VS_STORE_OK(bp, DR_TOK_SYNC, a.counters, 4)) add_release(a.counters, 1);
        }
        compute_bar();
      }

    int slot = 0;
    uint32_t par = 0, rs_parity = 0;
    auto weight_phase = [&](int l, int kind) {
      const Phase p = make_phase(a, kind, cta, ncta);
      const int seq = 1 + l * 5 + kind;
      if (warp == 0 && kind == PH_QKV) TOK_STAMP(0, l);
      const bool normed = a.use_rmsnorm && (kind == PH_QKV || kind == PH_GU || kind == PH_LM);
      float acc[ITEMS][4];
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) { acc[i][0] = 0.f; acc[i][1] = 0.f; acc[i][2] = 0.f; acc[i][3] = 0.f; }
      // where row g of a sub-tile's second half (the rotation partner, the up row, row g + 8), the next K block and the next
      // sub-tile lie in a stage
      const uint32_t hi_off = kind == PH_QKV ? 8 * MT * 128 : kind == PH_GU ? kStageW / 2 : 8 * 128;
      const uint32_t kb_stride = kind == PH_GU ? 8 * MT * 128 : 16 * MT * 128;
      const uint32_t m_off = (kind == PH_QKV || kind == PH_GU) ? 8 * 128 : 16 * 128;
      const int pg = pi(g);
      int tile = p.s0 / p.kst, kk = p.s0 - tile * p.kst, kk_begin = kk;
#pragma unroll 1
      for (int s = p.s0; s < p.s1; ++s) {
        const int len = min(KS, p.K - kk * KS);
        stage_wait(full(slot), par, abort_flag);
        if (warp == 0 && kind == PH_QKV && s == p.s0) TOK_STAMP(1, l);
        if (warp == 0 && kind == PH_QKV && s == p.s1 - 1) TOK_STAMP(2, l);
        const bool part_ends = kk + 1 == p.kst || s + 1 == p.s1;
        const int item = (warp - tile) & (kCW - 1);                    // the accumulator that this warp finishes, if there is one
        FinishIn in = {};
        if (part_ends && item < ITEMS && kk_begin == 0) in = finish_in<D>(a, l, kind, tile * MT + item / NT, item % NT, lane);
        const uint32_t xb = ring + slot * stage_bytes + kStageW;
        // the stage's weights: [K block of 64][rows][128 bytes, swizzled]; each warp takes 64 of K
        constexpr int KW = KS / kCW / 32;                              // 32s of K
        static_assert(KW == 2, "a warp takes a 64-element block");
        const uint32_t wb = ring + slot * stage_bytes + (uint32_t)warp * kb_stride + (uint32_t)pg * 128;
        if (warp * KW * 32 < len) {                                    // (a multiple of 64; what is left of KW 32s is zeros)
          uint4 xv[KW][NT], w0[KW][MT], w1[KW][MT];
#pragma unroll
          for (int kb = 0; kb < KW; ++kb) {
            const uint32_t cb = (uint32_t)(((kb * 4 + t4) ^ pg) << 4);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
              w0[kb][mt] = lds128(wb + (uint32_t)mt * m_off + cb);
              w1[kb][mt] = lds128(wb + (uint32_t)mt * m_off + hi_off + cb);
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) xv[kb][nt] = lds128(xb + (uint32_t)min(nt * 8 + g, rows - 1) * RS + (uint32_t)((warp * KW + kb) * 64 + t4 * 16));   // (columns beyond the rows: never stored)
          }
#pragma unroll
          for (int kb = 0; kb < KW; ++kb)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
              for (int mt = 0; mt < MT; ++mt) mma_bf16(acc[mt * NT + nt], w0[kb][mt].x, w1[kb][mt].x, w0[kb][mt].y, w1[kb][mt].y, xv[kb][nt].x, xv[kb][nt].y);
#pragma unroll
          for (int kb = 0; kb < KW; ++kb)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
              for (int mt = 0; mt < MT; ++mt) mma_bf16(acc[mt * NT + nt], w0[kb][mt].z, w1[kb][mt].z, w0[kb][mt].w, w1[kb][mt].w, xv[kb][nt].z, xv[kb][nt].w);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty(slot));
        if (++slot == stages) { slot = 0; par ^= 1u; }
        if (!part_ends) { ++kk; continue; }
        // the end of this CTA's part of the tile: the warps' partial sums meet in shared memory, each accumulator is
        // finished by one warp
        compute_bar();                                                 // (the tile before has been read)
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
          red[(warp * ITEMS + i) * 32 + lane] = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
          acc[i][0] = 0.f; acc[i][1] = 0.f; acc[i][2] = 0.f; acc[i][3] = 0.f;
        }
        compute_bar();
        if (normed) stage_wait(rs_bar, rs_parity, abort_flag);
        if (item < ITEMS) {
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int w = 0; w < kCW; ++w) {
            const float4 u = red[(w * ITEMS + item) * 32 + lane];
            v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
          }
          if (kk_begin > 0) {
            // the end of a tile that another CTA began: left for that CTA
            float4* dst = reinterpret_cast<float4*>(a.part) + ((size_t)cta * ITEMS + item) * 32 + lane;
            if (VS_STORE_OK(bp, DR_TOK, dst, 16)) __stcg(dst, v);
            __syncwarp();
            if (lane == 0 && VS_STORE_OK(bp, DR_TOK_SYNC, a.frag_flags + cta * 8 + item, 4)) st_release(a.frag_flags + cta * 8 + item, seq);
          } else {
          if (kk + 1 < p.kst) {
            const uint32_t total = (uint32_t)(p.tiles * p.kst);
#pragma unroll 1
            for (int c = cta + 1; c < ncta; ++c) {
              const uint32_t c0 = total * (uint32_t)c / (uint32_t)ncta, c1 = total * (uint32_t)(c + 1) / (uint32_t)ncta;
              if ((int)c0 >= (tile + 1) * p.kst) break;
              if (c0 == c1) continue;              // a CTA without work
              if (lane == 0) wait_count(a.frag_flags + c * 8 + item, seq, abort_flag);
              __syncwarp();
              const float4 u = __ldcg(reinterpret_cast<const float4*>(a.part) + ((size_t)c * ITEMS + item) * 32 + lane);
              v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
            }
          }
          finish_item<D, NT>(a, bp, l, kind, tile * MT + item / NT, item % NT, v, in, lane, rope_s, rsc_s, best_s);
          }
        }
        kk_begin = 0; kk = 0; ++tile;
      }
      if (normed && p.s0 < p.s1) rs_parity ^= 1u;
      if (kind == PH_LM) return;
      if (warp == 0 && kind == PH_QKV) TOK_STAMP(3, l);
      compute_bar();                                                   // every finisher's stores come before this point
      if (warp == 0 && kind == PH_QKV) TOK_STAMP(4, l);
      if (tid == 0 && VS_STORE_OK(bp, DR_TOK_SYNC, counter(a, l, kind), 4)) add_release(counter(a, l, kind), 1);
    };

    // ---- attention of layer l: unit = (token row, KV head, share of the keys) ------------------------------
    const int G = a.Hq / a.Hkv;
    const int kofs = 4 * (g >> 1) + (g & 1);       // S^T rows g and g + 8 are keys kofs and kofs + 2 of a 16-key tile
    struct Unit {
      int row, hkv, begin, end, fresh, hole, P, PB;     // keys begin .. end - 1; from `fresh` on the step's own; prefix ends at P, bank at PB
      size_t o_pre, o_bank, o_tail;                     // element offsets of the stream's and head's rows (bank and tail: of key 0)
    };
    auto make_unit = [&](int l, int u) {
      Unit x;
      const int split = u % a.nsplit, rh = u / a.nsplit;
      x.hkv = rh % a.Hkv; x.row = rh / a.Hkv;
      const int b = x.row / rps, tt = x.row - b * rps, sid = bp.entry[b].stream_id;
      const bool bank_full = a.M > 0 && bp.entry[b].count == a.M;
      int NB, TL;
      if (a.to_prefix) { x.P = bp.entry[b].prefix_len + tt + 1; NB = 0; TL = 0; }
      else { x.P = bp.entry[b].prefix_len; NB = (a.M == 0) ? 0 : (bank_full ? a.M + 1 : bp.entry[b].count); TL = bp.entry[b].text_len + tt + 1; }
      x.PB = x.P + NB;
      const int Lv = x.PB + TL;
      x.fresh = Lv - tt - 1;
      x.begin = Lv * split / a.nsplit; x.end = Lv * (split + 1) / a.nsplit;
      const size_t hoff = (size_t)sid * a.Hkv + x.hkv;
      x.o_pre = (size_t)l * a.ls_prefix + hoff * a.maxP * D;
      x.o_bank = (size_t)l * a.ls_bank + hoff * a.slots * D - (size_t)x.P * D;
      x.o_tail = (size_t)l * a.ls_tail + hoff * a.maxT * D - (size_t)x.PB * D;
      // the slot being refilled holds no carrier: fetched like any key, masked when the scores are formed
      x.hole = bank_full ? x.P + __ldcg(&a.meta[sid].free_slot) : -1;
      return x;
    };
    uint4 kr[2][KC], vr[4][VC];                    // a warp's 16 keys
    // late == false: the keys of earlier steps; late == true: the step's own (read past L1: written in this launch)
    auto load_tile = [&](const Unit& x, int v0, bool late) {
      auto row_of = [&](int v, const bf16* p, const bf16* bk, const bf16* t) {
        return reinterpret_cast<const uint4*>((v < x.P ? p + x.o_pre : (v < x.PB ? bk + x.o_bank : t + x.o_tail)) + (size_t)v * D);
      };
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int v = v0 + kofs + 2 * i;
        if (v < x.end && ((v >= x.fresh) == late)) {
          const uint4* kp = row_of(v, a.prefix_k, a.bank_k, a.tail_k);
#pragma unroll
          for (int c = 0; c < KC; ++c) kr[i][c] = __ldcg(kp + t4 + 4 * c);
        } else if (!late) {
#pragma unroll
          for (int c = 0; c < KC; ++c) kr[i][c] = make_uint4(0, 0, 0, 0);
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int v = v0 + 4 * t4 + r;
        if (v < x.end && ((v >= x.fresh) == late)) {
          const uint4* vp = row_of(v, a.prefix_v, a.bank_v, a.tail_v);
#pragma unroll
          for (int c = 0; c < VC; ++c) vr[r][c] = __ldcg(vp + g + 8 * c);
        } else if (!late) {
#pragma unroll
          for (int c = 0; c < VC; ++c) vr[r][c] = make_uint4(0, 0, 0, 0);
        }
      }
    };
    // `unit`: its first tile's stored keys are in kr and vr, or on their way (asked for ahead of the projection)
    auto attention_unit = [&](int l, int u, const Unit& unit) {
      const int row = unit.row, hkv = unit.hkv, begin = unit.begin, end = unit.end, fresh = unit.fresh, hole = unit.hole;
      const int rh = row * a.Hkv + hkv;
      const int n_tiles = (end - begin + kKeysPerTile - 1) / kKeysPerTile;
      float m[2] = {-INFINITY, -INFINITY}, ls[2] = {0.f, 0.f};               // heads 2 * t4 and 2 * t4 + 1
      float o[OT][4];
#pragma unroll
      for (int j = 0; j < OT; ++j) { o[j][0] = 0.f; o[j][1] = 0.f; o[j][2] = 0.f; o[j][3] = 0.f; }
#pragma unroll 1
      for (int ti = warp; ti == warp || ti < n_tiles; ti += kCW) {           // (every warp goes round once: the barriers)
        const int v0 = begin + ti * kKeysPerTile;
        if (ti != warp) {
          load_tile(unit, v0, false);
        } else {                                   // now the projection is needed: the query and the step's own keys
          if (warp == 0) TOK_STAMP(5, l);
          if (tid == 0) wait_count(counter(a, l, PH_QKV), ncta, abort_flag);
          compute_bar();
          if (warp == 0) TOK_STAMP(6, l);
        }
        if (v0 + kKeysPerTile > fresh) load_tile(unit, v0, true);
        if (ti == warp) {
#pragma unroll 1
          for (int i = tid; i < 2 * kHeads * (D / 8); i += kCT) {
            const int which = i / (kHeads * (D / 8)), r = i - which * (kHeads * (D / 8)), hd = r / (D / 8), c = r - hd * (D / 8);
            uint4 v = make_uint4(0, 0, 0, 0);
            if (hd < G) v = __ldcg(reinterpret_cast<const uint4*>((which ? a.q_lo : a.q) + ((size_t)row * a.Hq + (size_t)hkv * G + hd) * D) + c);
            q_s[which][hd][c ^ ((hd & 1) << 2)] = v;
          }
          compute_bar();
          if (warp == 0) TOK_STAMP(7, l);
          if (ti >= n_tiles) break;
        }
        float s[4] = {0.f, 0.f, 0.f, 0.f}, sl[4] = {0.f, 0.f, 0.f, 0.f};     // high and low query halves
#pragma unroll
        for (int c = 0; c < KC; ++c) {
          const int ch = (t4 + 4 * c) ^ ((g & 1) << 2);
          const uint4 qh = q_s[0][g][ch], ql = q_s[1][g][ch];
          mma_bf16(s, kr[0][c].x, kr[1][c].x, kr[0][c].y, kr[1][c].y, qh.x, qh.y);
          mma_bf16(sl, kr[0][c].x, kr[1][c].x, kr[0][c].y, kr[1][c].y, ql.x, ql.y);
          mma_bf16(s, kr[0][c].z, kr[1][c].z, kr[0][c].w, kr[1][c].w, qh.z, qh.w);
          mma_bf16(sl, kr[0][c].z, kr[1][c].z, kr[0][c].w, kr[1][c].w, ql.z, ql.w);
        }
        const int va = v0 + kofs, vb = va + 2;
        const bool ina = va < end && va != hole, inb = vb < end && vb != hole;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          s[e] = ina ? (s[e] + sl[e]) * a.scale_log2e : -INFINITY;
          s[2 + e] = inb ? (s[2 + e] + sl[2 + e]) * a.scale_log2e : -INFINITY;
          float mx = fmaxf(s[e], s[2 + e]);
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
          const float mn = fmaxf(m[e], mx);
          const float mu = (mn == -INFINITY) ? 0.f : mn;                     // masked keys alone so far
          const float sc = exp2f(m[e] - mu);
          s[e] = exp2f(s[e] - mu);
          s[2 + e] = exp2f(s[2 + e] - mu);
          ls[e] = ls[e] * sc + (s[e] + s[2 + e]);
          m[e] = mn;
#pragma unroll
          for (int j = 0; j < OT; ++j) { o[j][e] *= sc; o[j][2 + e] *= sc; }
        }
        const uint32_t pa = pack2(s[0], s[1]), pb = pack2(s[2], s[3]);
        const float2 fa = unpack2(pa), fb = unpack2(pb);
        const uint32_t ph0 = transpose_8x8(pa), ph1 = transpose_8x8(pb);
        const uint32_t pl0 = transpose_8x8(pack2(s[0] - fa.x, s[1] - fa.y)), pl1 = transpose_8x8(pack2(s[2] - fb.x, s[3] - fb.y));
#pragma unroll
        for (int j = 0; j < OT; ++j) {
          // tile j: row g = dim 8 g + j, row g + 8 = dim 64 + 8 g + j (D = 128) or 8 g + 4 + j (D = 64)
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
      if (warp == 0) TOK_STAMP(8, l);
      // warps -> CTA
      // (what the outputs of this thread will be added to and multiplied with, in case this CTA finishes the row)
      const int idx = 4 * tid, hd = idx / D, dim = idx - hd * D;               // outputs 4 tid .. + 3 of the group, all of one head
      const bool mine = hd < G;
      const size_t off = ((size_t)row * a.Hq + (size_t)hkv * G) * D + idx;
      uint2 hr = make_uint2(0u, 0u), gw = make_uint2(0u, 0u);
      const bf16* gain = (a.use_rmsnorm && !a.full && l + 1 < a.L) ? a.layers[l + 1].gain : nullptr;
      if (mine && a.residual && !a.full) {
        hr = __ldcg(reinterpret_cast<const uint2*>(layer_input(a, l) + off));
        if (gain != nullptr) { const uint32_t* gp = reinterpret_cast<const uint32_t*>(gain + (size_t)hkv * G * D + idx); gw = make_uint2(gp[0], gp[1]); }   // (4-byte aligned, like every reader of a gain on this path)
      }
      const int n_used = min(n_tiles, kCW);
      if (warp < n_used) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
#pragma unroll
          for (int off = 4; off < 32; off <<= 1) ls[e] += __shfl_xor_sync(0xffffffffu, ls[e], off);
          if (g == 0) st_ml[warp][2 * t4 + e] = make_float2(m[e], ls[e]);
          float4* dst = reinterpret_cast<float4*>(st_o) + (warp * kHeads + 2 * t4 + e) * (D / 4);
#pragma unroll
          for (int hh = 0; hh < 2; ++hh)
#pragma unroll
            for (int j = 0; j < OT; j += 4)
              dst[merge_unit(2 * t4 + e, (D == 128 ? hh * 16 + j / 4 : hh) + 2 * g)] =
                  make_float4(o[j][2 * hh + e], o[j + 1][2 * hh + e], o[j + 2][2 * hh + e], o[j + 3][2 * hh + e]);
        }
      }
      compute_bar();
      float M = -INFINITY, Ls = 0.f;
      float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
      if (mine) {
#pragma unroll
        for (int w = 0; w < kCW; ++w) if (w < n_used) M = fmaxf(M, st_ml[w][hd].x);
#pragma unroll
        for (int w = 0; w < kCW; ++w) {
          if (w < n_used) {
            const float2 ml = st_ml[w][hd];
            const float wt = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - M);
            const float4 v = reinterpret_cast<const float4*>(st_o)[(w * kHeads + hd) * (D / 4) + merge_unit(hd, dim / 4)];
            Ls = fmaf(ml.y, wt, Ls);
            O.x = fmaf(v.x, wt, O.x); O.y = fmaf(v.y, wt, O.y); O.z = fmaf(v.z, wt, O.z); O.w = fmaf(v.w, wt, O.w);
          }
        }
      }
      if (warp == 0) TOK_STAMP(9, l);
      if (a.nsplit > 1) {
        // the last share of this row and KV head to arrive combines them all, in order
        float* pp = a.att_part + (size_t)u * (kHeads * D + 2 * kHeads);
        if (mine) {
          if (VS_STORE_OK(bp, DR_TOK, pp + idx, 16)) __stcg(reinterpret_cast<float4*>(pp + idx), O);
          if (dim == 0 && VS_STORE_OK(bp, DR_TOK, pp + kHeads * D + 2 * hd, 8)) __stcg(reinterpret_cast<float2*>(pp + kHeads * D + 2 * hd), make_float2(M, Ls));
        }
        compute_bar();
        if (tid == 0) {
          const int t = VS_STORE_OK(bp, DR_TOK_SYNC, a.tickets + rh, 4) ? add_acq_rel(a.tickets + rh, 1) : 0;
          if (t == a.nsplit - 1) a.tickets[rh] = 0;                          // (the next layer's units start after this one's)
          *bcast = t;
        }
        compute_bar();
        if (warp == 0) TOK_STAMP(10, l);
        if (*bcast != a.nsplit - 1) return;
        if (mine) {
          const float* p0 = a.att_part + (size_t)rh * a.nsplit * (kHeads * D + 2 * kHeads);
          M = -INFINITY; Ls = 0.f; O = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
          for (int s0 = 0; s0 < a.nsplit; s0 += 4) {                           // four shares' loads in flight
            float2 ml[4];
            float4 v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float* ps = p0 + (size_t)min(s0 + j, a.nsplit - 1) * (kHeads * D + 2 * kHeads);
              ml[j] = __ldcg(reinterpret_cast<const float2*>(ps + kHeads * D + 2 * hd));
              v[j] = __ldcg(reinterpret_cast<const float4*>(ps + idx));
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              if (s0 + j >= a.nsplit || ml[j].x == -INFINITY) continue;
              const float Mn = fmaxf(M, ml[j].x), w0 = exp2f(M - Mn), w1 = exp2f(ml[j].x - Mn);     // (exp2f(-inf) = 0)
              M = Mn;
              Ls = Ls * w0 + ml[j].y * w1;
              O.x = O.x * w0 + v[j].x * w1; O.y = O.y * w0 + v[j].y * w1; O.z = O.z * w0 + v[j].z * w1; O.w = O.w * w0 + v[j].w * w1;
            }
          }
        }
      }
      if (warp == 0) TOK_STAMP(11, l);
      float sq = 0.f;
      if (mine) {
        const float inv = (Ls > 0.f) ? 1.f / Ls : 0.f;
        const float4 v = make_float4(O.x * inv, O.y * inv, O.z * inv, O.w * inv);
        if (a.full) {
          if (VS_STORE_OK(bp, DR_OBUF, a.attn_rows + off, 8)) *reinterpret_cast<uint2*>(a.attn_rows + off) = make_uint2(pack2(v.x, v.y), pack2(v.z, v.w));
        } else {
          const bool last = l + 1 == a.L;
          if (last) {
            if (a.out_fp32) *reinterpret_cast<float4*>(static_cast<float*>(a.out) + off) = v;
            else *reinterpret_cast<uint2*>(static_cast<bf16*>(a.out) + off) = make_uint2(pack2(v.x, v.y), pack2(v.z, v.w));
          }
          if (a.residual) {
            const float2 h0 = unpack2(hr.x), h1 = unpack2(hr.y);
            const uint2 hw = make_uint2(pack2(h0.x + v.x, h0.y + v.y), pack2(h1.x + v.z, h1.y + v.w));
            bf16* ho = a.hbuf[l & 1] + off;
            if (VS_STORE_OK(bp, (l & 1) ? DR_HBUF1 : DR_HBUF0, ho, 8)) *reinterpret_cast<uint2*>(ho) = hw;
            const float2 s0 = unpack2(hw.x), s1 = unpack2(hw.y);
            sq = (s0.x * s0.x + s0.y * s0.y) + (s1.x * s1.x + s1.y * s1.y);
            if (gain != nullptr) {
              const float2 g0 = unpack2(gw.x), g1 = unpack2(gw.y);
              if (VS_STORE_OK(bp, DR_XN, a.xn + off, 8))
                *reinterpret_cast<uint2*>(a.xn + off) = make_uint2(pack2(s0.x * g0.x, s0.y * g0.y), pack2(s1.x * g1.x, s1.y * g1.y));
            }
          }
        }
      }
      if (a.use_rmsnorm && !a.full) {
        // this head group's part of the row's sum of squares, in a fixed order
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
        if (lane == 0) sum_s[warp] = sq;
      }
      compute_bar();
      if (tid == 0) {
        if (a.use_rmsnorm && !a.full) {
          float t = 0.f;
#pragma unroll
          for (int i = 0; i < kCW; ++i) t += sum_s[i];
          float* sp = a.ss + (size_t)row * a.ss_cap + hkv;
          if (VS_STORE_OK(bp, DR_TOK, sp, 4)) *sp = t;
        }
        if (VS_STORE_OK(bp, DR_TOK_SYNC, counter(a, l, PH_ATT), 4)) add_release(counter(a, l, PH_ATT), 1);
      }
      if (warp == 0) TOK_STAMP(12, l);
    };

    const int units = a.vocab > 0 ? 0 : rows * a.Hkv * a.nsplit;
    Unit unit = {};
    for_phases([&](int l, int kind) {
      if (kind != PH_ATT) {
        if (kind == PH_QKV && cta < units) { unit = make_unit(l, cta); load_tile(unit, unit.begin + warp * kKeysPerTile, false); }
        weight_phase(l, kind);
      } else {
#pragma unroll 1
        for (int u = cta; u < units; u += ncta) {
          if (u != cta) { unit = make_unit(l, u); load_tile(unit, unit.begin + warp * kKeysPerTile, false); }
          attention_unit(l, u, unit);
        }
      }
    });
    if (a.vocab > 0) {
      compute_bar();
      if (tid < rows && a.next_token != nullptr && best_s[tid] != 0ull && VS_STORE_OK(bp, DR_LM_KEYS, a.lm_keys + tid, 8)) atomicMax(a.lm_keys + tid, best_s[tid]);
    }
  }

  // ---- the last CTA to finish leaves the counters as it found them (and turns the greedy keys into tokens) ----
  __syncthreads();
  if (tid == 0) {
    if (*abort_flag) atomicExch(a.status, VS_ERR_DEVICE_TIMEOUT);
    __threadfence();
    *bcast = VS_STORE_OK(bp, DR_TOK_SYNC, a.done, 4) ? atomicAdd(a.done, 1) : 0;
    __threadfence();
  }
  __syncthreads();
  if (*bcast == ncta - 1) {
    const int n_counters = 1 + 5 * a.L;
#pragma unroll 1
    for (int i = tid; i < n_counters; i += kThreads)
      if (VS_STORE_OK(bp, DR_TOK_SYNC, a.counters + (size_t)i * kCntStride, 4)) a.counters[(size_t)i * kCntStride] = 0;
#pragma unroll 1
    for (int i = tid; i < ncta * 8; i += kThreads)
      if (VS_STORE_OK(bp, DR_TOK_SYNC, a.frag_flags + i, 4)) a.frag_flags[i] = 0;
    if (tid == 0) *a.done = 0;
    if (a.vocab > 0 && a.next_token != nullptr && tid < rows) {
      const unsigned long long k = atomicExch(a.lm_keys + tid, 0ull);
      a.next_token[tid] = (k == 0ull) ? 0 : 0x7fffffff - (int)(uint32_t)(k & 0xffffffffull);
    }
  }
}

}  // namespace

namespace {
constexpr size_t kMaxDynSmem = 227 * 1024;
constexpr size_t kCtlBytes = 6144;
template <int D, int NT>
struct TokShape {
  static constexpr size_t kRS = (size_t)KS * 2 + 64, kW = (size_t)16 * MT * KS * 2;   // bytes of a token row and of the weights in a stage
  static constexpr size_t kRed = (size_t)kCW * MT * NT * 512, kO = (size_t)kCW * kHeads * D * 4;
  static constexpr size_t kFixed = (kRed > kO ? kRed : kO) + (size_t)NT * 8 * (D / 2) * 8 + kCtlBytes;
};
template <int D, int NT>
cudaError_t launch_shape(TokArgs a, const BatchParams& bp, int n_sms, cudaStream_t st) {
  using S = TokShape<D, NT>;
  const size_t stage = (S::kW + a.rows * S::kRS + 1023) / 1024 * 1024;     // the swizzle wants 1024-byte boundaries
  int stages = (int)((kMaxDynSmem - 1024 - S::kFixed) / stage);
  if (stages > kMaxStages) stages = kMaxStages;
  const long long widest = (long long)(a.vocab > 0 ? a.vocab : 2 * a.d_ff > (a.Hq + 2 * a.Hkv) * a.D ? 2 * a.d_ff : (a.Hq + 2 * a.Hkv) * a.D);
  const long long deepest = a.d_ff > a.d ? a.d_ff : a.d;
  if (stages < 2 || widest / 16 * (deepest / 256 + 1) * n_sms >= (1ll << 31)) return cudaErrorInvalidValue;
  a.stages = stages;
  a.ring_bytes = (uint32_t)(stages * stage);
  return launch_pdl(token_kernel<D, NT>, dim3(n_sms), dim3(kThreads), 1024 + a.ring_bytes + S::kFixed, st, a, bp);
}
template <int D>
cudaError_t init_head() {
  cudaError_t e = cudaSuccess;
  auto fits = [&](auto kernel) {       // one CTA of it on an SM
    int n = 0;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxDynSmem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kThreads, kMaxDynSmem);
    if (e == cudaSuccess && n < 1) e = cudaErrorInvalidConfiguration;
  };
  fits(token_kernel<D, 1>);
  fits(token_kernel<D, 2>);
  return e;
}
}  // namespace

cudaError_t token_step_init() {
  const cudaError_t e = init_head<128>();
  return e == cudaSuccess ? init_head<64>() : e;
}

int token_step_split(int max_keys, int rows, int n_kv_heads, int n_sms) {
  // eight warps take 128 keys in one go; every share a CTA of its own
  const int room = n_sms / (rows * n_kv_heads), wanted = (max_keys + 127) / 128;
  return wanted < 1 || room < 1 ? 1 : (wanted < room ? wanted : room);
}

cudaError_t launch_token_step(const TokArgs& a, const BatchParams& bp, int n_sms, cudaStream_t st) {
  if (a.rows < 1 || a.rows > TOK_MAX_ROWS || n_sms > TOK_MAX_CTAS) return cudaErrorInvalidValue;
  const int D = a.vocab > 0 ? 128 : a.D;
  if (D == 128) {
    if (a.rows <= 8) return launch_shape<128, 1>(a, bp, n_sms, st);
    return launch_shape<128, 2>(a, bp, n_sms, st);
  }
  if (D != 64) return cudaErrorInvalidValue;
  if (a.rows <= 8) return launch_shape<64, 1>(a, bp, n_sms, st);
  return launch_shape<64, 2>(a, bp, n_sms, st);
}

}  // namespace vs
