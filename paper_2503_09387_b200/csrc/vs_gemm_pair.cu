// The linear layers of a step of many token rows (a chunk of frames, a batch of streams) or of many output tiles (gate and up,
// the vocabulary projection): tcgen05.mma on CTA pairs, persistent, the epilogue of one tile under the main loop of the next.
//
// As in vs_gemm_tcgen05.cu the *features* take the MMA's M axis and the *tokens* its N axis.  A CTA pair (cta_group::2) shares
// one tile of 256 weight rows x tile_n tokens: each CTA stages its own 128 weight rows and *half* of the token columns, the
// tensor cores of both read both halves.  What bounds the main loop is then the MMA rate, not the L2 -> SM traffic:
// (128 + tile_n / 2) * 128 bytes per CTA and 64 of K, where a CTA alone needs (128 + tile_n) for half the weight rows.
// Tiles are dealt to persistent pairs, one CTA per SM; two accumulators in tensor memory (2 x tile_n columns) let the
// epilogue of one tile run under the main loop of the next.
// (One CTA per tile of 256 rows, epilogue after the main loop: 0.88 PFLOP/s on the 2720 rows of a 16-frame chunk through full
// decoder layers; this kernel 1.2, power-capped clocks included.)
//
// The epilogue (16 warps; with 8, two tokens a thread and chunk, five streams of 121 rows took 259 us for 6 layers, now 250, a full-model
// frame 4.11 and 4.09 ms) takes 32 tokens at a time through shared memory, so that a thread finishes both elements of four
// rotation pairs of a token and stores 8-byte pieces.
// Per CTA 18 warps.  Warp 0 lane 0 = TMA loader (weights are constant: a launch's first stages of them are requested before the
// wait on the stream's earlier kernels), warp 1 = TMEM allocator, its lane 0 in the pair's first CTA the MMA issuer, warps 2..17
// the epilogue (tcgen05.ld of the 32-lane quarter that warp % 4 allows).  Every wait is bounded; on expiry the CTA raises an
// abort flag, records VS_ERR_DEVICE_TIMEOUT, lets in-flight copies land, frees its tensor memory and exits.
// No copy is multicast: the halves each CTA loads are its own.
#include "vs_gemm_common.cuh"

namespace vs {

namespace {

using namespace gemm;

constexpr int kEpiWarps = 16;
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kThreads = 64 + kEpiThreads;
constexpr int kChunk = 32;                                      // tokens the epilogue stages at a time
constexpr int kPitch = GEMM_BLOCK_M + 4;                        // floats from token to token in the staging buffer
constexpr int kStagingBytes = 2 * kChunk * kPitch * 4;          // two buffers

// a load of one CTA of the pair: into its own shared memory, its bytes counted on the first CTA's barrier
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {      // `bar`: an address of the cluster's shared memory
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Instruction descriptor, kind::f16, both CTAs of a pair: D = fp32, A = B = bf16, both K-major, M = 256, N = n.
__device__ __forceinline__ uint32_t make_idesc_pair(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)((2 * GEMM_BLOCK_M) >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.u32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}
// arrives on the barrier at this offset in both CTAs once the MMAs issued so far have completed
__device__ __forceinline__ void umma_commit_pair(uint32_t bar, uint32_t elected) {
  asm volatile("{\n\t.reg .pred e;\n\tsetp.ne.u32 e, %2, 0;\n\t"
               "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}"
               ::"r"(bar), "h"((uint16_t)3), "r"(elected) : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}

struct PairParams {
  ProjectionOut o;
  int* status;
  int rows, E_out, tile_n, m_tiles, n_tiles, kblocks, stages, acc_cols;
  float inv_d;                  // 1 / K
};
struct Tile { int m0, n0; };

// The epilogue warps of one CTA: every tile's 128 x tile_n accumulator, in the order the issuer fills them.
template <int kFin, typename TileFn>
__device__ __forceinline__ void epilogue_role(const PairParams& p, const BatchParams& bp, uint32_t tmem, float* staging, float* rsc_all,
                                              volatile int* abort_flag, uint32_t acc_full0, uint32_t acc_empty0, int warp, int lane, int pair,
                                              int n_pairs, int n_items, TileFn tile) {
  const int te = (int)threadIdx.x - 64;                  // 0 .. 511
  const int quarter = warp & 3, eighth = (warp - 2) >> 2;  // TMEM lanes this warp may read; which 8 tokens of a chunk
  auto epi_bar = [] { asm volatile("bar.sync 1, 512;" ::: "memory"); };
  static_assert(kEpiThreads == 512 && kChunk == 32, "the named barrier above counts 512 threads, half a warp to a token");
  int j = 0, buf = 0;
#pragma unroll 1
  for (int i = pair; i < n_items; i += n_pairs, ++j) {
    const Tile t = tile(i);
    const int acc = j & 1;
    const uint32_t tm = tmem + (uint32_t)(acc * p.acc_cols) + ((uint32_t)(quarter * 32) << 16);
    float* rsc_s = rsc_all + acc * 256;
    const int n_tok = min(p.tile_n, p.rows - t.n0), n_blk = (n_tok + 15) >> 4;   // tokens of the tile that exist, in blocks of 16
    const Place pl = place_of(p.o, p.E_out, t.m0, te);
    float bb1[4], bb2[4];
    bias_of(p.o, pl, t.m0, bb1, bb2);
    // RMSNorm: the row scales of the tile's tokens, worked out while the main loop runs
    if (p.o.row_ss != nullptr) {
      for (int k = te; k < n_tok; k += kEpiThreads) {
        const float* src = p.o.row_ss + (size_t)(t.n0 + k) * p.o.ss_parts;
        float tot = 0.f;
        for (int q = 0; q < p.o.ss_parts; ++q) tot += src[q];
        rsc_s[k] = rsqrtf(tot * p.inv_d + p.o.norm_eps);
      }
    }
    const bool ok = __all_sync(0xffffffffu, mbar_wait(acc_full0 + 8u * (uint32_t)acc, (uint32_t)(j >> 1) & 1u, abort_flag));
    tcgen05_fence_after();
    VS_STAMP_BY(bp, 1, 2, 64);        // accumulator complete
#pragma unroll 1
    for (int c0 = 0; c0 < n_blk; c0 += 2) {              // 32 tokens at a time, two staging buffers
      const int tok = te >> 4, row = t.n0 + c0 * 16 + tok;
      const bool mine = pl.on && c0 + (tok >> 4) < n_blk && row < p.rows;
      FinishIn in;
      if (mine) in = finish_in<kFin>(p.o, pl, p.E_out, t.m0, row);
      float* st = staging + buf * (kChunk * kPitch);
      buf ^= 1;
      if (c0 + (eighth >> 1) < n_blk && ok) {
        uint32_t r[8];
        tmem_ld8(tm + (uint32_t)(c0 * 16 + eighth * 8), r);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        float* d = st + (8 * eighth) * kPitch + quarter * 32 + lane;
#pragma unroll
        for (int k = 0; k < 8; ++k) d[k * kPitch] = __uint_as_float(r[k]);
      }
      if (c0 + 2 >= n_blk) {
        // this warp has read its last part of the accumulator: once all have, the issuer may fill it again
        tcgen05_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_shared_rank(acc_empty0 + 8u * (uint32_t)acc, 0u));
      }
      // (one barrier a chunk: the buffer written next is the one read a chunk ago, which every thread has left by the barrier)
      epi_bar();
      if (mine && !*abort_flag) {
        const float4 a1 = *reinterpret_cast<const float4*>(st + tok * kPitch + pl.f1);
        const float4 a2 = *reinterpret_cast<const float4*>(st + tok * kPitch + pl.f2);
        // RMSNorm's row scale commutes with the projection: applied here, in fp32
        finish_row<kFin>(p.o, bp, pl, p.E_out, t.m0, row, a1, a2, p.o.row_ss != nullptr ? rsc_s[c0 * 16 + tok] : 1.f, bb1, bb2, in, te);
      }
    }
  }
}

template <int kFin>
__global__ void __launch_bounds__(kThreads, 1) __cluster_dims__(2, 1, 1)
pair_gemm_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
                 const __grid_constant__ CUtensorMap tm_w2, const __grid_constant__ PairParams p, const __grid_constant__ BatchParams bp) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // carve: [stages][A 16 KiB | B tile_n / 2 rows] | staging | row scales [2][256] | full, empty [stages], acc_full, acc_empty [2] |
  // tmem slot | abort
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t stage_bytes = kStageABytes + (uint32_t)p.tile_n * 64u;
  float* staging = reinterpret_cast<float*>(gen_base + (size_t)p.stages * stage_bytes);
  float* rsc_s = reinterpret_cast<float*>(gen_base + (size_t)p.stages * stage_bytes + kStagingBytes);
  uint8_t* ctl = reinterpret_cast<uint8_t*>(rsc_s + 2 * 256);
  const uint32_t bars = smem_u32(ctl);
  auto full_bar = [&](int s) { return bars + 8u * (uint32_t)s; };
  auto empty_bar = [&](int s) { return bars + 8u * (uint32_t)(p.stages + s); };
  auto acc_full = [&](int b) { return bars + 8u * (uint32_t)(2 * p.stages + b); };
  auto acc_empty = [&](int b) { return bars + 8u * (uint32_t)(2 * p.stages + 2 + b); };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(ctl + 16 * p.stages + 32);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(ctl + 16 * p.stages + 36);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)blockIdx.x & 1, pair = (int)blockIdx.x >> 1, n_pairs = (int)gridDim.x >> 1;
  const int n_items = p.m_tiles * p.n_tiles;
  // token tiles fastest: pairs side by side read the same weights at a time
  auto tile = [&](int i) {
    Tile t;
    const int mt = i / p.n_tiles;
    t.m0 = (mt * 2 + rank) * GEMM_BLOCK_M;
    t.n0 = (i - mt * p.n_tiles) * p.tile_n;
    return t;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), 2 * kEpiWarps); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_w) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_x) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"((uint32_t)(2 * p.acc_cols)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tcgen05_fence_before();
  __syncthreads();
  cluster_sync_all();               // both CTAs' barriers exist
  tcgen05_fence_after();
  const uint32_t tmem = *tmem_slot;
  VS_STAMP(bp, 1, 0);

  if (warp == 0) {
    // ---- TMA loader (each CTA: its 128 weight rows, its half of the tokens) --------------------------
    if (lane == 0) {
      auto load_w = [&](const Tile& t, int kb, int s) {
        const uint32_t dst = base + (uint32_t)s * stage_bytes, bar = map_shared_rank(full_bar(s), 0u);
        if (rank == 0) mbar_arrive_expect_tx(full_bar(s), 2u * stage_bytes);      // the bytes of both CTAs
        if constexpr (kFin == FIN_SWIGLU) {
          // a 128-row tile = 64 rows of the gate matrix, then the same 64 rows of the up matrix
          tma_load_2d_pair(dst, &tm_w, kb * GEMM_BLOCK_K, t.m0 >> 1, bar);
          tma_load_2d_pair(dst + kStageABytes / 2, &tm_w2, kb * GEMM_BLOCK_K, t.m0 >> 1, bar);
        } else {
          tma_load_2d_pair(dst, &tm_w, kb * GEMM_BLOCK_K, t.m0, bar);
        }
      };
      auto load_x = [&](const Tile& t, int kb, int s) {
        tma_load_2d_pair(base + (uint32_t)s * stage_bytes + kStageABytes, &tm_x, kb * GEMM_BLOCK_K, t.n0 + rank * (p.tile_n >> 1),
                         map_shared_rank(full_bar(s), 0u));
      };
      // the first stages' weights, then the wait for whoever wrote the token rows
      int ahead = 0;
      if (pair < n_items) {
        const Tile t = tile(pair);
        ahead = min(p.stages, p.kblocks);
        for (int i = 0; i < ahead; ++i) load_w(t, i, i);
      }
      pdl_wait();
      pdl_launch_dependents();
      VS_STAMP(bp, 1, 1);
      int s = 0;
      uint32_t par = 1;
      bool ok = true;
      for (int i = pair; i < n_items && ok; i += n_pairs) {
        const Tile t = tile(i);
        for (int kb = 0; kb < p.kblocks; ++kb) {
          if (ahead > 0) {
            --ahead;
            load_x(t, kb, s);
          } else {
            if (!mbar_wait(empty_bar(s), par, abort_flag)) { ok = false; break; }
            load_w(t, kb, s);
            load_x(t, kb, s);
          }
          if (++s == p.stages) { s = 0; par ^= 1u; }
        }
      }
      if (*abort_flag) {
        // let the copies in flight land before the shared memory is given up (their barrier may be the other CTA's)
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 2000000ull) __nanosleep(1000);
      }
    } else {
      pdl_wait();
    }
  } else if (warp == 1) {
    pdl_wait();
    if (rank == 0) {
      // ---- MMA issuer: one lane for both CTAs ---------------------------------------------------------
      const uint32_t idesc = make_idesc_pair(p.tile_n), elected = elect_lane();
      int s = 0, j = 0;
      uint32_t par = 0;
      bool ok = true;
      for (int i = pair; i < n_items && ok; i += n_pairs, ++j) {
        const uint32_t acc = tmem + (uint32_t)((j & 1) * p.acc_cols);
        ok = __all_sync(0xffffffffu, mbar_wait(acc_empty(j & 1), ((uint32_t)(j >> 1) & 1u) ^ 1u, abort_flag));
        for (int kb = 0; kb < p.kblocks && ok; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait(full_bar(s), par, abort_flag));
          if (!ok) break;
          tcgen05_fence_after();
          const uint64_t da = make_smem_desc(base + (uint32_t)s * stage_bytes), db = make_smem_desc(base + (uint32_t)s * stage_bytes + kStageABytes);
#pragma unroll
          for (int k = 0; k < GEMM_BLOCK_K / 16; ++k)      // 16 bf16 = 32 bytes further along K inside the 128-byte swizzle row
            umma_bf16_pair(acc, da + 2u * k, db + 2u * k, idesc, (uint32_t)((kb | k) != 0), elected);
          umma_commit_pair(empty_bar(s), elected);         // frees the stage in both CTAs once these MMAs have read it
          if (++s == p.stages) { s = 0; par ^= 1u; }
        }
        if (ok) umma_commit_pair(acc_full(j & 1), elected);
      }
    }
  } else {
    pdl_wait();
    epilogue_role<kFin>(p, bp, tmem, staging, rsc_s, abort_flag, acc_full(0), acc_empty(0), warp, lane, pair, n_pairs, n_items, tile);
  }

  tcgen05_fence_before();
  __syncthreads();
  cluster_sync_all();               // neither CTA's shared or tensor memory goes away while the pair's MMAs may read it
  if (warp == 1) {
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(2 * p.acc_cols)) : "memory");
  }
  if (threadIdx.x == 0 && *abort_flag) atomicExch(p.status, VS_ERR_DEVICE_TIMEOUT);
  VS_STAMP(bp, 1, 15);
}

size_t fixed_smem(int stages) { return 1024 + kStagingBytes + 2 * 256 * 4 + 16 * (size_t)stages + 64; }

using Kernel = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const PairParams, const BatchParams);
Kernel kernel_of(int mode) {
  switch (mode) {
    case FIN_RESIDUAL: return pair_gemm_kernel<FIN_RESIDUAL>;
    case FIN_SWIGLU: return pair_gemm_kernel<FIN_SWIGLU>;
    case FIN_LOGITS: return pair_gemm_kernel<FIN_LOGITS>;
    default: return pair_gemm_kernel<FIN_PROJECT>;
  }
}

}  // namespace

cudaError_t pair_gemm_init() {
  for (int mode : {(int)FIN_PROJECT, (int)FIN_RESIDUAL, (int)FIN_SWIGLU, (int)FIN_LOGITS}) {
    const cudaError_t e = cudaFuncSetAttribute((const void*)kernel_of(mode), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// CTA pairs of this kernel that can be resident at once on the current device; 0 if the query fails
int pair_gemm_max_pairs() {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * 128); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = kMaxDynSmem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  int pairs = 0;
  if (cudaOccupancyMaxActiveClusters(&pairs, kernel_of(FIN_PROJECT), &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  return pairs;
}

cudaError_t launch_pair_gemm(const GemmArgs& a, int max_pairs, const BatchParams& bp, cudaStream_t st) {
  PairParams p;
  p.o = a.out;
  p.status = a.status;
  p.rows = a.rows;
  p.E_out = a.E_out;
  p.tile_n = a.tile_n;
  p.inv_d = 1.f / (float)a.d;
  p.kblocks = a.d / GEMM_BLOCK_K;
  p.n_tiles = a.n_tiles;
  p.m_tiles = (a.E_out + 2 * GEMM_BLOCK_M - 1) / (2 * GEMM_BLOCK_M);
  if (a.tile_n < 16 || a.tile_n > 256 || (a.tile_n & 15) || 128 % a.out.D != 0 || max_pairs < 1) return cudaErrorInvalidValue;
  if (a.out.mode < 4 && a.out.rope == nullptr) return cudaErrorInvalidValue;
  const int stage_bytes = kStageABytes + a.tile_n * 64;
  int stages = (int)((kMaxDynSmem - fixed_smem(12)) / stage_bytes);
  if (stages > 12) stages = 12;
  p.stages = stages;
  int cols = 32;
  while (cols < a.tile_n) cols <<= 1;
  p.acc_cols = cols;
  const int items = p.m_tiles * p.n_tiles, pairs = items < max_pairs ? items : max_pairs;
  return launch_pdl(kernel_of(a.out.mode), dim3(2 * pairs), dim3(kThreads), (size_t)stages * stage_bytes + fixed_smem(stages), st, a.tm_w, a.tm_x, a.tm_w2, p, bp);
}

}  // namespace vs
