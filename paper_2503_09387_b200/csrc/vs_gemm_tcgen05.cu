// QKV projection (Eq. 1: Q = X W_Q, K = X W_K, V = X W_V) on the 5th-generation tensor
// cores: tcgen05.mma with the accumulator in tensor memory, operands staged in shared
// memory by TMA, one elected lane issuing the MMAs.
//
// Orientation.  A frame brings only N + 1 (<= 256) token rows but E_out = (Hq + 2 Hkv) D
// output features (4608 at the Qwen2-7B shape), so the *features* take the MMA's M axis
// (128 weight rows per accumulator, read K-major straight from the caller's [E_out, d] matrix)
// and the *tokens* take the MMA's N axis (any multiple of 16 up to 256: 170 tokens cost 176
// columns, 3.5 % padding instead of 33 % with 128-row token tiles).
//
// This kernel takes the launches of few rows (a frame, a short text step), whose output tiles alone do not fill the GPU;
// vs_gemm_pair.cu the others.  The reduction dimension d is split over `ksplit` CTAs so that m_tiles * n_tiles * ksplit
// comes close to the 148 SMs.  The tile's tokens, in blocks of 16, are dealt to the ksplit CTAs: every CTA stores
// the blocks it does not own of its fp32 partial accumulator to an exchange buffer in global memory (it stays in L2),
// counts itself in on the owners' flags, and an owner, once its flag shows ksplit - 1 arrivals, adds the
// peers' partials to its own.  All CTAs of the grid are resident at once (the launch checks
// it), so the wait on the flag ends; it is bounded like every other wait.
//
// The epilogue adds the bias, applies RoPE (a 128-row tile holds whole heads, so both elements
// of a rotation pair are at hand), writes Q as a bf16 hi + lo pair and K, V as bf16, and
// persists what the method keeps: the carrier row's K/V goes straight into the bank's free slot
// (Section 3.2: only the carrier keeps its K/V), text rows are appended to the prefix or to the
// turn's tail.
//
// Per CTA: 6, 10 or 18 warps.  Warp 0 lane 0 = TMA producer, warp 1 = TMEM allocator + MMA issuer
// (lane 0), warps 2.. = epilogue, 4, 8 or 16 of them (tcgen05.ld of the 32-lane quarter that
// warp % 4 allows; with 16, four warps per quarter take every fourth block of 16 columns).
// Every mbarrier wait is bounded; on expiry the CTA raises an abort flag, records
// VS_ERR_DEVICE_TIMEOUT, lets in-flight copies land, frees its tensor memory and exits.
#include "vs_gemm_common.cuh"

namespace vs {

namespace {

using namespace gemm;

constexpr int kMaxEpiWarps = 16;                 // 4 per scheduler: the epilogue is bound by instruction latency
constexpr int kMaxThreads = 64 + 32 * kMaxEpiWarps;
// Up to 16 rows without a table: ten warps of 80 registers and six stages, so that a CTA of the decode attention (eight warps of 128
// registers, 106 KB) fits beside this one and has its first keys when the projection is done.  (Sixteen finishing warps of 96, eight stages:
// 16 streams of 1150 keys 26.6 us, 25.7 this way.)
constexpr int kFewBound = 768, kFewWarps = 8, kFewStages = 6;   // (threads that would fill the register file at 80 each)
// The same beside the prefill attention (ten warps of 96 registers, 113 KB): whether a projection of 17 to 48 rows, or the W_o behind the
// attention, leaves room for one of its CTAs (leaves_room_for_attention), which then has its set-up and first keys behind it when the
// projection is done, as this block has its first weights when the attention is.  The price is depth, five stages of weights for eight.
// Registers: its ten warps of at most 96 take no more than half of the register file, as the attention's two blocks an SM do (a test asks
// few_row_linear_registers; a launch bound of 640 threads that forces it made 6 small full layers 268.4 -> 269.7 us).
constexpr int kSlimSmem = 113 * 1024;
// Instruction descriptor, kind::f16: D = fp32, A = B = bf16, both K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t make_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(GEMM_BLOCK_M >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.u32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}
struct KernelParams {
  ProjectionOut o;
  int* status;
  int rows, E_out, tile_n, total_kb, stages, tmem_cols, ksplit;
  float inv_d;                  // 1 / d_model
  uint32_t data_bytes;          // shared memory ahead of the barriers: max(pipeline stages, own fp32 slice)
  float* xchg;                  // [group][rank][tile_n][128] partial tiles of the K split
  int* flags;                   // [group][rank] peers that have delivered their part of slice `rank`
};

__device__ __forceinline__ int ld_acquire_gpu(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// first token block (of n_blk) that share r of a K split owns
__host__ __device__ inline int first_block(int r, int n_blk, int ksplit) { return (r * n_blk + ksplit - 1) / ksplit; }

template <int kFin, bool kOwnRope>   // kOwnRope: no RoPE table, every finishing thread derives the rotation of its one row
__global__ void __launch_bounds__(kOwnRope ? kFewBound : kMaxThreads, 1)
qkv_gemm_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
                const __grid_constant__ CUtensorMap tm_w2, KernelParams p, BatchParams bp) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // carve: [stages][A 16 KiB | B tile_n*128] (later reused for this CTA's own token slice of
  // the fp32 partial tile, [token][128 features]) | full[stages] | empty[stages] | tmem_full |
  // tmem slot | abort
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t stage_b_bytes = (uint32_t)p.tile_n * 128u;
  const uint32_t stage_bytes = kStageABytes + stage_b_bytes;
  const uint32_t bar_base = base + p.data_bytes;
  uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
  uint8_t* ctl = gen_base + p.data_bytes + 16 * p.stages;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(ctl + 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(ctl + 12);
  auto full_bar = [&](int s) { return bar_base + 8u * (uint32_t)s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (uint32_t)(p.stages + s); };
  const uint32_t tmem_full_bar = bar_base + 16u * (uint32_t)p.stages;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int epi_warps = ((int)blockDim.x >> 5) - 2;   // 4, 8 or 16
  const int tok_lanes = 2 * epi_warps;                // token rows finished side by side
  const int m0 = blockIdx.x * GEMM_BLOCK_M;
  const int n0 = blockIdx.y * p.tile_n;
  const int rank = (int)blockIdx.z;            // share of K
  const int kb0 = p.total_kb * rank / p.ksplit, kblocks = p.total_kb * (rank + 1) / p.ksplit - kb0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(tmem_full_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");   // (the only scope this fence has)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_w) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_x) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"((uint32_t)p.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem_acc = *tmem_slot;
  VS_STAMP(bp, 1, 0);
  auto load_w = [&](int kb) {
    const int s = kb % p.stages, kx = (kb0 + kb) * GEMM_BLOCK_K;
    const uint32_t a_dst = base + (uint32_t)s * stage_bytes;
    mbar_arrive_expect_tx(full_bar(s), stage_bytes);
    if constexpr (kFin == FIN_SWIGLU) {
      // a 128-row tile = 64 rows of the gate matrix, then the same 64 rows of the up matrix
      tma_load_2d(a_dst, &tm_w, kx, m0 >> 1, full_bar(s));
      tma_load_2d(a_dst + kStageABytes / 2, &tm_w2, kx, m0 >> 1, full_bar(s));
    } else {
      tma_load_2d(a_dst, &tm_w, kx, m0, full_bar(s));
    }
  };
  // weights are constant: the first stages' are requested before the wait on the stream's earlier kernels
  const int ahead = min(p.stages, kblocks);
  if (threadIdx.x == 0)
    for (int kb = 0; kb < ahead; ++kb) load_w(kb);
  pdl_wait();                       // earlier kernels of the stream have completed
  pdl_launch_dependents();
  VS_STAMP(bp, 1, 1);

  if (warp == 0) {
    if (lane == 0) {
      int issued = ahead;
      for (int kb = 0; kb < kblocks; ++kb) {
        const int s = kb % p.stages;
        if (kb >= ahead) {
          if (!mbar_wait(empty_bar(s), ((uint32_t)(kb / p.stages) & 1u) ^ 1u, abort_flag)) break;
          load_w(kb);
          issued = kb + 1;
        }
        tma_load_2d(base + (uint32_t)s * stage_bytes + kStageABytes, &tm_x, (kb0 + kb) * GEMM_BLOCK_K, n0, full_bar(s));
      }
      if (*abort_flag) {
        // let this CTA's copies land before its shared memory is given up
        for (int kb = (issued > p.stages ? issued - p.stages : 0); kb < issued; ++kb) {
          const unsigned long long t0 = global_ns();
          while (!mbar_try_wait(full_bar(kb % p.stages), (uint32_t)(kb / p.stages) & 1u)) {
            if (global_ns() - t0 > kWaitLimitNs) break;
          }
        }
      }
    }
  } else if (warp == 1) {
    const uint32_t idesc = make_idesc(p.tile_n), elected = elect_lane();
    bool ok = true;
    for (int kb = 0; kb < kblocks; ++kb) {
      const int s = kb % p.stages;
      ok = __all_sync(0xffffffffu, mbar_wait(full_bar(s), (uint32_t)(kb / p.stages) & 1u, abort_flag));
      if (!ok) break;
      tcgen05_fence_after();
      const uint64_t da = make_smem_desc(base + (uint32_t)s * stage_bytes), db = make_smem_desc(base + (uint32_t)s * stage_bytes + kStageABytes);
#pragma unroll
      for (int k = 0; k < GEMM_BLOCK_K / 16; ++k)      // 16 bf16 = 32 bytes further along K inside the 128-byte swizzle row
        umma_bf16(tmem_acc, da + 2u * k, db + 2u * k, idesc, (uint32_t)((kb | k) != 0), elected);
      umma_commit(empty_bar(s), elected);              // frees the stage once these MMAs have read it
    }
    if (ok) umma_commit(tmem_full_bar, elected);       // accumulator complete
  }

  // ---- epilogue ---------------------------------------------------------------------------
  // A  every CTA waits for its own accumulator (all its MMAs done, so all its TMA writes have
  //    landed and its stages are dead) and stores the token blocks it does not own, fp32, as [token][128 features], to its part
  //    of the exchange buffer.
  // B  it then counts itself in on the flag of every other owner, copies its own blocks into its shared memory, and waits
  //    until the ksplit - 1 peers have done the same on its own flag.
  // C  the owner of a block sums the ksplit partials of its tokens, adds the bias, rotates,
  //    rounds and stores.
  const int n_blk = (min(p.tile_n, p.rows - n0) + 15) >> 4;       // blocks that hold tokens
  const int blk0 = first_block(rank, n_blk, p.ksplit), blk1 = first_block(rank + 1, n_blk, p.ksplit);
  const int t_begin = blk0 * 16, slice = (blk1 - blk0) * 16;
  const int group = (int)(blockIdx.y * gridDim.x + blockIdx.x);
  // A step of a few rows brings no RoPE table: each finishing thread works out the (cos, sin) of
  // the four rotation pairs of its one row, in fp64 like the table kernel, while the main loop runs.
  float4 own_ra = make_float4(1.f, 0.f, 1.f, 0.f), own_rb = own_ra;
  if (kOwnRope && warp >= 2) {
    const int te = threadIdx.x - 64;
    const int half = p.o.D >> 1;
    const int p0 = (te & 15) * 4, hl = p0 / half, k0 = p0 - hl * half;
    const int row = n0 + t_begin + (te >> 4);
    if ((m0 + hl * p.o.D + k0) / p.o.D < p.o.Hq + p.o.Hkv && (te >> 4) < slice && row < p.rows) {
      const int b = row / bp.rows_per_stream;
      const double pos = (double)(bp.entry[b].pos_base + (row - b * bp.rows_per_stream));
      double sn, cs;
      float r[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        sincos(pos * p.o.inv_freq[k0 + i], &sn, &cs);
        r[2 * i] = (float)cs; r[2 * i + 1] = (float)sn;
      }
      own_ra = make_float4(r[0], r[1], r[2], r[3]);
      own_rb = make_float4(r[4], r[5], r[6], r[7]);
    }
  }
  // RMSNorm: the row scales of this CTA's token slice, worked out while the main loop runs
  float* rsc_s = reinterpret_cast<float*>(ctl + 64);             // [slice]
  if (warp >= 2 && p.o.row_ss != nullptr) {
    for (int t = threadIdx.x - 64; t < slice; t += (int)blockDim.x - 64) {
      const int row = n0 + t_begin + t;
      float tot = 0.f;
      if (row < p.rows)
        for (int i = 0; i < p.o.ss_parts; ++i) tot += p.o.row_ss[(size_t)row * p.o.ss_parts + i];
      rsc_s[t] = rsqrtf(tot * p.inv_d + p.o.norm_eps);
    }
  }
  bool acc_ok = true;
  if (warp >= 2) {
    acc_ok = __all_sync(0xffffffffu, mbar_wait(tmem_full_bar, 0, abort_flag));   // warp-uniform
  }
  tcgen05_fence_after();
  VS_STAMP_BY(bp, 1, 2, 64);          // accumulator complete

  float* part_local = reinterpret_cast<float*>(gen_base);      // [token - t_begin][128 features]
  // warp w may touch TMEM lanes 32*(w%4) .. +31 (lane = feature)
  const int quarter = warp & 3, w4 = (warp - 2) >> 2, nw4 = epi_warps >> 2;
  const uint32_t tmem_q = tmem_acc + ((uint32_t)(quarter * 32) << 16);
  if (p.ksplit > 1) {
    if (warp >= 2 && acc_ok) {
      float* dst_far = p.xchg + ((size_t)group * p.ksplit + rank) * p.tile_n * GEMM_BLOCK_M + quarter * 32 + lane;
      // the blocks of others, counted round the own ones
      for (int i = w4; i < n_blk - (blk1 - blk0); i += nw4) {
        const int blk = i < blk0 ? i : i + (blk1 - blk0);
        uint32_t r[16];
        tmem_ld16(tmem_q + (uint32_t)(blk * 16), r);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          float* d = dst_far + (size_t)(blk * 16 + j) * GEMM_BLOCK_M;
          if (VS_STORE_OK(bp, DR_GEMM_XCHG, d, 4)) *d = __uint_as_float(r[j]);
        }
      }
    }
    __syncthreads();
    VS_STAMP_BY(bp, 1, 3, 64);
    if (threadIdx.x == 64 && !*abort_flag) {
      // the barrier above ordered every thread's stores before this point; one cumulative fence
      // then orders them before the flag increments for whoever acquires a flag
      __threadfence();
      for (int s = 0; s < p.ksplit; ++s)
        if (s != rank && first_block(s, n_blk, p.ksplit) < first_block(s + 1, n_blk, p.ksplit) &&
            VS_STORE_OK(bp, DR_GEMM_FLAGS, p.flags + group * p.ksplit + s, 4)) atomicAdd(p.flags + group * p.ksplit + s, 1);
    }
  }
  if (warp >= 2 && acc_ok) {
    float* dst_own = part_local + quarter * 32 + lane;
    // (dealt from the last warp on: the first one has the flags to see to)
    for (int i = nw4 - 1 - w4; i < blk1 - blk0; i += nw4) {
      uint32_t r[16];
      tmem_ld16(tmem_q + (uint32_t)((blk0 + i) * 16), r);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int j = 0; j < 16; ++j) dst_own[(i * 16 + j) * GEMM_BLOCK_M] = __uint_as_float(r[j]);
    }
  }
  if (p.ksplit > 1 && threadIdx.x == 64 && blk0 < blk1) {
    int* mine = p.flags + group * p.ksplit + rank;
    uint32_t spins = 0;
    unsigned long long t0 = 0;
    while (!*abort_flag && ld_acquire_gpu(mine) < p.ksplit - 1) {
      if ((++spins & 255u) == 0u) {
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > kWaitLimitNs) *abort_flag = 1;
      }
    }
    if (VS_STORE_OK(bp, DR_GEMM_FLAGS, mine, 4)) *mine = 0;                                                 // next launch starts from zero
  }
  tcgen05_fence_before();
  __syncthreads();
  VS_STAMP_BY(bp, 1, 4, 64);

  // phase C.  Thread = (group of 4 rotation pairs, token lane).  The reads of a row -- float4
  // pieces of the own slice in shared memory and of the peers' partials in the exchange buffer,
  // and the row's RoPE entries -- are all issued before the arithmetic.
  if (warp >= 2 && !*abort_flag) {
    const int te = threadIdx.x - 64;               // 0 .. 32 * epi_warps - 1
    const Place pl = place_of(p.o, p.E_out, m0, te);
    const float* far = p.xchg + (size_t)group * p.ksplit * p.tile_n * GEMM_BLOCK_M;
    const size_t far_stride = (size_t)p.tile_n * GEMM_BLOCK_M;
    if (pl.on) {
      float bb1[4], bb2[4];
      bias_of(p.o, pl, m0, bb1, bb2);
      const int n_it = (slice - (te >> 4) + tok_lanes - 1) / tok_lanes;   // rows this thread finishes
      struct RowRegs { float4 v1[KSPLIT_MAX], v2[KSPLIT_MAX]; FinishIn in; float rsc; };
      auto valid_it = [&](int it) { return it < n_it && n0 + t_begin + (te >> 4) + tok_lanes * it < p.rows; };
      auto load_row = [&](RowRegs& R, int it) {
        const int t = t_begin + (te >> 4) + tok_lanes * it;
        const int row = n0 + t;
#pragma unroll
        for (int r = 0; r < KSPLIT_MAX; ++r) {
          if (r == rank) {
            R.v1[r] = *reinterpret_cast<const float4*>(part_local + (t - t_begin) * GEMM_BLOCK_M + pl.f1);
            R.v2[r] = *reinterpret_cast<const float4*>(part_local + (t - t_begin) * GEMM_BLOCK_M + pl.f2);
          } else if (r < p.ksplit) {
            // written by another SM during this launch: read past L1
            R.v1[r] = __ldcg(reinterpret_cast<const float4*>(far + r * far_stride + (size_t)t * GEMM_BLOCK_M + pl.f1));
            R.v2[r] = __ldcg(reinterpret_cast<const float4*>(far + r * far_stride + (size_t)t * GEMM_BLOCK_M + pl.f2));
          }
        }
        if (!kOwnRope || !pl.rotate) {
          R.in = finish_in<kFin>(p.o, pl, p.E_out, m0, row);
        } else {                         // the thread's only row (the launch checks it)
          R.in.ra = own_ra; R.in.rb = own_rb;
        }
        // RMSNorm's row scale commutes with the projection: applied here, in fp32
        R.rsc = (p.o.row_ss != nullptr) ? rsc_s[t - t_begin] : 1.f;
      };
      auto sum_row = [&](const RowRegs& R, int it) {
        const int t = t_begin + (te >> 4) + tok_lanes * it;
        const int row = n0 + t;
        float4 a1 = make_float4(0.f, 0.f, 0.f, 0.f), a2 = a1;
#pragma unroll
        for (int r = 0; r < KSPLIT_MAX; ++r) {
          if (r < p.ksplit) {
            a1.x += R.v1[r].x; a1.y += R.v1[r].y; a1.z += R.v1[r].z; a1.w += R.v1[r].w;
            a2.x += R.v2[r].x; a2.y += R.v2[r].y; a2.z += R.v2[r].z; a2.w += R.v2[r].w;
          }
        }
        finish_row<kFin>(p.o, bp, pl, p.E_out, m0, row, a1, a2, R.rsc, bb1, bb2, R.in, te);
      };
      // four warps per scheduler overlap one another's load latency; a thread holds one row at a time
#pragma unroll 1
      for (int it = 0; valid_it(it); ++it) {
        RowRegs A;
        load_row(A, it);
        sum_row(A, it);
      }
    }
  }

  __syncthreads();
  if (warp == 1) {
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_acc), "r"((uint32_t)p.tmem_cols) : "memory");
  }
  if (threadIdx.x == 0 && *abort_flag) atomicExch(p.status, VS_ERR_DEVICE_TIMEOUT);
  VS_STAMP(bp, 1, 15);
}

using Kernel = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, KernelParams, BatchParams);
Kernel kernel_of(int mode, bool own_rope) {
  switch (mode) {
    case FIN_RESIDUAL: return qkv_gemm_kernel<FIN_RESIDUAL, false>;
    case FIN_SWIGLU: return qkv_gemm_kernel<FIN_SWIGLU, false>;
    case FIN_LOGITS: return qkv_gemm_kernel<FIN_LOGITS, false>;
    default: return own_rope ? qkv_gemm_kernel<FIN_PROJECT, true> : qkv_gemm_kernel<FIN_PROJECT, false>;
  }
}

}  // namespace

// Whole steps, us without / with room, attention layers alone unless a full layer is named; keys before the question:
// * more than 48 rows: four stages and less, 64 rows 193 / 203; where K leaves no more stages than the room it costs nothing (8 layers of
//   width 1024, 17 to 48 rows: 0.5 to 3.5 % gained).
// * 33 to 48 rows gain (width 3584, 6 layers, one stream, 33 rows over 64 keys 1.3 %, over 1200 6.8 %; groups of eight 7 to 11 %), 25 to 32
//   where the attention takes three eighths of the SMs: it pays by its keys.  With a key tile to a CTA and a projection on nine tenths of
//   the SMs they lose: 4 x 8 rows over 64 keys 3.5 %, 25 rows 2.1 %, width 2560 2 x 13 rows 4 %; with two tiles 25 rows gain 0.9 %, with
//   three 3.1.  Projections on fewer SMs gain with one too (width 2048, 25 rows 7 %; 4096, 4 x 7 rows 3 %).
// * where a CTA's share of K is longer than the eight stages, an attention of so many CTAs that, with the projection's, there are
//   1.7 to an SM does not wait in the room but takes it: width 3584, 4 x 12 rows over 700 keys lose 5.1 %, 5 x 9 8.3 %, 12 x 4 3.4 %, 2 x 17
//   2.7 % (144 + 128 or more), one stream of 48 (144 + 96) gains 4.6 %; width 4096, 12 x 4 lose 4.5 % (120 + 192), 8 x 4 gain 2.7 (120 + 128).
// * there a full layer's W_o loses by itself (3 layers: 28 rows 321.4 / 324.2, 40 rows 321.7 / 326.5), and its projection gains with 144 + 64
//   (28 rows 321.4 / 317.1) and not with 144 + 96 (40 rows 321.7 / 326.5).
// Found the other way: width 3584, 6 x 8 rows over 64 keys (144 + 96) lose 3.0 %, 3 x 11 1.8.
bool leaves_room_for_attention(BesideAttention att, int rows, int blocks, int most_kb, int slim_stages, int n_sms) {
  if (att.ctas <= 0 || rows > 48) return false;
  if (most_kb <= slim_stages) return true;
  if (most_kb > 8 && (att.ahead || 20 * (att.ctas + blocks) > (att.full ? 29 : 34) * n_sms)) return false;
  if (rows > 32) return true;
  if (!att.full && att.tiles < 2 && 10 * blocks > 9 * n_sms) return false;
  return rows > 24 && 8 * att.ctas >= 3 * n_sms;
}

cudaError_t qkv_gemm_init() {
  for (int mode : {(int)FIN_PROJECT, (int)FIN_RESIDUAL, (int)FIN_SWIGLU, (int)FIN_LOGITS})
    for (bool own_rope : {false, true}) {
      const cudaError_t e = cudaFuncSetAttribute((const void*)kernel_of(mode, own_rope), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

// registers a thread of the kernels that may run beside the prefill attention, the most of them; 0 if the query fails
int few_row_linear_registers() {
  int most = 0;
  for (int mode : {(int)FIN_PROJECT, (int)FIN_RESIDUAL}) {
    cudaFuncAttributes at;
    if (cudaFuncGetAttributes(&at, (const void*)kernel_of(mode, false)) != cudaSuccess) { cudaGetLastError(); return 0; }
    most = at.numRegs > most ? at.numRegs : most;
  }
  return most;
}

cudaError_t launch_qkv_gemm(const GemmArgs& a, const BatchParams& bp, cudaStream_t st) {
  KernelParams p;
  p.o = a.out;
  p.status = a.status;
  p.rows = a.rows;
  p.E_out = a.E_out;
  p.tile_n = a.tile_n;
  p.ksplit = a.ksplit;
  p.inv_d = 1.f / (float)a.d;
  p.total_kb = a.d / GEMM_BLOCK_K;
  if (a.ksplit < 1 || a.ksplit > KSPLIT_MAX || a.ksplit > p.total_kb) return cudaErrorInvalidValue;
  if (a.tile_n < 16 || a.tile_n > 256 || (a.tile_n & 15) || 128 % a.out.D != 0) return cudaErrorInvalidValue;
  p.xchg = a.xchg;
  p.flags = a.flags;
  const bool own_rope = a.out.rope == nullptr && a.out.mode < 4;
  const int stage_bytes = kStageABytes + a.tile_n * 128, most_kb = (p.total_kb + a.ksplit - 1) / a.ksplit;
  int stages = (kMaxDynSmem - 3072) / stage_bytes;
  const int slim_stages = (kSlimSmem - 3072) / stage_bytes;
  const int blocks = (a.E_out + GEMM_BLOCK_M - 1) / GEMM_BLOCK_M * a.n_tiles * a.ksplit;
  const bool slim = !own_rope && leaves_room_for_attention(a.beside, a.rows, blocks, most_kb, slim_stages, a.n_sms);
  if (slim) stages = slim_stages;
  const int most = own_rope ? kFewStages : 8;
  if (stages > most) stages = most;
  if (stages > most_kb) stages = most_kb;
  if (stages < 1) return cudaErrorInvalidValue;
  p.stages = stages;
  int cols = 32;
  while (cols < a.tile_n) cols <<= 1;
  p.tmem_cols = cols;                      // a power of two, at most 512
  // the most tokens a share finishes
  const int n_blk = a.tile_n / 16, slice_rows = (n_blk + a.ksplit - 1) / a.ksplit * 16;
  size_t data = (size_t)stages * stage_bytes;
  const size_t own = (size_t)slice_rows * GEMM_BLOCK_M * 4;
  if (own > data) data = (own + 1023) / 1024 * 1024;
  p.data_bytes = (uint32_t)data;
  const size_t smem = 1024 + data + 16 * stages + 64 + 1024;     // + the slice's RMSNorm row scales
  if (smem > (size_t)kMaxDynSmem) return cudaErrorInvalidValue;
  // a step of few rows is finished by 4 or 8 warps; others by 16, which overlap one another's latency
  const int threads = 64 + 32 * (a.rows <= 8 ? 4 : (own_rope || slim ? kFewWarps : kMaxEpiWarps));
  // without a RoPE table every finishing thread must have at most one row
  if (own_rope && (a.out.inv_freq == nullptr || a.rows > 2 * (threads / 32 - 2))) return cudaErrorInvalidValue;
  const dim3 grid((a.E_out + GEMM_BLOCK_M - 1) / GEMM_BLOCK_M, a.n_tiles, a.ksplit);
  // the CTAs of a K split wait for one another: the whole grid has to be resident at once (a CTA an SM always fits)
  if (a.ksplit > 1 && (a.xchg == nullptr || a.flags == nullptr || (long long)grid.x * grid.y * grid.z > a.n_sms ||
                       (long long)grid.x * grid.y * grid.z > GEMM_XCHG_CTAS)) return cudaErrorInvalidValue;
  return launch_pdl(kernel_of(a.out.mode, own_rope), grid, dim3(threads), smem, st, a.tm_w, a.tm_x, a.tm_w2, p, bp);
}

}  // namespace vs
