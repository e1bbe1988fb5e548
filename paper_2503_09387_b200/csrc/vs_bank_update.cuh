// Bank update (Section 3.3, memory mechanism): evict-if-full, then append, as a device function
// run by spare CTAs of a frame step's attention launches (it needs the carrier embeddings, not the
// attention's result, so it runs beside it instead of after it): every layer's scores a share, the last one commits.
#pragma once

#include "vs_common.cuh"

namespace vs {

__device__ __forceinline__ double warp_tree_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// dot, |a|^2 and |b|^2 over d elements by one warp: lane p sums elements k = p (mod 32) in ascending k in fp64, then
// a butterfly 16, 8, 4, 2, 1; the results are the same in every lane.  A product of two bf16 values is exact in fp64, so the
// fused multiply-add rounds once, exactly where a separate addition would.  The loop is a chain of dependent fp64 adds fed
// by 2-byte loads, so what it costs is load latency: kU elements of every lane are requested before any is used (one at a
// time the scoring of a 1024-carrier bank took 33 us beside the attention of a one-layer frame step).
template <int kU>
__device__ __forceinline__ void warp_dot_norms(const bf16* va, const bf16* vb, int d, int lane, double& dot, double& na, double& nb) {
  dot = 0.0; na = 0.0; nb = 0.0;
  const unsigned short* pa = reinterpret_cast<const unsigned short*>(va) + lane;
  const unsigned short* pb = reinterpret_cast<const unsigned short*>(vb) + lane;
#pragma unroll 1
  for (int k0 = 0; k0 < d; k0 += 32 * kU) {
    unsigned short xa[kU], xb[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int k = k0 + 32 * u;                     // d is a multiple of 64: uniform over the warp
      xa[u] = (k < d) ? pa[k] : (unsigned short)0;   // (zeros add nothing: no sum is ever -0)
      xb[u] = (k < d) ? pb[k] : (unsigned short)0;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const double x = (double)__uint_as_float((uint32_t)xa[u] << 16);
      const double y = (double)__uint_as_float((uint32_t)xb[u] << 16);
      dot = __fma_rn(x, y, dot);
      na = __fma_rn(x, x, na);
      nb = __fma_rn(y, y, nb);
    }
  }
  dot = warp_tree_sum(dot); na = warp_tree_sum(na);
  nb = warp_tree_sum(nb);
}

// (out of line: a square root, a division and their special cases, once per row)
static __device__ __noinline__ double cosine_of(double dot, double na, double nb) {
  double s = 0.0;
  if (na != 0.0 && nb != 0.0) s = __ddiv_rn(dot, __dmul_rn(__dsqrt_rn(na), __dsqrt_rn(nb)));
  // a vector holding Inf or NaN has no cosine: counted as 0, like a zero vector
  if (!(s >= -2.0 && s <= 2.0)) s = 0.0;
  return s;
}

__host__ __device__ constexpr int bank_scratch_bytes(int nt) { return nt * 12 + 16; }

__device__ __forceinline__ void bank_cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}

// Scores bank rows j0 .. j1 - 1 against the incoming carrier (policy 0), four rows to a warp: a lane's sum is a chain of d / 32
// dependent fp64 operations, 9 clocks each at best, and every element costs a conversion of 9 to 14; four rows side by side fill
// the one with the other.  The rows stream through shared memory, 512 elements of each at a time, two chunks ahead; the incoming carrier is
// widened to fp64 once per block.  No one unit bounds it: of a frame step of 16 full banks of 1024 rows, 230 us, this loop's arithmetic and
// loads are 23; without the conversions it takes 224.6, without the rows' own norms 228.2, without either 221.6, so most of it is the chain of
// loads from shared memory and sums.  (Conversions by integer operations: 265 against 273 us of a longer such step, more instructions.)  Same
// sums in the same order as warp_dot_norms.  (One row a warp, staged whole: 16 banks of 1024 rows added 50 us to a batched frame step.)
constexpr int kScoreRows = 4, kScoreChunk = 512, kScoreStages = 3, kScoreWarpBytes = kScoreRows * kScoreStages * kScoreChunk * 2;
__device__ __forceinline__ int staged_warps(int d, uint32_t bytes) {
  const int left = (int)bytes - d * 8;
  return left > 0 ? min(left / kScoreWarpBytes, (int)blockDim.x >> 5) : 0;
}
__device__ __forceinline__ void staged_scores(const BankUpdateArgs& a, const BatchParams& bp, const bf16* emb, const int32_t* order, const bf16* emb_in,
                                              double* scores, int block, int n_blocks, int j1, uint8_t* smem, int n_warps) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, d = a.d;
  double* ys = reinterpret_cast<double*>(smem);
  uint8_t* ring = smem + (size_t)d * 8 + (size_t)warp * kScoreWarpBytes;     // [stage][row][512]
  const int step = n_blocks * n_warps, n_chunks = (d + kScoreChunk - 1) / kScoreChunk;
  int j = a.j0 + warp * n_blocks + block;                                    // rows j, j + step, j + 2 step, j + 3 step side by side
  const bf16* src[kScoreRows];
  auto pick = [&]() {
#pragma unroll
    for (int r = 0; r < kScoreRows; ++r) src[r] = j + r * step < j1 ? emb + (size_t)order[j + r * step] * d : nullptr;
  };
  auto fetch = [&](int c) {
    if (c < n_chunks) {
#pragma unroll
      for (int r = 0; r < kScoreRows; ++r) {
        if (src[r] == nullptr) continue;
        uint8_t* dst = ring + ((c % kScoreStages) * kScoreRows + r) * (kScoreChunk * 2);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int k = c * kScoreChunk + (lane + 32 * i) * 8;
          if (k < d) bank_cp_async16(dst + (lane + 32 * i) * 16, src[r] + k);
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (warp < n_warps) {
    pick();
#pragma unroll 1
    for (int c = 0; c < kScoreStages - 1; ++c) fetch(c);
  }
#pragma unroll 1
  for (int c = tid; c < d / 8; c += (int)blockDim.x) {
    const uint4 v = reinterpret_cast<const uint4*>(emb_in)[c];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      ys[c * 8 + 2 * i] = (double)__uint_as_float(w[i] << 16);
      ys[c * 8 + 2 * i + 1] = (double)__uint_as_float(w[i] & 0xffff0000u);
    }
  }
  __syncthreads();
  if (warp >= n_warps) return;
#pragma unroll 1
  while (j < j1) {
    double dot[kScoreRows], na[kScoreRows], nb = 0.0;
#pragma unroll
    for (int r = 0; r < kScoreRows; ++r) { dot[r] = 0.0; na[r] = 0.0; }
#pragma unroll 1
    for (int c = 0; c < n_chunks; ++c) {
      fetch(c + kScoreStages - 1);                     // into the stage that was read a chunk ago
      asm volatile("cp.async.wait_group %0;" ::"n"(kScoreStages - 1) : "memory");
      __syncwarp();
      const unsigned short* xs = reinterpret_cast<const unsigned short*>(ring + (c % kScoreStages) * kScoreRows * (kScoreChunk * 2)) + lane;
      const double* yc = ys + c * kScoreChunk + lane;
      const int n = min(kScoreChunk, d - c * kScoreChunk);
      // (64 elements a round: their twenty loads go out together -- one at a time the chain load, conversion, sum took 34 clocks a
      // row and element where the conversion's rate allows 10)
#pragma unroll 1
      for (int k = 0; k < n; k += 128) {
        double y[4];
        unsigned short xr[kScoreRows][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const bool in = k + 32 * i < n;              // (n is a multiple of 64; zeros add nothing)
          y[i] = in ? yc[k + 32 * i] : 0.0;
#pragma unroll
          for (int r = 0; r < kScoreRows; ++r) xr[r][i] = in ? xs[r * kScoreChunk + k + 32 * i] : (unsigned short)0;   // (a row that does not exist: whatever lies there)
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          nb = __fma_rn(y[i], y[i], nb);
#pragma unroll
          for (int r = 0; r < kScoreRows; ++r) {
            const double x = (double)__uint_as_float((uint32_t)xr[r][i] << 16);
            dot[r] = __fma_rn(x, y[i], dot[r]);
            na[r] = __fma_rn(x, x, na[r]);
          }
        }
      }
      __syncwarp();
    }
    nb = warp_tree_sum(nb);
    const int j_done = j;
    j += kScoreRows * step;
    if (j < j1) {
      pick();
#pragma unroll 1
      for (int c = 0; c < kScoreStages - 1; ++c) fetch(c);
    }
#pragma unroll 1
    for (int r = 0; r < kScoreRows; ++r) {
      // (row r's sums, picked without indexing registers)
      const double dr = r == 0 ? dot[0] : (r == 1 ? dot[1] : (r == 2 ? dot[2] : dot[3]));
      const double nr = r == 0 ? na[0] : (r == 1 ? na[1] : (r == 2 ? na[2] : na[3]));
      const int jr = j_done + r * step;
      if (jr >= j1) break;                             // uniform over the warp
      const double sc = cosine_of(warp_tree_sum(dr), warp_tree_sum(nr), nb);
      if (lane == 0 && VS_STORE_OK(bp, DR_SCORES, scores + jr, 8)) scores[jr] = sc;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Scores bank rows j0 .. j1 - 1 against their successors (policy 1; the last one's is the incoming carrier): a warp takes four
// neighbours and the row behind them, so that a row is read, widened and squared once for the two scores it has a part in (a
// score at a time: twice the conversions, and their latency bare -- a frame step with a bank of 22 rows took 65 us, not 56).
// Rows stream through shared memory as above; same sums in the same order as warp_dot_norms.  (Out of line: inlined, it cost the
// attention kernel's own code 2 %.)
constexpr int kAdjWarpBytes = (kScoreRows + 1) * kScoreStages * kScoreChunk * 2;
static __device__ __noinline__ void staged_adjacent_scores(const BankUpdateArgs& a, const BatchParams& bp, const bf16* emb, const int32_t* order,
                                                       const bf16* emb_in, double* scores, int block, int n_blocks, int j1, int count, uint8_t* smem,
                                                       int n_warps) {
  constexpr int R = kScoreRows + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, d = a.d;
  if (warp >= n_warps) return;
  uint8_t* ring = smem + (size_t)warp * kAdjWarpBytes;                       // [stage][row][512]
  const int n_chunks = (d + kScoreChunk - 1) / kScoreChunk;
#pragma unroll 1
  for (int j = a.j0 + (warp * n_blocks + block) * kScoreRows; j < j1; j += n_blocks * n_warps * kScoreRows) {
    const bf16* src[R];
#pragma unroll
    for (int r = 0; r < R; ++r) src[r] = j + r > j1 ? nullptr : (j + r < count ? emb + (size_t)order[j + r] * d : emb_in);
    auto fetch = [&](int c) {
      if (c < n_chunks) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (src[r] == nullptr) continue;
          uint8_t* dst = ring + ((c % kScoreStages) * R + r) * (kScoreChunk * 2);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int k = c * kScoreChunk + (lane + 32 * i) * 8;
            if (k < d) bank_cp_async16(dst + (lane + 32 * i) * 16, src[r] + k);
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll 1
    for (int c = 0; c < kScoreStages - 1; ++c) fetch(c);
    double dot[kScoreRows], sq[R];
#pragma unroll
    for (int r = 0; r < R; ++r) { sq[r] = 0.0; if (r < kScoreRows) dot[r] = 0.0; }
#pragma unroll 1
    for (int c = 0; c < n_chunks; ++c) {
      fetch(c + kScoreStages - 1);                     // into the stage that was read a chunk ago
      asm volatile("cp.async.wait_group %0;" ::"n"(kScoreStages - 1) : "memory");
      __syncwarp();
      const unsigned short* xs = reinterpret_cast<const unsigned short*>(ring + (c % kScoreStages) * R * (kScoreChunk * 2)) + lane;
      const int n = min(kScoreChunk, d - c * kScoreChunk);
#pragma unroll 1
      for (int k = 0; k < n; k += 64) {                // (n is a multiple of 64)
        unsigned short xr[2][R];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int r = 0; r < R; ++r) xr[i][r] = xs[r * kScoreChunk + k + 32 * i];    // (a row that does not exist: whatever lies there)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          double x[R];
#pragma unroll
          for (int r = 0; r < R; ++r) { x[r] = (double)__uint_as_float((uint32_t)xr[i][r] << 16); sq[r] = __fma_rn(x[r], x[r], sq[r]); }
#pragma unroll
          for (int r = 0; r < kScoreRows; ++r) dot[r] = __fma_rn(x[r], x[r + 1], dot[r]);
        }
      }
      __syncwarp();
    }
#pragma unroll
    for (int r = 0; r < R; ++r) sq[r] = warp_tree_sum(sq[r]);
#pragma unroll 1
    for (int r = 0; r < kScoreRows; ++r) {
      if (j + r >= j1) break;                          // uniform over the warp
      const double sc = cosine_of(warp_tree_sum(dot[0]), sq[0], sq[1]);
      if (lane == 0 && VS_STORE_OK(bp, DR_SCORES, scores + j + r, 8)) scores[j + r] = sc;
      // (the next row's sums move up: registers are not indexed)
      dot[0] = dot[1]; dot[1] = dot[2]; dot[2] = dot[3];
      sq[0] = sq[1]; sq[1] = sq[2]; sq[2] = sq[3]; sq[3] = sq[4];
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// One of the `n_blocks` thread blocks (any number of them, whole warps) that update the bank of listed stream b.
// scratch: 16-byte aligned shared memory, at least bank_scratch_bytes(NT); the more, the more rows are staged.
// Bank not full: block 0 appends; the other blocks return.
// Bank full: the warps of all blocks deal the temporal indexes j0 .. j1 - 1 among themselves and score cos(e_j, e_other) --
// e_other is the incoming carrier (policy 0) or the next carrier in temporal order (policy 1).  (A stack of layers shares
// the scoring out over the layers' launches; the last one commits.)  The fixed order of the fp64 sums makes the score, and
// with it the argmax, reproducible bit for bit.  The last block of a stream to finish picks the victim
// (largest score, oldest on ties), closes the gap in the temporal order and appends.
template <int kU, int NT>   // kU: loads in flight where nothing is staged; NT: threads that take part in the argmax, at most the block's
__device__ __forceinline__ void bank_update_block(const BankUpdateArgs& a, const BatchParams& bp, int b, int block, int n_blocks, void* scratch,
                                                  uint32_t scratch_bytes) {
  const int tid = threadIdx.x;
  const bool on = tid < NT;
  const int sid = bp.entry[b].stream_id;
  StreamMeta* meta = a.meta + sid;
  const bool meta_ok = VS_STORE_OK(bp, DR_META, meta, sizeof(StreamMeta));
  if (!a.commit && (a.M == 0 || bp.entry[b].count < a.M)) return;           // nothing to score
  if (a.M == 0) {
    if (block == 0 && tid == 0 && meta_ok) { meta->frames_seen += 1; meta->last_victim_frame = -1; }
    return;
  }
  int32_t* order = a.order + (size_t)sid * a.slots;
  int32_t* slot_frame = a.slot_frame + (size_t)sid * a.slots;
  int64_t* slot_pos = a.slot_pos + (size_t)sid * a.slots;
  const int count = bp.entry[b].count;
  const int incoming = (a.incoming_emb != nullptr) ? meta->free_slot : a.step_slot[sid];
  // chunked prefill, a launch per frame: the incoming embedding is read from where it is parked and moved into its slot
  // by whoever commits
  const bf16* emb_in = (a.incoming_emb != nullptr) ? a.incoming_emb
                                                   : a.emb + ((size_t)sid * a.slots + incoming) * a.d;
  auto adopt = [&]() {      // all threads of the committing block
    if (a.incoming_emb != nullptr) {
      bf16* dst = const_cast<bf16*>(a.emb) + ((size_t)sid * a.slots + incoming) * a.d;
#pragma unroll 1
      for (int k = tid; k < a.d; k += blockDim.x) if (VS_STORE_OK(bp, DR_EMB, dst + k, 2)) dst[k] = emb_in[k];
      if (tid == 0 && VS_STORE_OK(bp, DR_CHUNK_SLOT, a.record_slot + b, 4)) a.record_slot[b] = incoming;
      if (tid == 0 && VS_STORE_OK(bp, DR_CHUNK_VICTIM, a.record_victim + b, 4)) a.record_victim[b] = -1;
    }
  };
  const int64_t carrier_pos = bp.entry[b].pos_base + bp.rows_per_stream - 1;
  if (count < a.M) {
    if (block == 0) adopt();
    if (block == 0 && tid == 0) {
      if (VS_STORE_OK(bp, DR_ORDER, order + count, 4)) order[count] = incoming;
      if (VS_STORE_OK(bp, DR_SLOT_FRAME, slot_frame + incoming, 4)) slot_frame[incoming] = (int32_t)bp.entry[b].frame_id;
      if (VS_STORE_OK(bp, DR_SLOT_POS, slot_pos + incoming, 8)) slot_pos[incoming] = carrier_pos;
      if (meta_ok) {
        meta->count = count + 1;
        meta->free_slot = count + 1;        // slots fill in order until the bank is full
        meta->last_victim_frame = -1;
        meta->frames_seen += 1;
      }
    }
    return;
  }
  // ---- bank full: score, then the last block commits --------------------------------------
  double* scores = a.scores + (size_t)sid * a.slots;
  const int lane = tid & 31;
  const int j1 = min(a.j1, count);
  const int staged = a.policy == 0 ? staged_warps(a.d, scratch_bytes) : (a.policy == 1 ? min((int)scratch_bytes / kAdjWarpBytes, (int)blockDim.x >> 5) : 0);
  if (staged > 0 && a.policy == 1) {
    staged_adjacent_scores(a, bp, a.emb + (size_t)sid * a.slots * a.d, order, emb_in, scores, block, n_blocks, j1, count, static_cast<uint8_t*>(scratch), staged);
  } else if (staged > 0) {
    staged_scores(a, bp, a.emb + (size_t)sid * a.slots * a.d, order, emb_in, scores, block, n_blocks, j1, static_cast<uint8_t*>(scratch), staged);
  } else if (a.policy != 2) {
    const int n_warps = (int)blockDim.x >> 5;
#pragma unroll 1
    for (int j = a.j0 + (tid >> 5) * n_blocks + block; j < j1; j += n_blocks * n_warps) {
      const bf16* va = a.emb + ((size_t)sid * a.slots + order[j]) * a.d;
      const bf16* vb = (a.policy == 1 && j + 1 < count) ? a.emb + ((size_t)sid * a.slots + order[j + 1]) * a.d : emb_in;
      double dot, na, nb;
      warp_dot_norms<kU>(va, vb, a.d, lane, dot, na, nb);
      const double s = cosine_of(dot, na, nb);
      if (lane == 0 && VS_STORE_OK(bp, DR_SCORES, scores + j, 8)) scores[j] = s;
    }
  }
  if (!a.commit) return;                             // (its scores are read by the last layer's launch)
  // (the staged rows and the carrier are done with when a block takes its ticket)
  double* best_s = static_cast<double*>(scratch);                        // [NT]
  int* best_j = reinterpret_cast<int*>(best_s + NT);                     // [NT]
  int& is_last = best_j[NT];
  __threadfence();
  __syncthreads();
  if (tid == 0) is_last = meta_ok && (atomicAdd(&meta->score_ticket, 1) == n_blocks - 1);
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  double bs = -4.0; int bj = 0x7fffffff;   // every score lies in [-2, 2], so some thread takes an index < count
  if (on && a.policy != 2) {
#pragma unroll 1
    for (int i = tid; i < count; i += NT) {
      const double s = __ldcg(scores + i);
      if (s > bs) { bs = s; bj = i; }                 // ascending i: first maximum kept
    }
  }
  if (on) { best_s[tid] = bs; best_j[tid] = bj; }
  __syncthreads();
#pragma unroll 1
  for (int o = NT / 2; o > 0; o >>= 1) {
    if (tid < o) {
      const double s2 = best_s[tid + o]; const int j2 = best_j[tid + o];
      if (s2 > best_s[tid] || (s2 == best_s[tid] && j2 < best_j[tid])) {
        best_s[tid] = s2; best_j[tid] = j2;
      }
    }
    __syncthreads();
  }
  adopt();
  // the index stays inside the bank whatever the scores were
  const int v = (a.policy == 2 || (unsigned)best_j[0] >= (unsigned)count) ? 0 : best_j[0];
  const int victim_slot = order[v];
  const int victim_frame = slot_frame[victim_slot];
  __syncthreads();
  // close the gap in the temporal order, one chunk of NT at a time in ascending order: a chunk
  // reads [base+1, base+NT] before anything at or above base is written
#pragma unroll 1
  for (int base = v; base < count - 1; base += NT) {
    const int jj = base + tid;
    const int32_t next = (on && jj < count - 1) ? order[jj + 1] : 0;
    __syncthreads();
    if (on && jj < count - 1 && VS_STORE_OK(bp, DR_ORDER, order + jj, 4)) order[jj] = next;
    __syncthreads();
  }
  if (tid == 0) {
    if (VS_STORE_OK(bp, DR_ORDER, order + count - 1, 4)) order[count - 1] = incoming;
    if (VS_STORE_OK(bp, DR_SLOT_FRAME, slot_frame + victim_slot, 4)) slot_frame[victim_slot] = -1;
    if (VS_STORE_OK(bp, DR_SLOT_FRAME, slot_frame + incoming, 4)) slot_frame[incoming] = (int32_t)bp.entry[b].frame_id;
    if (VS_STORE_OK(bp, DR_SLOT_POS, slot_pos + incoming, 8)) slot_pos[incoming] = carrier_pos;
    if (a.log_cap > 0) {
      int32_t* e = a.evict_log + ((size_t)sid * a.log_cap + (meta->log_count % a.log_cap)) * 2;
      if (VS_STORE_OK(bp, DR_EVICT_LOG, e, 8)) { e[0] = (int32_t)bp.entry[b].frame_id; e[1] = victim_frame; }
    }
    meta->log_count += 1;
    meta->evictions += 1;
    meta->last_victim_frame = victim_frame;
    if (a.incoming_emb != nullptr && VS_STORE_OK(bp, DR_CHUNK_VICTIM, a.record_victim + b, 4))
      a.record_victim[b] = (victim_frame >= a.chunk_first_frame) ? a.chunk_l1 + (int)(victim_frame - a.chunk_first_frame)
                                                                 : victim_slot;
    meta->free_slot = victim_slot;
    meta->victim_logical = -1;
    meta->frames_seen += 1;
    meta->score_ticket = 0;
  }
}

}  // namespace vs
