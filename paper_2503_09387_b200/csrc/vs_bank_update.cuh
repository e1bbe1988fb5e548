// Bank update (Section 3.3, memory mechanism): evict-if-full, then append, as a device function
// run by spare CTAs of a frame step's last attention launch (it needs the carrier embeddings,
// not the attention's result, so it runs beside it instead of after it).
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

__device__ __forceinline__ double cosine_of(double dot, double na, double nb) {
  double s = 0.0;
  if (na != 0.0 && nb != 0.0) s = __ddiv_rn(dot, __dmul_rn(__dsqrt_rn(na), __dsqrt_rn(nb)));
  // a vector holding Inf or NaN has no cosine: counted as 0, like a zero vector
  if (!(s >= -2.0 && s <= 2.0)) s = 0.0;
  return s;
}

__device__ __forceinline__ void bank_cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}

// Scores bank rows j = first, first + step, ... < j1 against the incoming carrier (policy 0), a row per warp: the whole row is
// fetched into shared memory at once (two buffers a warp, the next row on its way while this one is summed), so a row costs one
// memory latency, and the incoming carrier is widened to fp64 once per block -- conversions to fp64 run at a sixteenth of
// the fp32 rate.  (With 16 two-byte loads in flight a lane, 64 rows took 6.5 us beside the attention of a one-layer frame step,
// longer than the attention; this way 3 us.)  Same sums in the same order as warp_dot_norms.
__device__ __forceinline__ int staged_warps(int d, uint32_t bytes) {
  const long long left = (long long)bytes - (long long)d * 8;
  const int n = left > 0 ? (int)(left / (4LL * d)) : 0;
  return min(n, (int)blockDim.x >> 5);
}
__device__ __forceinline__ void staged_scores(const BankUpdateArgs& a, const BatchParams& bp, const bf16* emb, const int32_t* order, const bf16* emb_in,
                                              double* scores, int block, int n_blocks, int j1, uint8_t* smem, int n_warps) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, d = a.d;
  double* ys = reinterpret_cast<double*>(smem);
  uint8_t* rows = smem + (size_t)d * 8 + (size_t)warp * 4 * d;
  const int step = n_blocks * n_warps;
  int j = a.j0 + warp * n_blocks + block;
  auto fetch = [&](int jj, int buf) {
    if (jj < j1) {
      const uint4* src = reinterpret_cast<const uint4*>(emb + (size_t)order[jj] * d);
      uint4* dst = reinterpret_cast<uint4*>(rows + (size_t)buf * 2 * d);
      for (int c = lane; c < d / 8; c += 32) bank_cp_async16(dst + c, src + c);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (warp < n_warps) { fetch(j, 0); fetch(j + step, 1); }
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
  double nb = 0.0;                                    // the incoming carrier's norm, summed with the first row
  bool first = true;
  for (int buf = 0; j < j1; j += step, buf ^= 1) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    const unsigned short* xs = reinterpret_cast<const unsigned short*>(rows + (size_t)buf * 2 * d);
    double dot = 0.0, na = 0.0;
    if (first) {
#pragma unroll 8
      for (int k = lane; k < d; k += 32) {
        const double x = (double)__uint_as_float((uint32_t)xs[k] << 16), y = ys[k];
        dot = __fma_rn(x, y, dot); na = __fma_rn(x, x, na); nb = __fma_rn(y, y, nb);
      }
      nb = warp_tree_sum(nb);
      first = false;
    } else {
#pragma unroll 8
      for (int k = lane; k < d; k += 32) {
        const double x = (double)__uint_as_float((uint32_t)xs[k] << 16);
        dot = __fma_rn(x, ys[k], dot); na = __fma_rn(x, x, na);
      }
    }
    __syncwarp();
    fetch(j + 2 * step, buf);
    const double sc = cosine_of(warp_tree_sum(dot), warp_tree_sum(na), nb);
    if (lane == 0 && VS_STORE_OK(bp, DR_SCORES, scores + j, 8)) scores[j] = sc;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// One of the `n_blocks` thread blocks (any number of them, whole warps) that update the bank of listed stream b.  smem:
// `smem_bytes` of dynamic shared memory for the scoring, 16-byte aligned, or null.
// Bank not full: block 0 appends; the other blocks return.
// Bank full: the warps of all blocks deal the temporal indexes j0 .. j1 - 1 among themselves and score cos(e_j, e_other) --
// e_other is the incoming carrier (policy 0) or the next carrier in temporal order (policy 1).  (A stack of layers shares
// the scoring out over the layers' launches; the last one commits.)  The fixed order of the fp64 sums makes the score, and
// with it the argmax, reproducible bit for bit.  The last block of a stream to finish picks the victim
// (largest score, oldest on ties), closes the gap in the temporal order and appends.
template <int kU, int NT>   // kU: loads in flight where nothing is staged; NT: threads that take part in the argmax, at most the block's
__device__ __forceinline__ void bank_update_block(const BankUpdateArgs& a, const BatchParams& bp, int b, int block, int n_blocks, uint8_t* smem,
                                                  uint32_t smem_bytes) {
  const int tid = threadIdx.x;
  const bool on = tid < NT;
  const int sid = bp.stream_id[b];
  StreamMeta* meta = a.meta + sid;
  if (!a.commit && (a.M == 0 || bp.count[b] < a.M)) return;           // nothing to score
  if (a.M == 0) {
    if (block == 0 && tid == 0) { meta->frames_seen += 1; meta->last_victim_frame = -1; }
    return;
  }
  int32_t* order = a.order + (size_t)sid * a.slots;
  int32_t* slot_frame = a.slot_frame + (size_t)sid * a.slots;
  int64_t* slot_pos = a.slot_pos + (size_t)sid * a.slots;
  const int count = bp.count[b];
  const int incoming = (a.incoming_emb != nullptr) ? meta->free_slot : a.step_slot[sid];
  // chunked prefill, a launch per frame: the incoming embedding is read from where it is parked and moved into its slot
  // by whoever commits
  const bf16* emb_in = (a.incoming_emb != nullptr) ? a.incoming_emb
                                                   : a.emb + ((size_t)sid * a.slots + incoming) * a.d;
  auto adopt = [&]() {      // all threads of the committing block
    if (a.incoming_emb != nullptr) {
      bf16* dst = const_cast<bf16*>(a.emb) + ((size_t)sid * a.slots + incoming) * a.d;
      for (int k = tid; k < a.d; k += blockDim.x) if (VS_STORE_OK(bp, DR_EMB, dst + k, 2)) dst[k] = emb_in[k];
      if (tid == 0) { a.record_slot[b] = incoming; a.record_victim[b] = -1; }
    }
  };
  const int64_t carrier_pos = bp.pos_base[b] + bp.rows_per_stream - 1;
  if (count < a.M) {
    if (block == 0) adopt();
    if (block == 0 && tid == 0) {
      if (VS_STORE_OK(bp, DR_ORDER, order + count, 4)) order[count] = incoming;
      if (VS_STORE_OK(bp, DR_SLOT_FRAME, slot_frame + incoming, 4)) slot_frame[incoming] = (int32_t)bp.frame_id[b];
      if (VS_STORE_OK(bp, DR_SLOT_POS, slot_pos + incoming, 8)) slot_pos[incoming] = carrier_pos;
      meta->count = count + 1;
      meta->free_slot = count + 1;          // slots fill in order until the bank is full
      meta->last_victim_frame = -1;
      meta->frames_seen += 1;
    }
    return;
  }
  // ---- bank full: score, then the last block commits --------------------------------------
  double* scores = a.scores + (size_t)sid * a.slots;
  const int lane = tid & 31;
  const int j1 = min(a.j1, count), staged = (smem != nullptr && a.policy == 0) ? staged_warps(a.d, smem_bytes) : 0;
  if (staged > 0) {
    staged_scores(a, bp, a.emb + (size_t)sid * a.slots * a.d, order, emb_in, scores, block, n_blocks, j1, smem, staged);
  } else if (a.policy != 2) {
    const int n_warps = (int)blockDim.x >> 5;
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
  __shared__ int is_last;
  __threadfence();
  __syncthreads();
  if (tid == 0) is_last = (atomicAdd(&meta->score_ticket, 1) == n_blocks - 1);
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  __shared__ double best_s[NT];
  __shared__ int best_j[NT];
  double bs = -4.0; int bj = 0x7fffffff;   // every score lies in [-2, 2], so some thread takes an index < count
  if (on && a.policy != 2) {
    for (int i = tid; i < count; i += NT) {
      const double s = __ldcg(scores + i);
      if (s > bs) { bs = s; bj = i; }                 // ascending i: first maximum kept
    }
  }
  if (on) { best_s[tid] = bs; best_j[tid] = bj; }
  __syncthreads();
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
    if (VS_STORE_OK(bp, DR_SLOT_FRAME, slot_frame + incoming, 4)) slot_frame[incoming] = (int32_t)bp.frame_id[b];
    if (VS_STORE_OK(bp, DR_SLOT_POS, slot_pos + incoming, 8)) slot_pos[incoming] = carrier_pos;
    if (a.log_cap > 0) {
      int32_t* e = a.evict_log + ((size_t)sid * a.log_cap + (meta->log_count % a.log_cap)) * 2;
      if (VS_STORE_OK(bp, DR_EVICT_LOG, e, 8)) { e[0] = (int32_t)bp.frame_id[b]; e[1] = victim_frame; }
    }
    meta->log_count += 1;
    meta->evictions += 1;
    meta->last_victim_frame = victim_frame;
    if (a.incoming_emb != nullptr)
      a.record_victim[b] = (victim_frame >= a.chunk_first_frame) ? a.chunk_l1 + (int)(victim_frame - a.chunk_first_frame)
                                                                 : victim_slot;
    meta->free_slot = victim_slot;
    meta->victim_logical = -1;
    meta->frames_seen += 1;
    meta->score_ticket = 0;
  }
}

}  // namespace vs
