// Frame-prefill / multi-token attention on the 5th-generation tensor cores
// (Eq. 1: Y = Softmax(Q K^T / sqrt(d_k)) V, grouped KV heads).
//
// One CTA = 16 query tokens x one KV head x one stream (x one share of the key tiles).  The G query heads of the group are
// stacked on the MMA's M axis (row = g * 16 + token, G * 16 <= 128), so K and V are staged once for the whole group.  Keys come
// from up to four segments -- prompt prefix, carrier bank (the free slot is masked), earlier text of the turn or carriers of a
// chunk's earlier frames, the step's own rows (causal) -- laid end to end, each starting on a multiple of 64 keys (the padding is
// masked), and cut into tiles of 64 keys, so that a tile lies in one segment.  The carrier is the last row of its frame
// (Section 3.2), so the causal rule alone gives it the whole frame.
// Per key tile:  S = Q K^T  (tcgen05.mma, M 128 x N 64, Q as a bf16 hi + lo pair)      -> TMEM, two buffers
//                softmax of the row in registers, P (bf16) -> TMEM, over the columns of S (tcgen05.st)
//                O += P V  (tcgen05.mma, A = P from TMEM, M 128 x N D, V read MN-major) -> TMEM; a row of O is
//                rescaled in TMEM only when its maximum grows by more than 2^8
// What bounds it: with many CTAs the tensor pipe (1040 clocks a key tile at 128 dims, three quarters of it the query's two halves: at
// N 64 the MMA waits for its operands from shared memory, 49 clocks where the arithmetic is 32; 1.2 us a tile to each of an SM's two
// CTAs is measured, 1.1 is what the pipe needs); with few the chain Q -> S -> softmax -> P V -> exchange -> stores.  Hence 64-key tiles
// and 112 KB of shared memory, 256 columns of TMEM and 320 threads a CTA: two CTAs fit an SM, and one's query fetch, softmax and
// stores run under the other's MMAs.  (S of two tiles by one MMA of N 128 needs a quarter less of the pipe, but its two buffers are then
// free only after the second P V, and nothing of a CTA's own runs under its softmax: 1.5 us a tile.)
// (One CTA an SM, 128-key tiles, four threads a row meeting at a barrier per tile, two K and V stages: 16 frames of 196 tokens
// over 320 keys took 106 us, 72 with two CTAs and 64-key tiles.)
// Warps 0..7: softmax, a warp per head of the group, its TMEM lanes in the shape of an MMA fragment: a quad of lanes holds two rows, whose
// maxima take two shuffles; fp32 pairs by one instruction each.  A row's stores come straight from there.  (A thread per row, four
// warps, and a CTA's rows through shared memory, half a warp to a row: 5.5 us from the last tile to the last store, 2.8 this way
// without a cluster; 28 layers of 170 rows over 747 keys 891 against 856 us, a chunk of eight frames 93.4 against 88.0.  A set-up with
// the barriers one after the other, divisions, and the query asked for behind the loader's first tiles: 856 against 841, 88.0 against 87.2.)
// Warp 8: one lane issues every MMA, one tile of Q K^T ahead of the softmax.  Warp 9: one thread fetches the query tile (bulk copies of the
// group's rows, 64 dims at a time, where the projection left it in operand
// layout) and the K and V tiles in the order they are used, through one ring of 16 KB stages, by bulk tensor copies (TMA, boxes of
// 64 keys x 64 dims through per-segment tensor maps, 128-byte swizzle as the MMA descriptors expect); tiles that hold only keys of
// earlier steps (prefix, bank, tail) are requested before the wait on the stream's earlier kernels.
// Few CTAs (a frame of one stream): the key tiles are shared by the CTAs of a thread-block cluster, each taking a contiguous run
// of tiles.  Each CTA finishes the rows of some tokens: the others send it theirs, unnormalised, with (max, denominator), by bulk
// copies from shared memory to shared memory, counted on a barrier of the owner's (to where the query was: dead once the owner's
// last S is there, which the first phase of the cluster's barrier tells).
// All mbarrier waits are bounded.
#include "vs_common.cuh"
#include "vs_ptx.cuh"
#include "vs_bank_update.cuh"

namespace vs {

namespace {

constexpr int kKeys = ATTN_KEY_BOX;   // keys per tile = key rows per bulk tensor copy
constexpr int kRows = 128;       // MMA M
constexpr int kTok = 16;         // query tokens per CTA

__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}
// untiled bulk copy: both addresses 16-byte aligned, size a multiple of 16
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// Shared-memory matrix descriptor, 128-byte swizzle, descriptor version 1.
//   K-major operand : rows of 128 bytes along K, 8-row groups `sbo` bytes apart.
//   MN-major operand: rows of 128 bytes along MN (64 elements), 8 K-rows per group, groups
//                     `sbo` bytes apart along K, 64-element MN blocks `lbo` bytes apart.
__device__ __forceinline__ uint64_t make_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// kind::f16 instruction descriptor: D fp32, A = B = bf16, M = 128, N = n; b_mn = 1 when B is MN-major.
__device__ __forceinline__ uint32_t make_idesc(int n, int b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn << 16) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(kRows >> 4) << 24);
}
__device__ __forceinline__ void umma_ss(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.u32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}
// A operand from tensor memory (128 lanes x 8 columns per 16 bf16 of K, two elements per column)
__device__ __forceinline__ void umma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc, uint32_t accumulate, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.u32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(db), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}
// 16 lanes x 64 columns of tensor memory, a thread with lane / 4 = g and lane % 4 = t: v[4 i + e] = (lane g, column 8 i + 2 t + e),
// v[4 i + 2 + e] = (lane g + 8, the same columns)
__device__ __forceinline__ void tmem_ld_16x64(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st_16x64(uint32_t taddr, const float (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]),
        "f"(v[8]), "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]),
        "f"(v[16]), "f"(v[17]), "f"(v[18]), "f"(v[19]), "f"(v[20]), "f"(v[21]), "f"(v[22]), "f"(v[23]),
        "f"(v[24]), "f"(v[25]), "f"(v[26]), "f"(v[27]), "f"(v[28]), "f"(v[29]), "f"(v[30]), "f"(v[31]) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// 16 lanes x 32 columns: r[2 i] = (lane g, column 4 i + t), r[2 i + 1] = (lane g + 8, the same column)
__device__ __forceinline__ void tmem_st_16x32(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// byte offset of 16-byte chunk c (8 bf16) of row r in a tile whose rows are `W` bf16 wide,
// stored as W/64 blocks of [rows x 128 bytes] with the 128-byte swizzle (chunk ^ (row & 7))
template <int ROWS>
__device__ __forceinline__ uint32_t sw_off(int r, int c) {
  return (uint32_t)((c >> 3) * (ROWS * 128) + r * 128 + (((c & 7) ^ (r & 7)) << 4));
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// two fp32 values side by side in a 64-bit register: one instruction for both
__device__ __forceinline__ uint64_t f32x2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 f32x2_parts(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// x / d by the reciprocal 2^32 / d + 1 (0: none that fits, or d = 1)
__device__ __forceinline__ int divide(int x, int d, uint32_t rcp) { return rcp != 0u ? (int)__umulhi((uint32_t)x, rcp) : (d == 1 ? x : x / d); }

// ---- thread-block cluster: the key splits of one (row tile, KV head, batch entry) -----------------------
// to a peer's shared memory, counted in bytes on a barrier of the peer's
__device__ __forceinline__ void st_async_f2(uint32_t addr, float2 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];"
               ::"r"(addr), "f"(v.x), "f"(v.y), "r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_shared_f2(uint32_t addr, float x, float y) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(x), "f"(y) : "memory");
}

constexpr int kSoftmaxWarps = 8;                         // one per head of the group: its 16 rows, a quad of lanes to two of them
constexpr int kIssuerWarp = kSoftmaxWarps, kLoaderWarp = kSoftmaxWarps + 1, kAllocWarp = kSoftmaxWarps - 1;
constexpr int kAttnThreads = 32 * (kSoftmaxWarps + 2);

template <int D>
struct Smem {
  static constexpr int kQBytes = kRows * D * 2;           // one of hi / lo
  static constexpr int kKVBytes = kKeys * D * 2;          // a K or V tile
  static constexpr int kStages = D == 128 ? 3 : 6;
  static constexpr int kQ = 0;                            // [hi | lo]; in a cluster, at the end, fp32 rows (see Exchange)
  static constexpr int kRing = 2 * kQBytes;               // [stage] K or V tile; in a cluster, at the end, rows on their way to peers
  static constexpr int kCtl = kRing + kStages * kKVBytes; // barriers, tmem slot, abort flag
  static constexpr int kPairs = kCtl + 80 + 16 * kStages;               // (max, denominator) of the peers' parts; weights; sums of squares
  static constexpr int kPairRows = D == 128 ? 108 : 128;  // (as many as two CTAs an SM leave room for)
  static constexpr int kTotal = kPairs + kPairRows * 8;
  static_assert(2 * (kTotal + 1024) <= 228 * 1024, "two CTAs an SM");
};

// Where a row tile's rows lie in the shared memory of CTA `split` of its cluster once the CTA's key tiles are done: byte offsets.
// The tile has n_tok tokens; CTA s finishes tokens s * tok_per ..., tok_per of them or what is left.  (Without a cluster a CTA finishes
// all of them out of its threads' registers, and nothing but the sums of squares has a place here.)
// Where the query was: the rows of its tokens, [CTA they come from][head][token].  At the top of the ring, on into the query's place
// where the ring does not hold them all: the rows that are on their way to the peers.  The peers' (max, denominator) pairs have a place
// of their own.  (With the pairs behind the rows a group of eight heads could not be split at all: its 128 rows fill the query's place.)
template <int D>
struct Exchange {
  using L = Smem<D>;
  int G, nsplit, n_tok, split, tok_per, my_tok;
  static constexpr int kRowBytes = D * 4;
  __host__ __device__ Exchange(int group, int nsplit_, int n_tok_, int split_)
      : G(group), nsplit(nsplit_), n_tok(n_tok_), split(split_), tok_per(nsplit_ == 1 ? kTok : (n_tok_ + nsplit_ - 1) / nsplit_) { my_tok = tokens_of(split_); }
  __host__ __device__ int tokens_of(int s) const {      // (none, perhaps)
    const int n = n_tok - s * tok_per;
    return n < 0 ? 0 : (n < tok_per ? n : tok_per);
  }
  // token tl of head g, as CTA s leaves it in the memory of the CTA that finishes it
  __host__ __device__ int rows() const { return nsplit * G * tok_per; }
  __host__ __device__ uint32_t row(int s, int g, int tl) const { return (uint32_t)(L::kQ + ((s * G + g) * tok_per + tl) * kRowBytes); }
  // ... with its pair, unless that is CTA `owner` itself: [head][token][peer].  A row's pairs give way to its weights, one a CTA, and
  // these, once the row is merged, to the sum of squares of the stored residual row.
  __host__ __device__ uint32_t stats(int g, int tl) const { return (uint32_t)(L::kPairs + (g * tok_per + tl) * (nsplit == 1 ? 4 : (nsplit - 1) * 8)); }
  __host__ __device__ uint32_t pair(int owner, int s, int g, int tl) const { return stats(g, tl) + 8u * (uint32_t)(s - (s > owner ? 1 : 0)); }
  // row `i` of those on their way, which may be read until the cluster's last barrier
  __host__ __device__ int staged_rows() const { return nsplit == 1 ? 0 : G * (n_tok - my_tok); }
  __host__ __device__ uint32_t staged(int i) const { return (uint32_t)(L::kCtl - (staged_rows() - i) * kRowBytes); }
};

// What a launch stores, known when the code is compiled: rows (fp32 or bf16), or the residual stream that they are added to; and whether the
// CTAs of a cluster share a row tile's keys.  (A CTA runs its stores once, and what lies between their parts is fetched for nothing: one
// layer of 170 rows 31.0 against 30.2 us by the stores, a chunk of eight frames 82.1, 78.7 and, with the cluster, 77.7.)
enum Stored { ST_ROWS_FP32, ST_ROWS_BF16, ST_RESIDUAL };
template <int D, int kStored, bool kCluster>
__global__ void __launch_bounds__(kAttnThreads, 2) prefill_attn_tc_kernel(const __grid_constant__ AttnArgs a,
                                                                          const __grid_constant__ BatchParams bp, int* status) {
  extern __shared__ __align__(1024) uint8_t gbase[];
  constexpr bool residual = kStored == ST_RESIDUAL, rows_out = !residual, rows_fp32 = kStored == ST_ROWS_FP32;
  const bool sums = residual && a.ss_out != nullptr;
  using L = Smem<D>;
  constexpr int CPR = D / 8, NS = L::kStages;
  const uint32_t base = smem_u32(gbase);
  const uint32_t ctl = base + L::kCtl;
  auto bar_s = [&](int i) { return ctl + 8u * (uint32_t)i; };             // S buffer ready (tcgen05.commit)
  // P of every second tile written (an arrival per head); P V of every second tile complete (tcgen05.commit).  (Two of each: a warp
  // may be done with a tile before another is with the one before, and a parity wait tells a phase only from the one before it.)
  auto bar_p = [&](int t) { return ctl + 16u + 8u * (uint32_t)(t & 1); };
  auto bar_o = [&](int t) { return ctl + 32u + 8u * (uint32_t)(t & 1); };
  constexpr uint32_t kRest = 48u + 16u * NS;
  const uint32_t bar_qb = ctl + kRest;                                      // query, first 64 dims, fetched by bulk copies (their bytes)
  const uint32_t bar_q = ctl + kRest + 8u;                                       // query, the other dims; or all of it, copied row by row (an arrival a softmax thread)
  auto bar_full = [&](int s) { return ctl + 48u + 8u * (uint32_t)s; };    // ring stage landed (its bytes)
  auto bar_free = [&](int s) { return ctl + 48u + 8u * (uint32_t)(NS + s); };    // ring stage read (tcgen05.commit)
  const uint32_t bar_recv = ctl + kRest + 16u;                                   // the peers' parts of this CTA's rows have arrived (their bytes)
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gbase + L::kCtl + kRest + 24);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + L::kCtl + kRest + 28);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // ---- bank update CTAs (frame steps), behind as many attention CTAs as run at once.  What they read -- carrier embeddings,
  // the bank's order and metadata -- was complete before the kernel ahead of this one let it start, and nothing else in this
  // launch touches what they write.  Their clusters hold no attention CTA, and they take part in no cluster barrier.
  if ((unsigned)((int)blockIdx.x - a.bank_pos) < (unsigned)a.bank_grid) {
    pdl_launch_dependents();
    const int bank_id = (int)blockIdx.x - a.bank_pos, stream = bank_id / a.bank_ctas;
    if (stream < bp.n_active)
      bank_update_block<16, 128>(a.bank, bp, stream, bank_id - stream * a.bank_ctas, a.bank_ctas, gbase, (uint32_t)L::kTotal);
    pdl_wait();      // so that this launch has completed only once the kernel ahead of it has
    return;
  }
  // ---- set-up that needs nothing from earlier kernels: barriers, tensor memory, the key axis ------------------
  // (Nothing of a block runs before its predecessor has left the SM, so this counts: a barrier a lane, divisions by the host's
  // reciprocals, the query asked for by the issuer and not behind the loader's first tiles.)
  if (warp == kIssuerWarp) {
    const uint32_t bar = ctl + 8u * (uint32_t)lane;                         // (all barriers side by side)
    if (bar <= bar_recv) mbar_init(bar, bar == bar_p(0) || bar == bar_p(1) ? (uint32_t)a.G : (bar == bar_q && a.q_tiled == nullptr ? 32u * kSoftmaxWarps : 1u));
    if (lane == 0) *abort_flag = (base & 1023u) != 0;      // (the swizzled layouts need the alignment that the declaration asks for)
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_proxy();
  } else if (warp == kAllocWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"(256u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else if (warp == kLoaderWarp) {
    if (lane < 2 * a.n_seg) asm volatile("prefetch.tensormap [%0];" ::"l"((lane & 1) ? &a.seg[lane >> 1].tv : &a.seg[lane >> 1].tk) : "memory");
  }
  // CTA id: key split (= rank in the cluster) fastest, then row tile, KV head, batch entry
  const int nsplit = kCluster ? a.nsplit : 1;                                // CTAs of the cluster = key splits of this row tile
  const int rps = bp.rows_per_stream, n_rt = (rps + kTok - 1) / kTok;
  const int id = (int)blockIdx.x - ((int)blockIdx.x >= a.bank_pos ? a.bank_grid : 0), id2 = divide(id, nsplit, a.rcp_split);
  const int split = id - id2 * nsplit, id3 = divide(id2, n_rt, a.rcp_rt), rt = id2 - id3 * n_rt, b = divide(id3, a.Hkv, a.rcp_hkv);
  const int hkv = id3 - b * a.Hkv, r0 = rt * kTok;
  const int sid = bp.entry[b].stream_id;
  const int G = a.G;
  const int count = a.chunk_mode ? a.chunk_count0 : bp.entry[b].count;
  const bool bank_full = (a.M > 0 && count == a.M);

  // the virtual key axis: segments end to end, each starting on a multiple of kKeys keys
  int seg_len[4], seg_beg[4], seg_kind[4];
  int ptotal = 0, bank_len = 0;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    int len = 0, kind = -1;
    if (s < a.n_seg) {
      kind = a.seg_kind[s];
      if (kind == 0) len = bp.entry[b].prefix_len;
      else if (kind == 1) { len = (a.M == 0) ? 0 : (bank_full ? a.M + 1 : count); bank_len = len; }
      else if (kind == 2) len = bp.entry[b].text_len;
      else if (kind == 4) len = (a.M == 0) ? 0 : b;                     // carriers of the chunk's frames before this one
      else len = min(rps, r0 + kTok);                                   // later keys are visible to no row of this tile
    }
    seg_kind[s] = kind; seg_len[s] = len; seg_beg[s] = ptotal / kKeys;
    ptotal += (len + kKeys - 1) & ~(kKeys - 1);
  }
  const int n_tiles_all = ptotal / kKeys;
  const int t_lo = (n_tiles_all * split) / nsplit, n_tiles = (n_tiles_all * (split + 1)) / nsplit - t_lo;   // this CTA's key tiles
  // segment of tile t_lo + t, and the index of the tile's first key in it
  auto find_seg = [&](int t, int& local) {
    int found = 0;
    local = 0;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (t_lo + t >= seg_beg[s] && seg_len[s] > (t_lo + t - seg_beg[s]) * kKeys) { found = s; local = (t_lo + t - seg_beg[s]) * kKeys; }
    }
    return found;
  };

  tc_fence_before();
  __syncthreads();                  // barriers initialised, tensor memory allocated
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tmem_o = tmem + 128u;                       // S (and P) buffers at columns 0 and 64, O at 128

  // ---- loader: the ring holds tiles in the order they are used: K(0), then K(t + 1), V(t) for every t
  auto element_of_k = [&](int t) { return t == 0 ? 0 : 2 * t - 1; };
  auto element_of_v = [&](int t) { return t == n_tiles - 1 ? 2 * n_tiles - 1 : 2 * t + 2; };
  const int n_elements = 2 * n_tiles;
  auto element_is_v = [&](int e) { return e == n_elements - 1 || (e > 0 && (e & 1) == 0); };
  // a walk over the tiles: the segment of the tile at hand, and the tile's first key in it
  struct Walk { int t, seg, local, len, kind; };
  auto enter = [&](Walk& w) {
    w.seg = find_seg(w.t, w.local);
#pragma unroll
    for (int i = 0; i < 4; ++i) if (i == w.seg) { w.len = seg_len[i]; w.kind = seg_kind[i]; }
  };
  auto advance = [&](Walk& w) {
    ++w.t;
    w.local += kKeys;
    if (w.local >= w.len) enter(w);
  };
  Walk walk = {0, 0, 0, 0, -1};
  enter(walk);
  int loaded = 0;
  const bool is_loader = (tid == kLoaderWarp * 32);
  Walk walk_v = walk;                        // the loader goes over the tiles twice: K with `walk`, V with this
  auto load_next = [&]() {
    const int s_ = loaded % NS;
    const bool is_v = element_is_v(loaded);
    const uint32_t dst = base + L::kRing + (uint32_t)s_ * L::kKVBytes;
    const int seg = is_v ? walk_v.seg : walk.seg, local = is_v ? walk_v.local : walk.local;
    const AttnSegment* sg = &a.seg[seg];
    const CUtensorMap* tm = is_v ? &sg->tv : &sg->tk;
    const int row = b * sg->rows_per_batch + local, z = sg->z0 + sid * sg->z_per_stream + hkv;
    mbar_arrive_expect_tx(bar_full(s_), (uint32_t)L::kKVBytes);
#pragma unroll
    for (int blk = 0; blk < D / 64; ++blk) tma_load_3d(dst + (uint32_t)(blk * (kKeys * 128)), tm, blk * 64, row, z, bar_full(s_));
    if (is_v) advance(walk_v); else advance(walk);
    ++loaded;
  };
  // keys of earlier steps only (prefix, bank, tail): nothing the kernel ahead of this one writes is
  // visible in such a tile (the bank slot it fills is masked or beyond the bank's count)
  if (is_loader)
    while (loaded < min(NS, n_elements) && (element_is_v(loaded) ? walk_v.kind : walk.kind) < 3) load_next();

  VS_STAMP(bp, 2, 0);
  pdl_wait();                       // earlier kernels of the stream have completed
  pdl_launch_dependents();
  VS_STAMP(bp, 2, 1);

  __syncwarp();
  // head of a softmax warp's 16 rows (rows 16 gg .. 16 gg + 15 of the MMA: the warp's quarter of the TMEM lanes, its lower or upper half)
  const int gg = 2 * (warp & 3) + (warp >> 2);
  const bool soft = warp < kSoftmaxWarps && gg < G;
  if (kCluster && !soft) cluster_arrive_release();   // (first phase; the softmax threads' arrival is the one that means something)
  // softmax threads: token rows lane / 4 and lane / 4 + 8.  m_run in the log2 domain (score * scale_log2e), the reference of P and O;
  // l_run the sum over this lane's own keys
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
  bool ok = true;
  if (warp == kLoaderWarp) {
    if (is_loader && n_tiles > 0) {
      while (loaded < n_elements) {
        if (loaded >= NS && !mbar_wait(bar_free(loaded % NS), (uint32_t)(loaded / NS - 1) & 1u, abort_flag)) break;
        load_next();
      }
      if (*abort_flag) {
        // let the copies in flight land before the shared memory is given up
        for (int e = max(loaded - NS, 0); e < loaded; ++e) {
          const unsigned long long t0 = global_ns();
          while (!mbar_try_wait(bar_full(e % NS), (uint32_t)(e / NS) & 1u)) { if (global_ns() - t0 > kWaitLimitNs) break; }
        }
      }
    }
  } else if (warp == kIssuerWarp) {
    // ---- MMA issuer.  MMAs run in the order they are issued: S of tile t + 1 may take the buffer that P of tile t - 1 was
    // read from as soon as the P V that reads it has been issued.
    if (n_tiles > 0) {
      const uint32_t elected = elect_lane();
      if (a.q_tiled != nullptr && lane == 0) {
        // the query tile as the projection left it, [hi | lo][64 dims] blocks in operand layout: the group's rows of each
        const bf16* tile = a.q_tiled + (((size_t)b * n_rt + (size_t)rt) * a.Hkv + hkv) * (size_t)(2 * kRows * D);
        const uint32_t bytes = (uint32_t)(G * kTok) * 128u;
#pragma unroll
        for (int blk = 0; blk < D / 64; ++blk) {
          const uint32_t bar = blk == 0 ? bar_qb : bar_q, off = (uint32_t)blk * (kRows * 128u);
          mbar_arrive_expect_tx(bar, 2u * bytes);
          bulk_load(base + L::kQ + off, tile + off / 2, bytes, bar);
          bulk_load(base + L::kQ + L::kQBytes + off, tile + (L::kQBytes + off) / 2, bytes, bar);
        }
      }
      __syncwarp();
      const uint32_t idesc_qk = make_idesc(kKeys, 0);
      const uint32_t idesc_pv = make_idesc(D, 1);
      const uint64_t dq = make_desc(base + L::kQ, 16, 1024);
      auto wait_all = [&](uint32_t bar, uint32_t parity) { return (bool)__all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)); };
      auto wait_full = [&](int e) { return wait_all(bar_full(e % NS), (uint32_t)(e / NS) & 1u); };
      auto issue_qk = [&](int t) {
        const int st = element_of_k(t) % NS;
        const uint32_t tmem_s = tmem + 64u * (uint32_t)(t & 1);
        const uint64_t dk = make_desc(base + L::kRing + (uint32_t)st * L::kKVBytes, 16, 1024);      // K tile, K-major
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          if (ks == 4 && t == 0 && a.q_tiled != nullptr && !wait_all(bar_q, 0)) return false;
          // k-step ks: block ks/4 of 64 elements, 32 bytes per step inside the 128-byte row
          const uint32_t qo = (uint32_t)((ks >> 2) * (kRows * 128) + (ks & 3) * 32) >> 4, ko = (uint32_t)((ks >> 2) * (kKeys * 128) + (ks & 3) * 32) >> 4;
          umma_ss(tmem_s, dq + qo, dk + ko, idesc_qk, (uint32_t)(ks != 0), elected);
          umma_ss(tmem_s, dq + ((uint32_t)L::kQBytes >> 4) + qo, dk + ko, idesc_qk, 1u, elected);
        }
        umma_commit(bar_s(t & 1), elected);
        umma_commit(bar_free(st), elected);
        return true;
      };
      bool go = wait_all(a.q_tiled != nullptr ? bar_qb : bar_q, 0) && wait_full(0);
      if (go) { tc_fence_after(); go = issue_qk(0); }
      for (int t = 0; t < n_tiles && go; ++t) {
        if (t + 1 < n_tiles) {      // the next S first: it has a whole softmax of lead time
          go = wait_full(element_of_k(t + 1));
          if (!go) break;
          tc_fence_after();
          issue_qk(t + 1);
        }
        const int ev = element_of_v(t), st = ev % NS;
        go = wait_all(bar_p(t), (uint32_t)(t >> 1) & 1u) && wait_full(ev);      // P(t) in place, O rescaled where needed; V(t)
        if (!go) break;
        tc_fence_after();
        const uint64_t dv = make_desc(base + L::kRing + (uint32_t)st * L::kKVBytes, kKeys * 128, 1024);   // V tile, MN-major
        const uint32_t tmem_p = tmem + 64u * (uint32_t)(t & 1);
#pragma unroll
        for (int kk = 0; kk < kKeys / 16; ++kk)
          // A = P from tensor memory: 16 keys = 8 columns.  B: 16 key rows = 2048 bytes further per step.  One accumulator for all tiles.
          umma_ts(tmem_o, tmem_p + 8u * (uint32_t)kk, dv + (uint64_t)((kk * 2048) >> 4), idesc_pv, (uint32_t)((t | kk) != 0), elected);
        umma_commit(bar_o(t), elected);
        umma_commit(bar_free(st), elected);
      }
      if (!go && a.q_tiled != nullptr) {
        // let the query's copies land before the shared memory is given up
        for (int blk = 0; blk < D / 64; ++blk) {
          const unsigned long long t0 = global_ns();
          while (!mbar_try_wait(blk == 0 ? bar_qb : bar_q, 0)) { if (global_ns() - t0 > kWaitLimitNs) break; }
        }
      }
    }
  } else {
    // ---- softmax: a warp per head, a quad of lanes per two rows -----------------------------------------------
    const int g8 = lane >> 2, t4 = lane & 3;
    if (a.q_tiled == nullptr && n_tiles > 0) {
      // Q rows (hi and lo) as a matrix-vector projection left them -> the operand layout in shared memory
      for (int idx = tid; idx < kRows * CPR; idx += 32 * kSoftmaxWarps) {
        const int r = idx / CPR, c = idx - r * CPR;
        const int qg = r >> 4, tt = r0 + (r & 15);
        const bool valid = (qg < G) && (tt < rps);
        const size_t off = valid ? (((size_t)b * rps + tt) * a.Hq + (size_t)hkv * G + qg) * D + c * 8 : 0;
        cp_async16(base + L::kQ + sw_off<kRows>(r, c), a.q + off, valid);
        cp_async16(base + L::kQ + L::kQBytes + sw_off<kRows>(r, c), a.q_lo + off, valid);
      }
      cp_async_commit();
      cp_async_wait<0>();
      fence_async_proxy();
      mbar_arrive(bar_q);
    }
    // a slot of the bank that no row sees: the one being refilled (in a chunk: the one that was free when it began)
    const int hole = bank_full ? (a.chunk_mode ? a.free_slot[0] : a.free_slot[sid * a.free_slot_stride]) : -1;
    // chunk of frames in one launch: whom the updates of the frames before this one evicted, two a lane, as bank-axis indexes
    int gone0 = -(1 << 20), gone1 = -(1 << 20);
    if (a.chunk_mode) {
      const int n = (a.M > 0) ? bank_len + b : 0;
      if (lane < b) { const int v = a.chunk_victim[lane]; if (v >= 0 && v < n) gone0 = v; }
      if (lane + 32 < b) { const int v = a.chunk_victim[lane + 32]; if (v >= 0 && v < n) gone1 = v; }
    }
    const float scale = a.scale_log2e;
    const uint64_t scale2 = f32x2(scale, scale);
    const uint32_t lane_base = (uint32_t)(16 * gg) << 16;           // warp w may touch TMEM lanes 32*(w%4)..+31
    // O accumulates in tensor memory over all tiles.  Its row -- and l -- are relative to m_run, which follows the row's
    // running maximum lazily: it moves (and the row of O is rescaled, in tensor memory) only when the maximum has grown by
    // more than 8, so 2^(score - m_run) <= 2^8.
    constexpr float kLazy = 8.f;
#pragma unroll 1
    for (int t = 0; t < n_tiles && soft; ++t) {
      if (t > 0) advance(walk);
      const int local = walk.local, len = walk.len, kind = walk.kind;
      // tiles with keys that some row does not see: the segment's end, the causal diagonal, the bank's free slot, what a chunk's frame
      // must not see (uniform over the warp)
      const bool masked = len - local < kKeys || (kind == 1 && (unsigned)(hole - local) < (unsigned)kKeys) || (kind == 3 && r0 - local + 1 < kKeys) ||
                          (a.chunk_mode && (kind == 1 || kind == 4));
      ok = mbar_wait(bar_s(t & 1), (uint32_t)(t >> 1) & 1u, abort_flag) && ok;
      __syncwarp();
      tc_fence_after();
      // (the last S: nothing will read this CTA's query again, its peers may store rows there)
      if (kCluster && t == n_tiles - 1) cluster_arrive_release();
      float sc[32];
      const uint32_t ts = tmem + 64u * (uint32_t)(t & 1) + lane_base;
      tmem_ld_16x64(ts, sc);
      tmem_ld_wait();
      if (masked) {
        uint32_t hide[2] = {0u, 0u};
        if (kind == 1) {
          const int hj = hole - local;
          if ((unsigned)hj < 32u) hide[0] = 1u << hj;
          else if ((unsigned)hj < 64u) hide[1] = 1u << (hj - 32);
        }
        if (a.chunk_mode && (kind == 1 || kind == 4)) {
          const int e = kind == 1 ? local : bank_len + local;                // index on the chunk's bank axis
          const unsigned d0 = (unsigned)(gone0 - e), d1 = (unsigned)(gone1 - e);
          hide[0] |= __reduce_or_sync(0xffffffffu, (d0 < 32u ? 1u << d0 : 0u) | (d1 < 32u ? 1u << d1 : 0u));
          hide[1] |= __reduce_or_sync(0xffffffffu, (d0 - 32u < 32u ? 1u << (d0 - 32u) : 0u) | (d1 - 32u < 32u ? 1u << (d1 - 32u) : 0u));
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int cnt = kind == 3 ? min(len - local, r0 + g8 + 8 * r - local + 1) : len - local;      // key i of the step is visible to rows >= i
          const uint32_t w0 = cnt >= 32 ? 0xffffffffu : (cnt <= 0 ? 0u : (1u << cnt) - 1u);
          const uint32_t w1 = cnt >= 64 ? 0xffffffffu : (cnt <= 32 ? 0u : (1u << (cnt - 32)) - 1u);
          // shifted so that bit 8 i is the lane's first key of column block i
          const uint32_t vis[2] = {(w0 & ~hide[0]) >> (2 * t4), (w1 & ~hide[1]) >> (2 * t4)};
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int c = 4 * (i >> 1) + 2 * r + (i & 1);
            sc[c] = ((vis[i >> 3] >> (8 * ((i >> 1) & 3) + (i & 1))) & 1u) ? sc[c] : -INFINITY;
          }
        }
      }
      float alpha[2];
      uint64_t minus_m[2];
      bool move = false;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float m0 = fmaxf(sc[2 * r], sc[2 * r + 1]), m1 = fmaxf(sc[2 * r + 4], sc[2 * r + 5]);
#pragma unroll
        for (int i = 2; i < 8; i += 2) {
          m0 = max3(m0, sc[4 * i + 2 * r], sc[4 * i + 2 * r + 1]);
          m1 = max3(m1, sc[4 * i + 4 + 2 * r], sc[4 * i + 4 + 2 * r + 1]);
        }
        float mx = fmaxf(m0, m1);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        mx *= scale;                                                         // scale > 0: max commutes with it
        const bool mv = mx > m_run[r] + kLazy || (m_run[r] == -INFINITY && mx > -INFINITY);
        const float m_new = mv ? mx : m_run[r];
        alpha[r] = mv ? ex2_approx(m_run[r] - m_new) : 1.f;                  // ex2(-inf) = 0: nothing accumulated yet
        m_run[r] = m_new;
        const float m_use = (m_new == -INFINITY) ? 0.f : -m_new;
        minus_m[r] = f32x2(m_use, m_use);
        move = move || mv;
      }
      // P, bf16 pairs, goes back into tensor memory over the first 32 columns of S: the warp has read its rows
      uint32_t pw[16];
      uint64_t rs[2][2] = {{0ull, 0ull}, {0ull, 0ull}};
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int r = i & 1;
        const float2 x = f32x2_parts(fma_f32x2(f32x2(sc[2 * i], sc[2 * i + 1]), scale2, minus_m[r]));
        const float p0 = ex2_approx(x.x), p1 = ex2_approx(x.y);
        rs[r][(i >> 1) & 1] = add_f32x2(rs[r][(i >> 1) & 1], f32x2(p0, p1));
        pw[i] = pack2(p0, p1);
      }
      tmem_st_16x32(ts, pw);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float2 sum = f32x2_parts(add_f32x2(rs[r][0], rs[r][1]));
        l_run[r] = l_run[r] * alpha[r] + (sum.x + sum.y);
      }
      // rows whose reference moved: O *= alpha (uniform over the warp), once the tile before has been added.  (S of this tile told of
      // the tile before that one.)
      if (t >= 1 && __any_sync(0xffffffffu, move)) {
        ok = mbar_wait(bar_o(t - 1), (uint32_t)((t - 1) >> 1) & 1u, abort_flag) && ok;
        __syncwarp();
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < D; c += 64) {
          float tv[32];
          tmem_ld_16x64(tmem_o + lane_base + (uint32_t)c, tv);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) tv[j] *= alpha[(j >> 1) & 1];
          tmem_st_16x64(tmem_o + lane_base + (uint32_t)c, tv);
        }
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_p(t));
    }
  }

  // ---- rows out -----------------------------------------------------------------------------------------------
  constexpr int F4 = D / 4, kWarps = kAttnThreads / 32, kRowBytes = D * 4;
  const int n_tok = min(kTok, rps - r0);                              // tokens of this row tile
  const Exchange<D> ex(G, nsplit, n_tok, split);
  const int tok_per = ex.tok_per, my_tok = ex.my_tok;
  const int g8 = lane >> 2, t4 = lane & 3;
  // element (token row r0, head 0 of the group, dim 0) of [rows][Hq * D]
  const size_t row0 = (((size_t)b * rps + r0) * a.Hq + (size_t)hkv * G) * D, tok_step = (size_t)a.Hq * D;
  VS_STAMP(bp, 2, 2);               // this CTA's tiles done
  if (soft) {
    // a lane's sums are over its own keys
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 1);
      l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 2);
    }
  }
  const uint32_t lane_base = (uint32_t)(16 * gg) << 16;
  auto wait_o = [&]() { return mbar_wait(bar_o(n_tiles - 1), (uint32_t)((n_tiles - 1) >> 1) & 1u, abort_flag); };      // all tiles added to O
  if constexpr (!kCluster) {
    // no peers: every thread stores what it holds of its two rows, eight bytes (fp32) or four at a time; a quad writes 32 bytes side by
    // side.  (Through shared memory, half a warp to a row: 5.5 us a CTA.)
    if (soft) {
      constexpr int NB = D / 64;
      size_t at[2];
      bool on[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) { at[r] = row0 + (size_t)(g8 + 8 * r) * tok_step + (size_t)gg * D + 2 * t4; on[r] = g8 + 8 * r < n_tok; }
      // the residual input is asked for before the wait for the last P V
      uint32_t hv[NB][16];
#pragma unroll
      for (int c = 0; c < NB; ++c)
#pragma unroll
        for (int i = 0; i < 16; ++i)
          hv[c][i] = (residual && on[i & 1]) ? *reinterpret_cast<const uint32_t*>(a.h_in + at[i & 1] + 64 * c + 8 * (i >> 1)) : 0u;
      ok = wait_o() && ok;
      __syncwarp();
      tc_fence_after();
      if (!ok) *abort_flag = 1;
      const float inv[2] = {l_run[0] > 0.f ? 1.f / l_run[0] : 0.f, l_run[1] > 0.f ? 1.f / l_run[1] : 0.f};
      float ss[2] = {0.f, 0.f};
#pragma unroll
      for (int c = 0; c < NB; ++c) {
        float v[32];
        __syncwarp();
        tmem_ld_16x64(tmem_o + lane_base + 64u * (uint32_t)c, v);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int r = i & 1;
          if (!on[r]) continue;
          const float v0 = v[2 * i] * inv[r], v1 = v[2 * i + 1] * inv[r];
          const size_t e = at[r] + 64 * c + 8 * (i >> 1);
          if constexpr (rows_out) {
            if constexpr (rows_fp32) {
              float* o = static_cast<float*>(a.out) + e;
              if (VS_STORE_OK(bp, a.out_region, o, 8)) *reinterpret_cast<float2*>(o) = make_float2(v0, v1);
            } else {
              bf16* o = static_cast<bf16*>(a.out) + e;
              if (VS_STORE_OK(bp, a.out_region, o, 4)) *reinterpret_cast<uint32_t*>(o) = pack2(v0, v1);
            }
          }
          if constexpr (residual) {
            const float2 h = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hv[c][i]));
            const uint32_t w = pack2(h.x + v0, h.y + v1);
            if (VS_STORE_OK(bp, a.h_out_region, a.h_out + e, 4)) *reinterpret_cast<uint32_t*>(a.h_out + e) = w;
            if (sums) {
              // RMSNorm of the next layer: its statistics are those of the rows as stored (bf16)
              const float2 s = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
              ss[r] += s.x * s.x + s.y * s.y;
              if (a.next_gain != nullptr) {
                // ... and, with a gain vector, the projection reads bf16(h * gain) instead of h
                const uint32_t graw = *reinterpret_cast<const uint32_t*>(a.next_gain + ((size_t)hkv * G + gg) * D + 64 * c + 8 * (i >> 1) + 2 * t4);
                const float2 g = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&graw));
                if (VS_STORE_OK(bp, DR_XN, a.xn_out + e, 4)) *reinterpret_cast<uint32_t*>(a.xn_out + e) = pack2(s.x * g.x, s.y * g.y);
              }
            }
          }
        }
      }
      if (sums) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          ss[r] += __shfl_xor_sync(0xffffffffu, ss[r], 1);
          ss[r] += __shfl_xor_sync(0xffffffffu, ss[r], 2);
          if (t4 == 0 && on[r]) *reinterpret_cast<float*>(gbase + ex.stats(gg, g8 + 8 * r)) = ss[r];
        }
      }
    }
  } else {
    // peers: rows to their owners, unnormalised, then every CTA merges the parts of its own rows
    constexpr int RPW = 32 / F4, U = 3;                // rows side by side in a warp; rows a lane has in hand at a time
    const int my_rows = G * my_tok, u = lane & (F4 - 1), hv = lane / F4;
    const uint32_t rcp_g = (65536u + (uint32_t)G - 1u) / (uint32_t)G;
    struct Row { int g, tl; bool on; size_t at; };
    auto row_of = [&](int j) {                         // row j of this CTA's: head j % G of token j / G
      Row r;
      r.tl = (int)(((uint32_t)j * rcp_g) >> 16); r.g = j - r.tl * G;
      r.on = j < my_rows;
      r.at = row0 + (size_t)(split * tok_per + r.tl) * tok_step + (size_t)r.g * D + 4 * u;
      return r;
    };
    auto load_res = [&](const Row& r) { return (residual && r.on) ? *reinterpret_cast<const uint2*>(a.h_in + r.at) : make_uint2(0u, 0u); };
    __syncwarp();
    if (soft && n_tiles == 0) cluster_arrive_release();
    if (tid == 0) mbar_arrive_expect_tx(bar_recv, (uint32_t)((nsplit - 1) * G * my_tok * (kRowBytes + 8)));
    uint2 h_first[U];                                  // the residual input of the first rows: asked for well ahead
#pragma unroll
    for (int k = 0; k < U; ++k) h_first[k] = load_res(row_of(warp * RPW + hv + k * kWarps * RPW));
    if (soft) {
      if (n_tiles > 0) ok = wait_o() && ok;
      __syncwarp();
      tc_fence_after();
      if (!ok) *abort_flag = 1;
    }
    __syncwarp();
    cluster_wait_acquire();                 // every peer's query is dead, and its barriers exist
    if (soft) {
      // Every row: into this CTA's own area if it finishes the row, else staged at the top of the ring, from where it goes to the owner
      // by bulk copies -- the rows of an owner's tokens lie side by side for every head.  (Stored straight into the peer's shared
      // memory, 16 bytes a lane scattered over 32 rows, they took 4 us.)
      const int theirs = n_tok - my_tok;                                // tokens of others, in order, numbered round this CTA's own
      uint32_t dst[2];
      bool on[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int tk = g8 + 8 * r, owner = tk / tok_per;
        on[r] = tk < n_tok;
        dst[r] = base + (owner == split ? ex.row(split, gg, tk - owner * tok_per) : ex.staged(gg * theirs + (tk < split * tok_per ? tk : tk - my_tok)));
        if (on[r] && owner != split && t4 == 0) {
          const uint32_t at = base + ex.pair(owner, split, gg, tk - owner * tok_per);
          st_async_f2(map_shared_rank(at, (uint32_t)owner), make_float2(m_run[r], l_run[r]), map_shared_rank(bar_recv, (uint32_t)owner));
        }
      }
#pragma unroll 1
      for (int c = 0; c < D; c += 64) {
        float v[32];
        __syncwarp();
        if (n_tiles > 0) {
          tmem_ld_16x64(tmem_o + lane_base + (uint32_t)c, v);
          tmem_ld_wait();
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = 0.f;
        }
        // (16-byte units XOR-swizzled by twice the token: eight rows of a quad's 32 bytes fall into different banks)
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int r = i & 1;
          if (on[r]) st_shared_f2(dst[r] + (uint32_t)(((((c + 8 * (i >> 1) + 2 * t4) >> 2) ^ (2 * g8)) << 4) + (t4 & 1) * 8), v[2 * i], v[2 * i + 1]);
        }
      }
      tc_fence_before();
      // a warp's rows are those of one head: it sends them on itself
      fence_async_proxy();
      __syncwarp();
      if (lane < nsplit && lane != split) {
        const int n = ex.tokens_of(lane), first = lane * tok_per, src = gg * theirs + (first < split * tok_per ? first : first - my_tok);
        if (n > 0) bulk_to_peer(map_shared_rank(base + ex.row(split, gg, 0), (uint32_t)lane), base + ex.staged(src), (uint32_t)(n * kRowBytes),
                                map_shared_rank(bar_recv, (uint32_t)lane));
      }
    }
    if (!mbar_wait(bar_recv, 0, abort_flag)) *abort_flag = 1;
    __syncwarp();
    if (soft) {
      // What each CTA's part of a row counts for, 2^(max_i - max) over the row's denominator: a part a lane, the rows of the warp's
      // head side by side.
      const int lg = nsplit > 4 ? 3 : (nsplit > 2 ? 2 : 1), wide = 1 << lg, tl = lane >> lg, s = lane & (wide - 1), tk = split * tok_per + tl;
      const float mA = __shfl_sync(0xffffffffu, m_run[0], 4 * (tk & 7)), mB = __shfl_sync(0xffffffffu, m_run[1], 4 * (tk & 7));
      const float lA = __shfl_sync(0xffffffffu, l_run[0], 4 * (tk & 7)), lB = __shfl_sync(0xffffffffu, l_run[1], 4 * (tk & 7));
      const bool row_on = tl < my_tok;
      float2 ml = make_float2(-INFINITY, 0.f);
      if (s == split) ml = tk < 8 ? make_float2(mA, lA) : make_float2(mB, lB);
      else if (row_on && s < nsplit) ml = *reinterpret_cast<const float2*>(gbase + ex.pair(split, s, gg, tl));
      float mm = ml.x;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) if (o < wide) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, o));
      const float w = (ml.x == -INFINITY) ? 0.f : ex2_approx(ml.x - mm);      // a CTA without visible keys adds nothing
      float den = 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float li = __shfl_sync(0xffffffffu, ml.y, i, wide), wi = __shfl_sync(0xffffffffu, w, i, wide);
        if (i < wide) den = fmaf(li, wi, den);
      }
      const float inv = (den > 0.f) ? 1.f / den : 0.f;
      if (row_on && s < nsplit) *(reinterpret_cast<float*>(gbase + ex.stats(gg, tl)) + s) = w * inv;
    }
    __syncthreads();
    cluster_arrive_release();               // this CTA has what it waited for
    VS_STAMP(bp, 2, 3);
    // F4 lanes per row, U rows of a lane side by side: their loads are all on their way before the first sum
#pragma unroll 1
    for (int jb = warp * RPW; jb < my_rows; jb += U * kWarps * RPW) {
      Row rw[U];
      float4 v[U];
      uint2 h[U];
#pragma unroll
      for (int k = 0; k < U; ++k) {
        // (a place without a row goes along with the warp's first one: another warp's weights may be giving way to its sums already)
        const int j = jb + hv + k * kWarps * RPW;
        rw[k] = row_of(j < my_rows ? j : jb);
        rw[k].on = j < my_rows;
        h[k] = jb == warp * RPW ? h_first[k] : load_res(rw[k]);
        v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll 1
      for (int s = 0; s < nsplit; ++s)
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const float w = reinterpret_cast<const float*>(gbase + ex.stats(rw[k].g, rw[k].tl))[s];
          const float4 o = *reinterpret_cast<const float4*>(gbase + ex.row(s, rw[k].g, rw[k].tl) + ((u ^ (2 * ((split * tok_per + rw[k].tl) & 7))) << 4));
          v[k].x = fmaf(o.x, w, v[k].x); v[k].y = fmaf(o.y, w, v[k].y); v[k].z = fmaf(o.z, w, v[k].z); v[k].w = fmaf(o.w, w, v[k].w);
        }
      float ss[U];
#pragma unroll
      for (int k = 0; k < U; ++k) {
        ss[k] = 0.f;
        if (!rw[k].on) continue;
        const size_t e = rw[k].at;
        if constexpr (rows_out) {
          if constexpr (rows_fp32) {
            if (VS_STORE_OK(bp, a.out_region, static_cast<float*>(a.out) + e, 16)) *reinterpret_cast<float4*>(static_cast<float*>(a.out) + e) = v[k];
          } else {
            const uint2 w = make_uint2(pack2(v[k].x, v[k].y), pack2(v[k].z, v[k].w));
            if (VS_STORE_OK(bp, a.out_region, static_cast<bf16*>(a.out) + e, 8)) *reinterpret_cast<uint2*>(static_cast<bf16*>(a.out) + e) = w;
          }
        }
        if constexpr (residual) {
          const float2 h0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h[k].x));
          const float2 h1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h[k].y));
          const uint2 w = make_uint2(pack2(h0.x + v[k].x, h0.y + v[k].y), pack2(h1.x + v[k].z, h1.y + v[k].w));
          if (VS_STORE_OK(bp, a.h_out_region, a.h_out + e, 8)) *reinterpret_cast<uint2*>(a.h_out + e) = w;
          if (sums) {
            // RMSNorm of the next layer: its statistics are those of the rows as stored (bf16)
            const float2 s0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.x)), s1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.y));
            ss[k] = (s0.x * s0.x + s0.y * s0.y) + (s1.x * s1.x + s1.y * s1.y);
            if (a.next_gain != nullptr) {
              // ... and, with a gain vector, the projection reads bf16(h * gain) instead of h
              const uint2 graw = *reinterpret_cast<const uint2*>(a.next_gain + ((size_t)hkv * G + rw[k].g) * D + 4 * u);
              const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&graw.x));
              const float2 g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&graw.y));
              if (VS_STORE_OK(bp, DR_XN, a.xn_out + e, 8))
                *reinterpret_cast<uint2*>(a.xn_out + e) = make_uint2(pack2(s0.x * g0.x, s0.y * g0.y), pack2(s1.x * g1.x, s1.y * g1.y));
            }
          }
        }
      }
      if (sums) {
#pragma unroll
        for (int k = 0; k < U; ++k) {
#pragma unroll
          for (int o = F4 / 2; o > 0; o >>= 1) ss[k] += __shfl_xor_sync(0xffffffffu, ss[k], o);
          if (u == 0 && rw[k].on) *reinterpret_cast<float*>(gbase + ex.stats(rw[k].g, rw[k].tl)) = ss[k];
        }
      }
    }
  }
  if (sums) {
    // the token's sum of squares over this KV head's query heads, in head order; the projection adds the KV heads' parts in
    // order
    __syncthreads();
    const int tl = tid - split * tok_per;
    if ((unsigned)tl < (unsigned)my_tok) {
      const uint8_t* part = gbase + ex.stats(0, tl);
      const uint32_t step = ex.stats(1, tl) - ex.stats(0, tl);
      float tot = 0.f;
#pragma unroll 4
      for (int g = 0; g < G; ++g, part += step) tot += *reinterpret_cast<const float*>(part);
      float* sp = a.ss_out + ((size_t)b * rps + r0 + tid) * a.Hkv + hkv;
      if (VS_STORE_OK(bp, DR_ROW_SS, sp, 4)) *sp = tot;
    }
  }
  // every CTA of the cluster has what it waited for: nobody's shared memory goes away while a copy may be reading it
  __syncwarp();
  if (kCluster) cluster_wait_acquire();
  tc_fence_before();
  __syncthreads();
  if (warp == kAllocWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
  }
  if (tid == 0 && *abort_flag) atomicExch(status, VS_ERR_DEVICE_TIMEOUT);
  VS_STAMP(bp, 2, 15);
}

using Kernel = void (*)(const AttnArgs, const BatchParams, int*);
template <int D, bool kCluster>
Kernel kernel_of(Stored what) {
  return what == ST_RESIDUAL ? prefill_attn_tc_kernel<D, ST_RESIDUAL, kCluster> : what == ST_ROWS_FP32 ? prefill_attn_tc_kernel<D, ST_ROWS_FP32, kCluster>
                                                                                : prefill_attn_tc_kernel<D, ST_ROWS_BF16, kCluster>;
}
template <int D>
Kernel kernel_of(Stored what, int nsplit) { return nsplit > 1 ? kernel_of<D, true>(what) : kernel_of<D, false>(what); }
template <int D>
cudaError_t init() {
  for (int i = 0; i < 6; ++i) {
    const void* k = reinterpret_cast<const void*>(kernel_of<D>((Stored)(i >> 1), 1 + (i & 1)));
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<D>::kTotal);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);   // two CTAs an SM
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t prefill_attention_tc_init() {
  const cudaError_t e = init<128>();
  return e != cudaSuccess ? e : init<64>();
}

// The byte ranges of an Exchange in CTA `split`, as (begin, end) pairs for a check on the host: the rows it finishes, the peers' pairs,
// the rows on their way to them, its sums of squares; the end of the query's place and of all.
void prefill_attention_ranges(int head_dim, int group, int nsplit, int n_tok, int split, int32_t* r) {
  auto fill = [&](auto ex, int q_end, int total) {
    const int n = ex.my_tok, row = ex.kRowBytes, first = split == 0 ? 1 : 0, last = split == nsplit - 1 ? nsplit - 2 : nsplit - 1, staged = ex.staged_rows();
    for (int i = 0; i < 8; ++i) r[i] = 0;
    if (n > 0) { r[6] = (int)ex.stats(0, 0); r[7] = (int)ex.stats(group - 1, n - 1) + 4; }
    if (n > 0 && nsplit > 1) {
      r[0] = (int)ex.row(0, 0, 0); r[1] = (int)ex.row(nsplit - 1, group - 1, n - 1) + row;
      r[2] = (int)ex.pair(split, first, 0, 0); r[3] = (int)ex.pair(split, last, group - 1, n - 1) + 8;
    }
    if (staged > 0) { r[4] = (int)ex.staged(0); r[5] = (int)ex.staged(staged - 1) + row; }
    r[8] = q_end; r[9] = total;
  };
  if (head_dim == 128) fill(Exchange<128>(group, nsplit, n_tok, split), Smem<128>::kRing, Smem<128>::kTotal);
  else fill(Exchange<64>(group, nsplit, n_tok, split), Smem<64>::kRing, Smem<64>::kTotal);
}

// Whether `nsplit` CTAs can share a row tile's keys: the rows that a CTA finishes have to fit where the query was, those on their way
// above them, the peers' pairs in their place (a tile of fewer tokens needs less of each); and nobody may be without tokens.  (Six
// for seven heads would fit with 64 dims, and lost to the eight that it was taken for: 170 rows over 427 keys, two KV heads, 20.5
// against 18.9 us a layer.)  Eight heads in four CTAs against one, 128 dims, four KV heads: 170 rows over 491 keys 35 against 41 us a
// layer, 32 rows over 608 keys 31 against 37; 64 dims, in eight CTAs, 32 rows: 17 against 26.
template <int D>
static bool can_split(int group, int nsplit) {
  const Exchange<D> ex(group, nsplit, kTok, nsplit - 1);
  if (nsplit == 6 && group > 6) return false;
  return ex.my_tok >= 1 && ex.rows() <= kRows && ex.rows() - group * ex.tok_per <= Smem<D>::kPairRows &&
         (ex.rows() + ex.staged_rows()) * ex.kRowBytes <= Smem<D>::kCtl;
}
bool prefill_attention_can_split(int head_dim, int group, int nsplit) {
  return head_dim == 128 ? can_split<128>(group, nsplit) : can_split<64>(group, nsplit);
}

cudaError_t launch_prefill_attention_tc(const AttnArgs& args, const BatchParams& bp, int* status, cudaStream_t st) {
  AttnArgs a = args;
  a.G = a.Hq / a.Hkv;
  if (a.nsplit < 1 || a.nsplit > ATTN_MAX_SPLIT || (a.nsplit > 1 && !prefill_attention_can_split(a.D, a.Hq / a.Hkv, a.nsplit))) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.bank_grid + ((bp.rows_per_stream + kTok - 1) / kTok) * a.nsplit * a.Hkv * bp.n_active);
  cfg.blockDim = dim3(kAttnThreads);
  // (exact while dividend and divisor multiply to less than 2^32)
  auto reciprocal = [&](uint32_t d) { return d > 1 && (uint64_t)cfg.gridDim.x * d < (1ull << 32) ? (uint32_t)((1ull << 32) / d + 1) : 0u; };
  a.rcp_split = reciprocal((uint32_t)a.nsplit); a.rcp_rt = reciprocal((uint32_t)((bp.rows_per_stream + kTok - 1) / kTok)); a.rcp_hkv = reciprocal((uint32_t)a.Hkv);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;            // the key splits of a row tile are one cluster
  attr[1].val.clusterDim.x = a.nsplit; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.nsplit > 1 ? 2 : 1;
  if ((a.out != nullptr) == (a.h_out != nullptr)) return cudaErrorInvalidValue;      // rows, or the residual stream (the last layer's rows have no next)
  const Stored what = a.h_out != nullptr ? ST_RESIDUAL : (a.out_fp32 ? ST_ROWS_FP32 : ST_ROWS_BF16);
  if (a.D == 128) { cfg.dynamicSmemBytes = Smem<128>::kTotal; return cudaLaunchKernelEx(&cfg, kernel_of<128>(what, a.nsplit), a, bp, status); }
  if (a.D == 64) { cfg.dynamicSmemBytes = Smem<64>::kTotal; return cudaLaunchKernelEx(&cfg, kernel_of<64>(what, a.nsplit), a, bp, status); }
  return cudaErrorInvalidValue;
}

// Clusters of `s` CTAs of this kernel that can be resident at once (a cluster's CTAs sit in one GPC); 0 if the query fails.
// (The query counts one CTA an SM for any kernel that allocates tensor memory; two of these share one, 256 columns each.)
// Asked once per handle.
int prefill_attention_max_clusters(int head_dim, int s) {
  if (s < 2 || s > ATTN_MAX_SPLIT) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(s * 64); cfg.blockDim = dim3(kAttnThreads);
  cfg.dynamicSmemBytes = head_dim == 128 ? Smem<128>::kTotal : Smem<64>::kTotal;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = s; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  int clusters = 0;
  const cudaError_t e = head_dim == 128 ? cudaOccupancyMaxActiveClusters(&clusters, kernel_of<128>(ST_RESIDUAL, s), &cfg)
                                        : cudaOccupancyMaxActiveClusters(&clusters, kernel_of<64>(ST_RESIDUAL, s), &cfg);
  if (e != cudaSuccess) { cudaGetLastError(); return 0; }
  return clusters;
}

}  // namespace vs
