// Weight-streaming GEMM for a few dozen tokens on sm_100a tensor cores (tcgen05 + TMEM), fed by TMA.
//
//   Y[t, n] = sum_k X[t, k] * W[n, k]      X: [rows <= 256, K] bf16 activations, W: [N, K] bf16 weights
//
// The verification forward is bound by the one pass over the weights (the paper's premise: checking dozens
// of tokens costs about as much as one, Section 3.2), so the kernel is organised around the weight stream:
//   * operands are swapped: a 128-row slab of W is the MMA's M side, the tokens (padded to a multiple of 16)
//     are its N side; the fp32 accumulator [128 x T] lives in TMEM;
//   * one persistent CTA per SM; the (tile, k-block) iteration space is cut into equal contiguous spans
//     (stream-K), so every SM streams the same number of bytes whatever N and K are;
//   * a span that covers only part of a tile's K range leaves a partial tile in scratch memory.  After its last
//     MMA every CTA adds up a share of the tokens of all such tiles, in ascending K order, and runs the epilogue on them.
//     The partial sums carry their own arrival (see EMPTY).  A CTA waits for the others' partials only
//     after it has published all of its own, so the waits cannot form a cycle (and they are bounded); the
//     result does not depend on arrival order;
//   * warp 0 issues TMA loads into a ring of shared-memory stages (128-byte swizzle), warp 1 issues
//     tcgen05.mma and releases stages with tcgen05.commit, warps 2-9 drain TMEM (double buffered) and run the
//     epilogue: plain store, residual add, or SiLU(gate)*up for the stacked gate/up matrices.
// The span boundaries depend on N, K and the grid only, never on the number of rows, and an output element
// is a function of its own row of X: a token's result is bitwise the same in a 1-row and in a 128-row call.
// Every mbarrier wait is bounded; on expiry the CTA raises the context's status word and drains.
#include <cuda.h>

#include <atomic>
#include <type_traits>

#include "ouro_internal.h"
#include "weight_stream.cuh"
#include "attn_fold.cuh"
#include "gemm_text.cuh"
#include "row_ops.cuh"

void ouro_set_global_error(const std::string &msg);   // api.cu

// Optional timeline of the GEMM launches (compile with -DOURO_TRACE, see paper_2402_13720_b200/trace.py): selected
// threads of every CTA stamp the global nanosecond timer at fixed points; ouro_trace_read_gemm copies the stamps
// of the most recent launch of every kind out.  Compiled out by default.
#ifdef OURO_TRACE
__device__ unsigned long long g_gemm_trace[8][160][16];
__device__ __forceinline__ unsigned long long trace_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)::"memory");
  return t;
}
#define TRACE(slot) do { if (blockIdx.x < 160) g_gemm_trace[p.trace_id & 7][blockIdx.x][slot] = trace_now(); } while (0)
extern "C" int ouro_trace_read_gemm(unsigned long long *out_host) {
  return (int)cudaMemcpyFromSymbol(out_host, g_gemm_trace, sizeof(g_gemm_trace));
}
#else
#define TRACE(slot) do { } while (0)
#endif

namespace {

using ws::BLOCK_K;
using ws::TILE_N;
using ws::Span;
constexpr int A_BYTES = TILE_N * BLOCK_K * 2;
constexpr int EPI_WARPS = 8;      // two per TMEM lane quarter
constexpr int EPI_THREADS = 32 * EPI_WARPS;
constexpr int ACT_WARP = 2 + EPI_WARPS;
constexpr int THREADS = 32 * (ACT_WARP + 1);   // warp 0 weight TMA, warp 1 MMA, warps 2..9 epilogue, warp 10 activation TMA
constexpr int MAX_GRID = 160;
constexpr uint32_t SPIN_LIMIT = 1u << 24;
constexpr unsigned long long HINT_EVICT_FIRST = 0x12F0000000000000ull;
constexpr unsigned long long HINT_EVICT_LAST = 0x14F0000000000000ull;

enum { MODE_STORE = 0, MODE_RESIDUAL = 1, MODE_SWIGLU = 2, MODE_HEAD = 3, MODE_QKV = 4 };
// HEAD: per-tile row maxima (+ optional logits).  QKV: rotary positions on q and k, q to its buffer, k and v appended to the cache.

struct GemmMaps {
  CUtensorMap a[3];   // weight matrices stacked along the output dimension (q|k|v), or gate and up
  CUtensorMap b;      // activations, box = 64 x t_pad
};
struct GemmParams {
  int a_tiles[3];     // tiles of each stacked matrix (MODE_STORE / MODE_RESIDUAL)
  int a_rows[3];      // output features of each stacked matrix
  int a_count;
  int mode;
  int tiles;          // total tiles
  int kb;             // k-blocks per tile (K / 64)
  int t0, per;        // tiles below t0 are handled whole; the others are cut into spans of `per` k-blocks (ws::cut)
  int sharers, sit_out;   // CTAs that share the cut tiles where not all do (else 0), and whether the first round of whole tiles leaves them out
  int finishers;      // CTAs (the first ones) that add up and finish the cut tiles' tokens, each a share of all of them
  int t_pad;          // tokens padded to a multiple of 16 (MMA N)
  int rows;           // valid tokens (an upper bound when rows_dev is set)
  const int *rows_dev;  // NULL, or where the block's true row count sits in device memory: the host then sizes the
                        // launch for the largest block the decoding parameters allow and never reads the count
  int stages;
  float *out_f32;     // MODE_STORE / MODE_RESIDUAL: [rows, ldo]
  int ldo;
  __nv_bfloat16 *out_bf16;  // MODE_SWIGLU: [rows, F]
  float *tile_max;    // MODE_HEAD: [tiles][128] largest logit of each token inside the tile ...
  int *tile_arg;      //            ... and its vocabulary index (smallest index among equals)
  // RMSNorm folded into the GEMMs around it: g*x/rms(x) feeds a GEMM as bf16(g*x), and the per-token factor
  // 1/rms(x) multiplies that GEMM's output instead.  The producer of x (a residual-add epilogue) leaves bf16(g*x)
  // and, per 128-column tile, each token's sum of squares; the consumer adds the tile sums in order.
  // MODE_QKV: stacked q|k|v tiles hold whole heads (head_dim 64 or 128); pairs (i, i + head_dim/2) are rotated by
  // the row's position; q goes to q_out [rows, dq], k and v to cache slots L + row of this layer
  const int32_t *pos;
  const float *cos_t, *sin_t;   // [max_seq, head_dim/2]
  __nv_bfloat16 *q_out, *k_out, *v_out;
  int head_dim, dq, dkv, L;
  const __nv_bfloat16 *gain;  // MODE_RESIDUAL: gain of the norm that follows (NULL: plain residual add)
  __nv_bfloat16 *xb;          // MODE_RESIDUAL: bf16(gain * x_new), [rows, ldo]
  float *ss_out;              // MODE_RESIDUAL: [tiles][OURO_TEXT_ROWS] per-tile sums of squares of x_new
  const float *ss_in;         // other modes: sums of squares of the activation rows (NULL: no scaling)
  int ss_tiles;
  float ss_inv_d, eps;
  float *scratch;     // [grid][2][128, or 256 in a wide launch][128] partial tiles; a word that holds no partial sum holds EMPTY
  int *status;        // context status word
  int trace_id;           // which GEMM of the layer this is (timeline builds only)
  uint32_t wait_limit;    // polls of a partial tile, or of packets, before the wait gives up (1 << 22 unless a test shortens it)
};

// A chain of GEMMs run by one persistent launch, each consuming what the one before produced (output projection ->
// gate/up -> down -> next layer's q,k,v or the LM head).  The weight producer runs straight on into the next GEMM's
// tiles; the activations of GEMM i + 1 are fetched once GEMM i has finished all its tiles, which the CTAs learn from
// a counter in global memory (one per chain position, counting finished tiles, never reset: the host passes the value
// it will have reached, both modulo 2^32).  All GEMMs of a chain have the same rows / t_pad / stages.
constexpr int MAX_CHAIN = 4;
struct ChainArgs {
  GemmParams g[MAX_CHAIN];
  int n;
  uint32_t *finished;         // [MAX_CHAIN + 1] tiles finished, per chain position; last: CTAs done folding
  uint32_t target[MAX_CHAIN]; // value finished[i] has when GEMM i of this launch is complete
  // The first GEMM's activations may be the attention output, still in per-span pieces: every CTA first folds a share
  // of the (row, head) pairs, and the first activation tile is fetched once all CTAs have.
  fold::Params fold;
  uint32_t fold_target;           // value finished[MAX_CHAIN] has once every CTA has done its share of the work in front
  // ... or the embedding rows of the block's tokens (first layer): gathered by all CTAs the same way.
  rowops::Embed embed;
};
struct ChainParams {
  GemmMaps maps[MAX_CHAIN];
  ChainArgs args;
};
static_assert(sizeof(ChainParams) <= 4096, "kernel parameters");
constexpr int MAX_CHAIN_ROWS = OURO_PART_ROWS;   // rows of a launch, the widest tcgen05 tile; more than OURO_MAX_ROWS are known text
constexpr int MISC_BYTES = 512 + 2 * MAX_CHAIN_ROWS * 4 + MAX_GRID * 4;   // barriers, flags, per-token factors and positions, cut tiles

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait: false when the limit ran out or another warp of the CTA has given up (the caller raises the status
// word and drains).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag, uint32_t limit = SPIN_LIMIT) {
  uint32_t addr = smem_u32(bar);
  for (uint32_t i = 0; i < limit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((i & 255) == 255 && abort_flag && *abort_flag) return false;
  }
  return false;
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y,
                                            unsigned long long hint) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(smem_u32(dst)),
      "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "l"(hint)
      : "memory");
}
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  // K-major operand in 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart.
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float *v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// order-preserving map float -> uint32 (and back), so that integer max picks the largest float
__device__ __forceinline__ uint32_t ordered_u32(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ordered_f32(uint32_t u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}
__device__ __forceinline__ void epi_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS) : "memory"); }
// Partial sums travel between CTAs without flags: a scratch word is EMPTY until its contributor has stored the sum, and
// whoever fetches it (exactly one thread of one CTA) empties it again.  The fetching thread polls the words themselves, so
// a partial tile costs one store and one load latency; with a fence, an arrival counter and a poll of that in between it
// was 4.5 us from the last contraction to the sum (7B output projection, 37 rows), now 3.3.  EMPTY is a NaN the tensor
// cores do not produce (theirs is 0x7fffffff).  A GEMM's stores into a slot come after the hand-over of the GEMM before it (or the
// end of the launch before it), which the fetching threads signal after having emptied their words.
constexpr uint32_t EMPTY = 0xffffffffu;
__device__ __forceinline__ void part_store(float *dst, float v) {
  const uint32_t u = __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(dst), "r"(u == EMPTY ? 0x7fffffffu : u) : "memory");
}
// Predicated inside the assembly: several of these in a row are in flight together, where a branch around each would wait
// for one before the next is requested.  A load that is left out gives zeros.
__device__ __forceinline__ uint4 part_load(const float *src, bool wanted) {
  uint4 v;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "mov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
      "@p ld.relaxed.gpu.global.v4.b32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "=&r"(v.x), "=&r"(v.y), "=&r"(v.z), "=&r"(v.w)
      : "l"(src), "r"((uint32_t)wanted)
      : "memory");
  return v;
}
__device__ __forceinline__ bool part_there(const uint4 &v) { return v.x != EMPTY && v.y != EMPTY && v.z != EMPTY && v.w != EMPTY; }
__device__ __forceinline__ void part_empty(float *src) {
  asm volatile("st.relaxed.gpu.global.v4.b32 [%0], {%1, %1, %1, %1};" ::"l"(src), "r"(EMPTY) : "memory");
}
// Tokens of a whole tile parked in shared memory at a time: fewer where the activation tiles are so large that a fourth
// stage of the ring hangs on it.
__host__ __device__ constexpr int stage_tokens(int rows) { return rows > OURO_MAX_ROWS ? 32 : 64; }
constexpr int STAGE_PITCH = TILE_N + 4;   // floats per parked token: 16-byte aligned rows that start 4 banks apart

// The schedule of this launch for CTA blockIdx.x (see weight_stream.cuh).
struct SpanWalker : ws::SpanWalker {
  __device__ SpanWalker(const GemmParams &p)
      : ws::SpanWalker(p.tiles, p.kb, p.t0, p.per, p.sharers, p.sit_out != 0, (int)gridDim.x, (int)blockIdx.x) {}
};

// Locates a tile: which stacked matrix, its first row there, and the first output column.
__device__ __forceinline__ void locate(const GemmParams &p, int tile, int &seg, int &row0, int &col0, int &valid) {
  seg = 0;
  col0 = 0;
  int t = tile;
  while (seg + 1 < p.a_count && t >= p.a_tiles[seg]) {
    t -= p.a_tiles[seg];
    col0 += p.a_rows[seg];
    ++seg;
  }
  row0 = t * TILE_N;
  col0 += row0;
  valid = min(TILE_N, p.a_rows[seg] - row0);
}

// Bounded wait until GEMM `i` of the chain has finished all its tiles (acquire).  The counters pass 2^31 after some hundred
// thousand forwards, so they are compared by their distance, and unsigned: a signed difference that overflows is no order.
__device__ __forceinline__ bool counter_wait(const uint32_t *counter, uint32_t target, const int *status, uint32_t limit) {
  for (uint32_t spin = 0; spin < limit; ++spin) {
    uint32_t seen;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
    if (seen - target < 0x80000000u) return true;
    if ((spin & 15) == 15 && *(volatile const int *)status != 0) return false;   // some CTA has given up: nobody waits on
  }
  return false;
}
__device__ __forceinline__ bool chain_wait(const ChainArgs &cp, int i) {
  return counter_wait(cp.finished + i, cp.target[i], cp.g[0].status, 1u << 22);
}

// The kernel by the block's size.  What a GEMM executes once per CTA it mostly waits for as instructions, so that the
// short blocks' kernel is kept short (and free of spills: a hundred bytes of them cost 4 % of a decoding step).
enum { ONE = 0, FEW = 1, SOME = 2, MANY = 3 };      // up to ONE_ROWS, FEW_ROWS, 128 and 256 rows (known text)
constexpr int ONE_ROWS = 32, FEW_ROWS = 48;
template <int SIZE>
__global__ void __launch_bounds__(THREADS, 1) gemm_tc_kernel(const __grid_constant__ ChainParams kp) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const ChainArgs &cp = kp.args;
  const GemmParams &p0 = cp.g[0];                 // rows, t_pad and stages are common to the chain
  const int n_stages = p0.stages, t_pad = p0.t_pad;
  const int b_bytes = t_pad * BLOCK_K * 2;
  constexpr int MAX_ROWS = SIZE == MANY ? MAX_CHAIN_ROWS : OURO_MAX_ROWS, stage_tok = stage_tokens(MAX_ROWS);
  constexpr int slot_floats = MAX_ROWS * TILE_N;  // (all slots together stay below 2^31 bytes)
  const int stage_bytes = A_BYTES + b_bytes;
  uint8_t *ring = smem;
  float *xchg = (float *)(ring + (size_t)n_stages * stage_bytes);          // [stage_tok tokens][128] accumulators of a whole tile
  uint64_t *bars = (uint64_t *)((uint8_t *)xchg + stage_tok * STAGE_PITCH * 4);
  uint64_t *full = bars, *empty = bars + 16, *acc_full = bars + 32, *acc_empty = bars + 34;
  uint32_t *tmem_base_p = (uint32_t *)(bars + 36);
  volatile int *abort_flag = (volatile int *)(bars + 37);
  volatile int *wait_flag = (volatile int *)(bars + 39);   // [0..1]: outcome of an accumulator wait; [2]: a fix-up gave up
  uint64_t *drain_bar = bars + 44;                          // give-up path: "every contraction issued so far has completed"
  float *rs = (float *)(bars + 56);                         // [256] per-token factor 1/rms of the consumed activations
  int *spos = (int *)(rs + MAX_CHAIN_ROWS);                 // [256] token positions (rotary table rows), QKV epilogue
  uint32_t *cuts = (uint32_t *)(spos + MAX_CHAIN_ROWS);     // [160] of every cut tile: first contributor | contributors << 16

  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int acc_cols = t_pad <= 32 ? 32 : t_pad <= 64 ? 64 : t_pad <= 128 ? 128 : 256;   // columns per accumulator buffer

  if (threadIdx.x == 0) {
    for (int s = 0; s < n_stages; ++s) {
      mbar_init(&full[s], 2);          // weight producer + activation producer, each with its byte count
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], EPI_WARPS);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_p)),
                 "r"((uint32_t)(2 * acc_cols)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = *tmem_base_p;
  if (threadIdx.x == 0) { const GemmParams &p = p0; TRACE(0); }
  uint32_t n_issued = 0;                           // producer lanes: stages they have issued copies into

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (elect_one()) {
      // The weights do not depend on the previous kernel, so this warp never waits for it: the ring fills with
      // weight tiles while the predecessor drains.  The activation tiles come from another warp, after its wait.
      // One thread runs this loop once per 16 KB stage; at 40 GB/s per SM that is every 0.4 us, so the loop carries
      // no division and nothing that is constant over a span: stage index and ring round are counted along.
      uint32_t n = 0, round = 0;
      int st = 0;
      bool ok = true;
      for (int ci = 0; ci < cp.n && ok; ++ci) {
      const GemmParams &p = cp.g[ci];
      const bool swiglu = p.mode == MODE_SWIGLU;
      SpanWalker w(p);
      Span s;
      while (ok && w.next(s)) {
        int seg = 0, row0 = s.tile * 64, col0, valid;
        if (!swiglu) locate(p, s.tile, seg, row0, col0, valid);
        const CUtensorMap *m0 = &kp.maps[ci].a[seg];
        uint8_t *sa = ring + (size_t)st * stage_bytes;
        for (int kb = s.kb0; kb < s.kb1; ++kb, ++n) {
          if (round > 0) {
            ok = mbar_wait(&empty[st], (round - 1) & 1, abort_flag) && !*abort_flag;
            if (!ok) break;
          }
          mbar_expect_tx(&full[st], A_BYTES);
          if (swiglu) {
            tma_load_2d(sa, &kp.maps[ci].a[0], &full[st], kb * BLOCK_K, row0, HINT_EVICT_FIRST);
            tma_load_2d(sa + A_BYTES / 2, &kp.maps[ci].a[1], &full[st], kb * BLOCK_K, row0, HINT_EVICT_FIRST);
          } else {
            tma_load_2d(sa, m0, &full[st], kb * BLOCK_K, row0, HINT_EVICT_FIRST);
          }
          sa += stage_bytes;
          if (++st == n_stages) { st = 0; ++round; sa = ring; }
        }
      }
      TRACE(8);
      }
      if (!ok) { *abort_flag = 1; atomicExch(p0.status, 1); }
      n_issued = n;
    }
  } else if (warp == ACT_WARP) {
    // ---------------------------------------------------------------- activation producer
    if (elect_one()) {
      pdl_wait();                                  // the first GEMM's activations are the previous kernel's output
      uint32_t n = 0, round = 0;
      int st = 0;
      uint8_t *sb = ring + A_BYTES;
      bool ok = true;
      if (cp.fold.part || cp.embed.table) {        // ... once every CTA has done its share of the fold / the gather
        ok = counter_wait(cp.finished + MAX_CHAIN, cp.fold_target, p0.status, 1u << 22);
        asm volatile("fence.proxy.async;" ::: "memory");
      }
      for (int ci = 0; ci < cp.n && ok; ++ci) {
        const GemmParams &p = cp.g[ci];
        if (ci > 0) {
          // they are what the GEMM before this one wrote: wait until all its tiles are finished, then make
          // those generic-proxy writes visible to the copy engine's reads
          ok = chain_wait(cp, ci - 1) && !*abort_flag;
          if (!ok) break;
          asm volatile("fence.proxy.async;" ::: "memory");
        }
        TRACE(1);
        SpanWalker w(p);
        Span s;
        while (ok && w.next(s)) {
          for (int kb = s.kb0; kb < s.kb1; ++kb, ++n) {
            if (round > 0) {
              ok = mbar_wait(&empty[st], (round - 1) & 1, abort_flag) && !*abort_flag;
              if (!ok) break;
            }
            mbar_expect_tx(&full[st], b_bytes);
            tma_load_2d(sb, &kp.maps[ci].b, &full[st], kb * BLOCK_K, 0, HINT_EVICT_LAST);
            sb += stage_bytes;
            if (++st == n_stages) { st = 0; ++round; sb = ring + A_BYTES; }
          }
        }
      }
      if (!ok) { *abort_flag = 1; atomicExch(p0.status, 1); }
      n_issued = n;
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (elect_one()) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p0.t_pad >> 3) << 17) | ((uint32_t)(TILE_N >> 4) << 24);
      uint32_t n = 0, item = 0, round = 0;
      int st = 0;
      uint32_t sa = smem_u32(ring);
      const uint32_t ring0 = sa;
      bool ok = true;
      for (int ci = 0; ci < cp.n && ok; ++ci) {
      const GemmParams &p = cp.g[ci];
      SpanWalker w(p);
      Span s;
      bool first = true;
      while (ok && w.next(s)) {
        int a = item & 1;
        if (item >= 2) ok = mbar_wait(&acc_empty[a], ((item >> 1) - 1) & 1, abort_flag) && !*abort_flag;
        if (!ok) break;
        fence_after_sync();
        uint32_t tmem_d = tmem_base + a * acc_cols;
        for (int kb = s.kb0; kb < s.kb1; ++kb, ++n) {
          ok = mbar_wait(&full[st], round & 1, abort_flag) && !*abort_flag;
          if (!ok) break;
          if (first) { TRACE(2); first = false; }
          fence_after_sync();
          const uint64_t da = smem_desc_sw128(sa), db = smem_desc_sw128(sa + A_BYTES);
#pragma unroll
          for (int k = 0; k < BLOCK_K / 16; ++k) mma_bf16(tmem_d, da + 2 * k, db + 2 * k, idesc, (kb > s.kb0 || k > 0) ? 1u : 0u);
          mma_commit(&empty[st]);
          sa += stage_bytes;
          if (++st == n_stages) { st = 0; ++round; sa = ring0; }
        }
        if (!ok) break;
        mma_commit(&acc_full[a]);
        ++item;
      }
      TRACE(3);
      }
      if (!ok) { *abort_flag = 1; atomicExch(p0.status, 1); }
    }
  } else {
    // ---------------------------------------------------------------- epilogue warps
    if (!cp.fold.part) pdl_wait();               // (the fold waits itself)
    const int q = warp & 3;                      // TMEM lane quarter this warp may read
    const int nl = q * 32 + lane;                // row of the tile held by this thread
    const int et = threadIdx.x - 64;             // 0..255 among the epilogue threads
    const int wh = (warp - 2) >> 2;              // which of the two warps of its lane quarter this is
    uint32_t item = 0;
    bool ok = true;
    float v[16];
    if (cp.fold.part || cp.embed.table) {
      const int gw = (int)blockIdx.x * EPI_WARPS + (warp - 2), nw = (int)gridDim.x * EPI_WARPS;
      if (cp.fold.part) {
        fold::run(cp.fold, gw, nw, lane);
      } else {
        rowops::embed(cp.embed, gw, nw, lane);
      }
      __threadfence();
      epi_barrier();
      if (et == 0) atomicAdd(cp.finished + MAX_CHAIN, 1u);
      if (cp.embed.table) {
        // the first GEMM's per-token factors are sums over what ALL CTAs gathered
        if (et == 0) wait_flag[0] = counter_wait(cp.finished + MAX_CHAIN, cp.fold_target, p0.status, 1u << 22) && !*abort_flag;
        epi_barrier();
        ok = wait_flag[0] != 0;
        epi_barrier();
        __threadfence();
      }
    }
    for (int ci = 0; ci < cp.n && ok; ++ci) {
    const GemmParams &p = cp.g[ci];
    const bool publish = ci + 1 < cp.n;          // a later GEMM of the chain consumes this one's output
    const int rows = p.rows_dev ? min(p.rows, __ldg(p.rows_dev)) : p.rows;
    SpanWalker w(p);
    Span s;
    // this CTA's share of the cut tiles is still to be finished  (spans as long as a tile: each is one tile, and whole)
    bool due = p.per > 0 && p.per < p.kb && (int)blockIdx.x < p.finishers;
    float *stage = xchg;                                         // [stage_tok tokens][STAGE_PITCH] fp32, 128 tile rows each

    // Finishing tokens of a tile.  Whatever produced the accumulator values - this CTA's own whole tile, parked
    // in shared memory token-major, or the partial tiles of all contributors in scratch - the last step is the
    // same: a warp walks over tokens, its 32 lanes holding the tile's 128 rows (= output
    // columns) four apiece, so every global access is a 16-byte piece of a contiguous 512-byte row.
    //   whole tile:  tokens t_base + (epilogue warp) + 8 i below t_lim (one staged chunk of tokens)
    //   cut tile:    tb tokens from t_base on, as far as they are below t_lim; the partials are added up in ascending K order as
    //                they arrive
    // Returns false (warp-uniform) when the wait for a partial gave up.
    auto finish = [&](auto split_c, int tile, float *stg, int tbn, int t_base, int t_lim) -> bool {
      constexpr bool SPLIT = decltype(split_c)::value;
      const bool swiglu = p.mode == MODE_SWIGLU;                     // tile rows 0..63: gate of 64 features, 64..127: up
      int seg = 0, row0 = 0, col0 = 0, valid = TILE_N;
      if (!swiglu) locate(p, tile, seg, row0, col0, valid);
      const int ng = lane;
      const int col = col0 + 4 * ng;
      // Every matrix has a multiple of 8 output features (the shape checks see to it), so a thread's four columns are
      // inside the matrix together or not at all.
      const bool full4 = 4 * ng < valid;
      const int cm = row0 + 4 * ng;                                  // first of this thread's 4 columns inside q, k or v
      const int half = p.head_dim >> 1;
      const bool res_norm = p.mode == MODE_RESIDUAL && p.gain != nullptr;
      const bool rope = p.mode == MODE_QKV && seg != 2;
      uint2 graw = make_uint2(0, 0);
      if (res_norm && full4) graw = *reinterpret_cast<const uint2 *>(p.gain + col);

      auto finish_token = [&](int t, const float4 acc) {
        if (res_norm) {
          // new residual stream, its bf16(gain * x) image for the next GEMM, and this tile's sums of squares
          float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
          if (full4) {
            float *x = p.out_f32 + (size_t)t * p.ldo + col;
            y = acc;
            if (!SPLIT) { const float4 x4 = *reinterpret_cast<const float4 *>(x); y.x += x4.x; y.y += x4.y; y.z += x4.z; y.w += x4.w; }
            *reinterpret_cast<float4 *>(x) = y;
            const __nv_bfloat162 g01 = *reinterpret_cast<const __nv_bfloat162 *>(&graw.x), g23 = *reinterpret_cast<const __nv_bfloat162 *>(&graw.y);
            __nv_bfloat162 lo = __floats2bfloat162_rn(__low2float(g01) * y.x, __high2float(g01) * y.y);
            __nv_bfloat162 hi = __floats2bfloat162_rn(__low2float(g23) * y.z, __high2float(g23) * y.w);
            *reinterpret_cast<uint2 *>(p.xb + (size_t)t * p.ldo + col) = make_uint2(*(uint32_t *)&lo, *(uint32_t *)&hi);
          }
          float sq = rowops::squares(y.x, y.y, y.z, y.w);
#pragma unroll
          for (int o = 16; o; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
          if (lane == 0) p.ss_out[(size_t)tile * OURO_TEXT_ROWS + t] = sq;
          return;
        }
        const float r = rs[t];
        float4 v4 = make_float4(acc.x * r, acc.y * r, acc.z * r, acc.w * r);
        if (swiglu || p.mode == MODE_QKV) {
          __nv_bfloat16 *dst;
          bool store = full4;
          if (swiglu || rope) {
            // the other half of the pair sits in another lane: gate with up, or dimension i with i + head_dim/2
            const int x = swiglu ? 16 : half >> 2;
            const float4 o4 = make_float4(__shfl_xor_sync(0xffffffffu, v4.x, x), __shfl_xor_sync(0xffffffffu, v4.y, x),
                                          __shfl_xor_sync(0xffffffffu, v4.z, x), __shfl_xor_sync(0xffffffffu, v4.w, x));
            if (swiglu) {
              const int feat = tile * 64 + 4 * ng;
              v4 = make_float4(rowops::silu(v4.x) * o4.x, rowops::silu(v4.y) * o4.y, rowops::silu(v4.z) * o4.z, rowops::silu(v4.w) * o4.w);
              dst = p.out_bf16 + (size_t)t * p.a_rows[0] + feat;
              store = ng < 16 && feat < p.a_rows[0];
            } else {
              const size_t ti = (size_t)spos[t] * half + (cm & (half - 1));
              const float4 cs = *reinterpret_cast<const float4 *>(p.cos_t + ti);
              float4 sn = *reinterpret_cast<const float4 *>(p.sin_t + ti);
              if ((cm & half) == 0) sn = make_float4(-sn.x, -sn.y, -sn.z, -sn.w);     // lower half: a cos - b sin
              v4 = make_float4(rowops::rotate(v4.x, o4.x, cs.x, sn.x), rowops::rotate(v4.y, o4.y, cs.y, sn.y),
                               rowops::rotate(v4.z, o4.z, cs.z, sn.z), rowops::rotate(v4.w, o4.w, cs.w, sn.w));
              dst = seg == 0 ? p.q_out + (size_t)t * p.dq + cm : p.k_out + (size_t)(p.L + t) * p.dkv + cm;
            }
          } else {
            dst = p.v_out + (size_t)(p.L + t) * p.dkv + cm;                          // v goes to the cache as it is
          }
          if (store) {
            __nv_bfloat162 lo = __floats2bfloat162_rn(v4.x, v4.y), hi = __floats2bfloat162_rn(v4.z, v4.w);
            *reinterpret_cast<uint2 *>(dst) = make_uint2(*(uint32_t *)&lo, *(uint32_t *)&hi);
          }
          return;
        }
        if (p.mode == MODE_HEAD) {                                   // the warp's 32 lanes hold the tile's 128 columns
          const float vals[4] = {v4.x, v4.y, v4.z, v4.w};
          uint32_t bu = 0;
          int bi = col;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const uint32_t uo = ordered_u32(vals[e]);
            if (full4 && uo > bu) { bu = uo; bi = col + e; }
          }
          const uint32_t mx = __reduce_max_sync(0xffffffffu, bu);
          const int src_lane = __ffs(__ballot_sync(0xffffffffu, bu == mx)) - 1;      // lowest lane = smallest index
          bi = __shfl_sync(0xffffffffu, bi, src_lane);
          if (lane == 0) {
            p.tile_max[(size_t)tile * OURO_MAX_ROWS + t] = ordered_f32(mx);
            p.tile_arg[(size_t)tile * OURO_MAX_ROWS + t] = bi;
          }
        }
        if (p.out_f32 && full4) {                                    // the row pitch is a multiple of 4 as well
          float *y = p.out_f32 + (size_t)t * p.ldo + col;
          if (p.mode == MODE_RESIDUAL) { const float4 y4 = *reinterpret_cast<const float4 *>(y); v4.x += y4.x; v4.y += y4.y; v4.z += y4.z; v4.w += y4.w; }
          *reinterpret_cast<float4 *>(y) = v4;
        }
      };

      if constexpr (!SPLIT) {
#pragma unroll 1
        for (int t = t_base + warp - 2; t < t_lim; t += EPI_WARPS)   // tokens are uniform inside a warp
          finish_token(t, *reinterpret_cast<const float4 *>(stg + (size_t)(t - t_base) * STAGE_PITCH + 4 * ng));
        return true;
      } else {
        // Twelve pieces are under way together: one token of twelve contributors, or, where there are more tokens than warps, four
        // tokens of three (7B prefill 13.2 -> 11.9 ms, 69 rows of the 34B shape 2.155 -> 2.130 ms).
        // With sixteen pieces the registers spill.  They are fetched without asking first whether they are there: a probe in
        // front is one more round trip to L2 between two GEMMs.
        const uint32_t of = cuts[tile - p.t0];
        const int first = of & 0xffff, n = of >> 16;
        float *slot = stg + (size_t)(warp - 2) * 4 * TILE_N + 4 * lane;       // this thread's 16 bytes of four parked tokens
        auto gather = [&](auto tb_c, int tb) -> bool {
          constexpr int TB = decltype(tb_c)::value, CB = 12 / TB;
          float4 acc[TB];
#pragma unroll
          for (int j = 0; j < TB; ++j) acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int c0 = 0; c0 < n; c0 += CB) {
            uint4 tmp[CB][TB];
            bool there = false;
            for (uint32_t spin = 0; spin < p.wait_limit; ++spin) {
              there = true;
#pragma unroll
              for (int cc = 0; cc < CB; ++cc) {
                const int owner = first + c0 + cc;
                const float *src = p.scratch + ((owner * 2 + w.owner_slot(tile, owner)) * slot_floats + tb * TILE_N + 4 * ng);
#pragma unroll
                for (int j = 0; j < TB; ++j)
                  tmp[cc][j] = part_load(src + j * TILE_N, c0 + cc < n && tb + j < t_lim);
              }
#pragma unroll
              for (int cc = 0; cc < CB; ++cc)
#pragma unroll
                for (int j = 0; j < TB; ++j) there = there && part_there(tmp[cc][j]);
              there = __all_sync(0xffffffffu, there);
              if (there) break;
              if ((spin & 15) == 15 && __any_sync(0xffffffffu, *abort_flag || *(volatile const int *)p.status != 0)) break;   // some CTA has given up
            }
            if (!there) return false;
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) {
              const int owner = first + c0 + cc;
              float *src = p.scratch + ((owner * 2 + w.owner_slot(tile, owner)) * slot_floats + tb * TILE_N + 4 * ng);
#pragma unroll
              for (int j = 0; j < TB; ++j) {
                if (c0 + cc < n && tb + j < t_lim) part_empty(src + j * TILE_N);
                acc[j].x += __uint_as_float(tmp[cc][j].x); acc[j].y += __uint_as_float(tmp[cc][j].y);
                acc[j].z += __uint_as_float(tmp[cc][j].z); acc[j].w += __uint_as_float(tmp[cc][j].w);
              }
            }
          }
          if (res_norm) {
            asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
            for (int j = 0; j < TB; ++j) {
              const float4 x = *reinterpret_cast<const float4 *>(slot + j * TILE_N);
              acc[j].x += x.x; acc[j].y += x.y; acc[j].z += x.z; acc[j].w += x.w;
            }
          }
#pragma unroll
          for (int j = 0; j < TB; ++j) *reinterpret_cast<float4 *>(slot + j * TILE_N) = acc[j];
          return true;
        };
        if (res_norm && full4) {
          for (int j = 0; j < tbn && t_base + j < t_lim; ++j)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(slot + j * TILE_N)),
                         "l"(p.out_f32 + (size_t)(t_base + j) * p.ldo + col) : "memory");
        }
        if (!(SIZE != ONE && tbn == 4 ? gather(std::integral_constant<int, SIZE == ONE ? 1 : 4>{}, t_base)
                                      : gather(std::integral_constant<int, 1>{}, t_base)))
          return false;
        if (et == 0) TRACE(12);
#pragma unroll 1
        for (int j = 0; j < tbn && t_base + j < t_lim; ++j)
          finish_token(t_base + j, *reinterpret_cast<const float4 *>(slot + j * TILE_N));
        return true;
      }
    };

    // Cut tiles.  Called once this CTA has published all its own partials, so waiting for the others cannot form a cycle.  The
    // (tile, tokens) pairs of all cut tiles are dealt out to all warps of the launch: with the contributors of a tile sharing its
    // tokens, the two tiles of a CTA whose span crosses a boundary decided how long it took (7B q,k,v, 37 rows: 7.5 us behind the
    // last contraction, now 5.6; output projection 5.8, now 3.9; 7B step 3221 -> 3154 us, 34B shape, 8 layers, 69 rows, 2121 ->
    // 2065 us).
    auto run_fixups = [&]() {
      const int n_cut = p.tiles - p.t0, warps = p.finishers * EPI_WARPS;
      // one token at a time, or four where there are more tokens than warps (7B step with 37 rows 3172 -> 3152 us; the longer code
      // costs a block that never needs it more: 19 rows of the 1.1B shape 5800 -> 5827 us, so up to ONE_ROWS there is none)
      const int tbn = SIZE != ONE && n_cut * rows > warps ? 4 : 1, items = n_cut * ((rows + tbn - 1) / tbn);
#pragma unroll 1
      for (int it = (warp - 2) * p.finishers + (int)blockIdx.x; it < items; it += warps) {
        const int group = it < n_cut ? 0 : it / n_cut;             // (one token: no division on the way to the next GEMM)
        if (!finish(std::true_type{}, p.t0 + it - group * n_cut, stage, tbn, group * tbn, rows)) {
          wait_flag[2] = 1;
          break;
        }
      }
      if (et == 0) TRACE(10);
      if (publish) __threadfence();                                // this thread's outputs, before the CTA's share counts as finished
      epi_barrier();
      if (et == 0 && publish && !wait_flag[2]) atomicAdd(cp.finished + ci, 1u);
      if (et == 0) TRACE(11);
      if (wait_flag[2]) ok = false;
      due = false;
    };

    if (ci > 0) {
      // this GEMM's per-token factors are sums over all tiles of the GEMM before it
      if (et == 0) wait_flag[0] = chain_wait(cp, ci - 1) && !*abort_flag;
      epi_barrier();
      ok = wait_flag[0] != 0;
      epi_barrier();
      if (!ok) break;
      __threadfence();
    }
    static_assert(EPI_THREADS >= MAX_CHAIN_ROWS, "one thread per token");
    if (et < MAX_CHAIN_ROWS) {
      float r = 1.0f;
      if (p.ss_in && et < rows) {
        float sum = 0.f;
        for (int i = 0; i < p.ss_tiles; ++i) sum += p.ss_in[(size_t)i * OURO_TEXT_ROWS + et];
        r = rowops::inv_rms(sum, p.ss_inv_d, p.eps);
      }
      rs[et] = r;
      spos[et] = (p.mode == MODE_QKV && et < rows) ? p.pos[et] : 0;
    }
    if (et == 0) wait_flag[2] = 0;
    if (p.per > 0 && et < p.tiles - p.t0) {                          // (fewer cut tiles than CTAs)
      const int first = et * p.kb / p.per;
      cuts[et] = (uint32_t)first | (uint32_t)((et * p.kb + p.kb - 1) / p.per - first + 1) << 16;
    }
    epi_barrier();

    for (;;) {
      const bool more = w.next(s);
      const int a = item & 1;
      // the stream-K spans come first: once the whole tiles start, this CTA has published all its partials and
      // can add up its share while the tensor cores work on the whole tile  (one call site: the routine is inlined)
      if (!more && et == 0) TRACE(5);
      if (due && (!more || s.whole)) run_fixups();
      if (!ok || !more) break;
      // one thread waits (bounded) and tells the others, so that all leave the loop together
      if (et == 0) wait_flag[a] = mbar_wait(&acc_full[a], (item >> 1) & 1, abort_flag) && !*abort_flag;
      epi_barrier();
      ok = wait_flag[a] != 0;
      if (!ok) break;
      if (et == 0) TRACE(4);                       // overwritten per item: the last accumulator's arrival remains
      fence_after_sync();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + a * acc_cols;
      if (s.whole) {
        // whole tile: the accumulators go to shared memory token-major, stage_tok tokens at a time, and are finished
        // from there; the TMEM buffer is handed back as soon as it has been read
        for (int c0 = 0; c0 < t_pad; c0 += stage_tok) {
          const int c1 = min(t_pad, c0 + stage_tok);
          for (int t0 = c0 + 16 * wh; t0 < c1; t0 += 32) {           // the quarter's two warps take 16 tokens in turn
            tmem_ld16(taddr + t0, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) stage[(t0 - c0 + i) * STAGE_PITCH + nl] = v[i];
          }
          if (c1 == t_pad) {
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[a]);
          }
          epi_barrier();
          finish(std::false_type{}, s.tile, stage, 0, c0, min(c1, rows));
          if (publish && c1 == t_pad) __threadfence();
          epi_barrier();
          if (publish && c1 == t_pad && et == 0) atomicAdd(cp.finished + ci, 1u);
        }
      } else {
        // partial tile: parked in this CTA's slot, for whoever finishes its tokens to fetch
        float *mine = p.scratch + ((int)blockIdx.x * 2 + s.slot) * slot_floats;
        for (int t0 = 16 * wh; t0 < rows; t0 += 32) {
          tmem_ld16(taddr + t0, v);
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (t0 + i < rows) part_store(mine + (size_t)(t0 + i) * TILE_N + nl, v[i]);
        }
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[a]);
      }
      ++item;
    }
    if (et == 0) TRACE(7);
    }
    if (!ok && et == 0) { *abort_flag = 1; atomicExch(p0.status, 1); }
  }
  // ------------------------------------------------------------------ teardown
  fence_before_sync();
  __syncthreads();
  if (*abort_flag && n_issued > 0) {               // (the two producer threads)
    // Somebody gave up: copies this lane issued may still be landing in this CTA's shared memory.  Wait (bounded) for
    // the last one of every stage before the CTA leaves; a stage whose other half was never requested cannot
    // complete its phase, which the limit covers (the bytes themselves arrive within microseconds).
    for (int st = 0; st < n_stages; ++st) {
      if (n_issued <= (uint32_t)st) continue;
      const uint32_t last = ((n_issued - 1 - st) / n_stages) * n_stages + st;      // last copy issued into this stage
      mbar_wait(&full[st], (last / n_stages) & 1, nullptr, 1u << 14);
    }
  }
  if (*abort_flag && warp == 1 && elect_one()) {   // ... and no contraction may still be running when TMEM is given back
    mma_commit(drain_bar);
    mbar_wait(drain_bar, 0, nullptr, 1u << 16);
  }
  __syncthreads();
  if (warp == 1) {
    fence_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)(2 * acc_cols)));
  }
}

// ------------------------------------------------------------------------------- host side
#include "gemm_rows.cuh"

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;

bool make_map(CUtensorMap *m, const void *base, int rows, int K, int box_rows) {
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  cuuint32_t box[2] = {BLOCK_K, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A matrix for the boxes of gemm_rows.cuh: rows of K values as [K / 64][rows][64], or, where a unit holds rotary pairs, as
// [K / 64][halves of heads][rows of a half][64].
bool make_map_rows(CUtensorMap *m, const void *base, int rows, int K, int box_rows, int nkb) {
  cuuint64_t dims[3] = {BLOCK_K, (cuuint64_t)rows, (cuuint64_t)(K / BLOCK_K)};
  cuuint64_t strides[2] = {(cuuint64_t)K * 2, BLOCK_K * 2};
  cuuint32_t box[3] = {BLOCK_K, (cuuint32_t)box_rows, (cuuint32_t)nkb};
  cuuint32_t es[3] = {1, 1, 1};
  return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool make_map_pairs(CUtensorMap *m, const void *base, int rows, int K, int half, int nkb) {
  cuuint64_t dims[4] = {BLOCK_K, (cuuint64_t)half, (cuuint64_t)(rows / half), (cuuint64_t)(K / BLOCK_K)};
  cuuint64_t strides[3] = {(cuuint64_t)K * 2, (cuuint64_t)half * K * 2, BLOCK_K * 2};
  cuuint32_t box[4] = {BLOCK_K, 8, 2, (cuuint32_t)nkb};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct LayerMaps {
  CUtensorMap wq, wk, wv, wo, wg, wu, wd;
  CUtensorMap hq, hk, hv, ho, hd;       // half tiles: boxes of 64 rows, as wg and wu have them
};
// What launches of gemm_rows.cuh need of a model: per kind of GEMM how it is dealt out, and its boxes.
enum { G_QKV = 0, G_WO = 1, G_GATEUP = 2, G_DOWN = 3, G_HEAD = 4 };
struct RowsModel {
  int x_bytes = 0;                    // (0: none)
  int slot = 0;                       // bytes of a ring slot
  rows_gemm::Plan plan[5];
  CUtensorMap head;
  struct Layer { CUtensorMap q, k, v, o, g, u, d; };
  std::vector<Layer> layers;
};
struct FastModel {
  bool ok = false;
  RowsModel rm;
  std::vector<LayerMaps> layers;
  CUtensorMap head;
  CUtensorMap kmap, vmap;               // K and V caches as [layers * max_seq][kv width], box 64 x 128 (tcgen05 attention)
  bool kv_maps = false;
  CUtensorMap x_d[16], x_q[16], x_f[16];   // activations normed [512, d], attention out [512, dq], SwiGLU out [512, F]; box rows 16, 32, .., 256
};
struct FastState {
  FastModel m[2];
  int grid = 0;
  int smem_max = 0;
  float *slots = nullptr;
  float *attn_part = nullptr;   // per-chunk softmax pieces of the split attention
  float *tile_max = nullptr;    // LM head: per-tile best logit and index of every token
  int *tile_arg = nullptr;
  float *ss = nullptr;          // per-tile sums of squares of the residual stream (RMSNorm folded into the GEMMs)
  uint32_t *finished = nullptr; // [MAX_CHAIN + 1] finished-tile counters of the chained GEMMs (device)
  uint32_t finished_host[MAX_CHAIN + 1] = {0, 0, 0, 0, 0};   // the values those counters have once everything launched so far is done
  ChainParams chain{};          // GEMMs collected for the next launch
  int chain_layer[MAX_CHAIN] = {0, 0, 0, 0}, chain_model = 0;
  uint4 *packets = nullptr;     // activations on their way: normed, attention out, SwiGLU out  (gemm_rows.cuh)
  size_t packets_size = 0;      // bytes
  uint32_t mark = 1;            // of the next launch's first packets; never zero, which an empty packet has
  uint32_t late = 0;            // test aid, see rows_gemm::Params
  uint32_t rows_launches = 0;   // of gemm_rows.cuh so far
  uint32_t few_launches = 0;    // of attn_few.cu
  float *squares = nullptr;     // squares of four columns each of the residual stream, as gemm_rows.cuh leaves them
  int chain_kind[MAX_CHAIN] = {0, 0, 0, 0};
  bool fuse = true;             // run consecutive GEMMs as one launch
  long pf_ffn_rows = 0;         // rows of gate and of up the attention kernel prefetches into L2 besides the output projection (< 0: nothing)
};
constexpr int MAX_TILES = 4096;
constexpr int CHAIN_BYTES = 256;           // the chain counters

size_t slots_bytes() { return (size_t)MAX_GRID * 2 * TILE_N * MAX_CHAIN_ROWS * sizeof(float); }
size_t tile_best_bytes() { return (size_t)MAX_TILES * OURO_MAX_ROWS * 4; }
constexpr int MAX_SS_TILES = 64;           // d_model <= 8192
// A token's activations, the widest of them, in the shared memory of a CTA of gemm_rows.cuh; 0: the model's single rows do not run
// there (nor do they where rows_pay says so).  What those kernels save is the latency between a layer's GEMMs, what they cost is a chain of steps per weight row, and the
// wider a layer, the more the stream of its weights hides of either.  One row behind 150 / 400 / 1800 keys, us a forward, gemm_tc.cu
// and here: two layers of 512 (4 MB a layer) 59, 63, 65 and 44, 48, 48; eight of the 1.1B shape (88 MB) 304, 305, 342 and 250, 250,
// 288; six of 2048 x 8192 (121 MB) 260, 261, 290 and 233, 234, 262; six of 2560 x 6912 (137 MB) 279, 280, 308 and 250, 252, 278;
// four of 3072 x 8192 (201 MB) 239, 255, 269 and 241, 247, 248; three of the 7B shape (405 MB) 285, 300, 322 and 290, 304, 325.
int rows_x_bytes(const ouro_model_desc &d) {
  const int dq = d.n_heads * d.head_dim, dkv = d.n_kv_heads * d.head_dim, x = 2 * std::max(std::max(d.d_model, dq), d.d_ffn);
  const size_t layer = 2 * (size_t)d.d_model * (2 * (size_t)(dq + dkv) + 3 * (size_t)d.d_ffn);
  return (d.head_dim == 64 || d.head_dim == 128) && layer <= (size_t)160 << 20 && x <= rows_gemm::MAX_X ? x : 0;
}
size_t squares_bytes() { return (size_t)MAX_SS_TILES * (TILE_N / 4) * sizeof(float); }
size_t packets_bytes(const ouro_model_desc &d) {
  return (size_t)(d.d_model + d.n_heads * d.head_dim + d.d_ffn) / 4 * sizeof(uint4);
}
size_t ss_bytes() { return (size_t)MAX_SS_TILES * OURO_TEXT_ROWS * sizeof(float); }

int stages_for(int t_pad, int smem_max) {
  int stage = A_BYTES + t_pad * BLOCK_K * 2;
  int fixed = 1024 + stage_tokens(t_pad) * STAGE_PITCH * 4 + MISC_BYTES;  // alignment slack, parked whole tile, the rest
  int s = (smem_max - fixed) / stage;
  return s > 12 ? 12 : s;
}

}  // namespace

struct ouro_fast { FastState s; };

size_t ouro_scratch_bytes(const ouro_model_desc *t, const ouro_model_desc *d) {
  size_t attn = attention_tc_scratch_bytes(*t);
  if (d && attention_tc_scratch_bytes(*d) > attn) attn = attention_tc_scratch_bytes(*d);
  return slots_bytes() + CHAIN_BYTES + 2 * tile_best_bytes() + ss_bytes() + attn;
}
size_t ouro_single_bytes(const ouro_model_desc *t, const ouro_model_desc *d) {
  return squares_bytes() + std::max(packets_bytes(*t), d ? packets_bytes(*d) : 0);
}

static bool shape_ok(const ouro_model_desc &d) {
  int dq = d.n_heads * d.head_dim;
  return d.dtype == OURO_BF16 && d.d_model % 64 == 0 && d.d_model <= MAX_SS_TILES * TILE_N && dq % 64 == 0 && d.d_ffn % 64 == 0 && d.vocab % 8 == 0 &&
         (d.vocab + TILE_N - 1) / TILE_N <= MAX_TILES && (2 * d.d_ffn + TILE_N - 1) / TILE_N <= MAX_TILES;
}

// All units of a pass lie in one tile, and are cut alike, where their number divides a tile's (a matrix begins at a multiple of four): the
// ring then takes the k-blocks of several pieces in turn.
static void rows_share(rows_gemm::Plan &pl, int kb, int per, int slots) {
  pl.max_pieces = per > 0 && per < kb ? std::min(kb, (kb - 1) / per + 2) : 1;
  pl.share = pl.up <= 2 || pl.up == 4 ? std::min(std::min(rows_gemm::CW / pl.up, pl.max_pieces), slots - 1) : 1;
  if (pl.up * pl.max_pieces > rows_gemm::PARKED) pl.share = 1;
}
// How a GEMM is dealt out to the CTAs, and how many k-blocks a ring slot holds.
static rows_gemm::Plan rows_plan(int kind, int units, int kb, int tiles, int grid, int slot) {
  rows_gemm::Plan pl{};
  const int chunk = (units + grid - 1) / grid;
  pl.units = units;
  pl.passes = (chunk + rows_gemm::MAX_UP - 1) / rows_gemm::MAX_UP;
  pl.up = (chunk + pl.passes - 1) / pl.passes;
  const ws::Cut cut = ws::cut(tiles, kb, std::min(grid, tiles * kb), std::min(grid, tiles * kb));
  const bool in_turn = cut.t0 == 0 && cut.per < kb && (pl.up <= 2 || pl.up == 4);      // (as launch_rows will have it, if the grid is what it is alone)
  const int len = in_turn ? cut.per : kb, fit = std::min(len, slot / (pl.up * rows_gemm::UNIT * 128)), steps = (len + fit - 1) / fit;
  pl.nkb = (len + steps - 1) / steps;
  pl.cut_per = cut.per;
  if (kind == G_QKV) { pl.su = rows_gemm::UNIT * pl.nkb; pl.sj = rows_gemm::UNIT; pl.sh = 8; }
  else if (kind == G_GATEUP) { pl.su = 8; pl.sj = 8 * pl.up; pl.sh = 8 * pl.up * pl.nkb; }
  else { pl.su = rows_gemm::UNIT; pl.sj = rows_gemm::UNIT * pl.up; pl.sh = 8; }
  return pl;
}
// Whether owned weight rows are faster than gemm_tc_kernel's cut tiles.  They save the tails and the hand-overs' round trips, 2 to 8 us a
// layer, and with head dim 128 in several spans of keys the attention in front as well (attention_few_pays).  They cost a chain: the k-blocks
// that the busiest warp of a GEMM takes one behind another, 0.1 us each, where gemm_tc_kernel deals a long K out to all SMs.  `beyond` is what
// a layer's chains take longer than the streams of their weights, in us; `late` the same against 0.4 of the streams, of which a long
// one on few warps does not hide all.  One row, three layers, gemm_tc.cu over here behind 150 / 1800 keys, of d_model x d_ffn (beyond, late),
// measured on 157 shapes:
//   head dim 128: 512 x 2048 1.05 / 1.22 (2.9, 3.2), 512 x 3072 1.05 / 1.22 (4.3, 5.1), 768 x 3072 0.96 / 1.13 (4.1, 5.4), 384 x 3072 0.94 / 1.10 (4.5,
//   5.1), 768 x 4608 0.92 / 1.09 (6.1, 7.3), 256 x 1792 with 2048 query columns 0.90 / 1.04 (5.7, 5.9), 512 x 28672 0.53 / 0.58 (40, 43); 2176 x 3968
//   1.04 / 1.20 (0, 3.1), 2560 x 7040 1.08 / 1.17 (0, 2.0), 1024 x 11264 1.14 / 1.28 (0, 1.9), 1536 x 9216 0.96 / 0.99 (0, 2.3), 1536 x 16896 0.93 / 0.93
//   (0.9, 6.6), 4096 x 2048 0.97 / 1.11 (0, 6.3)
//   head dim 64: 2048 x 5632 1.2 / 1.2 (0, 1.3), 256 x 1600 1.13 / 1.09 (2.5, 2.7), 2240 x 768 1.00 / 1.01 (3.1, 3.6), 384 x 3200 1.06 / 1.07 (4.7, 5.4), 384
//   x 1024 with 3072 query columns 0.95 / 0.96 (4.5, 4.8), 320 x 1600 0.97 / 0.96 (5.0, 5.2), 1984 x 256 0.88 / 0.90 (5.6, 6.0); 4096 x 4096 with 512
//   query columns 0.96 / 0.97 (0, 2.9): the worst that is let in
// The head costs up to 1 us more in each of its passes than it does there, which a layer's saving makes up for four of: one layer in front of 3 / 6
// passes 1.02 to 1.19 / 0.96 to 1.05, two in front of 6 / 12 1.01 to 1.16 / 0.96 to 1.05, three in front of 12 1.005 to 1.09 (256 to 2048 wide, 150 keys).
static bool rows_pay(const rows_gemm::Plan *plan, const int *kb, int head_dim, int n_layers) {
  double beyond = 0, late = 0;
  for (int k = 0; k < 4; ++k) {
    const rows_gemm::Plan &pl = plan[k];
    const int step = (pl.cut_per + pl.nkb - 1) / pl.nkb * pl.nkb;
    const double walk = 0.1 * pl.passes * (pl.share == 1 ? kb[k] : (pl.max_pieces + pl.share - 1) / pl.share * step);
    const double stream = (double)pl.units * rows_gemm::UNIT * kb[k] * BLOCK_K * 2 / 6.5e6;
    beyond += std::max(0.0, walk - stream);
    late += std::max(0.0, walk - 0.4 * stream);
  }
  return beyond <= (head_dim == 128 ? 4.4 : 3.3) && late <= 6.0 && plan[G_HEAD].passes <= 4 * n_layers;
}
static bool rows_setup(int grid, int smem_max, const ModelRt &M, RowsModel &rm) {
  const ouro_model_desc &d = M.d;
  const int dq = d.n_heads * d.head_dim, dkv = d.n_kv_heads * d.head_dim, half = d.head_dim / 2, U = rows_gemm::UNIT;
  auto tiles = [](int n) { return (n + TILE_N - 1) / TILE_N; };
  const int n_units[5] = {(dq + 2 * dkv) / U, d.d_model / U, d.d_ffn / 8, d.d_model / U, (d.vocab + U - 1) / U};
  const int n_tiles[5] = {tiles(dq) + 2 * tiles(dkv), tiles(d.d_model), tiles(2 * d.d_ffn), tiles(d.d_model), tiles(d.vocab)};
  const int K[5] = {d.d_model, dq, d.d_model, d.d_ffn, d.d_model};
  // A slot takes two k-blocks of gate and up, more than half of a layer's weights: with room for less or with some left over the ring is
  // shorter than it could be (one row behind 400 keys, us a forward with slots of 20 / 24 / 30 / 36 KB: eight layers of the 1.1B shape,
  // five units of gate and up a CTA, 248 / 259 / 270 / 279; six of 2560 x 6912, six units, 267 / 251 / 263 / 257; six of 2048 x 8192,
  // seven units, 242 / 240 / 237 / 243).
  rm.slot = rows_gemm::MIN_SLOT;
  const int gu = rows_plan(G_GATEUP, n_units[G_GATEUP], K[G_GATEUP] / BLOCK_K, n_tiles[G_GATEUP], grid, rm.slot).up;
  if (gu <= 8) rm.slot = std::max(rm.slot, 2 * gu * U * 128);
  int kb[5];
  for (int k = 0; k < 5; ++k) {
    kb[k] = K[k] / BLOCK_K;
    rm.plan[k] = rows_plan(k, n_units[k], kb[k], n_tiles[k], grid, rm.slot);
    rows_share(rm.plan[k], kb[k], rm.plan[k].cut_per, rows_gemm::slots_for(rm.slot, d.d_model + rows_x_bytes(d), smem_max));
  }
  if (!rows_pay(rm.plan, kb, d.head_dim, d.n_layers)) return true;
  auto plain = [&](CUtensorMap *m, const void *w, int rows, int kind) {
    return make_map_rows(m, w, rows, K[kind], rm.plan[kind].up * (kind == G_GATEUP ? 8 : U), rm.plan[kind].nkb);
  };
  bool ok = plain(&rm.head, M.lm_head, d.vocab, G_HEAD);
  rm.layers.resize(d.n_layers);
  for (int l = 0; l < d.n_layers && ok; ++l) {
    RowsModel::Layer &lm = rm.layers[l];
    ok = make_map_pairs(&lm.q, M.wq[l], dq, d.d_model, half, rm.plan[G_QKV].nkb) &&
         make_map_pairs(&lm.k, M.wk[l], dkv, d.d_model, half, rm.plan[G_QKV].nkb) &&
         make_map_pairs(&lm.v, M.wv[l], dkv, d.d_model, half, rm.plan[G_QKV].nkb) &&
         plain(&lm.o, M.wo[l], d.d_model, G_WO) && plain(&lm.g, M.w_gate[l], d.d_ffn, G_GATEUP) &&
         plain(&lm.u, M.w_up[l], d.d_ffn, G_GATEUP) && plain(&lm.d, M.w_down[l], d.d_model, G_DOWN);
  }
  rm.x_bytes = rows_x_bytes(d);
  return ok;
}

int ouro_fast_setup(ouro_ctx *c) {
  c->fast = nullptr;
  bool any = false;
  for (auto &M : c->m) any = any || (M.present && shape_ok(M.d));
  if (!any) return OURO_OK;
  int dev = 0, sms = 0, smem = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    c->err = "device attributes unavailable";
    return OURO_ECUDA;
  }
  if (!g_encode) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn) {
      c->err = "cuTensorMapEncodeTiled unavailable";
      return OURO_ECUDA;
    }
    g_encode = (EncodeTiledFn)fn;
  }
  ouro_fast *f = new ouro_fast();
  f->s.grid = sms < MAX_GRID ? sms : MAX_GRID;
  f->s.smem_max = smem;
  f->s.slots = c->a.scratch;
  f->s.finished = (uint32_t *)((char *)c->a.scratch + slots_bytes());
  {
    const char *e = getenv("OURO_FUSE");                       // OURO_FUSE=0: every GEMM is a launch of its own
    f->s.fuse = !(e && e[0] == '0');
    const char *pf = getenv("OURO_PF_ROWS");
    if (pf) f->s.pf_ffn_rows = atol(pf);
    const char *c0 = getenv("OURO_COUNT_START");                // test aid: what the hand-over counters start at
    if (c0) {
      for (uint32_t &v : f->s.finished_host) v = (uint32_t)strtoul(c0, nullptr, 0);
      f->s.mark = std::max(1u, (uint32_t)strtoul(c0, nullptr, 0));                   // (and the packets' marks)
    }
    const char *late = getenv("OURO_LATE_NS");                  // test aid: a late warp in gemm_rows.cuh, at most 0.1 ms a GEMM
    if (late) f->s.late = (uint32_t)std::min(strtoul(late, nullptr, 0), 100000ul);
  }
  f->s.tile_max = (float *)((char *)c->a.scratch + slots_bytes() + CHAIN_BYTES);
  f->s.tile_arg = (int *)((char *)f->s.tile_max + tile_best_bytes());
  f->s.ss = (float *)((char *)f->s.tile_arg + tile_best_bytes());
  f->s.attn_part = (float *)((char *)f->s.ss + ss_bytes());
  size_t packets = 0;                                           // (one model computes at a time)
  for (auto &M : c->m)
    if (M.present) packets = std::max(packets, packets_bytes(M.d));
  f->s.squares = c->a.single;
  f->s.packets = (uint4 *)((char *)f->s.squares + squares_bytes());
  f->s.packets_size = packets;
  if (cudaMemsetAsync(f->s.slots, 0xff, slots_bytes(), c->stream) != cudaSuccess ||
      cudaMemsetAsync(f->s.packets, 0, packets, c->stream) != cudaSuccess ||
      cudaMemcpyAsync(f->s.finished, f->s.finished_host, sizeof(f->s.finished_host), cudaMemcpyHostToDevice, c->stream) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<FEW>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<SOME>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<MANY>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaFuncSetAttribute(rows_gemm::gemm_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      text_gemm_setup() != OURO_OK || attention_tc_setup() != OURO_OK || attention_tm_setup() != OURO_OK || attention_few_setup() != OURO_OK) {
    delete f;
    c->err = "tensor-core GEMM set-up failed";
    return OURO_ECUDA;
  }
  for (int w = 0; w < 2; ++w) {
    ModelRt &M = c->m[w];
    if (!M.present || !shape_ok(M.d)) continue;
    const ouro_model_desc &d = M.d;
    FastModel &fm = f->s.m[w];
    const int dq = d.n_heads * d.head_dim, dkv = d.n_kv_heads * d.head_dim;
    bool ok = true;
    fm.layers.resize(d.n_layers);
    for (int l = 0; l < d.n_layers && ok; ++l) {
      LayerMaps &lm = fm.layers[l];
      ok = make_map(&lm.wq, M.wq[l], dq, d.d_model, TILE_N) && make_map(&lm.wk, M.wk[l], dkv, d.d_model, TILE_N) &&
           make_map(&lm.wv, M.wv[l], dkv, d.d_model, TILE_N) && make_map(&lm.wo, M.wo[l], d.d_model, dq, TILE_N) &&
           make_map(&lm.wg, M.w_gate[l], d.d_ffn, d.d_model, 64) && make_map(&lm.wu, M.w_up[l], d.d_ffn, d.d_model, 64) &&
           make_map(&lm.wd, M.w_down[l], d.d_model, d.d_ffn, TILE_N) && make_map(&lm.hq, M.wq[l], dq, d.d_model, 64) &&
           make_map(&lm.hk, M.wk[l], dkv, d.d_model, 64) && make_map(&lm.hv, M.wv[l], dkv, d.d_model, 64) &&
           make_map(&lm.ho, M.wo[l], d.d_model, dq, 64) && make_map(&lm.hd, M.w_down[l], d.d_model, d.d_ffn, 64);
    }
    ok = ok && make_map(&fm.head, M.lm_head, d.vocab, d.d_model, TILE_N);
    if (ok && attention_tm_supported(d)) {
      ok = make_map(&fm.kmap, M.k_cache, d.n_layers * d.max_seq, dkv, 128) && make_map(&fm.vmap, M.v_cache, d.n_layers * d.max_seq, dkv, 128);
      fm.kv_maps = ok;
    }
    for (int i = 0; i < 16 && ok; ++i)
      ok = make_map(&fm.x_d[i], c->a.xn, OURO_TEXT_ROWS, d.d_model, 16 * (i + 1)) &&
           make_map(&fm.x_q[i], c->a.att, OURO_TEXT_ROWS, dq, 16 * (i + 1)) &&
           make_map(&fm.x_f[i], c->a.act, OURO_TEXT_ROWS, d.d_ffn, 16 * (i + 1));
    if (ok && rows_x_bytes(d) > 0) ok = rows_setup(f->s.grid, smem, M, fm.rm);
    if (!ok) {
      delete f;
      c->err = "cuTensorMapEncodeTiled failed";
      return OURO_ECUDA;
    }
    fm.ok = true;
  }
  c->fast = f;
  return OURO_OK;
}

void ouro_fast_teardown(ouro_ctx *c) {
  delete c->fast;
  c->fast = nullptr;
}

// The weight side of one GEMM of the forward: which matrices, how they are tiled, how long K is.
struct WeightSide {
  CUtensorMap a[3];
  int a_tiles[3] = {0, 0, 0}, a_rows[3] = {0, 0, 0}, a_count = 1, tiles = 0, K = 0;
  bool swiglu = false;
};
static WeightSide weight_side(const ouro_model_desc &d, const FastModel &fm, int l, int kind) {
  auto tiles = [](int n) { return (n + TILE_N - 1) / TILE_N; };
  const int dq = d.n_heads * d.head_dim, dkv = d.n_kv_heads * d.head_dim;
  WeightSide w;
  switch (kind) {
    case G_QKV: {
      const LayerMaps &lm = fm.layers[l];
      w.a[0] = lm.wq; w.a[1] = lm.wk; w.a[2] = lm.wv;
      w.a_tiles[0] = tiles(dq); w.a_tiles[1] = tiles(dkv); w.a_tiles[2] = tiles(dkv);
      w.a_rows[0] = dq; w.a_rows[1] = dkv; w.a_rows[2] = dkv;
      w.a_count = 3;
      w.tiles = w.a_tiles[0] + w.a_tiles[1] + w.a_tiles[2];
      w.K = d.d_model;
      break;
    }
    case G_WO:
      w.a[0] = fm.layers[l].wo; w.a_tiles[0] = tiles(d.d_model); w.a_rows[0] = d.d_model;
      w.tiles = w.a_tiles[0];
      w.K = dq;
      break;
    case G_GATEUP:
      w.a[0] = fm.layers[l].wg; w.a[1] = fm.layers[l].wu; w.a_rows[0] = d.d_ffn; w.a_count = 2;
      w.tiles = (d.d_ffn + 63) / 64;
      w.K = d.d_model;
      w.swiglu = true;
      break;
    case G_DOWN:
      w.a[0] = fm.layers[l].wd; w.a_tiles[0] = tiles(d.d_model); w.a_rows[0] = d.d_model;
      w.tiles = w.a_tiles[0];
      w.K = d.d_ffn;
      break;
    default:
      w.a[0] = fm.head; w.a_tiles[0] = tiles(d.vocab); w.a_rows[0] = d.vocab;
      w.tiles = w.a_tiles[0];
      w.K = d.d_model;
      break;
  }
  return w;
}
struct Gemm : GemmParams { GemmMaps m; };
static void set_weights(Gemm &p, const WeightSide &w) {
  for (int i = 0; i < 3; ++i) { p.m.a[i] = w.a[i]; p.a_tiles[i] = w.a_tiles[i]; p.a_rows[i] = w.a_rows[i]; }
  p.a_count = w.a_count;
  p.tiles = w.tiles;
}
static int grid_for(const FastState &s, int tiles, int kb) {
  const long total = (long)tiles * kb;
  return total < s.grid ? (int)total : s.grid;
}
// What the hand-over counter of a GEMM advances by: one count per whole tile and one per CTA that has finished its share of the
// cut tiles.
static int finish_units(const GemmParams &g) { return g.per == g.kb ? g.tiles : g.t0 + (g.per > 0 ? g.finishers : 0); }
static bool rows_launch(const FastModel &fm, int rows) { return rows == 1 && fm.rm.x_bytes > 0; }
static void launch_rows(ouro_ctx *c) {
  FastState &s = c->fast->s;
  ChainArgs &cp = s.chain.args;
  const RowsModel &rm = s.m[s.chain_model].rm;
  const ouro_model_desc &d = c->m[s.chain_model].d;
  const int dq = d.n_heads * d.head_dim;
  rows_gemm::Params kp;
  kp.squares_bytes = d.d_model;
  kp.slot = rm.slot;
  kp.slots = rows_gemm::slots_for(rm.slot, d.d_model + rm.x_bytes, s.smem_max);
  if (s.mark > UINT32_MAX - (MAX_CHAIN + 1)) {                    // some hours of decoding: the marks begin anew, on empty packets
    if (cudaMemsetAsync(s.packets, 0, s.packets_size, c->stream) != cudaSuccess) return;   // (the layer finds the error; nothing begins anew)
    s.mark = 1;
  }
  kp.mark = s.mark;
  s.mark += MAX_CHAIN + 1;
  kp.late = s.late;
  uint4 *px = s.packets, *patt = px + d.d_model / 4, *pact = patt + dq / 4;
  const bool front = cp.fold.part || cp.embed.table;
  int grid = front ? s.grid : 1;
  for (int i = 0; i < cp.n; ++i) {
    const int kind = s.chain_kind[i];
    const GemmParams &g = cp.g[i];
    rows_gemm::Plan &pl = kp.told.plan[i];
    pl = rm.plan[kind];
    grid = std::max(grid, (pl.units + pl.up * pl.passes - 1) / (pl.up * pl.passes));
    rows_share(pl, g.kb, g.per, kp.slots);                        // (the cut is the chain's)
    pl.q_in = pl.q_out = s.squares;
    pl.x_in = (const __nv_bfloat16 *)(kind == G_WO ? c->a.att : kind == G_DOWN ? c->a.act : c->a.xn);
    if (i > 0 || front) pl.packets_in = kind == G_WO ? patt : kind == G_DOWN ? pact : px;
    if (i + 1 < cp.n) pl.packets_out = kind == G_GATEUP ? pact : px;
    const RowsModel::Layer *l = kind == G_HEAD ? nullptr : &rm.layers[s.chain_layer[i]];
    CUtensorMap *w = kp.w[i];
    switch (kind) {
      case G_QKV: w[0] = l->q; w[1] = l->k; w[2] = l->v; break;
      case G_WO: w[0] = l->o; break;
      case G_GATEUP: w[0] = l->g; w[1] = l->u; break;
      case G_DOWN: w[0] = l->d; break;
      default: w[0] = rm.head; break;
    }
  }
  kp.front = cp.fold.part ? patt : px;
  kp.told.args = cp;
  ++s.rows_launches;
  launch_pdl(rows_gemm::gemm_rows_kernel, grid, rows_gemm::THREADS, (size_t)s.smem_max, c->stream, kp);
}
// Launches the GEMMs collected so far as one chain.
static void flush_chain(ouro_ctx *c) {
  FastState &s = c->fast->s;
  ChainArgs &cp = s.chain.args;
  if (cp.n == 0) return;
  OURO_COUNT_LAUNCH();
  int grid = 1;
  for (int i = 0; i < cp.n; ++i) grid = std::max(grid, grid_for(s, cp.g[i].tiles, cp.g[i].kb));
  cp.finished = s.finished;
  for (int i = 0; i < cp.n; ++i) {
    const ws::Cut cut = ws::cut(cp.g[i].tiles, cp.g[i].kb, grid, grid);
    cp.g[i].t0 = cut.t0;
    cp.g[i].per = cut.per;
    cp.g[i].finishers = grid;
  }
  const bool few = rows_launch(s.m[s.chain_model], cp.g[0].rows);
  for (int i = 0; i + 1 < cp.n && !few; ++i) cp.target[i] = (s.finished_host[i] += finish_units(cp.g[i]));
  if (!few && (cp.fold.part || cp.embed.table)) cp.fold_target = (s.finished_host[MAX_CHAIN] += grid);
  const bool per_kind = cp.n == 1 && c->prof_class >= OURO_PROF_QKV && c->prof_class <= OURO_PROF_HEAD;
  static const int kind_class[5] = {OURO_PROF_QKV, OURO_PROF_WO, OURO_PROF_GATEUP, OURO_PROF_DOWN, OURO_PROF_HEAD};
  {
    ProfScope ps(c, per_kind ? kind_class[s.chain_kind[0]] : OURO_PROF_GEMM);
    const int t_pad = cp.g[0].t_pad;
    if (few) launch_rows(c);
    else launch_pdl(t_pad > OURO_MAX_ROWS ? gemm_tc_kernel<MANY> : t_pad > FEW_ROWS ? gemm_tc_kernel<SOME>
               : t_pad > ONE_ROWS ? gemm_tc_kernel<FEW> : gemm_tc_kernel<ONE>,
               grid, THREADS, (size_t)s.smem_max, c->stream, s.chain);
  }
  cp.n = 0;
  cp.fold.part = nullptr;
  cp.embed.table = nullptr;
}

// Adds a GEMM to the chain under construction; `last` launches the chain (something other than a GEMM follows).
static void push_gemm(ouro_ctx *c, int which, int layer, Gemm &p, int kind, const CUtensorMap *xmaps, int K, int rows, bool last) {
  FastState &s = c->fast->s;
  p.kb = K / BLOCK_K;
  p.rows = rows;
  p.t_pad = (rows + 15) & ~15;
  p.m.b = xmaps[p.t_pad / 16 - 1];
  p.stages = stages_for(p.t_pad, s.smem_max);
  p.scratch = s.slots;
  p.status = &c->st->status;
  p.rows_dev = c->cur_rows_dev;
  p.trace_id = kind;
  p.wait_limit = c->wait_limit;
  ChainArgs &cp = s.chain.args;
  if (cp.n > 0 && cp.g[0].rows != rows) flush_chain(c);             // cannot happen inside one forward
  s.chain_kind[cp.n] = kind;
  s.chain_layer[cp.n] = layer;
  s.chain_model = which;
  s.chain.maps[cp.n] = p.m;
  cp.g[cp.n++] = p;
  // one launch per GEMM when asked for, and while a single kind of GEMM is being timed
  const bool split = !s.fuse || (c->prof_class >= OURO_PROF_QKV && c->prof_class <= OURO_PROF_HEAD);
  if (last || split || cp.n == MAX_CHAIN) flush_chain(c);
}

// Forgets the chain under construction.
void ouro_fast_reset(ouro_ctx *c) {
  if (!c->fast) return;
  ChainArgs &cp = c->fast->s.chain.args;
  cp.n = 0;
  cp.fold.part = nullptr;
  cp.embed.table = nullptr;
}
// values[1..8] of ouro_debug_counts.
void ouro_fast_counts(const ouro_ctx *c, uint32_t *values) {
  if (!c->fast) return;
  const FastState &s = c->fast->s;
  static_assert(OURO_DEBUG_COUNTS == 4 + MAX_CHAIN + 1, "one value each");
  values[1] = s.rows_launches;
  values[2] = s.few_launches;
  values[3] = s.mark;
  for (int i = 0; i <= MAX_CHAIN; ++i) values[4 + i] = s.finished_host[i];
}
// What the launches so far leave behind if one of them has given up.
Leftovers ouro_leftovers(ouro_ctx *c) {
  Leftovers l;
  l.met = c->met_dev;
  if (!c->fast) return l;
  const FastState &s = c->fast->s;
  l.slots = (uint4 *)s.slots;
  l.n_slots = slots_bytes() / sizeof(uint4);
  l.empty = EMPTY;
  l.counters = s.finished;
  l.n_counters = MAX_CHAIN + 1;
  for (int i = 0; i <= MAX_CHAIN; ++i) l.value[i] = s.finished_host[i];
  return l;
}

// The row count of a candidate block may stay on the device when every kernel of the forward reads it from there:
// the tensor-core GEMMs with the rotary epilogue and one of the two tensor-core attention kernels.
bool ouro_fast_available(ouro_ctx *c, int which) {
  if (!c->fast || !c->fast->s.m[which].ok) return false;
  const ouro_model_desc &d = c->m[which].d;
  return d.head_dim == 64 || d.head_dim == 128;
}

bool ouro_fast_layers(ouro_ctx *c, int which) { return c->fast && c->fast->s.m[which].ok; }

// Blocks that run on the kernels of gemm_text.cu: those longer than a chained launch takes.  Up to there the chain is faster, beyond
// it would take two.  A prompt's prefill in us with the chain and with gemm_text.cu: 7B shape, four layers, 193 rows 501 and 656, 256
// rows 569 and 665, 257 rows 862 and 800, 300 rows 927 and 829, 512 rows 1228 and 912; 34B shape, two layers, 256 rows 430 and 454, 257
// rows 683 and 610; 1.1B shape, four layers, 256 rows 375 and 410, 257 rows 493 and 480; two layers of 512 x 512, 256 rows 106 and 108,
// 257 rows 136 and 99.  The widest shapes gain last: 70B, two layers, 257 rows 932 and 963, 384 rows 1035 and 1061, 512 rows 1238 and 1118.
static bool text_rows(int rows) { return rows > MAX_CHAIN_ROWS; }

// The embedding gather runs in front of the first layer's q,k,v GEMM, inside its launch.
int ouro_fast_embed(ouro_ctx *c, int which, int rows) {
  if (!c->fast || !c->fast->s.m[which].ok) return OURO_ESTATE;
  ModelRt &M = c->m[which];
  ChainArgs &cp = c->fast->s.chain.args;
  cp.n = 0;
  cp.fold.part = nullptr;
  rowops::Embed own, &e = text_rows(rows) ? own : cp.embed;
  e.table = (const __nv_bfloat16 *)M.embed;
  e.tok = M.blk.tok;
  e.gain = (const __nv_bfloat16 *)M.attn_norm[0];
  e.x = c->a.x;
  e.xb = (__nv_bfloat16 *)c->a.xn;
  e.ss = c->fast->s.ss;
  e.rows_dev = c->cur_rows_dev;
  e.rows = rows;
  e.d = M.d.d_model;
  e.ss_pitch = OURO_TEXT_ROWS;
  if (text_rows(rows)) launch_text_embed(own, c->sms, c->stream);
  return OURO_OK;
}

// One layer of a block of known text (text_rows) on the kernels of gemm_text.cu: the same values as in
// the decoding launches, which is why it asks where those cut a GEMM's tiles along K.
static int text_layer(ouro_ctx *c, int which, int l, int rows, bool kv_only) {
  FastState &fs = c->fast->s;
  ModelRt &M = c->m[which];
  FastModel &fm = fs.m[which];
  const ouro_model_desc &d = M.d;
  const int dq = d.n_heads * d.head_dim, dkv = d.n_kv_heads * d.head_dim;
  Activations &a = c->a;
  cudaStream_t s = c->stream;
  const LayerMaps &lm = fm.layers[l];
  static const int kind_class[4] = {OURO_PROF_QKV, OURO_PROF_WO, OURO_PROF_GATEUP, OURO_PROF_DOWN};
  const bool per_kind = c->prof_class >= OURO_PROF_QKV && c->prof_class <= OURO_PROF_HEAD;
  // the grid of the launch that has this GEMM while decoding: alone (the first q,k,v), or with the others of its chain
  auto grid_of = [&](int layer, int kind) {
    const WeightSide w = weight_side(d, fm, layer, kind);
    return grid_for(fs, w.tiles, w.K / BLOCK_K);
  };
  auto chain_grid = [&](int kind) {
    if (!fs.fuse || (kind == G_QKV && l == 0)) return grid_of(l, kind);
    const int first = kind == G_QKV ? l - 1 : l;                  // the chain begins with this layer's output projection
    return std::max(std::max(grid_of(first, G_WO), grid_of(first, G_GATEUP)),
                    std::max(grid_of(first, G_DOWN), first + 1 < d.n_layers ? grid_of(first + 1, G_QKV) : grid_of(0, G_HEAD)));
  };
  auto gemm = [&](TextGemm &g, int kind, const CUtensorMap *xmaps) {
    const WeightSide w = weight_side(d, fm, l, kind);
    for (int i = 0; i < 3; ++i) { g.w_tiles[i] = w.a_tiles[i]; g.w_rows[i] = w.a_rows[i]; }
    g.w_count = w.a_count;
    g.tiles = w.tiles;
    g.kb = w.K / BLOCK_K;
    const int grid = chain_grid(kind);
    const ws::Cut cut = ws::cut(g.tiles, g.kb, grid, grid);
    g.t0 = cut.t0;
    g.per = cut.per;
    g.a = xmaps[OURO_MAX_ROWS / 16 - 1];
    g.rows = rows;
    g.status = &c->st->status;
    ProfScope ps(c, per_kind ? kind_class[kind] : OURO_PROF_GEMM);
    launch_text_gemm(g, c->sms, s);
  };
  auto consume = [&](TextGemm &g) { g.ss_in = fs.ss; g.ss_tiles = (d.d_model + TILE_N - 1) / TILE_N; g.ss_inv_d = 1.0f / (float)d.d_model; g.eps = d.rms_eps; };
  auto produce = [&](TextGemm &g, const void *gain) {
    g.mode = TEXT_RESIDUAL;
    g.x = a.x; g.ldx = d.d_model;
    g.gain = (const __nv_bfloat16 *)gain; g.xb = (__nv_bfloat16 *)a.xn; g.ss_out = fs.ss;
  };
  {
    TextGemm g{};
    const size_t off = (size_t)l * d.max_seq * dkv;
    g.mode = TEXT_QKV;
    g.w[0] = lm.hq; g.w[1] = lm.hk; g.w[2] = lm.hv;
    consume(g);
    g.pos = M.blk.pos; g.cos_t = M.rope_cos; g.sin_t = M.rope_sin;
    g.q_out = (__nv_bfloat16 *)a.q;
    g.k_out = (__nv_bfloat16 *)M.k_cache + off;
    g.v_out = (__nv_bfloat16 *)M.v_cache + off;
    g.head_dim = d.head_dim; g.dq = dq; g.dkv = dkv; g.L = M.L;
    gemm(g, G_QKV, fm.x_d);
  }
  if (kv_only) return OURO_OK;
  {
    ProfScope ps(c, OURO_PROF_ATTENTION);
    // in one launch where every row's keys lie in one span, else in parts whose pieces are folded one after the other.  A cache
    // longer than the fold can take has no room for pieces in the workspace: the generic kernel, as in the decoding launches.
    const bool spans = attention_tc_supported(d), direct = !spans || fold::span_count(d.head_dim, M.L + rows) <= 1;
    for (int r0 = 0; r0 < rows; r0 += OURO_PART_ROWS) {
      const int n = direct ? rows : std::min<int>(OURO_PART_ROWS, rows - r0);
      BlockDev b = M.blk;
      b.tok += r0; b.pos += r0; b.group += r0; b.lin_end += r0; b.seg_start += r0; b.seg_len += r0; b.mask += 2 * r0;
      const __nv_bfloat16 *q = (const __nv_bfloat16 *)a.q + (size_t)r0 * dq;
      __nv_bfloat16 *out = (__nv_bfloat16 *)a.att + (size_t)r0 * dq;
      bool pieces = false;
      if (!spans) {
        launch_attention_simple(d, q, M.k_cache, M.v_cache, b, n, nullptr, l, out, s);
      } else if (fm.kv_maps) {
        L2Prefetch pf;
        if (r0 + n >= rows) { pf.ptr[0] = M.wo[l]; pf.bytes[0] = (size_t)d.d_model * dq * 2; }
        pieces = launch_attention_tm(d, q, &fm.kmap, &fm.vmap, M.k_cache, M.v_cache, b, n, 1, M.L + r0, M.L, M.L + r0 + n, l, fs.attn_part, out,
                                     &c->st->status, nullptr, pf, c->sms, s);
      } else {
        pieces = launch_attention_tc(d, q, M.k_cache, M.v_cache, b, n, M.L + r0, M.L, M.L + r0 + n, l, fs.attn_part, out, nullptr, c->sms, s);
      }
      if (pieces) {
        fold::Params f{};
        f.part = fs.attn_part;
        f.out = out;
        f.lin_end = b.lin_end;
        f.seg_len = b.seg_len;
        f.rows = n;
        f.H = d.n_heads;
        f.cap = fold::span_count(d.head_dim, d.max_seq);
        f.head_dim = d.head_dim;
        launch_text_fold(f, c->sms, s);
      }
      if (direct) break;
    }
  }
  {
    TextGemm g{};
    g.w[0] = lm.ho;
    produce(g, M.ffn_norm[l]);
    gemm(g, G_WO, fm.x_q);
  }
  {
    TextGemm g{};
    g.mode = TEXT_SWIGLU;
    g.w[0] = lm.wg; g.w[1] = lm.wu;
    consume(g);
    g.act = (__nv_bfloat16 *)a.act;
    gemm(g, G_GATEUP, fm.x_d);
  }
  {
    TextGemm g{};
    g.w[0] = lm.hd;
    produce(g, l + 1 < d.n_layers ? M.attn_norm[l + 1] : M.final_norm);
    gemm(g, G_DOWN, fm.x_f);
  }
  return OURO_OK;
}

// Whether a block of `rows` rows that sees up to `keys` keys is attended to by attn_few_kernel: rows in order that fill one
// small tile, whose chunks it takes side by side.  What it saves is attn_tm_kernel's chain; what it costs is that its CTAs, four chunks
// of K and V in flight each, share the HBM with the weights on their way to the next kernel, more of them the more kv heads and spans, and
// that P and O of all query rows go through shared memory.  Time of a forward of three layers with attn_tm_kernel over that with this one, both in
// one process (which differ by half a percent; where in memory a build's kernels lie makes one and the same kernel up to 2 % slower):
//   one chunk (behind 60 or 110 keys): 1.00 to 1.13 in all of 100 cases (7B shape, one row, 1.04; 16 rows 1.02)
//   one span, up to 8 query rows, behind 150 to 480 keys: 7B shape (32 kv heads) 1.02 to 1.00, 4096 wide with 16 / 8 / 4 kv heads of 1, 4 and 8
//   query heads 1.04 to 1.01 / 1.03 to 1.01 / 1.03 to 1.02, 34B shape 1.01 to 1.00, two layers of 512 1.04 to 1.15; the worst 0.99 (32 x 2 heads, 460 keys)
//   one span, 9 to 16 query rows: up to 2 kv heads 1.02 to 1.13; 4096 wide, 4 x 1 heads, 16 rows 0.98 to 0.96, 8 x 4, four rows 1.00 to 0.98; 34B shape, two
//   rows 1.00 to 0.98
//   several spans in front of gemm_tc_kernel: 4096 wide, 32 kv heads, 900 / 1800 keys 0.98 / 0.96
//   in front of gemm_rows.cuh, kv heads x spans up to 32: 1.03 to 1.18 (2048 wide, 4 x 8 heads behind 4000 keys 1.09); 64: 1024 wide, 8 x 4 behind 4000
//   keys 0.97, 16 x 1 behind 1800 1.02; 128: 8 x 4 behind 8000 keys 0.94; 512: 32 x 1 behind 8000 keys 0.83
static bool attention_few_pays(const FastModel &fm, const ouro_model_desc &d, int rows, int keys, bool candidates) {
  if (candidates || !attention_few_supported(d, rows)) return false;
  const int spans = fold::span_count(d.head_dim, keys);
  if (keys <= fold::CHUNK) return true;
  if (rows_launch(fm, rows)) return spans * d.n_kv_heads <= 32;
  return spans <= 1 && (d.n_heads / d.n_kv_heads * rows <= 8 || d.n_kv_heads <= 2);
}

// One decoder layer with the tensor-core GEMMs (kv_only: up to its keys and values); OURO_ESTATE when the model does not
// qualify.
int ouro_fast_layer(ouro_ctx *c, int which, int l, int rows, bool kv_only) {
  if (!c->fast || !c->fast->s.m[which].ok) return OURO_ESTATE;
  if (text_rows(rows)) {
    const int rc = text_layer(c, which, l, rows, kv_only);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
      c->err = std::string("text layer launch: ") + cudaGetErrorString(e);
      return OURO_ECUDA;
    }
    return rc;
  }
  ModelRt &M = c->m[which];
  FastModel &fm = c->fast->s.m[which];
  const ouro_model_desc &d = M.d;
  const int dq = d.n_heads * d.head_dim, dkv = d.n_kv_heads * d.head_dim;
  Activations &a = c->a;
  cudaStream_t s = c->stream;
  auto tiles = [](int n) { return (n + TILE_N - 1) / TILE_N; };
  // a.xn holds bf16(attn_norm * x) and ss the sums of squares, left by the embedding or the previous layer's down GEMM
  float *ss = c->fast->s.ss;
  const int ss_tiles = tiles(d.d_model);
  auto consume = [&](GemmParams &p) { p.ss_in = ss; p.ss_tiles = ss_tiles; p.ss_inv_d = 1.0f / (float)d.d_model; p.eps = d.rms_eps; };
  auto produce = [&](GemmParams &p, const void *gain) { p.gain = (const __nv_bfloat16 *)gain; p.xb = (__nv_bfloat16 *)a.xn; p.ss_out = ss; };
  {
    Gemm p{};
    set_weights(p, weight_side(d, fm, l, G_QKV));
    consume(p);
    const bool fused_rope = d.head_dim == 64 || d.head_dim == 128;   // tiles then hold whole heads
    if (fused_rope) {
      const size_t off = (size_t)l * d.max_seq * dkv;
      p.mode = MODE_QKV;
      p.pos = M.blk.pos; p.cos_t = M.rope_cos; p.sin_t = M.rope_sin;
      p.q_out = (__nv_bfloat16 *)a.q;
      p.k_out = (__nv_bfloat16 *)M.k_cache + off;
      p.v_out = (__nv_bfloat16 *)M.v_cache + off;
      p.head_dim = d.head_dim; p.dq = dq; p.dkv = dkv; p.L = M.L;
    } else {
      p.mode = MODE_STORE;
      p.out_f32 = a.qkv;
      p.ldo = dq + 2 * dkv;
    }
    push_gemm(c, which, l, p, G_QKV, fm.x_d, d.d_model, rows, true);       // closes the chain the previous layer began
    if (!fused_rope) {
      ProfScope pr(c, OURO_PROF_ROPE);
      launch_rope_append(d, a.qkv, M.blk.pos, M.rope_cos, M.rope_sin, rows, M.L, l, a.q, M.k_cache, M.v_cache, s);
    }
  }
  if (!kv_only) {
    ProfScope ps(c, OURO_PROF_ATTENTION);
    bool pieces = false;             // the attention output is still in per-span pieces
    if (c->fast->s.m[which].kv_maps) {
      // what the launch after the attention streams first: the output projection, then the first rows of gate and up
      L2Prefetch pf;
      const size_t row_bytes = (size_t)d.d_model * 2, head = std::min<size_t>((size_t)d.d_ffn, c->fast->s.pf_ffn_rows) * row_bytes;
      if (c->fast->s.pf_ffn_rows >= 0) {
        pf.ptr[0] = M.wo[l]; pf.bytes[0] = (size_t)d.d_model * dq * 2;
        pf.ptr[1] = M.w_gate[l]; pf.bytes[1] = head;
        pf.ptr[2] = M.w_up[l]; pf.bytes[2] = head;
      }
      if (attention_few_pays(fm, d, rows, M.L + rows, M.blk_is_candidate)) {
        ++c->fast->s.few_launches;
        pieces = launch_attention_few(d, a.q, M.k_cache, M.v_cache, M.blk, rows, M.L, M.L + rows, l, c->fast->s.attn_part, a.att, c->cur_rows_dev, pf, s);
      } else {
        pieces = launch_attention_tm(d, a.q, &c->fast->s.m[which].kmap, &c->fast->s.m[which].vmap, M.k_cache, M.v_cache, M.blk, rows,
                                   M.blk_is_candidate ? 1 + std::max(1, c->p.K) : 1, M.L, M.L, M.L + rows, l, c->fast->s.attn_part, a.att,
                                   &c->st->status, c->cur_rows_dev, pf, c->sms, s);
      }
    }
    else if (attention_tc_supported(d))
      pieces = launch_attention_tc(d, a.q, M.k_cache, M.v_cache, M.blk, rows, M.L, M.L, M.L + rows, l, c->fast->s.attn_part, a.att,
                                   c->cur_rows_dev, c->sms, s);
    else
      launch_attention_simple(d, a.q, M.k_cache, M.v_cache, M.blk, rows, c->cur_rows_dev, l, a.att, s);
    if (pieces) {                    // folded by the output projection's launch, all its CTAs taking part
      fold::Params &f = c->fast->s.chain.args.fold;
      f.part = c->fast->s.attn_part;
      f.out = (__nv_bfloat16 *)a.att;
      f.lin_end = M.blk.lin_end;
      f.seg_len = M.blk.seg_len;
      f.rows_dev = c->cur_rows_dev;
      f.rows = rows;
      f.H = d.n_heads;
      f.cap = fold::span_count(d.head_dim, d.max_seq);
      f.head_dim = d.head_dim;
    }
  }
  if (!kv_only) {
    Gemm p{};
    set_weights(p, weight_side(d, fm, l, G_WO));
    p.mode = MODE_RESIDUAL;
    p.out_f32 = a.x;
    p.ldo = d.d_model;
    produce(p, M.ffn_norm[l]);
    push_gemm(c, which, l, p, G_WO, fm.x_q, dq, rows, false);
  }
  if (!kv_only) {
    Gemm p{};
    set_weights(p, weight_side(d, fm, l, G_GATEUP));
    p.mode = MODE_SWIGLU;
    p.out_bf16 = (__nv_bfloat16 *)a.act;
    consume(p);
    push_gemm(c, which, l, p, G_GATEUP, fm.x_d, d.d_model, rows, false);
  }
  if (!kv_only) {
    Gemm p{};
    set_weights(p, weight_side(d, fm, l, G_DOWN));
    p.mode = MODE_RESIDUAL;
    p.out_f32 = a.x;
    p.ldo = d.d_model;
    produce(p, l + 1 < d.n_layers ? M.attn_norm[l + 1] : M.final_norm);
    push_gemm(c, which, l, p, G_DOWN, fm.x_f, d.d_ffn, rows, false);     // the next layer's q,k,v or the LM head completes the chain
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    c->err = std::string("tensor-core layer launch: ") + cudaGetErrorString(e);
    return OURO_ECUDA;
  }
  return OURO_OK;
}

// Final norm, LM head and greedy choice.  The GEMM's epilogue keeps, per 128-entry vocabulary tile, each
// token's best logit and index; a small kernel then picks the best tile per token.  logits may be NULL.
// With `tidy` (the static scratch, which calls share) no partial sums are left for the next call, whatever this call or one that
// overlapped with it has left there.
struct Tidy {
  float *slots = nullptr;      // [n_slots][128][128]; a call of `rows` rows has used the first rows x 128 words of each
  int n_slots = 0;
};
__global__ void argmax_tiles_kernel(const float *tile_max, const int *tile_arg, int tiles, int32_t *out, const Tidy tidy) {
  pdl_trigger();
  pdl_wait();
  const int t = blockIdx.x;
  for (int s = threadIdx.x >> 5; s < tidy.n_slots; s += blockDim.x >> 5)
    part_empty(tidy.slots + ((size_t)s * OURO_MAX_ROWS + t) * TILE_N + 4 * (threadIdx.x & 31));
  // compared through the same order-preserving integer image as inside the tiles (-0.0 below +0.0), so that the
  // choice does not depend on where a tile boundary falls
  uint32_t bv = 0;
  int bi = INT_MAX;
  for (int i = threadIdx.x; i < tiles; i += blockDim.x) {
    uint32_t v = ordered_u32(tile_max[(size_t)i * OURO_MAX_ROWS + t]);
    int a = tile_arg[(size_t)i * OURO_MAX_ROWS + t];
    if (v > bv || (v == bv && a < bi)) { bv = v; bi = a; }
  }
  __shared__ uint32_t sv[8];
  __shared__ int si[8];
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    uint32_t ov = __shfl_xor_sync(0xffffffffu, bv, o);
    int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
  }
  if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = bv; si[threadIdx.x >> 5] = bi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
      if (sv[w] > bv || (sv[w] == bv && si[w] < bi)) { bv = sv[w]; bi = si[w]; }
    out[t] = bi == INT_MAX ? 0 : bi;
  }
}

int ouro_fast_head(ouro_ctx *c, int which, int rows, float *logits, int32_t *argmax_dev) {
  if (!c->fast || !c->fast->s.m[which].ok) return OURO_ESTATE;
  ModelRt &M = c->m[which];
  FastModel &fm = c->fast->s.m[which];
  const ouro_model_desc &d = M.d;
  {
    Gemm p{};
    set_weights(p, weight_side(d, fm, 0, G_HEAD));
    p.mode = MODE_HEAD;
    p.out_f32 = logits;
    p.ldo = d.vocab;
    p.tile_max = c->fast->s.tile_max;
    p.tile_arg = c->fast->s.tile_arg;
    p.ss_in = c->fast->s.ss; p.ss_tiles = (d.d_model + TILE_N - 1) / TILE_N; p.ss_inv_d = 1.0f / (float)d.d_model; p.eps = d.rms_eps;
    push_gemm(c, which, 0, p, G_HEAD, fm.x_d, d.d_model, rows, true);
  }
  {
    ProfScope ps(c, OURO_PROF_ARGMAX);
    OURO_COUNT_LAUNCH();
    const rows_gemm::Plan &pl = fm.rm.plan[G_HEAD];
    const int entries = rows_launch(fm, rows) ? (pl.units + pl.up - 1) / pl.up : (d.vocab + TILE_N - 1) / TILE_N;
    launch_pdl(argmax_tiles_kernel, rows, 128, 0, c->stream, (const float *)c->fast->s.tile_max, (const int *)c->fast->s.tile_arg,
               entries, argmax_dev, Tidy());
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    c->err = std::string("tensor-core head launch: ") + cudaGetErrorString(e);
    return OURO_ECUDA;
  }
  return OURO_OK;
}

// ===================================================================================================
// ouro_lm_head_static: the LM-head pass for callers that must not allocate.
//
// Some users of this library cannot give it a workspace: a serving process that handed all device memory to
// its own arena at start-up (a later cudaMalloc simply fails), or a latency-critical loop that must not run
// into the implicit device synchronisation an allocation can cause.  For them this one call keeps everything
// the GEMM needs besides its inputs and outputs - the partial-tile slots of the split-K schedule, the per-tile
// maxima and a status word - in a fixed array that is part of the library image.
// Every GPU that loads the library carries these 5 MiB until the process exits.
//
// The array's name is only meaningful in device code.  Host code must ask the runtime for its device address
// (cudaGetSymbolAddress) with the right device current; that is done once per device by the first call.
// ===================================================================================================
namespace {
constexpr int NA_SPLITTERS = 32;                   // CTAs that may leave partial tiles (two slots each)
constexpr int NA_MAX_TILES = 512;                  // vocabulary <= 65536
constexpr size_t NA_SLOT_BYTES = (size_t)NA_SPLITTERS * 2 * TILE_N * OURO_MAX_ROWS * sizeof(float);
constexpr size_t NA_OFF_STATUS = NA_SLOT_BYTES;
constexpr size_t NA_OFF_TMAX = NA_OFF_STATUS + 256;
constexpr size_t NA_OFF_TARG = NA_OFF_TMAX + (size_t)NA_MAX_TILES * OURO_MAX_ROWS * sizeof(float);
constexpr size_t NA_BYTES = NA_OFF_TARG + (size_t)NA_MAX_TILES * OURO_MAX_ROWS * sizeof(int);
static_assert(NA_BYTES <= (5u << 20), "the static scratch is documented as 5 MiB");
constexpr int NA_MAX_DEVICES = 64;
}  // namespace

static __device__ __align__(256) unsigned char g_static_scratch[NA_BYTES];

namespace {
unsigned char *g_na_ptr[NA_MAX_DEVICES] = {};      // device address of g_static_scratch, per device
int g_na_smem[NA_MAX_DEVICES] = {};
int g_na_sms[NA_MAX_DEVICES] = {};
std::atomic<bool> g_na_ready[NA_MAX_DEVICES] = {};  // the slots are empty and the status word is zero, and every call leaves them so

// Once per device, with that device current: resolve the array's device address and size the kernel's
// shared memory.  Returns OURO_OK or an error with a text for ouro_last_error(NULL).
int na_setup(int dev) {
  if (g_na_ptr[dev]) return OURO_OK;
  void *ptr = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_scratch);
  if (e != cudaSuccess || !ptr) {
    ouro_set_global_error(std::string("cudaGetSymbolAddress(static scratch): ") + cudaGetErrorString(e));
    return OURO_ECUDA;
  }
  int smem = 0, sms = 0;
  if ((e = cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(gemm_tc_kernel<SOME>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) {
    ouro_set_global_error(std::string("static-scratch set-up: ") + cudaGetErrorString(e));
    return OURO_ECUDA;
  }
  if (!g_encode) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn) {
      ouro_set_global_error("cuTensorMapEncodeTiled unavailable");
      return OURO_ECUDA;
    }
    g_encode = (EncodeTiledFn)fn;
  }
  g_na_smem[dev] = smem;
  g_na_sms[dev] = sms;
  g_na_ptr[dev] = (unsigned char *)ptr;
  return OURO_OK;
}
}  // namespace

extern "C" int ouro_debug_static_scratch(void **dev_ptr, size_t *slot_bytes) {
  int dev = 0;
  if (!dev_ptr || !slot_bytes) return OURO_EINVAL;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) return OURO_ECUDA;
  const int rc = na_setup(dev);
  if (rc != OURO_OK) return rc;
  *dev_ptr = g_na_ptr[dev];
  *slot_bytes = NA_SLOT_BYTES;
  return OURO_OK;
}

extern "C" int ouro_lm_head_static(const void *x_dev, const void *lm_head_dev, int32_t rows, int32_t d_model, int32_t vocab,
                                   int32_t *argmax_dev, float *logits_dev, void *cuda_stream) {
  if (!x_dev || !lm_head_dev || !argmax_dev) {
    ouro_set_global_error("ouro_lm_head_static: null pointer");
    return OURO_EINVAL;
  }
  if (rows < 1 || rows > OURO_MAX_ROWS || d_model < 64 || d_model % 64 != 0 || vocab < 8 || vocab % 8 != 0 ||
      (vocab + TILE_N - 1) / TILE_N > NA_MAX_TILES || (((uintptr_t)x_dev | (uintptr_t)lm_head_dev) & 15)) {
    ouro_set_global_error("ouro_lm_head_static: size beyond the static scratch (rows 1..128, d_model a multiple of 64, "
                          "vocab a multiple of 8 and at most 65536) or pointers not 16-byte aligned");
    return OURO_EINVAL;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) {
    ouro_set_global_error("ouro_lm_head_static: no usable current device");
    return OURO_ECUDA;
  }
  int rc = na_setup(dev);
  if (rc != OURO_OK) return rc;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  unsigned char *base = g_na_ptr[dev];
  const int tiles = (vocab + TILE_N - 1) / TILE_N;
  // The slots are empty (see EMPTY) and the status word is zero: cleared by the first call on the device and by the one after
  // a give-up.  The second kernel of every call empties the slots that the call has used, so that what calls that overlapped
  // against the rules did to one another ends with them.
  cudaError_t e = cudaSuccess;
  const bool clear = !g_na_ready[dev].load(std::memory_order_acquire);
  if (clear) {
    e = cudaMemsetAsync(base, 0xff, NA_SLOT_BYTES, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(base + NA_OFF_STATUS, 0, NA_OFF_TMAX - NA_OFF_STATUS, s);
  }
  ChainParams kp{};
  ChainArgs &cp = kp.args;
  cp.n = 1;
  GemmParams &p = cp.g[0];
  GemmMaps &m = kp.maps[0];
  const int t_pad = (rows + 15) & ~15;
  if (e != cudaSuccess || !make_map(&m.a[0], lm_head_dev, vocab, d_model, TILE_N) || !make_map(&m.b, x_dev, rows, d_model, t_pad)) {
    ouro_set_global_error("ouro_lm_head_static: could not describe the operands to the copy engine");
    return OURO_ECUDA;
  }
  p.a_tiles[0] = tiles; p.a_rows[0] = vocab; p.a_count = 1;
  p.mode = MODE_HEAD;
  p.tiles = tiles;
  p.kb = d_model / BLOCK_K;
  p.t_pad = t_pad;
  p.rows = rows;
  p.stages = stages_for(t_pad, g_na_smem[dev]);
  p.out_f32 = logits_dev;
  p.ldo = vocab;
  p.tile_max = (float *)(base + NA_OFF_TMAX);
  p.tile_arg = (int *)(base + NA_OFF_TARG);
  p.wait_limit = 1u << 22;
  p.scratch = (float *)base;
  p.status = (int *)(base + NA_OFF_STATUS);
  // Which tiles are cut, and where, is that of a launch over the 32 CTAs that have slots, whoever streams the others: a tile
  // summed along K in pieces is nearer to the exact sum than one long chain in the tensor cores (relative error, 37 rows of
  // width 4096: vocabulary 32000 4.23e-6, all tiles in one chain 4.37e-6; vocabulary 6000 3.73e-6 and 4.37e-6).  Whole
  // tiles need no scratch; all SMs stream them, those behind the CTAs that share the cut tiles first.  Bound by the weight
  // stream: 32000 x 4096 with 37 rows took 207 us on 32 CTAs (1.3 TB/s, what 32 rings can ask for) and takes 89 us on all
  // SMs.  The cut costs time where one tile per SM would do: 18944 x 4096 79 us, with its 148 tiles whole 65 us.
  const int sms = std::min(g_na_sms[dev], MAX_GRID), sharers = std::min(tiles * p.kb, NA_SPLITTERS);
  const ws::Cut cut = ws::cut(tiles, p.kb, sharers, sharers);
  const int cut_by = cut.per ? ((tiles - cut.t0) * p.kb + cut.per - 1) / cut.per : 0;
  const int grid = std::min(cut_by + cut.t0, sms);
  p.t0 = cut.t0;
  p.per = cut.per;
  p.sharers = cut_by % grid;
  p.finishers = cut_by;
  // A sharer's pieces cost it up to a tile and the round trip of their sum: where the whole tiles need no further round
  // without it, it sits the first one out (32000 x 1024, 128 rows: 66 -> 56 us; 50000 x 8192, 37 rows: 178 -> 171 us).
  const int others = grid - p.sharers, rounds = (cut.t0 + grid - 1) / grid;
  p.sit_out = p.sharers > 0 && others > 0 && others + (rounds - 1) * grid >= cut.t0 && rounds > 1;
  gemm_tc_kernel<SOME><<<grid, THREADS, g_na_smem[dev], s>>>(kp);
  Tidy tidy;
  tidy.slots = p.scratch;
  tidy.n_slots = 2 * cut_by;
  argmax_tiles_kernel<<<rows, 128, 0, s>>>(p.tile_max, p.tile_arg, tiles, argmax_dev, tidy);
  int status = 0;
  if ((e = cudaGetLastError()) != cudaSuccess ||
      (e = cudaMemcpyAsync(&status, p.status, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
      (e = cudaStreamSynchronize(s)) != cudaSuccess) {
    ouro_set_global_error(std::string("ouro_lm_head_static: ") + cudaGetErrorString(e));
    return OURO_ECUDA;
  }
  if (status != 0) {                             // (only the call that has cleared the array may call it clear)
    g_na_ready[dev].store(false, std::memory_order_release);
    ouro_set_global_error("ouro_lm_head_static: a bounded device-side wait gave up");
    return OURO_ETIMEOUT;
  }
  if (clear) g_na_ready[dev].store(true, std::memory_order_release);
  return OURO_OK;
}
