// Weight GEMMs of long blocks of known text (up to 512 rows of a prompt) on pairs of SMs: tcgen05 with cta_group::2.
//
//   Y[t, n] = sum_k X[t, k] * W[n, k]      X: [rows <= 512, K] bf16 activations, W: [N, K] bf16 weights
//
// Known text is bound by the tensor cores and by what L2 can bring into an SM, not by the one pass over the weights that
// gemm_tc.cu is built around: with 256 tokens beside every 128 weight rows an SM took 48 KB in for 512 cycles of contraction,
// and the partial tiles of the K split, 128 KB each, took as long to add up as the contraction itself (7B layer, 256 rows:
// 95 us of contraction in 197 us).  Here
//   * a pair of CTAs (a cluster) works on 256 tokens x 128 or 256 weight rows.  The tokens are the MMA's M side, 128 of them
//     in each CTA; the weight rows are its N side, half of every tile in each CTA's shared memory: 32 KB per 512 cycles;
//   * every tile is contracted along its whole K by one pair.  No partial sum leaves an SM.
// What bounds it is L2: 24 to 32 KB per k-block at about 50 bytes per cycle into every SM (0.26 to 0.33 us), and 10 to 20 us of
// beginning and end per launch.  7B shape, 466 rows, before in two blocks of 256: q,k,v 110 -> 64 us, output projection 64 -> 35,
// gate / up 125 -> 91, down 85 -> 63; a prompt of 467 tokens through 32 layers 12.2 -> 8.3 ms.
// A token's values must not depend on the block it comes in, so the sum over K is cut where the decoding launches cut it
// (ws::cut): the contraction goes on into another accumulator at each cut, and the thread that owns (token, tile) adds the pieces
// up in its registers in ascending order, while the next piece is being contracted.
// Two threads share a token's 128 columns of a tile, 16 columns each in turn: dimensions 32 or 64 apart - rotary pairs, gate and
// up - are in one thread, and each holds 64 sums (with all 128 in one thread 1.2 KB of them were spilled).  The kernel with two tiles
// per pair has 576 threads of 96 registers and still spills (300 bytes stored, 432 loaded); the one with a single tile does not.
//
// Warp 0 fetches (TMA; weights before, activations after the dependency wait), warp 1 of the pair's first CTA contracts, the
// others drain and finish: eight warps per weight tile.  Every mbarrier wait is bounded; on expiry the CTA raises the status word and
// drains.
#include "gemm_text.cuh"

#include <algorithm>
#include <type_traits>

namespace {

constexpr int BLOCK_K = 64, TILE_N = 128;
constexpr int CTA_TOK = 128, UNIT_TOK = 2 * CTA_TOK;
constexpr int MAX_TT = OURO_TEXT_ROWS / UNIT_TOK;
constexpr int A_BYTES = CTA_TOK * BLOCK_K * 2;
constexpr int W_BYTES = TILE_N / 2 * BLOCK_K * 2;       // this CTA's half of a weight tile
constexpr int MAX_STAGES = 8;
// A finishing warp turns 16 columns of its 32 tokens around in shared memory: one token per lane as they come out of TMEM, several
// lanes per token on the way to memory.
constexpr int PITCH = 20;                                // floats per token: 16-byte pieces that start in different banks
constexpr uint32_t SPIN_LIMIT = 1u << 24;
constexpr unsigned long long HINT_EVICT_LAST = 0x14F0000000000000ull;
template <int WT> constexpr int EPI_THREADS = 256 * WT;      // two per token and weight tile
template <int WT> constexpr int THREADS = 64 + EPI_THREADS<WT>;
template <int WT> constexpr int STAGE_BYTES = A_BYTES + WT * W_BYTES;
template <int WT> constexpr int STAGES = WT == 1 ? 8 : 5;
template <int WT> constexpr int SMEM_BYTES = 1024 + STAGES<WT> * STAGE_BYTES<WT> + EPI_THREADS<WT> * PITCH * 4;
static_assert(STAGES<1> <= MAX_STAGES && STAGES<2> <= MAX_STAGES, "barriers of the ring");
static_assert(SMEM_BYTES<1> <= 216 * 1024 && SMEM_BYTES<2> <= 216 * 1024, "beside 11 KB of static shared memory");

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// the same place in the shared memory of the pair's first CTA
__device__ __forceinline__ uint32_t in_leader(uint32_t addr) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive_leader(uint64_t *bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(in_leader(smem_u32(bar))) : "memory");
}
// Bounded wait: false when the limit ran out or another warp of the CTA has given up.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag, uint32_t limit = SPIN_LIMIT) {
  const uint32_t addr = smem_u32(bar);
  for (uint32_t i = 0; i < limit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((i & 255) == 255 && abort_flag && *abort_flag) return false;
  }
  return false;
}
// A tile into this CTA's shared memory; the bytes are counted by the pair's first CTA.
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap *map, uint32_t leader_bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(map), "r"(leader_bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tma_load_pair_keep(uint32_t dst, const CUtensorMap *map, uint32_t leader_bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(dst),
      "l"(map), "r"(leader_bar), "r"(x), "r"(y), "l"(HINT_EVICT_LAST)
      : "memory");
}
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  // K-major operand in 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart.
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}
__device__ __forceinline__ void mma_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the barrier at this place in both CTAs (or those of the mask) once every contraction issued so far has completed.
__device__ __forceinline__ void mma_commit_pair(uint64_t *bar, uint16_t ctas = 3) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
               "h"(ctas)
               : "memory");
}
// 16 columns of this warp's lane quarter
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float *v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
               "tcgen05.wait::ld.sync.aligned;"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Where the pieces of a tile along K end: at `end` for the piece that begins at the tile's front, then every `per` k-blocks.
__device__ __forceinline__ int first_end(const TextGemm &p, int tile) {
  if (tile < p.t0) return p.kb;
  const int past = (tile - p.t0) * p.kb % p.per;
  return min(p.kb, p.per - past);
}
// Which stacked matrix a tile belongs to, its first row there, and the first output column.
__device__ __forceinline__ void locate(const TextGemm &p, int tile, int &seg, int &row0, int &col0) {
  seg = 0;
  col0 = 0;
  while (seg + 1 < p.w_count && tile >= p.w_tiles[seg]) {
    tile -= p.w_tiles[seg];
    col0 += p.w_rows[seg];
    ++seg;
  }
  row0 = tile * TILE_N;
  col0 += row0;
}

// Turns 16 columns of a warp's 32 tokens around: `own` are the lane's (one token per lane), v[i] afterwards columns 4 (lane mod 4) on
// of token 8 i + lane / 4 - four lanes per token, whose accesses to memory are 64 bytes in a row.
__device__ __forceinline__ void turn(float *piece, int lane, const float *own, float4 *v) {
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 16; i += 4) *reinterpret_cast<float4 *>(piece + lane * PITCH + i) = make_float4(own[i], own[i + 1], own[i + 2], own[i + 3]);
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = *reinterpret_cast<const float4 *>(piece + (8 * i + (lane >> 2)) * PITCH + 4 * (lane & 3));
}
__device__ __forceinline__ float4 times(const float4 &v, float r) { return make_float4(v.x * r, v.y * r, v.z * r, v.w * r); }
__device__ __forceinline__ void store_bf16(__nv_bfloat16 *dst, const float4 &v) {
  *reinterpret_cast<uint2 *>(dst) = make_uint2(rowops::pack(v.x, v.y), rowops::pack(v.z, v.w));
}
__device__ __forceinline__ float4 rotate(const float4 &own, const float4 &other, const float4 &c, const float4 &s) {
  return make_float4(rowops::rotate(own.x, other.x, c.x, s.x), rowops::rotate(own.y, other.y, c.y, s.y),
                     rowops::rotate(own.z, other.z, c.z, s.z), rowops::rotate(own.w, other.w, c.w, s.w));
}

template <int WT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS<WT>, 1) gemm_text_kernel(const __grid_constant__ TextGemm p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[MAX_STAGES], empty[MAX_STAGES], acc_full[WT][2], acc_empty[WT][2], drain_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  __shared__ float rs[MAX_TT][CTA_TOK];            // per-token factor 1/rms of the consumed activations
  __shared__ float halves[2][WT][CTA_TOK][4];      // sums of squares on their way from a tile's one warp to the other
  __shared__ int spos[MAX_TT][CTA_TOK];            // token positions
  constexpr int NS = STAGES<WT>, SB = STAGE_BYTES<WT>;
  volatile int *abort_flag = &abort_s;
  const uint32_t ring = (smem_u32(smem_raw) + 1023) & ~1023u;
  float *turn_base = reinterpret_cast<float *>(smem_raw + (ring - smem_u32(smem_raw)) + NS * SB);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t rank;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int j = 0; j < WT; ++j)
      for (int b = 0; b < 2; ++b) {
        mbar_init(&acc_full[j][b], 1);
        mbar_init(&acc_empty[j][b], 16);           // eight warps of each CTA
      }
    mbar_init(&drain_bar, 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  pdl_trigger();
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"((uint32_t)(256 * WT)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::);
  }
  fence_before_sync();
  __syncthreads();
  cluster_sync();
  fence_after_sync();
  const uint32_t tmem = tmem_base_s;
  uint32_t n_issued = 0;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer, one per CTA
    if (elect_one()) {
      const int units = pair < p.units ? (p.units - pair + n_pairs - 1) / n_pairs : 0, total = units * p.kb;
      // One thread runs this loop once per k-block, so what is constant over a unit is worked out once per unit.
      const CUtensorMap *map[WT];
      int y[WT], ya = 0;
      auto unit = [&](int u) {
#pragma unroll
        for (int j = 0; j < WT; ++j) {
          const int tile = min(u / p.token_tiles * WT + j, p.tiles - 1);
          int seg = (int)rank, row0 = tile * 64, col0;
          if (p.mode != TEXT_SWIGLU) {
            locate(p, tile, seg, row0, col0);
            row0 += 64 * (int)rank;
          }
          map[j] = &p.w[seg];
          y[j] = row0;
        }
        ya = u % p.token_tiles * UNIT_TOK + (int)rank * CTA_TOK;
      };
      auto weights = [&](int st, int kb) {
        const uint32_t bar = in_leader(smem_u32(&full[st]));
#pragma unroll
        for (int j = 0; j < WT; ++j) tma_load_pair(ring + st * SB + A_BYTES + j * W_BYTES, map[j], bar, kb * BLOCK_K, y[j]);
      };
      auto activations = [&](int st, int kb) {
        tma_load_pair_keep(ring + st * SB, &p.a, in_leader(smem_u32(&full[st])), kb * BLOCK_K, ya);
      };
      // the first stages' weights do not wait for the previous kernel, whose output the activations are
      const int ahead = min(NS, min(total, p.kb));
      if (total > 0) unit(pair);
      for (int i = 0; i < ahead; ++i) {
        if (rank == 0) mbar_expect_tx(&full[i], 2 * SB);
        weights(i, i);
      }
      pdl_wait();
      asm volatile("fence.proxy.async;" ::: "memory");
      for (int i = 0; i < ahead; ++i) activations(i, i);
      n_issued = ahead;
      bool ok = true;
      int u = pair, kb = ahead, st = ahead % NS;
      uint32_t round = ahead / NS;
      for (int i = ahead; i < total; ++i) {
        if (kb == p.kb) { kb = 0; u += n_pairs; unit(u); }
        if (round > 0) {
          ok = mbar_wait(&empty[st], (round - 1) & 1, abort_flag) && !*abort_flag;
          if (!ok) break;
        }
        if (rank == 0) mbar_expect_tx(&full[st], 2 * SB);
        weights(st, kb);
        activations(st, kb);
        n_issued = i + 1;
        ++kb;
        if (++st == NS) { st = 0; ++round; }
      }
      if (!ok) { *abort_flag = 1; atomicExch(p.status, 1); }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- contraction, by the pair's first CTA
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TILE_N >> 3) << 17) | ((uint32_t)(UNIT_TOK >> 4) << 24);
      int st = 0;
      uint32_t round = 0, item[WT];
#pragma unroll
      for (int j = 0; j < WT; ++j) item[j] = 0;
      bool ok = true;
      for (int u = pair; u < p.units && ok; u += n_pairs) {
        int begin[WT], end[WT];
#pragma unroll
        for (int j = 0; j < WT; ++j) {
          begin[j] = 0;
          end[j] = first_end(p, min(u / p.token_tiles * WT + j, p.tiles - 1));
        }
        for (int kb = 0; kb < p.kb; ++kb) {
#pragma unroll
          for (int j = 0; j < WT; ++j)
            if (kb == begin[j] && item[j] >= 2) ok = ok && mbar_wait(&acc_empty[j][item[j] & 1], ((item[j] >> 1) - 1) & 1, abort_flag);
          ok = ok && mbar_wait(&full[st], round & 1, abort_flag) && !*abort_flag;
          if (!ok) break;
          fence_after_sync();
          const uint32_t base = ring + st * SB;
          const uint64_t da = smem_desc_sw128(base);
#pragma unroll
          for (int j = 0; j < WT; ++j) {
            const uint64_t db = smem_desc_sw128(base + A_BYTES + j * W_BYTES);
            const uint32_t d = tmem + (uint32_t)((2 * j + (item[j] & 1)) * TILE_N);
#pragma unroll
            for (int k = 0; k < BLOCK_K / 16; ++k) mma_pair(d, da + 2 * k, db + 2 * k, idesc, (kb > begin[j] || k > 0) ? 1u : 0u);
          }
          mma_commit_pair(&empty[st]);
#pragma unroll
          for (int j = 0; j < WT; ++j)
            if (kb + 1 == end[j]) {
              mma_commit_pair(&acc_full[j][item[j] & 1]);
              ++item[j];
              begin[j] = end[j];
              end[j] = min(p.kb, end[j] + p.per);
            }
          if (++st == NS) { st = 0; ++round; }
        }
      }
      if (!ok) { *abort_flag = 1; atomicExch(p.status, 1); }
    }
  } else {
    // ---------------------------------------------------------------- adding up and finishing: eight warps per weight tile
    pdl_wait();
    const int j = (warp - 2) >> 3, h = (warp - 2) >> 2 & 1, q = warp & 3;  // tile of the unit, half of its columns, lane quarter
    const int tok = 32 * q + lane, et = threadIdx.x - 64;                  // TMEM lane = token of this CTA
    for (int i = et; i < p.token_tiles * CTA_TOK; i += EPI_THREADS<WT>) {
      const int t = i / CTA_TOK * UNIT_TOK + (int)rank * CTA_TOK + i % CTA_TOK;
      float r = 1.0f;
      if (p.ss_in && t < p.rows) {
        float sum = 0.f;
#pragma unroll 8
        for (int k = 0; k < p.ss_tiles; ++k) sum += __ldcg(p.ss_in + (size_t)k * OURO_TEXT_ROWS + t);
        r = rowops::inv_rms(sum, p.ss_inv_d, p.eps);
      }
      rs[i / CTA_TOK][i % CTA_TOK] = r;
      spos[i / CTA_TOK][i % CTA_TOK] = p.mode == TEXT_QKV && t < p.rows ? p.pos[t] : 0;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS<WT>) : "memory");
    uint32_t item = 0, odd = 0;
    bool ok = true;
    for (int u = pair; u < p.units && ok; u += n_pairs, odd ^= 1) {
      const int tt = u % p.token_tiles, want = u / p.token_tiles * WT + j, tile = min(want, p.tiles - 1);
      const int t = tt * UNIT_TOK + (int)rank * CTA_TOK + tok;
      const bool split = tile >= p.t0;
      float acc[64];
#pragma unroll
      for (int i = 0; i < 64; ++i) acc[i] = 0.f;
      int end = first_end(p, tile);
      for (int begin = 0; begin < p.kb; begin = end, end = min(p.kb, end + p.per)) {
        ok = mbar_wait(&acc_full[j][item & 1], (item >> 1) & 1, abort_flag) && !*abort_flag;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        fence_after_sync();
        const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)((2 * j + (item & 1)) * TILE_N + 16 * h);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          float v[16];
          tmem_ld16(taddr + 32 * m, v);
          if (split) {
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[16 * m + i] += v[i];
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[16 * m + i] = v[i];
          }
        }
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive_leader(&acc_empty[j][item & 1]);
        ++item;
      }
      if (!ok) {
        // the warp with the tile's other columns may be waiting for this one's sums: it sees the flag behind this barrier
        *abort_flag = 1;
        __threadfence_block();
        __syncwarp();
        if (p.mode == TEXT_RESIDUAL) asm volatile("bar.arrive %0, 64;" ::"r"(2 + 4 * j + q) : "memory");
        break;
      }
      if (want >= p.tiles && p.mode != TEXT_RESIDUAL) continue;       // (an odd number of tiles: the last one is contracted twice)
      // From here on a lane holds four columns of four of the warp's 32 tokens, those from t0w on: columns 32 m + 16 h + lc of tokens
      // 8 i + lt.
      const int t0w = t - lane, n_tok = want < p.tiles ? min(32, p.rows - t0w) : 0;
      const int lt = lane >> 2, lc = 4 * (lane & 3);
      float *piece = turn_base + (warp - 2) * 32 * PITCH;
      const float *r = &rs[tt][32 * q + lt];
      int seg = 0, row0 = 0, col0 = 0;
      if (p.mode != TEXT_SWIGLU) locate(p, tile, seg, row0, col0);
      const int live = p.mode != TEXT_SWIGLU && row0 + TILE_N > p.w_rows[seg] ? 2 : 4;   // chunks inside the matrix, which has a multiple of 64 rows
      float4 a[4];
      if (p.mode == TEXT_RESIDUAL) {
        // new residual stream, its bf16(gain * x) image for the next GEMM, and this tile's sums of squares
        float sq[4][2];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int c = col0 + 32 * m + 16 * h + lc;
          turn(piece, lane, acc + 16 * m, a);
          float4 x4[4];
          uint2 graw = make_uint2(0, 0);
          if (m < live) graw = *reinterpret_cast<const uint2 *>(p.gain + c);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (8 * i + lt < n_tok && m < live) x4[i] = *reinterpret_cast<const float4 *>(p.x + (size_t)(t0w + 8 * i + lt) * p.ldx + c);
          const float2 g0 = rowops::unpack(graw.x), g1 = rowops::unpack(graw.y);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float s = 0.f;
            if (8 * i + lt < n_tok && m < live) {
              const float4 y = make_float4(a[i].x + x4[i].x, a[i].y + x4[i].y, a[i].z + x4[i].z, a[i].w + x4[i].w);
              const size_t at = (size_t)(t0w + 8 * i + lt) * p.ldx + c;
              *reinterpret_cast<float4 *>(p.x + at) = y;
              store_bf16(p.xb + at, make_float4(g0.x * y.x, g0.y * y.y, g1.x * y.z, g1.y * y.w));
              s = rowops::squares(y.x, y.y, y.z, y.w);
            }
            sq[i][m & 1] = m < 2 ? s : sq[i][m & 1] + s;              // groups of four columns 64 apart ...
          }
        }
        // ... 32, then (in the other warp) 16, then 8 and 4 columns apart
        if (h == 1) {
#pragma unroll
          for (int i = 0; i < 4; ++i) halves[odd][j][32 * q + 8 * i + lt][lane & 3] = sq[i][0] + sq[i][1];
        }
        asm volatile("bar.sync %0, 64;" ::"r"(2 + 4 * j + q) : "memory");
        if (h == 0) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float s = (sq[i][0] + sq[i][1]) + halves[odd][j][32 * q + 8 * i + lt][lane & 3];
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            if ((lane & 3) == 0 && 8 * i + lt < n_tok) p.ss_out[(size_t)tile * OURO_TEXT_ROWS + t0w + 8 * i + lt] = s;
          }
        }
        continue;
      }
      if (p.mode == TEXT_SWIGLU) {                                    // chunks 0 and 1: gate of 64 features, 2 and 3: up
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          float4 b[4];
          turn(piece, lane, acc + 16 * m, a);
          turn(piece, lane, acc + 16 * (m + 2), b);
          __nv_bfloat16 *dst = p.act + (size_t)(t0w + lt) * p.w_rows[0] + tile * 64 + 32 * m + 16 * h + lc;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 g = times(a[i], r[8 * i]), up = times(b[i], r[8 * i]);
            if (8 * i + lt < n_tok)
              store_bf16(dst + (size_t)(8 * i) * p.w_rows[0], make_float4(rowops::silu(g.x) * up.x, rowops::silu(g.y) * up.y, rowops::silu(g.z) * up.z, rowops::silu(g.w) * up.w));
          }
        }
        continue;
      }
      const size_t pitch = seg == 0 ? p.dq : p.dkv;
      __nv_bfloat16 *dst = (seg == 0 ? p.q_out + (size_t)(t0w + lt) * p.dq : (seg == 1 ? p.k_out : p.v_out) + (size_t)(p.L + t0w + lt) * p.dkv) +
                           row0 + 16 * h + lc;
      if (seg == 2) {                                                 // v goes to the cache as it is
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          if (m >= live) break;
          turn(piece, lane, acc + 16 * m, a);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (8 * i + lt < n_tok) store_bf16(dst + 32 * m + 8 * i * pitch, times(a[i], r[8 * i]));
        }
        continue;
      }
      // the columns of chunk m with those of chunk m + apart: 64 (one head of 128) or 32 (two heads of 64) columns on
      auto rotated = [&](auto m_c, auto apart_c) {
        constexpr int m = decltype(m_c)::value, apart = decltype(apart_c)::value, half = 32 * apart;
        float4 b[4];
        turn(piece, lane, acc + 16 * m, a);
        turn(piece, lane, acc + 16 * (m + apart), b);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const size_t at = (size_t)spos[tt][32 * q + 8 * i + lt] * half + (apart == 2 ? 32 * m : 0) + 16 * h + lc;
          const float4 c = *reinterpret_cast<const float4 *>(p.cos_t + at), s = *reinterpret_cast<const float4 *>(p.sin_t + at);
          const float4 lo = times(a[i], r[8 * i]), hi = times(b[i], r[8 * i]);
          if (8 * i + lt < n_tok) {
            store_bf16(dst + 32 * m + 8 * i * pitch, rotate(lo, hi, c, make_float4(-s.x, -s.y, -s.z, -s.w)));
            store_bf16(dst + 32 * (m + apart) + 8 * i * pitch, rotate(hi, lo, c, s));
          }
        }
      };
      using std::integral_constant;
      if (p.head_dim == 128) {
        rotated(integral_constant<int, 0>{}, integral_constant<int, 2>{});
        rotated(integral_constant<int, 1>{}, integral_constant<int, 2>{});
      } else {
        rotated(integral_constant<int, 0>{}, integral_constant<int, 1>{});
        if (live == 4) rotated(integral_constant<int, 2>{}, integral_constant<int, 1>{});
      }
    }
    if (!ok) { *abort_flag = 1; atomicExch(p.status, 1); }
  }
  // ------------------------------------------------------------------ teardown
  // Nothing may still be on its way to this CTA when it leaves: the last contraction on every stage has released it in both CTAs.
  if (n_issued > 0) {                              // (the producer)
    for (uint32_t st = 0; st < (uint32_t)NS && st < n_issued; ++st) {
      const uint32_t last = (n_issued - 1 - st) / NS * NS + st;      // last fetch into this stage
      if (!mbar_wait(&empty[st], (last / NS) & 1, abort_flag, SPIN_LIMIT)) { *abort_flag = 1; atomicExch(p.status, 1); }
    }
    if (*abort_flag)                               // somebody gave up: fetches that nobody contracts land within microseconds
      for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  fence_before_sync();
  __syncthreads();
  if (*abort_flag && warp == 1 && rank == 0 && elect_one()) {          // ... and no contraction may still be running
    mma_commit_pair(&drain_bar, 1);                // (this CTA's barrier alone: the other one may be about to leave)
    mbar_wait(&drain_bar, 0, nullptr, 1u << 16);
    for (int i = 0; i < 64; ++i) __nanosleep(1000);                    // the last arrivals in the other CTA land within microseconds
  }
  __syncwarp();
  cluster_sync();
  if (warp == 1) {
    fence_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(256 * WT)));
  }
}

__global__ void __launch_bounds__(256) text_embed_kernel(const rowops::Embed e) {
  pdl_trigger();
  pdl_wait();
  rowops::embed(e, blockIdx.x * 8 + (threadIdx.x >> 5), gridDim.x * 8, threadIdx.x & 31);
}
__global__ void __launch_bounds__(256) text_fold_kernel(const fold::Params f) {
  fold::run(f, blockIdx.x * 8 + (threadIdx.x >> 5), gridDim.x * 8, threadIdx.x & 31);
}

}  // namespace

int text_gemm_setup() {
  return cudaFuncSetAttribute(gemm_text_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES<1>) == cudaSuccess &&
                 cudaFuncSetAttribute(gemm_text_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES<2>) == cudaSuccess
             ? OURO_OK
             : OURO_ECUDA;
}

// One or two weight tiles per unit: a k-block brings 32 or 24 KB into each SM, about 600 or 450 cycles.  What decides is the number
// of rounds: 7B q,k,v, 466 rows, two rounds of two tiles or three of one; its output projection has 32 units of two tiles or 64 of one for
// 74 pairs.
void launch_text_gemm(TextGemm &g, int sms, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  const int pairs = std::max(1, sms / 2);
  g.token_tiles = (g.rows + UNIT_TOK - 1) / UNIT_TOK;
  const int units1 = g.tiles * g.token_tiles, units2 = (g.tiles + 1) / 2 * g.token_tiles;
  const int cost1 = (units1 + pairs - 1) / pairs * 450, cost2 = (units2 + pairs - 1) / pairs * 600;
  const bool two = cost2 <= cost1;
  g.units = two ? units2 : units1;
  const int grid = 2 * std::min(pairs, g.units);
  if (two) launch_pdl(gemm_text_kernel<2>, grid, THREADS<2>, SMEM_BYTES<2>, s, g);
  else launch_pdl(gemm_text_kernel<1>, grid, THREADS<1>, SMEM_BYTES<1>, s, g);
}

void launch_text_embed(const rowops::Embed &e, int sms, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  launch_pdl(text_embed_kernel, std::max(1, std::min(4 * sms, (e.rows * ((e.d + 127) / 128) + 7) / 8)), 256, 0, s, e);
}

void launch_text_fold(const fold::Params &f, int sms, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  launch_pdl(text_fold_kernel, std::max(1, std::min(4 * sms, (f.rows * f.H + 7) / 8)), 256, 0, s, f);
}
