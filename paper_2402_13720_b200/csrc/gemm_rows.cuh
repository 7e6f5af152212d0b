// Weight-streaming GEMMs for one token (plain decoding, drafting) of a model with small layers: part of gemm_tc.cu, which has the
// chain, the schedule that says where a tile is cut along K, and the rules that say which models run here (rows_x_bytes, rows_pay).
//
// At one token a GEMM of gemm_tc_kernel is latency: a tile of 128 weight rows is cut along K among several CTAs, whose
// partial sums cross the chip before anybody can finish the token (3 us of the 5 to 10 of a GEMM of the 1.1B shape), and
// the outputs cross it again behind a fence and a counter (2 us).  Here a CTA owns its weight rows for the whole of K: groups of 16
// (a unit), as many per CTA as an equal split over the SMs gives, so that only finished activations leave it.  They travel
// in packets that say themselves that they are there (row_ops.cuh), and every CTA gathers all of them into its shared memory.
// 1.1B draft, four forwards behind 389 keys: 3156 -> 2497 us; a layer 36 -> 28 us, of which 13.5 are its 88 MB at the copy peak and
// the rest four hand-overs, the attention and two launches.
//
// The tensor cores are used through mma.sync (16 weight rows x 8 tokens x 16 values of K, operands by ldmatrix): its fragments
// are as small as a unit, where a tcgen05 tile has 128 rows of which 16 to 80 would be the CTA's, and the sums are in
// registers the moment they are complete.  The rate does not matter: a token is 2 flop per weight byte.
// The sums are those of gemm_tc_kernel to the last bit: one chain over K in steps of 16, begun anew where the schedule cuts the
// tile, the pieces added up in ascending order.  (A step of 16 gives the same sum in either instruction: results agree bit
// for bit on random operands of all magnitudes, and the tests compare blocks on either kernel.)
//
// Warp 0 streams weights into the ring (boxes of [k-blocks][rows][64]), warp 1 works out the token's factor of the norm, CW warps
// contract.  What they execute is latency as well: a step of a chain waits 47 cycles for the one before, and a warp spends about 4
// cycles on every other instruction.  So a stage is as large as a slot of the ring (12 KB slots: draft 5061 us) and a slot two k-blocks of the
// largest GEMM (see rows_setup), a stage is looked at by the warps that contract it only (one per unit), where all units of a CTA
// are cut alike the ring takes the k-blocks of several pieces in turn, each for other warps, and the two warps that finish a GEMM's
// sums leave the next one's activations to the others (2953 -> 2622 us).  Two groups of eight tokens, or the activations of several
// tokens beside the weights in the ring, were slower than gemm_tc_kernel (two small layers, 13 rows: step 91 -> 129 us; five rows
// of the 1.1B shape 867 -> 1288).

namespace rows_gemm {

constexpr int CW = 10, CTHREADS = 32 * CW;        // contracting warps (twelve warps in all leave 168 registers)
constexpr int THREADS = 32 * (2 + CW);
constexpr int UNIT = 16;                          // weight rows of a unit: 16 outputs, 8 gate/up pairs or 8 rotary pairs
constexpr int PARKED = 24;                        // sums of a unit's piece parked at a time
constexpr int MIN_SLOT = 20 * 1024;               // bytes of a ring slot, at the least
constexpr int MAX_UP = 10;                        // units contracted at a time
constexpr uint32_t TAKERS = 2520;                 // arrivals that free a slot: divisible by every number of units up to MAX_UP
static_assert(MAX_UP <= CW && MAX_UP * UNIT * 128 <= MIN_SLOT, "one warp per unit, one k-block per slot");
constexpr int MAX_SLOTS = 10;
constexpr int MAX_X = 64 * 1024;                  // bytes of a token's activations, as a CTA keeps them
constexpr int GATHERERS = CW - 2, GTHREADS = 32 * GATHERERS;     // warps that fetch the activations: all but the two that finish
static_assert(4 * MAX_UP <= CTHREADS - GTHREADS, "one thread per four columns");

struct Plan {
  int units, up, passes;      // units of the GEMM; a CTA takes up x passes consecutive ones, `up` at a time
  int nkb;                    // k-blocks per ring slot
  int cut_per;                // k-blocks of a piece along K if this GEMM is a launch of its own (host)
  int su, sj, sh;             // 128-byte lines from a unit to the next, from a k-block to the next, to the unit's upper eight rows
  int share, max_pieces;      // warps that share a unit's pieces (more than one: the ring takes k-blocks of as many in turn); most pieces a unit has
  const float *q_in;          // squares of four columns each [d / 4] of activations in memory
  float *q_out;               // MODE_RESIDUAL: the same of what this GEMM leaves in memory
  const __nv_bfloat16 *x_in;  // activations in memory, or, of the same launch, as packets
  const uint4 *packets_in;
  uint4 *packets_out;         // where the packets of this GEMM go (NULL: its output goes to memory)
};
// What a launch says of its GEMMs, kept in shared memory.
struct alignas(16) Told {
  ChainArgs args;
  Plan plan[MAX_CHAIN];
};
struct Params {
  CUtensorMap w[MAX_CHAIN][3];
  Told told;
  int slots, slot;            // of the ring, and the bytes of one
  int squares_bytes;          // the squares of the activations; those are behind them
  uint4 *front;               // where the work in front leaves its packets
  uint32_t mark;              // of those; GEMM i leaves those with mark + 1 + i
  uint32_t late;              // test aid: ns that the warp of the factors sleeps before it looks at a GEMM (0)
};
static_assert(sizeof(Params) <= 4096, "kernel parameters");

constexpr int PARK_BYTES = PARKED * UNIT * 4;
constexpr int HEAD_BYTES = 1024, MISC = HEAD_BYTES + (int)sizeof(Told);     // barriers, factors, maxima; Told
inline int slots_for(int slot, int x_bytes, int smem_max) { return std::min(MAX_SLOTS, (smem_max - 1024 - PARK_BYTES - MISC - x_bytes) / slot); }

__device__ __forceinline__ void load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(smem_u32(dst)),
      "l"(map), "r"(smem_u32(bar)), "r"(0), "r"(y), "r"(z), "l"(HINT_EVICT_FIRST)
      : "memory");
}
__device__ __forceinline__ void load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int y, int z, int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4, %5, %6}], [%2], %7;" ::"r"(smem_u32(dst)),
      "l"(map), "r"(smem_u32(bar)), "r"(0), "r"(y), "r"(z), "r"(w), "l"(HINT_EVICT_FIRST)
      : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t *r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16(float *c, const uint32_t *a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mbar_arrive_n(uint64_t *bar, uint32_t n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(n) : "memory");
}
// Bounded wait of a warp (see mbar_wait): all its lanes get the same answer.
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag) {
  const uint32_t addr = smem_u32(bar);
  for (uint32_t i = 0; i < SPIN_LIMIT; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (__all_sync(0xffffffffu, ok != 0)) return true;
    if ((i & 255) == 255 && __any_sync(0xffffffffu, *abort_flag)) return false;
  }
  return false;
}
__device__ __forceinline__ void warps_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(CTHREADS) : "memory"); }
// A barrier of the contracting warps that tells all of them alike whether one of them has given up.
__device__ __forceinline__ bool warps_any(bool failed) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}" : "=r"(r) : "r"((uint32_t)failed), "n"(CTHREADS) : "memory");
  return r != 0;
}

// Which stacked matrix a unit belongs to, its number there, and the tile of gemm_tc_kernel's schedule that holds it.
__device__ __forceinline__ int locate_unit(const GemmParams &p, int u, int &seg, int &tile) {
  seg = 0;
  tile = 0;
  if (p.mode == MODE_QKV) {
    while (seg + 1 < p.a_count && u >= p.a_rows[seg] / UNIT) {
      u -= p.a_rows[seg] / UNIT;
      tile += p.a_tiles[seg];
      ++seg;
    }
  }
  tile += u / (TILE_N / UNIT);
  return u;
}
// Where the first of a unit's pieces along K ends (kb: there is one piece), and how many there are.
__device__ __forceinline__ int first_cut(const GemmParams &p, int u) {
  int seg, tile;
  locate_unit(p, u, seg, tile);
  return tile < p.t0 ? p.kb : min(p.kb, p.per - (tile - p.t0) * p.kb % p.per);
}
__device__ __forceinline__ int pieces_of(const GemmParams &p, int first) { return first == p.kb ? 1 : 1 + (p.kb - first + p.per - 1) / p.per; }

// The pieces of the units of a pass that are all cut alike.  The ring takes them `share` at a time, and of those nkb k-blocks each in
// turn, for as many rounds as the longest needs (a shorter one's last stages may be empty).
struct Pieces {
  int kbs, per, cut, n;
  __device__ Pieces(const GemmParams &p, int u0) : kbs(p.kb), per(p.per), cut(first_cut(p, u0)), n(pieces_of(p, cut)) {}
  __device__ int begin(int q) const { return q == 0 ? 0 : cut + (q - 1) * per; }
  __device__ int end(int q) const { return min(kbs, cut + q * per); }
  // rounds of the pieces [q, q + m)
  __device__ int rounds(int q, int m, int nkb) const {
    const int longest = n == 1 ? kbs : m > 2 || (q > 0 && q + m < n) ? (n > 2 ? per : max(cut, kbs - cut)) : max(end(q) - begin(q), end(q + m - 1) - begin(q + m - 1));
    return (longest + nkb - 1) / nkb;
  }
};

// Activations into shared memory, and the squares for the norm's factor beside them.  What this launch computed itself arrives in
// packets: the poll that finds them has them.
__device__ __forceinline__ bool gather(const GemmParams &p, const Plan &pl, uint32_t mark, uint32_t limit, float *squares, uint8_t *xs, int gt) {
  const int n = p.kb * (BLOCK_K / 4);
  const bool norm = p.ss_in != nullptr;
  uint2 *dst = reinterpret_cast<uint2 *>(xs);
  if (!pl.packets_in) {
    for (int i = gt; i < n; i += GTHREADS) {
      dst[i] = __ldcg(reinterpret_cast<const uint2 *>(pl.x_in) + i);
      if (norm) squares[i] = __ldcg(pl.q_in + i);
    }
    return true;
  }
  const uint4 *src = pl.packets_in;
  constexpr int BATCH = 4;
  for (int i0 = gt; i0 < n; i0 += BATCH * GTHREADS) {
    rowops::Packet v[BATCH];
    bool there = false;
    for (uint32_t spin = 0; spin < limit; ++spin) {
      there = true;
#pragma unroll
      for (int b = 0; b < BATCH; ++b)
        if (i0 + b * GTHREADS < n) v[b] = rowops::get_packet(src + i0 + b * GTHREADS);
#pragma unroll
      for (int b = 0; b < BATCH; ++b) there = there && (i0 + b * GTHREADS >= n || v[b].mark == mark);
      if (there) break;
      if ((spin & 15) == 15 && *(volatile const int *)p.status != 0) return false;   // some CTA has given up
    }
    if (!there) return false;
#pragma unroll
    for (int b = 0; b < BATCH; ++b)
      if (i0 + b * GTHREADS < n) {
        dst[i0 + b * GTHREADS] = make_uint2(v[b].lo, v[b].hi);
        if (norm) squares[i0 + b * GTHREADS] = __uint_as_float(v[b].extra);
      }
  }
  return true;
}

__global__ void __launch_bounds__(THREADS, 1) gemm_rows_kernel(const __grid_constant__ Params kp) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *ring = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int slots = kp.slots, slot_bytes = kp.slot;
  float *park = (float *)(ring + (size_t)slots * slot_bytes);                     // [PARKED][UNIT]
  uint64_t *full = (uint64_t *)((uint8_t *)park + PARK_BYTES), *empty = full + MAX_SLOTS;
  uint64_t *factors_full = empty + MAX_SLOTS, *x_full = factors_full + 1;   // the factor, the activations of a GEMM are there
  volatile int *abort_flag = (volatile int *)(x_full + 1);
  float *rs = (float *)(x_full + 2);                                        // 1/rms of the consumed activations
  uint2 *best = (uint2 *)(rs + 2);                                          // [4 MAX_UP] LM head: the largest of four logits, its index
  static_assert((2 * MAX_SLOTS + 4) * 8 + 8 + 4 * MAX_UP * 8 <= HEAD_BYTES, "room");
  Told *told = (Told *)((uint8_t *)park + PARK_BYTES + HEAD_BYTES);
  const ChainArgs &cp = told->args;
  const Plan *plans = told->plan;
  const GemmParams &p0 = cp.g[0];
  float *squares = (float *)((uint8_t *)told + sizeof(Told));

  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < slots; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], TAKERS);
    }
    mbar_init(factors_full, 1);
    mbar_init(x_full, GATHERERS + 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < (int)(sizeof(Told) / 16); i += THREADS)
    reinterpret_cast<uint4 *>(told)[i] = reinterpret_cast<const uint4 *>(&kp.told)[i];
  __syncthreads();
  if (threadIdx.x == 0) { const GemmParams &p = p0; TRACE(0); }
  uint8_t *xs = (uint8_t *)squares + kp.squares_bytes;
  uint32_t n_issued = 0;

  if (warp == 0) {
    // ---------------------------------------------------------------- weights: they depend on no kernel, so nothing is waited for
    if (elect_one()) {
      uint32_t round = 0, n = 0;
      int st = 0;
      uint8_t *slot = ring;
      bool ok = true;
      for (int ci = 0; ci < cp.n && ok; ++ci) {
        const GemmParams &p = cp.g[ci];
        const Plan &pl = plans[ci];
        const CUtensorMap *w = kp.w[ci];
        const int mode = p.mode, up = pl.up, unit_bytes = pl.nkb * UNIT * 128, half = p.head_dim >> 1;
        for (int pass = 0; pass < pl.passes && ok; ++pass) {
          const int u0 = ((int)blockIdx.x * pl.passes + pass) * up, nu = min(up, pl.units - u0);
          if (nu <= 0) break;
          int seg0 = 0, y0 = 0, h0 = 0;                  // (rotary pairs) the first unit: matrix, dimension and half of a head
          if (mode == MODE_QKV) {
            int tile;
            const int u = locate_unit(p, u0, seg0, tile), per_head = p.head_dim / UNIT;
            h0 = u / per_head;
            y0 = (u - h0 * per_head) * 8;
            h0 *= 2;
          }
          const uint32_t bytes = (mode == MODE_QKV ? nu : up) * unit_bytes;
          auto stage = [&](int kb, bool empty_stage) -> bool {
            if (round > 0 && !(mbar_wait(&empty[st], (round - 1) & 1, abort_flag) && !*abort_flag)) return false;
            ++n;
            if (empty_stage) {
              mbar_arrive(&full[st]);
            } else {
              mbar_expect_tx(&full[st], bytes);
              if (mode == MODE_QKV) {
                int seg = seg0, y = y0, h = h0;
                uint8_t *dst = slot;
                for (int i = 0; i < nu; ++i, dst += unit_bytes) {
                  load_4d(dst, w + seg, &full[st], y, h, kb);
                  if ((y += 8) == half) {
                    y = 0;
                    if ((h += 2) * half == p.a_rows[seg]) { h = 0; ++seg; }
                  }
                }
              } else if (mode == MODE_SWIGLU) {
                load_3d(slot, w, &full[st], u0 * 8, kb);
                load_3d(slot + up * unit_bytes / 2, w + 1, &full[st], u0 * 8, kb);
              } else {
                load_3d(slot, w, &full[st], u0 * UNIT, kb);
              }
            }
            slot += slot_bytes;
            if (++st == slots) { st = 0; ++round; slot = ring; }
            return true;
          };
          const int nkb = pl.nkb, share = pl.share, kbs = p.kb;
          if (share == 1) {
            for (int kb = 0; kb < kbs && ok; kb += nkb) ok = stage(kb, false);
          } else {
            const Pieces pc(p, u0);
            for (int q = 0; q < pc.n && ok; q += share) {
              const int m = min(share, pc.n - q), rounds = pc.rounds(q, m, nkb);
              for (int r = 0; r < rounds && ok; ++r)
                for (int i = 0; i < m && ok; ++i) {
                  const int kb = pc.begin(q + i) + r * nkb;
                  ok = stage(kb, kb >= pc.end(q + i));
                }
            }
          }
        }
        TRACE(8);
      }
      if (!ok) { *abort_flag = 1; atomicExch(p0.status, 1); }
      n_issued = n;
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- the factor 1/rms of the activations
    // This warp looks at every phase of x_full, but nobody waits for its answer where a GEMM has no norm.  So it is one of those
    // whose arrival completes the next phase: were it late by a GEMM and a hand-over, it would find the parity it waits for
    // as it was a phase ago, and wait until its limit.
    bool ok = true;
    uint32_t gathered = 0;
    for (int ci = 0; ci < cp.n && ok; ++ci) {
      const GemmParams &p = cp.g[ci];
      const Plan &pl = plans[ci];
      if ((int)blockIdx.x * pl.passes * pl.up >= pl.units) continue;
      if (lane == 0) {
        if (kp.late) __nanosleep(kp.late);
        mbar_arrive(x_full);                                       // has seen the phase before
      }
      __syncwarp();
      ok = warp_wait(x_full, gathered++ & 1, abort_flag);
      if (!ok || !p.ss_in) continue;
      float sum = 0.f;
      for (int i0 = 0; i0 < p.ss_tiles; i0 += 8) {                 // tile sums in halves, then tile by tile
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int c = (i0 + i) * 32 + lane;
          v[i] = 4 * c < p.kb * BLOCK_K ? squares[c] : 0.f;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i0 + i < p.ss_tiles) sum += v[i];
      }
      if (lane == 0) {
        *rs = rowops::inv_rms(sum, p.ss_inv_d, p.eps);
        mbar_arrive(factors_full);
      }
    }
  } else {
    // ---------------------------------------------------------------- contraction and epilogue
    const int w = warp - 2, ct = threadIdx.x - 64;
    if (cp.fold.part) fold::run<true>(cp.fold, (int)blockIdx.x * CW + w, (int)gridDim.x * CW, lane, {kp.front, kp.mark});    // (waits itself)
    else pdl_wait();
    if (cp.embed.table) rowops::embed_packets(cp.embed, (int)blockIdx.x * CW + w, (int)gridDim.x * CW, lane, kp.front, kp.mark);
    int st = 0;
    uint32_t round = 0, n_factors = 0, n_gathered = 0;
    bool ok = true;
    for (int ci = 0; ci < cp.n && ok; ++ci) {
      const GemmParams &p = cp.g[ci];
      const Plan &pl = plans[ci];
      const int mode = p.mode, share = pl.share, nkb = pl.nkb, kbs = p.kb, sj = pl.sj * 128, max_pieces = pl.max_pieces;
      for (int pass = 0; pass < pl.passes && ok; ++pass) {
        const int u0 = ((int)blockIdx.x * pl.passes + pass) * pl.up, nu = min(pl.up, pl.units - u0);
        if (nu <= 0) break;
        // ---- everything that can be known ahead of the activations.  The first threads finish four columns each, or two of the pairs.
        const bool finishes = ct < 4 * nu;
        const int fu = u0 + (ct >> 2), sub = ct & 3, half = p.head_dim >> 1;
        const uint32_t mark = kp.mark + 1 + ci;
        float4 pre = make_float4(0.f, 0.f, 0.f, 0.f);
        uint2 pre_g = make_uint2(0, 0);
        int np = 1, seg = 0;
        size_t at = 0;                               // where the result goes
        if (finishes) {
          if (share > 1) np = pieces_of(p, first_cut(p, fu));
          if (mode == MODE_RESIDUAL) {
            at = fu * UNIT + 4 * sub;
            pre = *reinterpret_cast<const float4 *>(p.out_f32 + at);
            pre_g = *reinterpret_cast<const uint2 *>(p.gain + at);
          } else if (mode == MODE_SWIGLU) {
            at = fu * 8 + 2 * sub;
          } else if (mode == MODE_QKV) {
            int tile;
            const int u = locate_unit(p, fu, seg, tile), per_head = p.head_dim / UNIT, h = u / per_head, i = (u - h * per_head) * 8 + 2 * sub;
            at = h * p.head_dim + i + (seg == 0 ? (size_t)0 : (size_t)p.L * p.dkv);
            if (seg != 2) {
              const size_t ti = (size_t)*p.pos * half + i;
              const float2 c = *reinterpret_cast<const float2 *>(p.cos_t + ti), s = *reinterpret_cast<const float2 *>(p.sin_t + ti);
              pre = make_float4(c.x, c.y, s.x, s.y);
            }
          }
        }
        const int us = w / share, member = w - us * share;
        const bool mine = us < nu;
        float acc[4];
        const int r8 = lane & 7;
        const uint32_t a_lane = smem_u32(ring) + (uint32_t)(us * pl.su + ((lane >> 3) & 1) * pl.sh + r8) * 128;
        const uint32_t b_lane = smem_u32(xs) + (lane >> 3) * 16;     // (all eight tokens of a step are the one: seven sums are left alone)
        uint32_t xo[4];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) xo[kk] = ((2 * kk + (lane >> 4)) ^ r8) << 4;
        const Pieces pc(p, mine ? u0 + us : u0);
        const uint32_t taken = TAKERS / nu;
        // ---- the activations
        bool good = true;
        if (pass == 0) {
          if (ct == 0) TRACE(1);
          if (w >= CW - GATHERERS) {
            good = __all_sync(0xffffffffu, gather(p, pl, kp.mark + ci, p.wait_limit, squares, xs, ct - (CTHREADS - GTHREADS)));
            if (lane == 0) mbar_arrive(x_full);
          }
          if (good) good = warp_wait(x_full, n_gathered & 1, abort_flag);
          ++n_gathered;
          if (ct == 0) TRACE(4);
        }
        // ---- contraction
        auto clear = [&]() {
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[i] = 0.f;
        };
        auto skip = [&](int n) {                                     // past n slots of the ring
          st += n;
          while (st >= slots) { st -= slots; ++round; }
        };
        auto contract = [&](uint32_t al, int kb, int n_kb) {       // k-blocks from kb on, the first at `al`
#pragma unroll 1
          for (uint32_t bl = b_lane + kb * 128; n_kb > 0; --n_kb, al += sj, bl += 128) {
            uint32_t a[4][4], b[8];
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) ldsm4(al + xo[kk], a[kk]);
            ldsm4(bl, b);
            ldsm4(bl + 64, b + 4);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) mma16(acc, a[kk], b[2 * kk], b[2 * kk + 1]);
          }
        };
        auto park_sums = [&](int slot) {                             // (token 0 of the eight)
          if ((lane & 3) == 0) {
            park[slot * UNIT + (lane >> 2)] = acc[0];
            park[slot * UNIT + (lane >> 2) + 8] = acc[2];
          }
        };
        if (share == 1) {
          if (mine && member == 0) {
            float tot[4] = {-0.f, -0.f, -0.f, -0.f};
            clear();
            int next = pc.cut;
            for (int k0 = 0; k0 < kbs && good; k0 += nkb) {
              good = warp_wait(&full[st], round & 1, abort_flag);
              if (!good) break;
              if (k0 == 0 && ct == 0) TRACE(2);
              const uint32_t base = a_lane + (uint32_t)(st * slot_bytes);
              const int k1 = min(kbs, k0 + nkb);
              for (int k = k0; k < k1;) {
                const int e = min(k1, next);
                contract(base + (uint32_t)((k - k0) * sj), k, e - k);
                k = e;
                if (e == next) {                                     // the piece is complete: added to those before it
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    tot[i] += acc[i];
                    acc[i] = e == kbs ? tot[i] : 0.f;
                  }
                  next = min(kbs, next + pc.per);
                }
              }
              if (lane == 0) mbar_arrive_n(&empty[st], taken);
              skip(1);
            }
            park_sums(us);
          } else {
            skip((kbs + nkb - 1) / nkb);
          }
        } else {
          for (int q = 0; q < pc.n && good; q += share) {
            const int m = min(share, pc.n - q), rounds = pc.rounds(q, m, nkb);
            if (mine && member < m) {
              const int end = pc.end(q + member);
              int kb = pc.begin(q + member);
              clear();
              skip(member);
              for (int r = 0; r < rounds; ++r, kb += nkb) {
                // A warp passes over the stages of others, so it has not seen what the slot held before.  That must have been freed
                // before the phase of `full` can be told from the one before: `empty` can, as its next phase wants this warp, and
                // the one before was over when the stage was asked for (before this warp's last: `share` is below `slots`).
                if (round > 0) good = warp_wait(&empty[st], (round - 1) & 1, abort_flag);
                if (good) good = warp_wait(&full[st], round & 1, abort_flag);
                if (!good) break;
                if (q == 0 && r == 0 && ct == 0) TRACE(2);
                contract(a_lane + (uint32_t)(st * slot_bytes), kb, min(nkb, end - kb));
                if (lane == 0) mbar_arrive_n(&empty[st], taken);
                skip(r + 1 < rounds ? m : m - member);
              }
              park_sums(us * max_pieces + q + member);
            } else {
              skip(rounds * m);
            }
          }
        }
        __syncwarp();
        if (ct == 0) TRACE(3);
        // ---- the sums are parked (and the factors known): finish
        if (good && p.ss_in && pass == 0) {
          good = warp_wait(factors_full, n_factors & 1, abort_flag);
          ++n_factors;
        }
        if (!good && lane == 0) { *abort_flag = 1; atomicExch(p0.status, 1); }
        ok = !warps_any(!good);
        if (!ok) break;
        if (ct == 0) TRACE(5);
        if (finishes) {
          // four columns: the pieces in ascending order
          auto total = [&](int column) {
            const float *src = park + (ct >> 2) * (share == 1 ? 1 : max_pieces) * UNIT + column;
            float4 v = *reinterpret_cast<const float4 *>(src);
            for (int i = 1; i < np; i += 4) {
              float4 o[4];
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (i + j < np) o[j] = *reinterpret_cast<const float4 *>(src + (i + j) * UNIT);
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (i + j < np) { v.x += o[j].x; v.y += o[j].y; v.z += o[j].z; v.w += o[j].w; }
            }
            return v;
          };
          if (mode == MODE_RESIDUAL) {
            float4 y = total(4 * sub);
            y.x += pre.x; y.y += pre.y; y.z += pre.z; y.w += pre.w;
            const float2 g01 = rowops::unpack(pre_g.x), g23 = rowops::unpack(pre_g.y);
            const uint2 xb = make_uint2(rowops::pack(g01.x * y.x, g01.y * y.y), rowops::pack(g23.x * y.z, g23.y * y.w));
            const float sq = rowops::squares(y.x, y.y, y.z, y.w);
            if (pl.packets_out) {
              rowops::put_packet(pl.packets_out + at / 4, xb.x, xb.y, __float_as_uint(sq), mark);
            } else {
              *reinterpret_cast<uint2 *>(p.xb + at) = xb;
              pl.q_out[at / 4] = sq;
            }
            *reinterpret_cast<float4 *>(p.out_f32 + at) = y;
          } else if (mode == MODE_HEAD) {
            const float r = *rs;
            const int col = fu * UNIT + 4 * sub;
            float4 v = total(4 * sub);
            v.x *= r; v.y *= r; v.z *= r; v.w *= r;
            uint32_t bu = 0;
            int bi = col;
            if (col < p.a_rows[0]) {                                 // (a multiple of 8)
              if (p.out_f32) *reinterpret_cast<float4 *>(p.out_f32 + col) = v;
              const float vals[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const uint32_t uo = ordered_u32(vals[e]);
                if (uo > bu) { bu = uo; bi = col + e; }
              }
            }
            best[ct] = make_uint2(bu, (uint32_t)bi);
          } else {
            // two pairs: gate and up of two features, or dimensions i and i + head_dim/2 of a head
            // (fetched as four columns: this lane's are the lower or the upper two of them)
            const float4 a4 = total(sub & 2 ? 4 : 0), b4 = total(sub & 2 ? 12 : 8);
            const float r = *rs;
            float2 a = sub & 1 ? make_float2(a4.z, a4.w) : make_float2(a4.x, a4.y), b = sub & 1 ? make_float2(b4.z, b4.w) : make_float2(b4.x, b4.y);
            a.x *= r; a.y *= r; b.x *= r; b.y *= r;
            if (mode == MODE_SWIGLU) {
              const uint32_t v = rowops::pack(rowops::silu(a.x) * b.x, rowops::silu(a.y) * b.y);
              if (pl.packets_out) {                                  // two lanes make a packet
                const int live = 4 * nu - (ct - lane);
                const uint32_t o = __shfl_down_sync(live >= 32 ? 0xffffffffu : (1u << live) - 1u, v, 1);
                if ((sub & 1) == 0) rowops::put_packet(pl.packets_out + at / 4, v, o, 0u, mark);
              } else {
                *reinterpret_cast<uint32_t *>(p.out_bf16 + at) = v;
              }
            } else {
              float2 lo = a, hi = b;
              if (seg != 2) {
                lo = make_float2(rowops::rotate(a.x, b.x, pre.x, -pre.z), rowops::rotate(a.y, b.y, pre.y, -pre.w));
                hi = make_float2(rowops::rotate(b.x, a.x, pre.x, pre.z), rowops::rotate(b.y, a.y, pre.y, pre.w));
              }
              __nv_bfloat16 *dst = (seg == 0 ? p.q_out : seg == 1 ? p.k_out : p.v_out) + at;
              *reinterpret_cast<uint32_t *>(dst) = rowops::pack(lo.x, lo.y);
              *reinterpret_cast<uint32_t *>(dst + half) = rowops::pack(hi.x, hi.y);
            }
          }
        }
        if (mode == MODE_HEAD) {
          warps_barrier();
          if (ct == 0) {
            uint2 b = best[0];
            for (int i = 1; i < 4 * nu; ++i) {
              const uint2 o = best[i];
              if (o.x > b.x) b = o;                                  // the columns ascend: the smallest index among equals
            }
            p.tile_max[(size_t)(u0 / pl.up) * OURO_MAX_ROWS] = ordered_f32(b.x);
            p.tile_arg[(size_t)(u0 / pl.up) * OURO_MAX_ROWS] = (int)b.y;
          }
        }
        if (ct == 0) TRACE(10);
        if (pass + 1 < pl.passes) warps_barrier();   // the parked sums are read  (behind the last pass the next GEMM's activations come first)
      }
    }
  }
  __syncthreads();
  if (*abort_flag && n_issued > 0) {              // (the producer thread) copies may still be landing in shared memory
    for (int st = 0; st < slots; ++st) {
      if (n_issued <= (uint32_t)st) continue;
      const uint32_t last = ((n_issued - 1 - st) / slots) * slots + st;
      mbar_wait(&full[st], (last / slots) & 1, nullptr, 1u << 14);
    }
  }
  __syncthreads();
}

}  // namespace rows_gemm
