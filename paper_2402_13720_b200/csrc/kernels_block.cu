// Integer side of one Ouroboros step: phrase pool, candidate packing, greedy acceptance,
// KV compaction, phrase harvest, row argmax.  All latency-bound kernels of one warp or one block.
#include "ouro_internal.h"

#define FULL 0xffffffffu

// ------------------------------------------------------------------------------- phrase pool
// sets x ways table; a phrase lives in the set selected by its first token (Section 3.2: phrases are
// retrieved by the draft's last token).  One warp works on one set, lanes stride over the ways.
// Every insert or refresh takes the next value of a global counter as stamp; stamps are unique.
//
// A kernel's operations form a list; each inserts one phrase (in place of another, or not) and so takes one value of the
// counter: the i-th operation's stamp is known without the others.  Operations on different sets do not see one another, so the
// list is shared by the warps of a block, a set's operations staying in order in one warp (pool_apply).  One operation is
// three round trips to memory, which one warp made one after the other: 458 phrases of four tokens took 529 us, of nine 730, and take
// 29 and 34.  (Together with the acceptance below: a step of two small layers 92.8 -> 91.9 us, the 1.1B draft with its window 5825 ->
// 5794 us, a 34B-shaped step of eight layers 2139 -> 2116 us.)

__device__ __forceinline__ int pool_set(const PoolDev &P, int32_t key) {
  int bits = 31 - __clz(P.sets);
  return bits ? (int)(((uint32_t)key * 2654435761u) >> (32 - bits)) : 0;
}

__device__ __forceinline__ int warp_min_int(int v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = min(v, __shfl_xor_sync(FULL, v, o));
  return v;
}

// way holding exactly this phrase, or INT_MAX.  phrase[] is warp-uniform.
__device__ int pool_find(const PoolDev &P, int set, const int32_t *phrase) {
  int lane = threadIdx.x & 31, best = INT_MAX;
  for (int w = lane; w < P.ways; w += 32) {
    int e = set * P.ways + w;
    bool hit = P.key[e] == phrase[0];
    for (int i = 0; hit && i < P.S; ++i) hit = P.suf[(size_t)e * P.S + i] == phrase[1 + i];
    if (hit) best = min(best, w);
  }
  return warp_min_int(best);
}

__device__ void pool_insert(const PoolDev &P, u64 stamp, const int32_t *phrase) {
  int lane = threadIdx.x & 31;
  int set = pool_set(P, phrase[0]);
  int w = pool_find(P, set, phrase);
  if (w == INT_MAX) {
    int free_w = INT_MAX;
    u64 old = ~0ull;
    int old_w = INT_MAX;
    for (int c = lane; c < P.ways; c += 32) {
      int e = set * P.ways + c;
      if (P.key[e] < 0) {
        free_w = min(free_w, c);
      } else if (P.stamp[e] < old) {
        old = P.stamp[e];
        old_w = c;
      }
    }
    free_w = warp_min_int(free_w);
    if (free_w != INT_MAX) {
      w = free_w;
    } else {  // least recently stamped entry of the set
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        u64 s2 = __shfl_xor_sync(FULL, old, o);
        int w2 = __shfl_xor_sync(FULL, old_w, o);
        if (s2 < old) { old = s2; old_w = w2; }
      }
      w = old_w;
    }
  }
  __syncwarp();
  if (lane == 0) {
    int e = set * P.ways + w;
    P.key[e] = phrase[0];
    for (int i = 0; i < P.S; ++i) P.suf[(size_t)e * P.S + i] = phrase[1 + i];
    P.stamp[e] = stamp;
  }
  __syncwarp();
}

__device__ void pool_erase(const PoolDev &P, const int32_t *phrase) {
  int set = pool_set(P, phrase[0]);
  int w = pool_find(P, set, phrase);
  __syncwarp();
  if (w != INT_MAX && (threadIdx.x & 31) == 0) P.key[set * P.ways + w] = -1;
  __syncwarp();
}

// Operations 0 .. n-1 by all warps of the block.  key(op) is the first token of its phrase, phrase(op, ph, old) writes the phrase
// (whole warp, between warp barriers) and says whether `old`, which has the same first token, goes.  buf: two phrases per warp.
template <typename Key, typename Phrase>
__device__ __forceinline__ void pool_apply(const PoolDev &P, DevState *st, int n, int32_t (*buf)[2][OURO_MAX_BETA], const Key &key, const Phrase &phrase) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const u64 clock = st->clock;
  for (int op0 = 0; op0 < n; op0 += 32) {
    const bool mine = op0 + lane < n && pool_set(P, key(op0 + lane)) % warps == warp;
    for (unsigned left = __ballot_sync(FULL, mine); left; left &= left - 1) {
      const int op = op0 + __ffs(left) - 1;
      __syncwarp();
      const bool erase = phrase(op, buf[warp][0], buf[warp][1]);
      __syncwarp();
      if (erase) pool_erase(P, buf[warp][1]);
      pool_insert(P, clock + 1 + op, buf[warp][0]);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) st->clock = clock + n;
}

// Up to K suffixes of phrases starting with key, newest first.  Returns the number found.
__device__ int pool_lookup(const PoolDev &P, int32_t key, int K, int32_t *suffix_out) {
  int lane = threadIdx.x & 31;
  int set = pool_set(P, key);
  if (P.ways <= 32) {
    // One way per lane: key and stamp are read once, the K newest are picked with shuffles alone, and all their
    // suffixes are fetched together: two round trips to memory whatever K is.  (Stamps start at 1 and are unique.)
    u64 mine = 0;
    if (lane < P.ways) {
      const int e = set * P.ways + lane;
      if (P.key[e] == key) mine = P.stamp[e];
    }
    int found = 0, sel = -1;                       // lane f remembers the way of the f-th newest phrase
    for (; found < K; ++found) {
      u64 best = mine;
      int best_w = mine ? lane : -1;
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        u64 s2 = __shfl_xor_sync(FULL, best, o);
        int w2 = __shfl_xor_sync(FULL, best_w, o);
        if (s2 > best) { best = s2; best_w = w2; }
      }
      if (best_w < 0) break;
      if (lane == best_w) mine = 0;
      if (lane == found) sel = best_w;
    }
    for (int idx0 = 0; idx0 < found * P.S; idx0 += 32) {
      const int idx = idx0 + lane, f = min(idx / P.S, found - 1);
      const int w = __shfl_sync(FULL, sel, f);
      if (idx < found * P.S) suffix_out[idx] = P.suf[(size_t)(set * P.ways + w) * P.S + (idx - f * P.S)];
    }
    return found;
  }
  u64 bound = ~0ull;
  int found = 0;
  for (; found < K; ++found) {
    u64 best = 0;
    int best_w = -1;
    for (int c = lane; c < P.ways; c += 32) {
      int e = set * P.ways + c;
      if (P.key[e] == key && P.stamp[e] < bound && P.stamp[e] > best) {
        best = P.stamp[e];
        best_w = c;
      }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      u64 s2 = __shfl_xor_sync(FULL, best, o);
      int w2 = __shfl_xor_sync(FULL, best_w, o);
      if (s2 > best) { best = s2; best_w = w2; }
    }
    if (best_w < 0) break;
    bound = best;
    for (int i = lane; i < P.S; i += 32) suffix_out[found * P.S + i] = P.suf[(size_t)(set * P.ways + best_w) * P.S + i];
  }
  return found;
}

__global__ void pool_clear_kernel(PoolDev P, DevState *st) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < P.sets * P.ways) {
    P.key[i] = -1;
    P.stamp[i] = 0;
  }
  if (i == 0) st->clock = 0;
}

__global__ void pool_lookup_kernel(PoolDev P, const int32_t *key_dev, int key_index, int32_t key_value, int K,
                                   int32_t *suffix, int32_t *count) {
  int32_t key = key_dev ? key_dev[key_index] : key_value;
  int n = (key < 0 || P.S == 0) ? 0 : pool_lookup(P, key, K, suffix);
  if (threadIdx.x == 0) *count = n;
}

// n beta-grams, the g-th starting at ngrams + g*stride (stride 1 = sliding windows over a text).
__global__ void __launch_bounds__(1024) pool_update_kernel(PoolDev P, DevState *st, const int32_t *ngrams, int n, int beta, int stride) {
  __shared__ int32_t buf[32][2][OURO_MAX_BETA];
  pool_apply(P, st, n, buf, [&](int g) { return ngrams[(size_t)g * stride]; },
             [&](int g, int32_t *ph, int32_t *) {
               const int i = threadIdx.x & 31;
               if (i < beta) ph[i] = ngrams[(size_t)g * stride + i];
               return false;
             });
}

void launch_pool_clear(const PoolDev &P, DevState *st, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  int n = P.sets * P.ways;
  pool_clear_kernel<<<(n + 255) / 256, 256, 0, s>>>(P, st);
}
void launch_pool_lookup(const PoolDev &P, const int32_t *key_dev, int key_index, int32_t key_value, int K,
                        int32_t *suffix, int32_t *count, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  pool_lookup_kernel<<<1, 32, 0, s>>>(P, key_dev, key_index, key_value, K, suffix, count);
}
void launch_pool_update(const PoolDev &P, DevState *st, const int32_t *ngrams, int n, int beta, int stride,
                        cudaStream_t s) {
  if (n <= 0) return;
  OURO_COUNT_LAUNCH();
  pool_update_kernel<<<1, 32 * (n < 32 ? n : 32), 0, s>>>(P, st, ngrams, n, beta, stride);
}

// --------------------------------------------------------------------------- candidate packing
// Eq. 7: rows [pending, d_1..d_gamma, p^1_2..beta, .., p^K'_2..beta].  Trunk row b: position L+b, sees
// slots [0, L+b].  Suffix row (j, i): position L+gamma+i, sees slots [0, L+gamma] and its own
// candidate's rows (j, 1..i), which sit at slots L+1+gamma+j*S .. (Eq. 8).
__device__ __forceinline__ void assemble_candidates_body(const BlockDev &b, DevState *st, const int32_t *draft,
                                                         const int32_t *suffix, const int32_t *count, int L, int gamma,
                                                         int S, int K) {
  int nc = S > 0 ? min(*count, K) : 0;
  int B = 1 + gamma + nc * S;
  int r = threadIdx.x;
  if (r == 0) {
    st->n_cand = nc;
    st->n_rows = B;
  }
  if (r >= B) return;
  u64 m0 = 0, m1 = 0;
  if (r <= gamma) {
    b.tok[r] = r == 0 ? st->pending : draft[r - 1];
    b.pos[r] = L + r;
    b.group[r] = 0;
    b.lin_end[r] = L + r + 1;
    b.seg_start[r] = 0;
    b.seg_len[r] = 0;
    for (int c = 0; c <= r; ++c) (c < 64 ? m0 : m1) |= 1ull << (c & 63);
  } else {
    int j = (r - 1 - gamma) / S, i = (r - 1 - gamma) % S + 1;
    b.tok[r] = suffix[j * S + i - 1];
    b.pos[r] = L + gamma + i;
    b.group[r] = 1 + j;
    b.lin_end[r] = L + gamma + 1;
    b.seg_start[r] = L + 1 + gamma + j * S;
    b.seg_len[r] = i;
    for (int c = 0; c <= gamma; ++c) (c < 64 ? m0 : m1) |= 1ull << (c & 63);
    for (int c = 1 + gamma + j * S; c <= r; ++c) (c < 64 ? m0 : m1) |= 1ull << (c & 63);
  }
  b.mask[2 * r] = m0;
  b.mask[2 * r + 1] = m1;
}

__global__ void assemble_candidates_kernel(BlockDev b, DevState *st, const int32_t *draft, const int32_t *suffix,
                                           const int32_t *count, int L, int gamma, int S, int K) {
  assemble_candidates_body(b, st, draft, suffix, count, L, gamma, S, K);
}

// Lookup with key d_gamma (warp 0) and packing in one launch.
__global__ void lookup_assemble_kernel(PoolDev P, BlockDev b, DevState *st, const int32_t *draft, int32_t *suffix,
                                       int32_t *count, int L, int gamma, int S, int K) {
  pdl_wait();            // launched while the kernel before it drains; it never lets its own successor start early (the
                         // forward's kernels read the block description before their dependency wait)
  if (threadIdx.x < 32) {
    int32_t key = draft[gamma - 1];
    int n = (key < 0 || P.S == 0) ? 0 : pool_lookup(P, key, K, suffix);
    if (threadIdx.x == 0) *count = n;
  }
  __syncthreads();
  assemble_candidates_body(b, st, draft, suffix, count, L, gamma, S, K);
}

__global__ void assemble_causal_kernel(BlockDev b, const int32_t *tokens, int n, int L) {
  int r = threadIdx.x;
  if (r >= n) return;
  b.tok[r] = tokens[r];
  b.pos[r] = L + r;
  b.group[r] = 0;
  b.lin_end[r] = L + r + 1;
  b.seg_start[r] = 0;
  b.seg_len[r] = 0;
  u64 m0 = 0, m1 = 0;                      // (a block of known text may be longer than the masks, which nobody reads then)
  for (int c = 0; c <= min(r, OURO_MAX_ROWS - 1); ++c) (c < 64 ? m0 : m1) |= 1ull << (c & 63);
  b.mask[2 * r] = m0;
  b.mask[2 * r + 1] = m1;
}

void launch_assemble_candidates(const BlockDev &b, DevState *st, const int32_t *draft, const int32_t *suffix,
                                const int32_t *count, int L, int gamma, int S, int K, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  assemble_candidates_kernel<<<1, OURO_MAX_ROWS, 0, s>>>(b, st, draft, suffix, count, L, gamma, S, K);
}
void launch_lookup_assemble(const PoolDev &P, const BlockDev &b, DevState *st, const int32_t *draft, int32_t *suffix,
                            int32_t *count, int L, int gamma, int S, int K, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  launch_pdl(lookup_assemble_kernel, 1, OURO_MAX_ROWS, 0, s, P, b, st, draft, suffix, count, L, gamma, S, K);
}
void launch_assemble_causal(const BlockDev &b, const int32_t *tokens, int n, int L, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  assemble_causal_kernel<<<1, OURO_TEXT_ROWS, 0, s>>>(b, tokens, n, L);
}

// ------------------------------------------------------------------------------- acceptance
// Eq. 3: A = longest a with d_1..a equal to the target's outputs at rows 0..a-1.  Eq. 9 (only when
// A == gamma): candidate j's chain is o[gamma], then the outputs at its own suffix rows; m_j counts
// its leading suffix tokens equal to that chain; the largest m_j wins, earliest j on ties.  The step
// accepts the matched tokens plus the chain's next output.
//
// All of it is comparisons of a row's token with the output of the row in front of it (of row gamma, for the first of a
// suffix): one thread per row fetches and compares, and what is left are leading ones of a 128-bit mask.
struct Verdict {
  int32_t tok[OURO_MAX_ROWS], o[OURO_MAX_ROWS];
  uint32_t match[OURO_MAX_ROWS / 32 + 1];
  int A, chosen, m, n_cand;
};
// Rows a, a+1, .. that match, up to n of them (n <= 32).
__device__ __forceinline__ int matching(const Verdict &v, int a, int n) {
  const uint32_t bits = __funnelshift_r(v.match[a >> 5], v.match[(a >> 5) + 1], a & 31);
  return min(n, bits == FULL ? 32 : __ffs(~bits) - 1);
}
// Whole block of at least OURO_MAX_ROWS threads; `v` is complete behind it.
__device__ __forceinline__ void decide(const BlockDev &b, const DevState *st, const int32_t *o, int gamma, int S, Verdict &v) {
  const int r = threadIdx.x;
  const int nc = st->n_cand, rows = 1 + gamma + nc * S;
  if (r < OURO_MAX_ROWS) {
    v.tok[r] = r < rows ? b.tok[r] : 0;
    v.o[r] = r < rows ? o[r] : 0;
  }
  __syncthreads();
  if (r < OURO_MAX_ROWS) {
    const bool first = r > gamma && S > 0 && (r - 1 - gamma) % S == 0;
    const uint32_t bits = __ballot_sync(FULL, r >= 1 && r < rows && v.tok[r] == v.o[first ? gamma : r - 1]);
    if ((r & 31) == 0) v.match[r >> 5] = bits;
  }
  if (r == 0) v.match[OURO_MAX_ROWS / 32] = 0;
  __syncthreads();
  if (r == 0) {
    const int A = matching(v, 1, gamma);
    int chosen = -1, best = -1;
    if (A == gamma)
      for (int j = 0; j < nc; ++j) {
        const int mj = matching(v, 1 + gamma + j * S, S);
        if (mj > best) { best = mj; chosen = j; }
      }
    v.A = A;
    v.chosen = chosen;
    v.m = max(best, 0);
    v.n_cand = nc;
  }
  __syncthreads();
}

// ------------------------------------------------------------------------------ KV compaction
// Slots L..L+A (pending token and accepted draft) already sit where they belong.  An accepted suffix of
// candidate j sits at slots L+1+gamma+j*S+[0,m) and moves to L+1+gamma+[0,m).  Source and destination
// ranges never overlap (j*S >= S >= m), so all rows move in parallel (accept_compact_harvest_kernel below).
// ---------------------------------------------------------------------------------- harvest
// Pool updates after a verification (Section 3.3), serialised in a fixed order by one warp:
//  1. when the draft was fully accepted: every tried phrase (d_gamma, p^j_2..beta), j ascending, is
//     replaced by (d_gamma, o[gamma], o at suffix rows (j,1..S-1)), the target's own continuation under
//     that candidate's context; an unchanged phrase is just refreshed;
//  2. when it was not: for every trunk row s in the discarded region (A+1 <= s <= gamma-1) whose
//     following draft tokens agree with the target outputs for at least max(1, beta-2) positions, the
//     beta-gram (t_s, o_s, .., o_{s+beta-2}) is inserted;
//  3. extension: every beta-window of the text that ends inside the newly accepted tokens.
struct Harvest {
  int16_t op[OURO_MAX_ROWS];                            // 0 .. 15: candidate; 16 ..: 16 + trunk row; 64 ..: 64 + accepted token
  int32_t text[2 * OURO_MAX_BETA + OURO_MAX_GAMMA];     // the beta - 1 tokens in front of the accepted ones, then those
  int n;
};
static_assert(OURO_MAX_K <= 16 && OURO_MAX_GAMMA <= 48, "codes of the operations");

// Acceptance, compaction and harvest in one launch.  Block 0 decides (Eq. 3, Eq. 9), posts the result and harvests.
// Blocks 1..: one (layer, K or V, suffix slot) each; every such block decides for itself instead of
// waiting for block 0, then moves its cache row if the row belongs to the accepted suffix.
constexpr int ACCEPT_THREADS = 256;
__global__ void __launch_bounds__(ACCEPT_THREADS) accept_compact_harvest_kernel(BlockDev b, DevState *st, PoolDev P, const int32_t *o, int32_t *seq_dev,
                                              unsigned char *k_cache, unsigned char *v_cache, int L, int gamma, int S,
                                              int max_seq, int row_bytes, unsigned flags, int32_t *mbox, int32_t seq) {
  __shared__ Verdict v;
  pdl_wait();            // its blocks are in place while the kernel that writes `o` finishes
  const int t = threadIdx.x;
  if (blockIdx.x == 0) {
    __shared__ Harvest hv;
    __shared__ int32_t buf[ACCEPT_THREADS / 32][2][OURO_MAX_BETA];
    const int beta = S + 1, n_seq = st->n_seq, status = st->status;
    if (t < S && n_seq - S + t >= 0) hv.text[t] = seq_dev[n_seq - S + t];
    decide(b, st, o, gamma, S, v);
    const int A = v.A, m = v.m, n = A + m + 1, suffix = 1 + gamma + v.chosen * S;
    const int32_t bonus = v.chosen < 0 || m == 0 ? v.o[A] : v.o[suffix + m - 1];
    // the record A .. n_cand_last, one value per thread
    constexpr int ACC = OURO_MAX_GAMMA + OURO_MAX_BETA, REC = 4 + ACC + 2;
    if (t < REC) {
      const int i = t - 4;
      const int32_t token = i < A ? v.tok[1 + max(i, 0)] : i < A + m ? v.tok[suffix + i - A] : bonus;
      const int32_t value = t == 0 ? A : t == 1 ? v.chosen : t == 2 ? m : t == 3 ? n : t < 4 + ACC ? token : t == 4 + ACC ? status : v.n_cand;
      const bool live = t < 4 + n || t >= 4 + ACC;
      if (mbox && live) mbox[MBOX_ACCEPT + 1 + t] = value;
      if (live && t != 4 + ACC) (&st->A)[t] = value;
      if (t >= 4 && t < 4 + n) {
        seq_dev[n_seq + i] = token;
        hv.text[S + i] = token;
      }
    }
    __syncthreads();
    if (t == 0) {
      if (mbox) {
        // what the host is polling for: behind the words of all threads, which the barrier has put in front of this fence
        __threadfence_system();
        *(volatile int32_t *)(mbox + MBOX_ACCEPT) = seq;
      }
      st->pending = bonus;
      st->n_seq = n_seq + n;
      int k = 0;
      if ((flags & OURO_HARVEST_CANDIDATES) && A == gamma)
        for (int j = 0; j < v.n_cand; ++j) hv.op[k++] = j;
      if ((flags & OURO_HARVEST_MATCHED) && A < gamma)
        for (int r = A + 1; r < gamma; ++r)
          if (matching(v, r + 1, gamma - r) >= max(1, beta - 2)) hv.op[k++] = 16 + r;
      if (flags & OURO_HARVEST_ACCEPTED)
        for (int i = 0; i < n; ++i)
          if (n_seq + i - S >= 0) hv.op[k++] = 64 + i;
      hv.n = k;
    }
    __syncthreads();
    pool_apply(P, st, hv.n, buf,
               [&](int op) {
                 const int c = hv.op[op];
                 return c < 16 ? v.tok[gamma] : c < 64 ? v.tok[c - 16] : hv.text[c - 64];
               },
               [&](int op, int32_t *ph, int32_t *old) {
                 const int c = hv.op[op], i = t & 31;             // token i of the phrase
                 bool differs = false;
                 if (i < beta) {
                   if (c < 16) {
                     const int base = 1 + gamma + c * S;
                     ph[i] = i == 0 ? v.tok[gamma] : i == 1 ? v.o[gamma] : v.o[base + i - 2];
                     old[i] = i == 0 ? v.tok[gamma] : v.tok[base + i - 1];
                     differs = ph[i] != old[i];
                   } else if (c < 64) {
                     ph[i] = i == 0 ? v.tok[c - 16] : v.o[c - 16 + i - 1];
                   } else {
                     ph[i] = hv.text[c - 64 + i];
                   }
                 }
                 return __any_sync(FULL, differs) != 0;
               });
    return;
  }
  decide(b, st, o, gamma, S, v);
  const int idx = blockIdx.x - 1, slot = idx % S, ly = idx / S;    // ly = 2 * layer + (0: K, 1: V)
  if (v.chosen <= 0 || slot >= v.m) return;                        // candidate 0 already sits next to the trunk
  unsigned char *base = ((ly & 1) ? v_cache : k_cache) + (size_t)(ly >> 1) * max_seq * row_bytes;
  const uint4 *src = (const uint4 *)(base + (size_t)(L + 1 + gamma + v.chosen * S + slot) * row_bytes);
  uint4 *dst = (uint4 *)(base + (size_t)(L + 1 + gamma + slot) * row_bytes);
  for (int i = t; i < row_bytes / 16; i += blockDim.x) dst[i] = src[i];
}

void launch_accept_compact_harvest(const BlockDev &b, DevState *st, const PoolDev &P, const int32_t *o, int32_t *seq_dev,
                                   const ouro_model_desc &d, void *k_cache, void *v_cache, int L, int gamma, int S,
                                   unsigned flags, int32_t *mbox, int32_t seq, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  const int es = d.dtype == OURO_BF16 ? 2 : 4;
  launch_pdl(accept_compact_harvest_kernel, 1 + S * d.n_layers * 2, ACCEPT_THREADS, 0, s, b, st, P, o, seq_dev, (unsigned char *)k_cache,
             (unsigned char *)v_cache, L, gamma, S, (int)d.max_seq, d.n_kv_heads * d.head_dim * es, flags, mbox, seq);
}

// ------------------------------------------------------------- phrase-level drafting (Section 3.1)
// A drafting round of the draft model.  Rows 0..n-1 are text it is fed (tokens[0..n-1], no verification needed),
// then the suffixes of up to K pool phrases that start with tokens[n-1], packed as in Eq. 7 / Eq. 8 with the
// n text rows in the role of the trunk.
__global__ void draft_lookup_assemble_kernel(PoolDev P, BlockDev b, DevState *st, const int32_t *tokens, int n,
                                             int32_t *suffix, int32_t *count, int L, int S, int K) {
  if (threadIdx.x < 32) {
    int32_t key = tokens[n - 1];
    int found = (key < 0 || P.S == 0 || S == 0) ? 0 : pool_lookup(P, key, K, suffix);
    if (threadIdx.x == 0) *count = found;
  }
  __syncthreads();
  const int nc = S > 0 ? min(*count, K) : 0, B = n + nc * S, r = threadIdx.x;
  if (r == 0) {
    st->d_cand = nc;
    st->d_rows = B;
  }
  if (r >= B) return;
  u64 m0 = 0, m1 = 0;
  if (r < n) {
    b.tok[r] = tokens[r];
    b.pos[r] = L + r;
    b.group[r] = 0;
    b.lin_end[r] = L + r + 1;
    b.seg_start[r] = 0;
    b.seg_len[r] = 0;
    for (int c = 0; c <= r; ++c) (c < 64 ? m0 : m1) |= 1ull << (c & 63);
  } else {
    const int j = (r - n) / S, i = (r - n) % S + 1;
    b.tok[r] = suffix[j * S + i - 1];
    b.pos[r] = L + n - 1 + i;
    b.group[r] = 1 + j;
    b.lin_end[r] = L + n;
    b.seg_start[r] = L + n + j * S;
    b.seg_len[r] = i;
    for (int c = 0; c < n; ++c) (c < 64 ? m0 : m1) |= 1ull << (c & 63);
    for (int c = n + j * S; c <= r; ++c) (c < 64 ? m0 : m1) |= 1ull << (c & 63);
  }
  b.mask[2 * r] = m0;
  b.mask[2 * r + 1] = m1;
}

// The round's outcome.  The draft model's next greedy token is o[n-1]; candidate j's chain continues from it as
// in Eq. 9; the longest match wins (earliest on ties) and the round yields its m tokens plus the chain's next
// one, cut to what the draft still lacks.  Block 0 writes the tokens; blocks 1.. each re-derive the choice and
// move one row of the draft cache next to the text (candidate 0 already sits there).
__global__ void draft_accept_compact_kernel(BlockDev b, DevState *st, const int32_t *o, int32_t *out_dev, int have,
                                            int gamma, unsigned char *k_cache, unsigned char *v_cache, int L, int n, int S,
                                            int max_seq, int row_bytes) {
  __shared__ int s_chosen, s_m;
  __shared__ int32_t s_bonus;
  if (threadIdx.x == 0) {
    const int nc = st->d_cand;
    int chosen = -1, best = -1;
    int32_t bonus = o[n - 1];
    for (int j = 0; j < nc; ++j) {
      int base = n + j * S, mj = 0;
      int32_t v = o[n - 1];
      while (mj < S && b.tok[base + mj] == v) { v = o[base + mj]; ++mj; }
      if (mj > best) { best = mj; chosen = j; bonus = v; }
    }
    s_chosen = chosen;
    s_m = best < 0 ? 0 : best;
    s_bonus = bonus;
  }
  __syncthreads();
  const int m = s_m, keep = min(m + 1, gamma - have), cached = min(m, keep);
  if (blockIdx.x == 0) {
    if (threadIdx.x < keep) out_dev[have + threadIdx.x] = (int)threadIdx.x < m ? b.tok[n + s_chosen * S + threadIdx.x] : s_bonus;
    if (threadIdx.x == 0) {
      st->d_keep = keep;
      st->d_cached = cached;
    }
    return;
  }
  const int idx = blockIdx.x - 1, t = idx % S, ly = idx / S;       // ly = 2 * layer + (0: K, 1: V)
  if (s_chosen <= 0 || t >= cached) return;
  unsigned char *base = ((ly & 1) ? v_cache : k_cache) + (size_t)(ly >> 1) * max_seq * row_bytes;
  const uint4 *src = (const uint4 *)(base + (size_t)(L + n + s_chosen * S + t) * row_bytes);
  uint4 *dst = (uint4 *)(base + (size_t)(L + n + t) * row_bytes);
  for (int i = threadIdx.x; i < row_bytes / 16; i += blockDim.x) dst[i] = src[i];
}

void launch_draft_lookup_assemble(const PoolDev &P, const BlockDev &b, DevState *st, const int32_t *tokens, int n,
                                  int32_t *suffix, int32_t *count, int L, int S, int K, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  draft_lookup_assemble_kernel<<<1, OURO_MAX_ROWS, 0, s>>>(P, b, st, tokens, n, suffix, count, L, S, K);
}
void launch_draft_accept_compact(const BlockDev &b, DevState *st, const int32_t *o, int32_t *out_dev, int have, int gamma,
                                 const ouro_model_desc &d, void *k_cache, void *v_cache, int L, int n, int S,
                                 cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  const int es = d.dtype == OURO_BF16 ? 2 : 4;
  draft_accept_compact_kernel<<<1 + (S > 0 ? S : 0) * d.n_layers * 2, 128, 0, s>>>(
      b, st, o, out_dev, have, gamma, (unsigned char *)k_cache, (unsigned char *)v_cache, L, n, S, d.max_seq,
      d.n_kv_heads * d.head_dim * es);
}

// ------------------------------------------- phrase generation during the draft forward (Section 3.1)
// A draft forward with a lookahead window: rows 0..n-1 are text the draft model is fed, rows n..n+W-1 hold the
// window's guesses for the W positions that follow, packed like one candidate suffix (window row i sees the text and
// window rows 1..i).  An empty window (after a reset) is first filled from the end of the text.
__global__ void draft_window_assemble_kernel(BlockDev b, DevState *st, const int32_t *tokens, int n, int32_t *win, int W,
                                             const int32_t *seq_dev, int L) {
  const int r = threadIdx.x;
  if (!st->win_valid) {
    const int n_seq = st->n_seq;
    if (r < W) {
      const int src = n_seq - W + r;                      // the text's last W tokens; a short text repeats its last one in front
      win[r] = seq_dev[src >= 0 ? src : n_seq - 1];
    }
  }
  __syncthreads();
  if (r == 0) st->win_valid = 1;
  if (r >= n + W) return;
  u64 m0 = 0, m1 = 0;
  if (r < n) {
    b.tok[r] = tokens[r];
    b.pos[r] = L + r;
    b.group[r] = 0;
    b.lin_end[r] = L + r + 1;
    b.seg_start[r] = 0;
    b.seg_len[r] = 0;
    for (int c = 0; c <= r; ++c) (c < 64 ? m0 : m1) |= 1ull << (c & 63);
  } else {
    const int i = r - n + 1;
    b.tok[r] = win[i - 1];
    b.pos[r] = L + n - 1 + i;
    b.group[r] = 1;
    b.lin_end[r] = L + n;
    b.seg_start[r] = L + n;
    b.seg_len[r] = i;
    for (int c = 0; c <= r; ++c) (c < 64 ? m0 : m1) |= 1ull << (c & 63);
  }
  b.mask[2 * r] = m0;
  b.mask[2 * r + 1] = m1;
}

// After that forward: chain[0] = o[n-1] is the next draft token; chain[i] = o[n-1+i] is the prediction after window
// guess i.  The beta-grams along the diagonal, (src[i], chain[i], .., chain[i+S-1]) for i = 0 .. W-S+1 with src[0] the
// last text token and src[i] guess i, enter the pool in that order; then the window becomes chain[1..W].
__global__ void __launch_bounds__(512) draft_window_harvest_kernel(BlockDev b, DevState *st, PoolDev P, const int32_t *o, int32_t *out, int n, int W,
                                            int32_t *win) {
  __shared__ int32_t buf[16][2][OURO_MAX_BETA], src[OURO_MAX_WINDOW + 1], chain[OURO_MAX_WINDOW + 1];
  pdl_wait();
  const int t = threadIdx.x, S = P.S;
  if (t <= W) {
    src[t] = b.tok[n - 1 + t];
    chain[t] = o[n - 1 + t];
    if (t > 0) win[t - 1] = o[n - 1 + t];
    if (t == 0 && out) *out = o[n - 1];
  }
  __syncthreads();
  if (S >= 1 && W - S + 2 > 0)
    pool_apply(P, st, W - S + 2, buf, [&](int i) { return src[i]; },
               [&](int i, int32_t *ph, int32_t *) {
                 const int q = t & 31;
                 if (q <= S) ph[q] = q == 0 ? src[i] : chain[i + q - 1];
                 return false;
               });
}

void launch_draft_window_assemble(const BlockDev &b, DevState *st, const int32_t *tokens, int n, int32_t *win, int W,
                                  const int32_t *seq_dev, int L, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  draft_window_assemble_kernel<<<1, OURO_MAX_ROWS, 0, s>>>(b, st, tokens, n, win, W, seq_dev, L);
}
void launch_draft_window_harvest(const BlockDev &b, DevState *st, const PoolDev &P, const int32_t *o, int32_t *out_or_null,
                                 int n, int W, int32_t *win, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  launch_pdl(draft_window_harvest_kernel, 1, 512, 0, s, b, st, P, o, out_or_null, n, W, win);
}

// ----------------------------------------------------------------------------------- argmax
// Greedy choice per row; equal maxima resolve to the smallest token id.
__global__ void argmax_kernel(const float *logits, int vocab, int32_t *out) {
  const float *row = logits + (size_t)blockIdx.x * vocab;
  float best = -INFINITY;
  int idx = INT_MAX;
  for (int i = threadIdx.x; i < vocab; i += blockDim.x) {
    float v = row[i];
    if (v > best || (v == best && i < idx)) { best = v; idx = i; }
  }
  __shared__ float sv[32];
  __shared__ int si[32];
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    float v2 = __shfl_xor_sync(FULL, best, o);
    int i2 = __shfl_xor_sync(FULL, idx, o);
    if (v2 > best || (v2 == best && i2 < idx)) { best = v2; idx = i2; }
  }
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) { sv[warp] = best; si[warp] = idx; }
  __syncthreads();
  if (warp == 0) {
    int nw = blockDim.x >> 5;
    best = lane < nw ? sv[lane] : -INFINITY;
    idx = lane < nw ? si[lane] : INT_MAX;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      float v2 = __shfl_xor_sync(FULL, best, o);
      int i2 = __shfl_xor_sync(FULL, idx, o);
      if (v2 > best || (v2 == best && i2 < idx)) { best = v2; idx = i2; }
    }
    if (lane == 0) out[blockIdx.x] = idx == INT_MAX ? 0 : idx;
  }
}

void launch_argmax(const float *logits, int rows, int vocab, int32_t *out, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  argmax_kernel<<<rows, 256, 0, s>>>(logits, vocab, out);
}

// Plain greedy decoding: the row-0 output becomes the next pending token and joins the text.
__global__ void vanilla_accept_kernel(DevState *st, const int32_t *o, int32_t *seq_dev) {
  st->pending = o[0];
  seq_dev[st->n_seq] = o[0];
  st->n_seq += 1;
}
void launch_vanilla_accept(DevState *st, const int32_t *o, int32_t *seq_dev, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  vanilla_accept_kernel<<<1, 1, 0, s>>>(st, o, seq_dev);
}

__global__ void pick_token_kernel(const int32_t *src, int index, int32_t *dst) {
  pdl_wait();
  *dst = src[index];
}
void launch_pick_token(const int32_t *src, int index, int32_t *dst, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  launch_pdl(pick_token_kernel, 1, 1, 0, s, src, index, dst);
}

// A drafted token joins the draft and is the whole of the next block: one launch instead of two, in place while the
// forward before drains.  The kernels after it start when it has finished (it does not trigger them), as they expect of
// an assembling kernel.
__global__ void pick_assemble_kernel(BlockDev b, const int32_t *src, int index, int32_t *dst, int L) {
  pdl_wait();
  const int32_t token = src[index];
  *dst = token;
  b.tok[0] = token;
  b.pos[0] = L;
  b.group[0] = 0;
  b.lin_end[0] = L + 1;
  b.seg_start[0] = 0;
  b.seg_len[0] = 0;
  b.mask[0] = 1;
  b.mask[1] = 0;
}
void launch_pick_assemble(const BlockDev &b, const int32_t *src, int index, int32_t *dst, int L, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  launch_pdl(pick_assemble_kernel, 1, 1, 0, s, b, src, index, dst, L);
}

// Text of n_seq tokens ending in the pending token; with fill, the earlier positions are recorded as 0.  The status word is
// cleared, and with it what a launch that raised it left behind: nobody need have read the status in between.
__global__ void set_state_kernel(DevState *st, int32_t *seq_dev, int n_seq, int pending, int fill, const Leftovers left) {
  const int status = blockIdx.x == 0 ? *(volatile const int32_t *)&st->status : 0;     // (asked for first, needed last)
  if (fill)
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_seq - 1; i += gridDim.x * blockDim.x) seq_dev[i] = 0;
  if (blockIdx.x != 0) return;
  if (threadIdx.x == 0) {
    seq_dev[n_seq - 1] = pending;
    st->pending = pending;
    st->n_seq = n_seq;
    st->n_cand = 0;
    st->n_rows = 0;
    st->win_valid = 0;
  }
  if (status != 0) {
    for (size_t i = threadIdx.x; i < left.n_slots; i += blockDim.x) left.slots[i] = make_uint4(left.empty, left.empty, left.empty, left.empty);
    if ((int)threadIdx.x < left.n_counters) left.counters[threadIdx.x] = left.value[threadIdx.x];
    if (left.met && threadIdx.x < 2) left.met[threadIdx.x] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) st->status = 0;
}
void launch_set_state(DevState *st, int32_t *seq_dev, int n_seq, int pending, int fill, const Leftovers &left, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  set_state_kernel<<<8, 256, 0, s>>>(st, seq_dev, n_seq, pending, fill, left);
}
