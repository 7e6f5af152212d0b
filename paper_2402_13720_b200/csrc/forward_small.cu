// One forward of a small generic model (fp32, or bf16 shapes the tensor-core kernels do not take) as ONE launch.
//
// Such a model's weights are read in microseconds; what a forward costs is its chain of dependent steps, eight launches a
// layer as kernels of their own (5.6 us each on the fp32 pair of 128-wide layers).  Here one CTA per SM stays for the
// whole forward and the steps are separated by grid barriers.  A warp takes a unit of a step: one, two or four output
// columns for a tile of rows; four warps take one (row, head) of the attention (one warp each: 2815 us for 64 tokens, four:
// 2391).  One cluster of 16 CTAs with its barrier in hardware was slower (2511 us): the units then queue for its warps.
// RMSNorm has no step of its own: the warp that contracts a row with the weights has just read the row, and sums its
// squares first.
//
// The rule of kernels_layer.cu holds: a value depends on its own row and on the keys that row sees, in fixed groups.
//
// The barriers are bounded: on expiry the CTA raises the context's status word and leaves, and so do the others.  Their counts
// begin and end a launch at zero, on the device alone: a launch that was refused, or one replayed from a graph, needs
// no book-keeping on the host.
#include <algorithm>
#include <type_traits>

#include "ouro_internal.h"
#include "generic.cuh"
#include "row_ops.cuh"

namespace {

constexpr int THREADS = 256;
constexpr int WARPS = THREADS / 32;
constexpr int QUAD = 4;                  // warps that share one (row, head) of the attention: warp j takes key groups j, j + 4, ..
constexpr int MAX_LAYERS = 40;           // layer pointers travel as kernel parameters

struct LayerPtrs { const void *attn_norm, *wq, *wk, *wv, *wo, *ffn_norm, *w_gate, *w_up, *w_down; };
struct SmallParams {
  LayerPtrs layer[MAX_LAYERS];
  const void *embed, *final_norm, *lm_head;
  void *k_cache, *v_cache;
  const float *cos_t, *sin_t;
  BlockDev b;
  int n_layers, d, H, Hkv, h, F, V, max_seq, L;
  float eps, scale;
  int rows;
  const int *rows_dev;     // NULL, or the block's true row count in device memory (`rows` is then an upper bound)
  float *x;                // residual stream [rows][d]
  void *q, *att, *act;     // [rows][dq], [rows][dq], [rows][F]
  float *logits;           // [rows][V]
  int32_t *argmax;         // [rows]; NULL: the last layer ends with its keys and values
  uint32_t *met;           // [2] CTAs arrived: at all barriers but the last, and at the last
  uint32_t wait_limit;     // polls of a barrier before it gives up
  int *status;
};
static_assert(sizeof(SmallParams) <= 4096, "kernel parameters");

// All CTAs of the grid (one per SM, launched cooperatively) meet; writes before are visible after.  False: given up, by this
// launch or by one before it (gave_up), whose counts then stand where it left them.
// Nobody arrives at the last barrier before having left those in front of it, so the count of those goes back to zero
// behind it; the last one's goes back to zero before the next launch's first barrier (see the kernel's beginning).
__device__ __forceinline__ bool grid_barrier(const SmallParams &p, uint32_t &target, bool last, int gave_up, int *flag) {
  uint32_t *const count = p.met + (last ? 1 : 0);
  target = last ? gridDim.x : target + gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    int ok = 0;
    for (uint32_t spin = 0; spin < p.wait_limit && !gave_up; ++spin) {
      uint32_t seen;
      asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
      if (seen >= target) { ok = 1; break; }
      if ((spin & 63) == 63 && *(volatile const int *)p.status != 0) break;
    }
    if (!ok) atomicExch(p.status, 1);
    else if (last && blockIdx.x == 0) *(volatile uint32_t *)p.met = 0;
    *flag = ok;
  }
  __syncthreads();
  return *flag != 0;
}

// Contractions of a tile of rows with C weight rows, the rows normalised on the way (gain != NULL):
//   acc[c][i] = sum_k T(gain[k] * x[i][k] / rms(x[i])) * w[c][k], lanes stride over k, the same order for any tile.
template <typename T, int C, int RT, typename Row>
__device__ __forceinline__ void contract(const Row &row, const T *gain, float eps, const T *const *w, int n_rows, int K, float (*acc)[RT]) {
  constexpr int V = Vec<T>::N;
  const int lane = threadIdx.x & 31;
  float inv[RT];
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    inv[i] = 0.f;
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c][i] = 0.f;
  }
  if (RT <= 2 && K <= 32 * V) {
    // a row is one vector per lane: everything is fetched at once and read once (the same sums in the same order)
    const int k = lane * V;
    const bool in = k < K;
    Vec<T> wv[C], gv;
    float xv[RT][V];
    if (in) {
#pragma unroll
      for (int c = 0; c < C; ++c) wv[c].load(w[c] + k);
      if (gain) gv.load(gain + k);
#pragma unroll
      for (int i = 0; i < RT; ++i)
        if (i < n_rows) row(i, k, xv[i]);
#pragma unroll
      for (int i = 0; i < RT; ++i)
        if (gain && i < n_rows) {
#pragma unroll
          for (int e = 0; e < V; ++e) inv[i] = fmaf(xv[i][e], xv[i][e], inv[i]);
        }
    }
    if (gain) {
#pragma unroll
      for (int i = 0; i < RT; ++i)
        if (i < n_rows) inv[i] = 1.0f / sqrtf(warp_sum(inv[i]) / (float)K + eps);
    }
    if (in) {
#pragma unroll
      for (int i = 0; i < RT; ++i)
        if (i < n_rows) {
#pragma unroll
          for (int e = 0; e < V; ++e) {
            const float a = gain ? to_f<T>(from_f<T>(gv.get(e) * (xv[i][e] * inv[i]))) : xv[i][e];
#pragma unroll
            for (int c = 0; c < C; ++c) acc[c][i] = fmaf(a, wv[c].get(e), acc[c][i]);
          }
        }
    }
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int i = 0; i < RT; ++i)
        if (i < n_rows) acc[c][i] = warp_sum(acc[c][i]);
    return;
  }
  // Rows beyond the tile's last repeat it (their sums are not used): the rows' loads are then under way together, where a branch
  // around each would wait for one before the next is requested.
  if (gain) {
    for (int k = lane * V; k < K; k += 32 * V) {
      float xv[RT][V];
#pragma unroll
      for (int i = 0; i < RT; ++i) row(min(i, n_rows - 1), k, xv[i]);
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int e = 0; e < V; ++e) inv[i] = fmaf(xv[i][e], xv[i][e], inv[i]);
    }
#pragma unroll
    for (int i = 0; i < RT; ++i) inv[i] = 1.0f / sqrtf(warp_sum(inv[i]) / (float)K + eps);
  }
#pragma unroll (RT <= 2 ? 2 : 1)
  for (int k = lane * V; k < K; k += 32 * V) {
    Vec<T> wv[C], gv;
#pragma unroll
    for (int c = 0; c < C; ++c) wv[c].load(w[c] + k);
    if (gain) gv.load(gain + k);
    float xv[RT][V];
#pragma unroll
    for (int i = 0; i < RT; ++i) row(min(i, n_rows - 1), k, xv[i]);
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const float a = gain ? to_f<T>(from_f<T>(gv.get(e) * (xv[i][e] * inv[i]))) : xv[i][e];
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c][i] = fmaf(a, wv[c].get(e), acc[c][i]);
      }
  }
#pragma unroll
  for (int c = 0; c < C; ++c)
#pragma unroll
    for (int i = 0; i < RT; ++i) acc[c][i] = warp_sum(acc[c][i]);
}

// Lane i's value of a tile's rows.
template <int RT>
__device__ __forceinline__ float of_row(const float (&acc)[RT], int lane) {
  float v = acc[0];
#pragma unroll
  for (int i = 1; i < RT; ++i) v = lane == i ? acc[i] : v;
  return v;
}

// WIDE: steps with work for many warps may take larger units (by_rows and the head).  A kernel of its own, so that the short
// blocks of a narrow model, which wait for their instructions as much as for anything else, run the shorter code.
template <typename T, bool WIDE>
__global__ void __launch_bounds__(THREADS, 1) forward_small_kernel(const __grid_constant__ SmallParams p) {
  __shared__ float sq[WARPS][128];         // attention: a warp's copy of its query, then its unnormalised output
  __shared__ float2 sml[WARPS];            // ... and its score maximum and sum
  __shared__ int flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gw = warp * gridDim.x + blockIdx.x, nw = gridDim.x * WARPS;   // (a short step is spread over the SMs)
  const int rows = p.rows_dev ? min(p.rows, __ldg(p.rows_dev)) : p.rows;
  const int d = p.d, h = p.h, half = h >> 1, dq = p.H * h, dkv = p.Hkv * h;
  uint32_t target = 0;
  int gave_up = 0;
  if (threadIdx.x == 0) gave_up = *(volatile const int *)p.status;
  if (blockIdx.x == 0 && threadIdx.x == 0) *(volatile uint32_t *)(p.met + 1) = 0;    // (made visible by the first barrier's arrival)
  T *q = (T *)p.q, *att = (T *)p.att, *act = (T *)p.act;

  // Rows of a unit, for a step of n columns (groups of them, pairs): two, so that a short block is spread over many warps (64
  // tokens of the fp32 pair: 2264 us, four rows 2365); eight where more than half the warps have a unit even so, since a unit
  // reads its weights once for all its rows (fp32, 512 x 2048, vocabulary 32000, 128 rows: 11.9 ms with two rows and one
  // column of the head a unit, 1.96 ms with eight and four; a row's sums are the same either way).
  auto by_rows = [&](int n, auto body) {
    if constexpr (WIDE)
      if (rows > 2 && n * ((rows + 7) / 8) > nw / 2) return body(std::integral_constant<int, 8>{});
    body(std::integral_constant<int, 2>{});
  };

  // a row of the residual stream: in front of the first layer still the token's embedding.  (Rows come through L1: the units of
  // a tile read the same ones, and the barrier's acquire makes what other SMs wrote visible.)
  int r0 = 0;
  bool embedded = true;
  auto residual = [&](int i, int k, float *xv) {
    constexpr int V = Vec<T>::N;
    if (embedded) {
      Vec<T> e;
      e.load((const T *)p.embed + (size_t)p.b.tok[r0 + i] * d + k);
#pragma unroll
      for (int j = 0; j < V; ++j) xv[j] = e.get(j);
    } else {
#pragma unroll
      for (int j = 0; j < V; j += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(p.x + (size_t)(r0 + i) * d + k + j);
        xv[j] = v.x; xv[j + 1] = v.y; xv[j + 2] = v.z; xv[j + 3] = v.w;
      }
    }
  };
  auto stored = [&](const T *base, int K) {
    return [=](int i, int k, float *xv) {
      constexpr int V = Vec<T>::N;
      Vec<T> e;
      e.load(base + (size_t)i * K + k);
#pragma unroll
      for (int j = 0; j < V; ++j) xv[j] = e.get(j);
    };
  };

  for (int l = 0; l < p.n_layers; ++l) {
    const LayerPtrs &w = p.layer[l];
    const size_t layer_off = (size_t)l * p.max_seq * dkv;
    // ---- q, k, v of the normalised rows, rotary positions, cache append.  A unit: dimensions i and i + half of a head
    const int pairs = (p.H + 2 * p.Hkv) * half;
    by_rows(pairs, [&](auto rt) {
    constexpr int RT = decltype(rt)::value;
    const int tiles = (rows + RT - 1) / RT;
    for (int u = gw; u < pairs * tiles; u += nw) {
      const int head = (u % pairs) / half, i = (u % pairs) % half;
      r0 = u / pairs * RT;
      const int n = min(RT, rows - r0);
      const bool is_q = head < p.H, is_v = head >= p.H + p.Hkv;
      const int hh = is_q ? head : is_v ? head - p.H - p.Hkv : head - p.H;
      const T *base = (const T *)(is_q ? w.wq : is_v ? w.wv : w.wk) + ((size_t)hh * h + i) * d;
      const T *const ws[2] = {base, base + (size_t)half * d};
      // What the last step of a unit needs besides is asked for in front of its contraction: round trips to L2, one after the
      // other, are what a short step consists of (here, in `project`, and in the unrolling of the sums over keys and of the greedy
      // choice; 64 tokens of the fp32 pair, mean of three prompts, 2.13 -> 2.07 ms).
      float c = 1.f, s = 0.f;
      if (lane < n && !is_v) {
        const size_t ti = (size_t)p.b.pos[r0 + lane] * half + i;
        c = p.cos_t[ti];
        s = p.sin_t[ti];
      }
      float acc[2][RT];
      contract<T, 2, RT>(residual, (const T *)w.attn_norm, p.eps, ws, n, d, acc);
      if (lane < n) {
        const int r = r0 + lane;
        const float a = of_row<RT>(acc[0], lane), b = of_row<RT>(acc[1], lane);
        float ra = a, rb = b;
        if (!is_v) {
          ra = rowops::rotate(a, b, c, -s);
          rb = rowops::rotate(b, a, c, s);
        }
        T *dst = is_q ? q + (size_t)r * dq + hh * h
                      : (T *)(is_v ? p.v_cache : p.k_cache) + layer_off + (size_t)(p.L + r) * dkv + hh * h;
        dst[i] = from_f<T>(ra);
        dst[i + half] = from_f<T>(rb);
      }
    }
    });
    if (!p.argmax && l + 1 == p.n_layers) return;
    if (!grid_barrier(p, target, false, gave_up, &flag)) return;
    // ---- attention, four warps per (row, head): keys by virtual position in groups of 32, online softmax over a warp's
    //      groups; the four warps' pieces are added in their order
    const int quad = warp / QUAD, qw = warp % QUAD;
    for (int u = blockIdx.x * (WARPS / QUAD) + quad; u < rows * p.H; u += gridDim.x * (WARPS / QUAD)) {
      const int r = u / p.H, a = u % p.H, kvh = a / (p.H / p.Hkv);
      float *myq = sq[warp];
      for (int i = lane; i < h; i += 32) myq[i] = to_f<T>(__ldcg(q + (size_t)r * dq + a * h + i));
      __syncwarp();
      const int lin_end = p.b.lin_end[r], seg_start = p.b.seg_start[r], n_vis = lin_end + p.b.seg_len[r];
      const T *kb = (const T *)p.k_cache + layer_off + kvh * h, *vb = (const T *)p.v_cache + layer_off + kvh * h;
      float m = -INFINITY, sum = 0.f;
      float o[4] = {0.f, 0.f, 0.f, 0.f};                 // dims lane, lane + 32, .. (h <= 128)
      const int nd = h >> 5;
      for (int p0 = 32 * qw; p0 < n_vis; p0 += 32 * QUAD) {
        const int pos = p0 + lane;
        const bool valid = pos < n_vis;
        const int slot = pos < lin_end ? pos : seg_start + (pos - lin_end);
        float sc = -INFINITY;
        if (valid) {
          const T *kr = kb + (size_t)slot * dkv;
          float acc = 0.f;
#pragma unroll 8
          for (int i = 0; i < h; i += Vec<T>::N) {
            Vec<T> kv;
            kv.v = __ldcg(reinterpret_cast<const decltype(kv.v) *>(kr + i));
#pragma unroll
            for (int e = 0; e < Vec<T>::N; ++e) acc = fmaf(myq[i + e], kv.get(e), acc);
          }
          sc = acc * p.scale;
        }
        const float m_new = fmaxf(m, warp_max(sc));
        const float at = m_new == -INFINITY ? 0.f : m_new;      // all this warp's scores so far overflowed: weights zero, not NaN
        const float corr = expf(m - at);
        const float pw = valid ? expf(sc - at) : 0.f;
        sum = sum * corr + warp_sum(pw);
#pragma unroll
        for (int dd = 0; dd < 4; ++dd) o[dd] *= corr;
        const int cnt = min(32, n_vis - p0);
#pragma unroll 16
        for (int t = 0; t < cnt; ++t) {
          const float pt = __shfl_sync(FULL, pw, t);
          const int st = __shfl_sync(FULL, slot, t);
          const T *vr = vb + (size_t)st * dkv;
#pragma unroll
          for (int dd = 0; dd < 4; ++dd)
            if (dd < nd) o[dd] = fmaf(pt, to_f<T>(__ldcg(vr + lane + 32 * dd)), o[dd]);
        }
        m = m_new;
      }
      __syncwarp();
#pragma unroll
      for (int dd = 0; dd < 4; ++dd)
        if (dd < nd) myq[lane + 32 * dd] = o[dd];
      if (lane == 0) sml[warp] = make_float2(m, sum);
      __syncwarp();
      asm volatile("barrier.sync %0, %1;" ::"r"(1 + quad), "n"(32 * QUAD) : "memory");
      // the four pieces together: a warp without keys has the weight zero (the first always has one)
      const int w0 = quad * QUAD;
      float mx = sml[w0].x, l_all = 0.f, wt[QUAD];
#pragma unroll
      for (int j = 1; j < QUAD; ++j) mx = fmaxf(mx, sml[w0 + j].x);
#pragma unroll
      for (int j = 0; j < QUAD; ++j) {
        wt[j] = expf(sml[w0 + j].x - mx);
        l_all += sml[w0 + j].y * wt[j];
      }
      const float inv = 1.0f / l_all;
      for (int dim = 32 * qw + lane; dim < h; dim += 32 * QUAD) {
        float v = 0.f;
#pragma unroll
        for (int j = 0; j < QUAD; ++j) v += sq[w0 + j][dim] * wt[j];
        att[(size_t)r * dq + a * h + dim] = from_f<T>(v * inv);
      }
      __syncwarp();
      asm volatile("barrier.sync %0, %1;" ::"r"(1 + quad), "n"(32 * QUAD) : "memory");
    }
    if (!grid_barrier(p, target, false, gave_up, &flag)) return;
    // ---- a column of a projection back into the residual stream
    auto project = [&](const T *src, const void *weight, int K) {
      by_rows(d, [&](auto rt) {
        constexpr int RT = decltype(rt)::value;
        const int tiles = (rows + RT - 1) / RT;
        for (int u = gw; u < d * tiles; u += nw) {
          const int n_col = u % d;
          r0 = u / d * RT;
          const int n = min(RT, rows - r0);
          const T *const ws[1] = {(const T *)weight + (size_t)n_col * K};
          float old = 0.f;
          if (lane < n)
            old = embedded ? to_f<T>(((const T *)p.embed)[(size_t)p.b.tok[r0 + lane] * d + n_col]) : __ldcg(p.x + (size_t)(r0 + lane) * d + n_col);
          float acc[1][RT];
          contract<T, 1, RT>(stored(src + (size_t)r0 * K, K), (const T *)nullptr, 0.f, ws, n, K, acc);
          if (lane < n) __stcg(p.x + (size_t)(r0 + lane) * d + n_col, old + of_row<RT>(acc[0], lane));
        }
      });
    };
    project(att, w.wo, dq);
    embedded = false;
    if (!grid_barrier(p, target, false, gave_up, &flag)) return;
    // ---- SiLU(gate) * up
    by_rows(p.F, [&](auto rt) {
      constexpr int RT = decltype(rt)::value;
      const int tiles = (rows + RT - 1) / RT;
      for (int u = gw; u < p.F * tiles; u += nw) {
        const int n_col = u % p.F;
        r0 = u / p.F * RT;
        const int n = min(RT, rows - r0);
        const T *const ws[2] = {(const T *)w.w_gate + (size_t)n_col * d, (const T *)w.w_up + (size_t)n_col * d};
        float acc[2][RT];
        contract<T, 2, RT>(residual, (const T *)w.ffn_norm, p.eps, ws, n, d, acc);
        if (lane < n) {
          const float g = of_row<RT>(acc[0], lane), up = of_row<RT>(acc[1], lane);
          act[(size_t)(r0 + lane) * p.F + n_col] = from_f<T>(g / (1.0f + expf(-g)) * up);
        }
      }
    });
    if (!grid_barrier(p, target, false, gave_up, &flag)) return;
    project(act, w.w_down, p.F);
    if (!grid_barrier(p, target, !p.argmax && l + 2 == p.n_layers, gave_up, &flag)) return;
  }
  // ---- LM head: four columns of a unit where all warps have one even so
  auto head = [&](auto cols, auto rt) {
    constexpr int CN = decltype(cols)::value, RT = decltype(rt)::value;
    const int tiles = (rows + RT - 1) / RT, groups = (p.V + CN - 1) / CN;
    for (int u = gw; u < groups * tiles; u += nw) {
      const int col = u % groups * CN;
      r0 = u / groups * RT;
      const int n = min(RT, rows - r0);
      const T *ws[CN];
#pragma unroll
      for (int c = 0; c < CN; ++c) ws[c] = (const T *)p.lm_head + (size_t)min(col + c, p.V - 1) * d;
      float acc[CN][RT];
      contract<T, CN, RT>(residual, (const T *)p.final_norm, p.eps, ws, n, d, acc);
      if (lane < n) {
#pragma unroll
        for (int c = 0; c < CN; ++c)
          if (col + c < p.V) __stcg(p.logits + (size_t)(r0 + lane) * p.V + col + c, of_row<RT>(acc[c], lane));
      }
    }
  };
  bool fours = false;
  if constexpr (WIDE) {
    fours = p.V >= 4 * nw;
    if (fours) by_rows(p.V / 4, [&](auto rt) { head(std::integral_constant<int, 4>{}, rt); });
  }
  if (!fours) by_rows(p.V, [&](auto rt) { head(std::integral_constant<int, 1>{}, rt); });
  if (!grid_barrier(p, target, true, gave_up, &flag)) return;
  // ---- greedy choice, a warp per row; the smallest index among equals
  for (int r = gw; r < rows; r += nw) {
    float best = -INFINITY;
    int idx = INT_MAX;
#pragma unroll 16
    for (int i = lane; i < p.V; i += 32) {
      const float v = __ldcg(p.logits + (size_t)r * p.V + i);
      if (v > best || (v == best && i < idx)) { best = v; idx = i; }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const float v2 = __shfl_xor_sync(FULL, best, o);
      const int i2 = __shfl_xor_sync(FULL, idx, o);
      if (v2 > best || (v2 == best && i2 < idx)) { best = v2; idx = i2; }
    }
    if (lane == 0) p.argmax[r] = idx == INT_MAX ? 0 : idx;
  }
}

}  // namespace

// Narrow models, as far as both sides were measured: at the bound (512 x 2048, vocabulary 32000, four layers) one launch
// takes 272 us for one row and 1.96 ms for 128 behind 64 keys, the single kernels 543 us and 3.40 ms; at 128 x 344 it is 39
// and 138 us against 87 and 547.  The choice hangs on the model alone: the two sum a row's squares in another order.
bool forward_small_supported(const ouro_model_desc &d) { return d.n_layers <= MAX_LAYERS && d.d_model <= 512 && d.d_ffn <= 2048; }

int launch_forward_small(ouro_ctx *c, int which, int rows, const int *rows_dev, int32_t *argmax, float *logits) {
  ModelRt &M = c->m[which];
  const ouro_model_desc &d = M.d;
  SmallParams p{};
  for (int l = 0; l < d.n_layers; ++l)
    p.layer[l] = {M.attn_norm[l], M.wq[l], M.wk[l], M.wv[l], M.wo[l], M.ffn_norm[l], M.w_gate[l], M.w_up[l], M.w_down[l]};
  p.embed = M.embed; p.final_norm = M.final_norm; p.lm_head = M.lm_head;
  p.k_cache = M.k_cache; p.v_cache = M.v_cache;
  p.cos_t = M.rope_cos; p.sin_t = M.rope_sin;
  p.b = M.blk;
  p.n_layers = d.n_layers; p.d = d.d_model; p.H = d.n_heads; p.Hkv = d.n_kv_heads; p.h = d.head_dim; p.F = d.d_ffn;
  p.V = d.vocab; p.max_seq = d.max_seq; p.L = M.L;
  p.eps = d.rms_eps;
  p.scale = 1.0f / sqrtf((float)d.head_dim);
  p.rows = rows; p.rows_dev = rows_dev;
  p.x = c->a.x; p.q = c->a.q; p.att = c->a.att; p.act = c->a.act;
  p.logits = logits; p.argmax = argmax;
  p.met = c->met_dev;
  p.wait_limit = c->wait_limit;
  p.status = &c->st->status;
  // as many CTAs as the widest step has units for: a barrier of fewer CTAs is no dearer
  const long tiles = (rows + 1) / 2;
  const long units = tiles * std::max<long>(std::max<long>(d.d_ffn, argmax ? d.vocab : 0), (d.n_heads + 2 * d.n_kv_heads) * (d.head_dim / 2));
  const int grid = (int)std::max<long>(1, std::min<long>(c->sms, (units + WARPS - 1) / WARPS));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = THREADS;
  cfg.stream = c->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const long nw = (long)grid * WARPS, pairs = (d.n_heads + 2 * d.n_kv_heads) * (d.head_dim / 2);
  const long widest = std::max(std::max<long>(d.d_model, pairs), std::max<long>(d.d_ffn, argmax ? d.vocab : 0));
  const bool wide = (argmax && d.vocab >= 4 * nw) || (rows > 2 && widest * ((rows + 7) / 8) > nw / 2);
  OURO_COUNT_LAUNCH();
  const auto kernel = d.dtype == OURO_BF16 ? (wide ? forward_small_kernel<__nv_bfloat16, true> : forward_small_kernel<__nv_bfloat16, false>)
                                           : (wide ? forward_small_kernel<float, true> : forward_small_kernel<float, false>);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, p);
  if (e != cudaSuccess) {
    c->err = std::string("one-launch forward: ") + cudaGetErrorString(e);
    return OURO_ECUDA;
  }
  return OURO_OK;
}
