// Attention over the KV cache for the few query rows of a decoding step without candidates (bf16, head dim 128).
//
// attn_tm_kernel walks a span of keys chunk by chunk: scores into TMEM, softmax, P to shared memory, P V into TMEM, each
// behind the one before, and a tile of 128 query rows of which a single token fills one.  That chain, 1.75 us a chunk behind
// 2 us of set-up, is what plain decoding spends on attention whatever the keys are.  (One row, us a forward, attn_tm_kernel and this
// one: two layers of 512 behind 150 keys 62.7 and 59.2, behind 400 69.0 and 62.6; three layers of the 7B shape behind 100 keys 289 and
// 283; where it is used and where it would be slower: attention_few_pays in gemm_tc.cu.)  Here up to 16 query rows of a kv head (rows x query heads) are one mma.sync tile, and the four chunks of a
// span are worked on at the same time, each by four warps:
//     S = Q K^T     a warp has 32 of the chunk's keys, their K straight in registers (one 8-byte piece per step and key),
//     maxima        of all four chunks through shared memory: every chunk then knows the running maximum it would have met,
//     P = exp2(S - running maximum), O_c = P V with V in shared memory (a warp has 32 of the dims),
//     O = O a + O_c in chunk order, at the end.
// K and V that were complete before the forward began are fetched ahead of the dependency wait.  The arithmetic of a row is
// attn_tm_kernel's to the last bit: the same chunks and spans, the same maxima and partial sums in the same order, steps of 16
// (which give the same sum in mma.sync and tcgen05.mma, in whatever order the 16 are laid out), pieces for the same fold.
#include "ouro_internal.h"
#include "row_ops.cuh"
#include "attn_fold.cuh"

// Optional timeline (compile with -DOURO_TRACE): the points of attn_tm_kernel's, see trace.py.
#ifdef OURO_TRACE
__device__ unsigned long long g_attn_few_trace[512][8];
__device__ __forceinline__ unsigned long long attn_few_trace_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)::"memory");
  return t;
}
#define TRACE(slot) do { const int cta_ = blockIdx.y * gridDim.x + blockIdx.x; if (threadIdx.x == 0 && cta_ < 512) g_attn_few_trace[cta_][slot] = attn_few_trace_now(); } while (0)
extern "C" int ouro_trace_read_attn_few(unsigned long long *out_host) {
  return (int)cudaMemcpyFromSymbol(out_host, g_attn_few_trace, sizeof(g_attn_few_trace));
}
#else
#define TRACE(slot) do { } while (0)
#endif

namespace {

constexpr int HD = 128, CH = fold::CHUNK, CHUNKS = fold::LONG_CHUNKS;
constexpr int TEAM = 4;                           // warps of a chunk
constexpr int THREADS = 32 * TEAM * CHUNKS;
constexpr int QR = 16;                            // query rows of the tile
constexpr int ROWB = HD * 2;
constexpr int P_HALF = 68;                        // floats of half a row of P in 32 bits: the threads that add them up hit different banks
constexpr int O_PITCH = HD + 4;
constexpr int OFF_P = CHUNKS * CH * ROWB;                                   // V in front: [chunk][key][dim]
constexpr int OFF_F = OFF_P + CHUNKS * QR * CH * 2;                         // P in 32 bits, then O_c: [chunk][row][..]
constexpr int F_FLOATS = QR * (2 * P_HALF > O_PITCH ? 2 * P_HALF : O_PITCH);
constexpr int OFF_MAX = OFF_F + CHUNKS * F_FLOATS * 4;                      // [chunk][row][warp of the team]
constexpr int OFF_SUM = OFF_MAX + CHUNKS * QR * TEAM * 4;                   // [chunk][row][half]
constexpr int BYTES = OFF_SUM + CHUNKS * QR * 2 * 4;

struct FewParams {
  const __nv_bfloat16 *q;          // [rows][H * HD] rotated queries
  const __nv_bfloat16 *k, *v;      // this layer's cache: [max_seq][Hkv * HD]
  const int32_t *lin_end, *seg_len;
  int rows, H, Hkv, cap;
  int ready;                       // cache rows that were complete before the forward began
  float scale_log2;
  float *part;
  __nv_bfloat16 *out;
  int direct;                      // every row's keys lie in span 0
  const int *rows_dev;
  const uint8_t *pf_ptr[3];        // brought into L2 for the kernel that follows (see L2Prefetch): each CTA asks for an equal share
  uint32_t pf_bytes[3];
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t *r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t *r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16(float *d, const uint32_t *a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// 2^x for x <= 0, as in attn_tm_kernel.
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void team_barrier(int team) { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(32 * TEAM) : "memory"); }

__global__ void __launch_bounds__(THREADS, 1) attn_few_kernel(const FewParams p) {
  extern __shared__ __align__(128) uint8_t smem[];
  const uint32_t sm_u = smem_u32(smem);
  float *s_max = (float *)(smem + OFF_MAX), *s_sum = (float *)(smem + OFF_SUM);
  pdl_trigger();
  TRACE(0);
  const int tid = threadIdx.x, lane = tid & 31, team = tid / (32 * TEAM), tw = (tid >> 5) & (TEAM - 1);
  const int sc = blockIdx.x, kvh = blockIdx.y, dkv = p.Hkv * HD, g = p.H / p.Hkv;
  if (tid == 0) {
    const uint32_t u = blockIdx.y * gridDim.x + blockIdx.x, U = gridDim.x * gridDim.y;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      if (p.pf_bytes[r] == 0) continue;
      const uint32_t share = ((p.pf_bytes[r] + U - 1) / U + 15u) & ~15u, off = u * share;
      if (off < p.pf_bytes[r])
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.pf_ptr[r] + off), "r"(min(share, p.pf_bytes[r] - off)) : "memory");
    }
  }
  // (the block's description and the cache below `ready` were complete before the forward pass began)
  const int rows = p.rows_dev ? min(p.rows, __ldg(p.rows_dev)) : p.rows, M = g * rows;
  int keys = 0;                                     // any row sees
  for (int r = 0; r < rows; ++r) keys = max(keys, p.lin_end[r] + p.seg_len[r]);
  const int span0 = fold::span_start(HD, sc), c0 = span0 + team * CH;
  if (span0 >= keys) return;                        // (the whole CTA)
  const bool on = c0 < keys;                        // somebody sees keys of this team's chunk
  // rows of this thread in the tile: lane / 4 and + 8
  int nv[2], rr[2], hh[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int m = (lane >> 2) + 8 * i;
    rr[i] = m < M ? m % rows : 0;
    hh[i] = m < M ? kvh * g + m / rows : 0;
    nv[i] = m < M ? p.lin_end[rr[i]] + p.seg_len[rr[i]] : 0;
  }
  // ---- K of this warp's keys into registers, V of the chunk into shared memory: first what may be read ahead of the wait
  const int t4 = lane & 3;
  uint2 kf[4][HD / 16];                             // [8 keys][step]: dims 16 s + 4 t .. + 3 of key lane / 4
#pragma unroll
  for (int n = 0; n < 4; ++n)
#pragma unroll
    for (int s = 0; s < HD / 16; ++s) kf[n][s] = make_uint2(0u, 0u);
  auto fetch = [&](int lo, int hi) {                // keys [lo, hi)
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const int pos = c0 + tw * 32 + 8 * n + (lane >> 2);
      if (pos >= lo && pos < hi) {
        const uint2 *src = reinterpret_cast<const uint2 *>(p.k + (size_t)pos * dkv + kvh * HD) + t4;
#pragma unroll
        for (int s = 0; s < HD / 16; ++s) kf[n][s] = __ldcg(src + 4 * s);
      }
    }
    for (int i = tw * 32 + lane; i < CH * 16; i += 32 * TEAM) {
      const int row = i >> 4, ch = i & 15, pos = c0 + row;
      if (pos >= lo && pos < hi)
        cp_async16(sm_u + (team * CH + row) * ROWB + ((ch ^ (row & 7)) << 4), p.v + (size_t)pos * dkv + kvh * HD + ch * 8);
    }
  };
  const int early = min(keys, p.ready);
  if (on) {
    fetch(c0, early);
    for (int i = tw * 32 + lane; i < CH * 16; i += 32 * TEAM)       // keys nobody sees
      if (c0 + (i >> 4) >= keys) *reinterpret_cast<uint4 *>(smem + (team * CH + (i >> 4)) * ROWB + ((i & 15) << 4)) = make_uint4(0, 0, 0, 0);
  }
  TRACE(1);
  pdl_wait();
  TRACE(2);
  float s[4][4];
#pragma unroll
  for (int n = 0; n < 4; ++n) s[n][0] = s[n][1] = s[n][2] = s[n][3] = 0.f;
  if (on) {
    uint2 qf[2][HD / 16];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int st = 0; st < HD / 16; ++st) {
        qf[i][st] = make_uint2(0u, 0u);
        if (nv[i] > 0) qf[i][st] = __ldcg(reinterpret_cast<const uint2 *>(p.q + ((size_t)rr[i] * p.H + hh[i]) * HD) + 4 * st + t4);
      }
    if (early < keys && c0 + CH > early) fetch(early, keys);
    // ---- S = Q K^T
#pragma unroll
    for (int st = 0; st < HD / 16; ++st) {
      const uint32_t a[4] = {qf[0][st].x, qf[1][st].x, qf[0][st].y, qf[1][st].y};
#pragma unroll
      for (int n = 0; n < 4; ++n) mma16(s[n], a, kf[n][st].x, kf[n][st].y);
    }
    TRACE(3);
    // ---- this warp's row maxima
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float mx = -INFINITY;
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (c0 + tw * 32 + 8 * n + 2 * t4 + e < nv[i]) mx = fmaxf(mx, s[n][2 * i + e]);
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      if (t4 == 0) s_max[(team * QR + (lane >> 2) + 8 * i) * TEAM + tw] = mx;
    }
  }
  __syncthreads();
  // the running maximum (log2 domain) of a row that sees n keys, behind chunk c of the span
  auto running = [&](int row, int n, int c) {
    float m = -INFINITY;
    for (int i = 0; i <= c; ++i)
      if (span0 + i * CH < n) {
        const float4 v = *reinterpret_cast<const float4 *>(s_max + (i * QR + row) * TEAM);
        m = fmaxf(m, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)) * p.scale_log2);
      }
    return m;
  };
  float *fl = (float *)(smem + OFF_F) + team * F_FLOATS;
  if (on) {
    // ---- P, as bf16 for the contraction and in 32 bits for the sums
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int row = (lane >> 2) + 8 * i;
      const float mn = running(row, nv[i], team);
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const int kc = tw * 32 + 8 * n + 2 * t4;                     // key within the chunk
        const float p0 = c0 + kc < nv[i] ? ex2(__fmaf_rn(s[n][2 * i], p.scale_log2, -mn)) : 0.f;
        const float p1 = c0 + kc + 1 < nv[i] ? ex2(__fmaf_rn(s[n][2 * i + 1], p.scale_log2, -mn)) : 0.f;
        *reinterpret_cast<float2 *>(fl + (2 * row + (kc >> 6)) * P_HALF + (kc & 63)) = make_float2(p0, p1);
        *reinterpret_cast<uint32_t *>(smem + OFF_P + (team * QR + row) * (CH * 2) + (((kc >> 3) ^ (row & 7)) << 4) + 2 * (kc & 7)) = rowops::pack(p0, p1);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    team_barrier(team);
    // ---- row sums: of each half of the chunk four interleaved sums over ascending keys, then those
    {
      const int i = tw * 32 + lane;
      const float *src = fl + (i >> 2) * P_HALF + t4;
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 16; ++j) sum += src[4 * j];
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      if (t4 == 0) s_sum[team * QR * 2 + (i >> 2)] = sum;
    }
    // ---- O_c = P V for this warp's 32 dims
    float o[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
    const int mi = lane >> 3;
#pragma unroll
    for (int kk = 0; kk < CH / 16; ++kk) {
      uint32_t a[4], b[2][4];
      const int row = (lane & 7) + ((mi & 1) << 3);
      ldsm_x4(sm_u + OFF_P + (team * QR + row) * (CH * 2) + (((2 * kk + (mi >> 1)) ^ (row & 7)) << 4), a);
      const int key = 16 * kk + row;
#pragma unroll
      for (int h = 0; h < 2; ++h)
        ldsm_x4_t(sm_u + (team * CH + key) * ROWB + (((4 * tw + 2 * h + (mi >> 1)) ^ (key & 7)) << 4), b[h]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        mma16(o[2 * h], a, b[h][0], b[h][1]);
        mma16(o[2 * h + 1], a, b[h][2], b[h][3]);
      }
    }
    team_barrier(team);                             // P in 32 bits has been added up: O_c goes there
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int i = 0; i < 2; ++i)
        *reinterpret_cast<float2 *>(fl + ((lane >> 2) + 8 * i) * O_PITCH + tw * 32 + 8 * n + 2 * t4) = make_float2(o[n][2 * i], o[n][2 * i + 1]);
  }
  __syncthreads();
  TRACE(4);
  // ---- the span's piece: a warp per row, four dims a lane
  {
    const int row = tid >> 5, d = 4 * lane;
    if (row >= M) return;
    const int r = row % rows, hq = kvh * g + row / rows, n = p.lin_end[r] + p.seg_len[r];
    if (n <= span0) return;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    float m = -INFINITY, l0 = 0.f, l1 = 0.f;
    for (int c = 0; c < CHUNKS && span0 + c * CH < n; ++c) {
      const float mn = running(row, n, c), a = m == -INFINITY ? 0.f : ex2(m - mn);
      const float4 v = *reinterpret_cast<const float4 *>((float *)(smem + OFF_F) + c * F_FLOATS + row * O_PITCH + d);
      const float2 sm = *reinterpret_cast<const float2 *>(s_sum + (c * QR + row) * 2);
      o = make_float4(__fmaf_rn(o.x, a, v.x), __fmaf_rn(o.y, a, v.y), __fmaf_rn(o.z, a, v.z), __fmaf_rn(o.w, a, v.w));
      l0 = __fmaf_rn(l0, a, sm.x);
      l1 = __fmaf_rn(l1, a, sm.y);
      m = mn;
    }
    const float l = l0 + l1;
    const size_t at = (size_t)r * p.H + hq;
    if (p.direct) {
      const float inv = 1.0f / l;                   // what the fold would compute from this single span
      *reinterpret_cast<uint2 *>(p.out + at * HD + d) = make_uint2(rowops::pack(o.x * inv, o.y * inv), rowops::pack(o.z * inv, o.w * inv));
    } else {
      float *dst = p.part + (at * p.cap + sc) * fold::PIECE<HD>;
      if (lane == 0) *reinterpret_cast<float2 *>(dst) = make_float2(m, l);
      *reinterpret_cast<float4 *>(dst + 4 + d) = o;
    }
  }
  TRACE(5);
}

}  // namespace

int attention_few_setup() {
  return cudaFuncSetAttribute(attn_few_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BYTES) == cudaSuccess ? OURO_OK : OURO_ECUDA;
}

// Blocks of one group (rows in order) whose query rows of a kv head fill one tile.
bool attention_few_supported(const ouro_model_desc &d, int rows) { return attention_tm_supported(d) && d.n_heads / d.n_kv_heads * rows <= QR; }

bool launch_attention_few(const ouro_model_desc &d, const void *q, const void *k_cache, const void *v_cache, const BlockDev &b, int rows, int ready,
                          int n_vis_max, int layer, float *part, void *out, const int *rows_dev, const L2Prefetch &pf, cudaStream_t s) {
  OURO_COUNT_LAUNCH();
  FewParams p;
  const size_t off = (size_t)layer * d.max_seq * d.n_kv_heads * d.head_dim;
  p.q = (const __nv_bfloat16 *)q;
  p.k = (const __nv_bfloat16 *)k_cache + off;
  p.v = (const __nv_bfloat16 *)v_cache + off;
  p.lin_end = b.lin_end; p.seg_len = b.seg_len;
  p.rows = rows; p.H = d.n_heads; p.Hkv = d.n_kv_heads; p.ready = ready;
  p.cap = fold::span_count(HD, d.max_seq);
  p.scale_log2 = 1.4426950408889634f / sqrtf((float)d.head_dim);
  p.part = part;
  p.out = (__nv_bfloat16 *)out;
  const int n_spans = fold::span_count(HD, n_vis_max);
  p.direct = n_spans <= 1;
  p.rows_dev = rows_dev;
  for (int r = 0; r < 3; ++r) {
    const bool ok = pf.ptr[r] && pf.bytes[r] > 0 && pf.bytes[r] < (1ull << 31) && pf.bytes[r] % 16 == 0 && ((uintptr_t)pf.ptr[r] & 15) == 0;
    p.pf_ptr[r] = ok ? (const uint8_t *)pf.ptr[r] : nullptr;
    p.pf_bytes[r] = ok ? (uint32_t)pf.bytes[r] : 0u;
  }
  launch_pdl(attn_few_kernel, dim3(n_spans, d.n_kv_heads), THREADS, BYTES, s, p);
  return !p.direct;
}
