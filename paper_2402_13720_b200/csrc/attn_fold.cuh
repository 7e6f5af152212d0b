// Folding the per-span pieces of the split attention into the block's attention output.
//
// Both tensor-core attention kernels cut a row's keys into spans and leave, per (row, head, span), the span's score maximum
// (log2 domain), its sum of exponentials and its unnormalised output.  A (row, head) pair is folded by one warp: first the
// largest span maximum, then one weighted sum over the spans in ascending order.  The arithmetic involves the pair's own
// spans only, so it does not matter which kernel, CTA or warp runs it; it runs in the kernel that consumes the attention
// output (the output projection), spread over all its CTAs.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "row_ops.cuh"

namespace fold {

// The spans, by absolute position.  Head dim 64 (mma.sync kernel): the first 1024 keys in spans of one chunk of 128, since a
// CTA walks its chunks one after the other (2 to 2.5 us each) and a short context would keep a few CTAs busy; the others in
// spans of four, so that a long context leaves few pieces to fold (1.1B draft, 389 keys: 3981 -> 3573 us, with a window
// over 521 keys 6971 -> 6347 us).  Head dim 128 (tcgen05 kernel): spans of four throughout - what a short span saves there
// (three passes of 1.75 us of one CTA) the set-up of the additional CTAs and the fold cost again (7B step 3526 us, with
// short spans 3549; prefill 12.4 ms and 13.3).
constexpr int CHUNK = 128, LONG_CHUNKS = 4, LONG_KEYS = LONG_CHUNKS * CHUNK;
constexpr int MAX_SPANS = 64;            // two per lane of the folding warp
constexpr int MAX_KEYS = 32 * LONG_KEYS;
__host__ __device__ constexpr int short_spans(int head_dim) { return head_dim == 64 ? 8 : 0; }
__host__ __device__ constexpr int span_count(int head_dim, int keys) {     // spans that hold the keys [0, keys)
  return keys <= short_spans(head_dim) * CHUNK ? (keys + CHUNK - 1) / CHUNK
                                               : short_spans(head_dim) + (keys - short_spans(head_dim) * CHUNK + LONG_KEYS - 1) / LONG_KEYS;
}
__host__ __device__ constexpr int span_chunks(int head_dim, int s) { return s < short_spans(head_dim) ? 1 : LONG_CHUNKS; }
__host__ __device__ constexpr int span_start(int head_dim, int s) {
  return s < short_spans(head_dim) ? s * CHUNK : short_spans(head_dim) * CHUNK + (s - short_spans(head_dim)) * LONG_KEYS;
}
static_assert(span_count(64, MAX_KEYS) <= MAX_SPANS, "spans of the longest context");

struct Params {
  const float *part;               // [rows][H][cap][PIECE]; NULL: nothing to fold
  __nv_bfloat16 *out;              // [rows][H * HD]
  const int32_t *lin_end, *seg_len;   // per block row: keys seen = lin_end + seg_len
  const int *rows_dev;             // NULL, or the block's true row count in device memory
  int rows, H, cap, head_dim;
};

// A piece: the span's score maximum and sum in front, two words of padding, then the output, so that a lane fetches its
// dims of a piece with one 16-byte (head dim 64: 8-byte) load.
template <int HD> constexpr int PIECE = HD + 4;
template <int HD> struct Dims { typedef float4 V; };
template <> struct Dims<64> { typedef float2 V; };
__device__ __forceinline__ void add_scaled(float4 &a, const float4 &o, float w) {
  a = make_float4(__fmaf_rn(o.x, w, a.x), __fmaf_rn(o.y, w, a.y), __fmaf_rn(o.z, w, a.z), __fmaf_rn(o.w, w, a.w));
}
__device__ __forceinline__ void add_scaled(float2 &a, const float2 &o, float w) { a = make_float2(__fmaf_rn(o.x, w, a.x), __fmaf_rn(o.y, w, a.y)); }
__device__ __forceinline__ void store_bf16(__nv_bfloat16 *dst, const float4 &a, float s) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(a.x * s, a.y * s), hi = __floats2bfloat162_rn(a.z * s, a.w * s);
  *reinterpret_cast<uint2 *>(dst) = make_uint2(*(uint32_t *)&lo, *(uint32_t *)&hi);
}
__device__ __forceinline__ void store_bf16(__nv_bfloat16 *dst, const float2 &a, float s) {
  *reinterpret_cast<__nv_bfloat162 *>(dst) = __floats2bfloat162_rn(a.x * s, a.y * s);
}
// One row's output as packets (row_ops.cuh) instead of `out`: this lane's dims, from dim `at` on (a pair of lanes fills a packet
// where a lane has two).
struct Packets { uint4 *dst; uint32_t mark; };
__device__ __forceinline__ void put(const Packets &k, size_t at, const float4 &a, float s) {
  rowops::put_packet(k.dst + at / 4, rowops::pack(a.x * s, a.y * s), rowops::pack(a.z * s, a.w * s), 0u, k.mark);
}
__device__ __forceinline__ void put(const Packets &k, size_t at, const float2 &a, float s) {
  const uint32_t lo = rowops::pack(a.x * s, a.y * s), hi = __shfl_down_sync(0xffffffffu, lo, 1);
  if (at % 4 == 0) rowops::put_packet(k.dst + at / 4, lo, hi, 0u, k.mark);
}

// Pairs first, first + step, .. (pair = row * H + head).  Lane c fetches the maxima and sums of spans c and c + 32 while
// every lane fetches its dims of up to UNR spans: one round trip to L2 up to 16 spans, then one more per 16.
template <int HD, bool PACKETS>
__device__ __forceinline__ void pairs(const Params &p, int rows, int first, int step, int lane, int keys, const Packets &k) {
  typedef typename Dims<HD>::V V;
  constexpr int PW = PIECE<HD>, DPL = HD / 32, UNR = 16;
  const int n_pairs = rows * p.H;
#pragma unroll 1
  for (int q = first; q < n_pairs; q += step) {
    if (q != first) keys = p.lin_end[q / p.H] + p.seg_len[q / p.H];
    const int ns = span_count(HD, keys);
    const float *src = p.part + (size_t)q * p.cap * PW;
    float2 ml = make_float2(-INFINITY, 0.f), ml2 = ml;
    if (lane < ns) ml = __ldcg(reinterpret_cast<const float2 *>(src + lane * PW));
    if (lane + 32 < ns) ml2 = __ldcg(reinterpret_cast<const float2 *>(src + (lane + 32) * PW));
    float l = 0.f;
    V acc{};
#pragma unroll 1
    for (int c0 = 0; c0 < ns; c0 += UNR) {
      V o[UNR];
#pragma unroll
      for (int cc = 0; cc < UNR; ++cc) {
        o[cc] = V{};
        if (c0 + cc < ns) o[cc] = __ldcg(reinterpret_cast<const V *>(src + (size_t)(c0 + cc) * PW + 4 + DPL * lane));
      }
      if (c0 == 0) {
        float mx = fmaxf(ml.x, ml2.x);
#pragma unroll
        for (int s = 16; s; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
        ml.x = (ml.x == -INFINITY) ? 0.f : exp2f(ml.x - mx);         // the spans' weights; mx is finite: the first span holds a
        ml2.x = (ml2.x == -INFINITY) ? 0.f : exp2f(ml2.x - mx);      // visible key
      } else if (c0 == 32) {
        ml = ml2;
      }
#pragma unroll
      for (int cc = 0; cc < UNR; ++cc) {
        if (c0 + cc >= ns) break;                                    // uniform in the warp
        const float w = __shfl_sync(0xffffffffu, ml.x, c0 + cc);     // (lane: modulo 32)
        l = __fmaf_rn(__shfl_sync(0xffffffffu, ml.y, c0 + cc), w, l);
        add_scaled(acc, o[cc], w);
      }
    }
    if constexpr (PACKETS) put(k, (size_t)q * HD + DPL * lane, acc, 1.0f / l);
    else store_bf16(p.out + (size_t)q * HD + DPL * lane, acc, 1.0f / l);
  }
}

// The dependency wait is in here: what a warp needs to know of the block (its rows, the keys its first pair sees) was written
// before the forward pass began and is fetched ahead of it (1.1B draft 3235 -> 3212 us).
template <bool PACKETS = false>
__device__ __forceinline__ void run(const Params &p, int first, int step, int lane, const Packets &k = Packets()) {
  const int r = min(first / p.H, p.rows - 1);
  const int rows = p.rows_dev ? min(p.rows, __ldg(p.rows_dev)) : p.rows, keys = p.lin_end[r] + p.seg_len[r];
  pdl_wait();
  if (p.head_dim == 128) pairs<128, PACKETS>(p, rows, first, step, lane, keys, k);
  else pairs<64, PACKETS>(p, rows, first, step, lane, keys, k);
}

}  // namespace fold
