// Arithmetic on rows that several kernels share.  A token's values must not depend on the kernel that computes them, so what
// the compiler could contract in more than one way is spelled out.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace rowops {

// x * sigmoid(x) with the fast exponential and reciprocal (the result is rounded to bf16 right after)
__device__ __forceinline__ float silu(float x) { return __fdividef(x, 1.0f + __expf(-x)); }
// One dimension of a rotated pair: own * cos + other * (+-sin).
__device__ __forceinline__ float rotate(float own, float other, float c, float s) { return __fmaf_rn(own, c, __fmul_rn(other, s)); }
// Sum of squares of four columns; those of a tile of 128 are added over the 32 groups of four in halves (16, 8, 4, 2, 1 apart).
__device__ __forceinline__ float squares(float a, float b, float c, float d) {
  return __fmaf_rn(d, d, __fmaf_rn(c, c, __fmaf_rn(b, b, __fmul_rn(a, a))));
}
__device__ __forceinline__ float inv_rms(float sum, float inv_d, float eps) { return 1.0f / sqrtf(__fmaf_rn(sum, inv_d, eps)); }
__device__ __forceinline__ uint32_t pack(float lo, float hi) {
  const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&t);
}
__device__ __forceinline__ float2 unpack(uint32_t v) {
  const __nv_bfloat162 t = *reinterpret_cast<const __nv_bfloat162 *>(&v);
  return make_float2(__low2float(t), __high2float(t));
}

// Four bf16 values on their way from the CTA that computed them to all that need them, in one 128-bit word: a poll that finds
// the mark has the values as well, so that a hand-over costs one store and one load (no fence, no counter, no second load).
// A mark is used once until the host clears all packets and begins anew, before the 32 bits run out: nothing is reset between launches,
// and what a launch that gave up left behind is not taken for anything.
struct Packet { uint32_t lo, hi, extra, mark; };
__device__ __forceinline__ void put_packet(uint4 *dst, uint32_t lo, uint32_t hi, uint32_t extra, uint32_t mark) {
  asm volatile(
      "{\n\t.reg .b128 v;\n\t.reg .b64 a, b;\n\t"
      "mov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\tmov.b128 v, {a, b};\n\t"
      "st.relaxed.gpu.global.b128 [%0], v;\n\t}" ::"l"(dst), "r"(lo), "r"(hi), "r"(extra), "r"(mark) : "memory");
}
__device__ __forceinline__ Packet get_packet(const uint4 *src) {
  Packet p;
  asm volatile(
      "{\n\t.reg .b128 v;\n\t.reg .b64 a, b;\n\t"
      "ld.relaxed.gpu.global.b128 v, [%4];\n\t"
      "mov.b128 {a, b}, v;\n\tmov.b64 {%0, %1}, a;\n\tmov.b64 {%2, %3}, b;\n\t}"
      : "=r"(p.lo), "=r"(p.hi), "=r"(p.extra), "=r"(p.mark) : "l"(src) : "memory");
  return p;
}

// Embedding rows of a block's tokens into the residual stream, plus what the first norm's consumer needs: bf16(gain * x) and
// the sums of squares per 128-column tile.
struct Embed {
  const __nv_bfloat16 *table;   // [vocab][d]; NULL: nothing to gather
  const int32_t *tok;           // [rows]
  const __nv_bfloat16 *gain;    // first norm's gain [d]
  float *x;                     // residual stream [rows][d]
  __nv_bfloat16 *xb;            // bf16(gain * x) [rows][d]
  float *ss;                    // [d / 128][ss_pitch] sums of squares per 128-column tile
  const int *rows_dev;
  int rows, d, ss_pitch;
};
// One warp per (row, tile): four columns per lane.  Items first, first + step, ..
__device__ __forceinline__ void embed(const Embed &e, int first, int step, int lane) {
  const int rows = e.rows_dev ? min(e.rows, __ldg(e.rows_dev)) : e.rows, tiles = (e.d + 127) / 128;
  for (int it = first; it < rows * tiles; it += step) {
    const int r = it / tiles, col = (it - r * tiles) * 128 + 4 * lane;
    float sq = 0.f;
    if (col < e.d) {                                            // d is a multiple of 64: four columns are in or out together
      const uint2 raw = __ldg(reinterpret_cast<const uint2 *>(e.table + (size_t)__ldg(e.tok + r) * e.d + col));
      const uint2 graw = __ldg(reinterpret_cast<const uint2 *>(e.gain + col));
      const float2 a = unpack(raw.x), b = unpack(raw.y), ga = unpack(graw.x), gb = unpack(graw.y);
      *reinterpret_cast<float4 *>(e.x + (size_t)r * e.d + col) = make_float4(a.x, a.y, b.x, b.y);
      *reinterpret_cast<uint2 *>(e.xb + (size_t)r * e.d + col) = make_uint2(pack(ga.x * a.x, ga.y * a.y), pack(gb.x * b.x, gb.y * b.y));
      // (bf16 values: each square is exact in 32 bits, and this is their sum two by two, however it is contracted)
      sq = __fadd_rn(__fmaf_rn(a.x, a.x, __fmul_rn(a.y, a.y)), __fmaf_rn(b.x, b.x, __fmul_rn(b.y, b.y)));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) e.ss[(size_t)(it - r * tiles) * e.ss_pitch + r] = sq;
  }
}

// The same for one row, as packets: its values and each four columns' squares, instead of xb and ss.
__device__ __forceinline__ void embed_packets(const Embed &e, int first, int step, int lane, uint4 *packets, uint32_t mark) {
  for (int it = first; it < (e.d + 127) / 128; it += step) {
    const int col = it * 128 + 4 * lane;
    if (col >= e.d) continue;
    const uint2 raw = __ldg(reinterpret_cast<const uint2 *>(e.table + (size_t)__ldg(e.tok) * e.d + col));
    const uint2 graw = __ldg(reinterpret_cast<const uint2 *>(e.gain + col));
    const float2 a = unpack(raw.x), b = unpack(raw.y), ga = unpack(graw.x), gb = unpack(graw.y);
    *reinterpret_cast<float4 *>(e.x + col) = make_float4(a.x, a.y, b.x, b.y);
    const float sq = __fadd_rn(__fmaf_rn(a.x, a.x, __fmul_rn(a.y, a.y)), __fmaf_rn(b.x, b.x, __fmul_rn(b.y, b.y)));
    put_packet(packets + col / 4, pack(ga.x * a.x, ga.y * a.y), pack(gb.x * b.x, gb.y * b.y), __float_as_uint(sq), mark);
  }
}

}  // namespace rowops
