// The weight-streaming schedule of the tensor-core GEMM: which (tile, k-block) pieces a CTA works on, in which
// order.  It depends on the problem shape and the grid only, never on the number of tokens, which is what makes a
// token's result independent of the block it is verified in.
#pragma once

#include <cuda.h>

namespace ws {

constexpr int TILE_N = 128;       // weight rows per tile (MMA M)
constexpr int BLOCK_K = 64;       // bf16 elements per k-block: one 128-byte swizzle row

struct Span {  // one piece of a CTA's work: k-blocks [kb0, kb1) of `tile`
  int tile, kb0, kb1, slot;
  bool whole;                     // all of the tile's k-blocks: no partial sum
};

// Work of one CTA.  The last R = tiles mod grid tiles are cut stream-K fashion into equal contiguous spans of
// the (tile, k-block) space and come first, so that their partial sums are added up while the whole tiles
// (tile c, c + grid, ...) that follow are still streaming.  Where only the first `sharers` CTAs share the cut tiles, the
// whole tiles are dealt out from the first CTA behind them, round by round; `sit_out` leaves the sharers out of the first
// round.  Depends on (tiles, kb, grid, splitters) only.
// The host works the cut out (GemmParams::t0, ::per): a walker is built by four warps of every CTA for every GEMM, and
// each integer division by a run-time number there is 0.1 us in front of the first load.
struct SpanWalker {
  int kb, per, t0, it, end, whole, step, grid, cta;
  __device__ SpanWalker(int tiles, int kb_, int t0_, int per_, int sharers, bool sit_out, int grid_, int cta_) {
    kb = kb_;
    grid = grid_;
    cta = cta_;
    t0 = t0_;                                                // tiles [0, t0) are handled whole
    per = per_;                                              // k-blocks per CTA of the others' (0: there are none)
    const int total = (tiles - t0) * kb;
    it = min(total, cta * per);
    end = min(total, it + per);
    const int first = sit_out ? grid - sharers : grid;       // whole tiles of the first round
    whole = cta >= sharers ? cta - sharers : first + cta + (sit_out ? grid : 0) - sharers;
    step = cta >= sharers ? first : grid;
  }
  __device__ int owner_slot(int tile, int owner) const { return ((tile - t0) * kb <= owner * per) ? 0 : 1; }
  __device__ bool next(Span &s) {
    if (it < end) {
      int rel = it / kb;
      s.tile = t0 + rel;
      s.kb0 = it - rel * kb;
      s.kb1 = min(kb, s.kb0 + (end - it));
      s.whole = s.kb0 == 0 && s.kb1 == kb;
      s.slot = owner_slot(s.tile, cta);                      // first or last piece of this CTA
      it += s.kb1 - s.kb0;
      return true;
    }
    if (whole < t0) {
      s.tile = whole;
      s.kb0 = 0;
      s.kb1 = kb;
      s.whole = true;
      s.slot = 0;
      whole += step;
      step = grid;
      return true;
    }
    return false;
  }
};

// The cut of `tiles` tiles of kb k-blocks for a launch of `grid` CTAs.  `splitters` CTAs share the remainder: all of them
// where scratch memory holds two partial tiles per CTA, fewer (or none: the remainder is then handled whole as well)
// where it does not.
struct Cut { int t0, per; };
inline Cut cut(int tiles, int kb, int grid, int splitters) {
  Cut c{tiles, 0};
  if (splitters > 0 && tiles % grid != 0) {
    c.t0 = tiles / grid * grid;
    c.per = ((tiles - c.t0) * kb + splitters - 1) / splitters;
  }
  return c;
}

}  // namespace ws
