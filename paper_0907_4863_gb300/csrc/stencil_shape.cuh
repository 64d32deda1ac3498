// Launch shapes of the level-0 stencil passes (internal; host arithmetic only).
#pragma once

#include <algorithm>

namespace saamg {

// Launch shape of the level-0 stencil passes of one precision (every row's arithmetic is the
// same under every shape, so the results are too): K chunks of 32 rows per warp step (1, 2,
// 4), packed (1: 32 regular-run rows per warp from the row list, then the table rows 32 at a
// time; 0: the line chunks), threads per block (128, 256) and blocks per SM (8, 16, 32).  fit: the
// default, which a small operator launches with fewer chunks a step and smaller blocks; a shape
// that a caller sets, or the autotuner times, runs as it stands.
struct StencilCfg {
  int k, packed, block, per_sm;
  bool fit = false;

  bool same_shape(const StencilCfg& o) const {
    return k == o.k && packed == o.packed && block == o.block && per_sm == o.per_sm;
  }
};

// Chunks per warp step of the shape on a pass of `units` chunks.  The default takes several only
// where a resident warp (64 per SM) has eight or more: fewer, longer steps leave SMs idle below that
// (32^3 solve 986 us with one chunk per step, 1063 with two).
inline int stencil_chunks(const StencilCfg& c, long long units, int sms) {
  return c.fit && units < 8LL * 64 * sms ? 1 : c.k;
}

struct StencilLaunch {
  int k, block, blocks;
};

// What a pass of `units` chunks launches.  The default spreads a small level over the SMs in blocks
// of down to 64 threads (an SM takes FP64 instructions of one warp per quarter at a time).
inline StencilLaunch stencil_launch(const StencilCfg& c, long long units, int sms) {
  StencilLaunch l;
  l.k = stencil_chunks(c, units, sms);
  l.block = c.block;
  while (c.fit && l.block > 64 && units * 32 < (long long)sms * l.block) l.block >>= 1;
  const long long step = (long long)(l.block / 32) * l.k;
  l.blocks = (int)std::max<long long>(
      1, std::min<long long>((units + step - 1) / step, (long long)sms * c.per_sm));
  return l;
}

}  // namespace saamg
