// Rules of the verify attention that are plain arithmetic: the kernel applies
// them, and they compile for the host by themselves.
#pragma once

#ifdef __CUDACC__
#define LIBRASPEC_HD __host__ __device__ __forceinline__
#else
#define LIBRASPEC_HD inline
#endif

namespace libraspec {

// First tile of part k of a row group of `tiles` tiles that p CTAs share
// (k = p: the end): floor(tiles k / p), whose product would pass 2^31 from 15
// million tiles on (a billion keys, which pages may repeat).
LIBRASPEC_HD int group_part(int tiles, int k, int p) { return tiles / p * k + tiles % p * k / p; }

// Buffers of split-group partials: layer l writes buffer l % 3, so layer l's
// merge may run until layer l + 2 starts, a layer after the one it overlaps.
constexpr int kAttnPartBufs = 3;

// Whether a CTA may let layer + 1 begin to write partials, over those of layer
// - 2 in the same buffer: all `chunks` merge chunks of each layer that used
// the buffer are merged, by the CTA's counts done[buffer]. One count over all
// buffers would not do: with two merge warps a chunk of layer - 1 can be done
// while one of layer - 2 is still being read.
LIBRASPEC_HD bool part_buf_free(const volatile int* done, int layer, int chunks) {
  const int old = layer + 1 - kAttnPartBufs;
  return old < 0 || done[old % kAttnPartBufs] >= (old / kAttnPartBufs + 1) * chunks;
}

}  // namespace libraspec
