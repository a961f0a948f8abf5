// The mask of blocked candidates that the CTAs of an on-demand walk build up together in global memory (engine.cu,
// walk_csc.cu): two masks of `pitch` words, used in turns.
//
// The conflicts found in batch i are OR-ed into mask i & 1, and behind the batch's barrier every CTA ORs that mask into its
// own copy.  With a single mask a CTA that is ahead writes batch i + 1's conflicts into the words a late one is still
// reading for batch i: the late one sees some of them, picks another next batch than the rest, and the serial part of the
// walk is no longer the same in every CTA.  With two, the mask that is read behind barrier i is written again in batch i + 2
// only, behind barrier i + 1, which the late reader has to reach first.  Bits are never taken back within a walk, so the union
// of both masks over the batches is what one mask would hold.
//
// (Plain C++, so that the scheme can be run on the host: tests/test_walk_mask.py.)
#pragma once

#ifdef __CUDACC__
#define WALK_MASK_FN __host__ __device__ __forceinline__
#else
#define WALK_MASK_FN inline
#endif

namespace strads {

constexpr int kWalkMasks = 2;

// First word of the mask that batch `batch` of a walk writes and every CTA reads behind its barrier.
WALK_MASK_FN int walk_mask_at(unsigned int batch, int pitch) { return (int)(batch % kWalkMasks) * pitch; }

}  // namespace strads
