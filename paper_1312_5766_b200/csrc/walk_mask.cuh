// The mask of blocked candidates that the CTAs of an on-demand walk build up together in global memory (engine_csc.cuh,
// walk_csc.cu): two masks of `pitch` words, used in turns.
//
// walk_csc.cu: the conflicts found in batch i are OR-ed into mask i & 1, and behind the batch's barrier every CTA ORs that mask into its
// own copy.  With a single mask a CTA that is ahead writes batch i + 1's conflicts into the words a late one is still
// reading for batch i: the late one sees some of them, picks another next batch than the rest, and the serial part of the
// walk is no longer the same in every CTA.  With two, the mask that is read behind barrier i is written again in batch i + 2
// only, behind barrier i + 1, which the late reader has to reach first.  Bits are never taken back within a walk, so the union
// of both masks over the batches is what one mask would hold.
//
// engine_csc.cuh: 32 consecutive candidates, a word, have one owner, which keeps the word as it is so far and writes the whole of it
// in every batch, changed or not, so that a mask is complete behind the batch's barrier whatever it held before (nothing clears it) and
// the next batch is picked from it alone.  Two masks in turns for the same reason.
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

// engine_csc.cuh: whether the CTAs still have to meet at the end of a walk that began with the grid barrier's target at `begun` and has it at
// `target` now: it had no batch's barrier.  (Not arriving at the start and waiting at the end: with the first batch's arrival on top of
// that one, a CTA still at the barrier before would see the counter run past the range in which it may pass.)
WALK_MASK_FN bool walk_to_meet(unsigned int begun, unsigned int target) { return begun == target; }

}  // namespace strads
