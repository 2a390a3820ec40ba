// fmm_ring.h -- sizes of the brick scheduler's rings and the claim of a scan's
// chunk: plain C++, shared by the kernels, the host code and a host model of the
// scheduler.
#pragma once

#ifdef __CUDACC__
#define FMM_HOST_DEVICE __host__ __device__
#else
#define FMM_HOST_DEVICE
#endif

namespace fmmgb {

// Slots of the waiting ring of a grid of nbricks bricks.  A scan appends the
// entries it keeps behind the region it empties, so between the first position
// of that region and the tail lie at most one entry of each brick that waited
// at the raise and one of each brick that was appended since: two per brick.
// With that many slots an append never finds its slot taken.  (With one slot
// per brick a scan of more than half of the bricks can wait for a slot that it
// has to empty itself, and never ends.)
FMM_HOST_DEVICE constexpr unsigned long long waiting_slots(long long nbricks)
{
    return 2ull * (unsigned long long)nbricks;
}

// The chunks of a scan: raise number << 32 | count.  A claim is what the shared
// counter (raise number << 32 | next chunk) held before it was advanced.  Its
// chunk is the claimer's only if it belongs to that raise: a claim past the last
// chunk holds nothing back, so two raises later the word may describe another
// scan with more chunks.  Returns the chunk, or -1.  (A chunk that was claimed
// keeps its scan open, so the word cannot change under a valid claim.)
FMM_HOST_DEVICE constexpr unsigned long long chunk_word(unsigned raise, unsigned count)
{
    return ((unsigned long long)raise << 32) | count;
}
FMM_HOST_DEVICE constexpr int claimed_chunk(unsigned long long claim, unsigned long long chunks)
{
    return claim >> 32 == chunks >> 32 && (unsigned)claim < (unsigned)chunks ? (int)(unsigned)claim : -1;
}

}  // namespace fmmgb
