// fmm_ring.h -- sizes of the brick scheduler's rings: plain C++, shared by the
// kernels, the host code and a host model of the scheduler.
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

}  // namespace fmmgb
