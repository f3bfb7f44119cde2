// Named barriers of the attention kernel and the rule by which P changes hands through them, also
// after a wait gave up.  Compiled for the device and, in the test of the rule, for the host.
#pragma once

#include <stdint.h>

#ifndef UNSTEP_HD
#if defined(__CUDACC__)
#define UNSTEP_HD __host__ __device__ __forceinline__
#else
#define UNSTEP_HD inline
#endif
#endif

namespace unstep {

// Barrier 0 is __syncthreads.  Group barriers: the 4 warps of softmax group a.  Turn barriers: the
// two issuing warps, one waiting for its turn (a), the other handing it over.
constexpr int kGroupBarrier = 1, kPReadyBarrier = 3, kTurnBarrier = 7;

// P of a key tile: 4 softmax warps of group a and the issuing warp a, two barriers per group used in
// turn.  The issuer always waits at the barrier of a tile; a softmax warp passes it without waiting
// (arrive) as long as its own waits succeed, and waits there (sync) once one of them gave up.
//
// Barriers only count arrivals, so a phase must never take two from one warp.  None does: a warp that
// arrives for tile i+1 without waiting has seen S of tile i+1, which the issuer commits behind tile
// i's phase; a warp that gave up waits out every phase it enters, and the phase of tile i, in which it
// may still have arrived without waiting, is on the other barrier than tile i+1's.  Its entry into
// tile i+2 comes behind the phase of tile i+1, which the issuer enters behind tile i's.  So every
// phase takes one arrival of each of the five warps, whatever gave up where, and all of them end.
// With one barrier per group a warp could arrive for tile i, give up on S of tile i+1 and arrive
// again in the phase of tile i, which then completes without one of the others: the issuer is left a
// phase behind, at a barrier that nobody comes to any more.
UNSTEP_HD int p_ready_barrier(int a, uint32_t tile) { return kPReadyBarrier + a + 2 * static_cast<int>(tile & 1u); }
UNSTEP_HD bool p_ready_waits(bool gave_up) { return gave_up; }

}  // namespace unstep
