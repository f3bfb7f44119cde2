// Named barriers of the attention kernel and the rule by which S and P change hands through them, also
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

// Barrier 0 is __syncthreads.  Group barriers: the 4 warps of softmax group a.  Swap barrier: all 8, in front of
// the exchange of partial results in a cluster.
constexpr int kGroupBarrier = 1, kPReadyBarrier = 3, kSFreeBarrier = 7, kSwapBarrier = 11;

// Per key tile of group a: S read (its 4 warps and the Q K^T issuer) and then P of the tile ready (its 4 warps
// and the P V issuer), two barriers of each kind per group used in turn.  The issuers always wait at the
// barriers, the Q K^T issuer at that of one tile's S before it issues the next one (the groups in turn), the
// P V issuer at that of a tile's P.  A softmax warp passes both without waiting (arrive) as long as its own
// waits succeed, and waits there (sync) once one of them gave up.
//
// Barriers only count arrivals, so a phase must never take two from one warp.  None does.  A warp that
// passes the S barrier of tile i+1 without waiting has seen S of tile i+1, which is issued behind tile i's
// phase; one that passes the P barrier of tile i+1 without waiting has seen the P V of tile i complete,
// which is issued behind tile i's phase.  A warp that gave up waits out every phase it enters, and a phase
// of tile i, in which it may still have arrived without waiting, is on the other barrier than tile i+1's.
// Its entry into tile i+2 comes behind the phase of tile i+1, which the issuer enters behind tile i's.  So
// every phase takes one arrival of each of the five warps, whatever gave up where, and, as all warps
// meet the barriers in one order (tile by tile, S before P), all of them end.
// With one barrier per group and kind a warp could arrive for tile i, give up, and arrive again for tile
// i+1 in the same phase, which then completes without one of the others: the issuer is left a phase
// behind, at a barrier that nobody comes to any more.
UNSTEP_HD int p_ready_barrier(int a, uint32_t tile) { return kPReadyBarrier + a + 2 * static_cast<int>(tile & 1u); }
UNSTEP_HD int s_free_barrier(int a, uint32_t tile) { return kSFreeBarrier + a + 2 * static_cast<int>(tile & 1u); }
UNSTEP_HD bool p_ready_waits(bool gave_up) { return gave_up; }

}  // namespace unstep
