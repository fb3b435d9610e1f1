// A wait on the barriers of a ring of shared-memory slots that bulk copies fill: its rule alone, without the hardware.
// np_pipe.cuh puts mbarriers under it, tests/test_ring_replay.py a model that replays it on the host.
//
// A slot has two barriers: `full` (the lane that fills the ring arms it, the copies complete it) and `empty` (its readers).  A
// barrier's parity tells the phase before the current one from the current one and nothing older, so a wait means what it says only
// while the ring keeps step: no slot is armed while copies are on their way into it.  Else `full` loses count of its phases, and
// with it the last means to tell when the block's shared memory is its own again; the block could leave before its copies.
//
// So a wait on these two barriers is not skipped once another wait of the block has run out, as all others are.  (If readers passed
// slots that they have not waited for, they would give them back ahead of the ring, and the filler's wait for a free slot would be
// over at once, on the parity of another use.)  Nor need it be: what it waits for are copies, and warps of this block that wait for
// nothing else then.  After kLimit polls it lowers the block's flag itself; the warps it waits for may then be at the start of a
// wait as long as that, so it goes on for 2 kLimit and pauses in between.  If that does not end it either, copies are lost;
// then the block gives up its ring.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define NP_RING_FN __device__ __forceinline__
#else
#define NP_RING_FN inline
#endif

namespace npp {

// The step behind a poll that has found the phase not complete; `polls` counts these.  True: the wait is given up.
// Block: stands() tells whether its flag does and lower() lowers it, pause(), given_up() tells whether the ring was given up, give_up().
template <uint32_t kLimit, class Block>
NP_RING_FN bool ring_wait_step(uint32_t& polls, Block& b) {
  if (!b.stands()) {
    if (b.given_up()) return true;
    b.pause();
    if (polls > 3 * kLimit) b.give_up();
  }
  if (++polls == kLimit) b.lower();
  return false;
}

}  // namespace npp
