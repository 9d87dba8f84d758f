// Equal shares of a march for a fixed number of channel groups ("slots").
//
// One channel a slot in turn leaves SMs idle at the end: 512 channels on 152
// SMs take four rounds, the last with 56 channels.  Here the channels' steps lie
// one after the other on a line, channel after channel, and each slot takes an
// equal part of it (McNaughton's wrap-around rule).  A channel that a boundary
// cuts runs its first steps at the start of the upper slot's share and the rest
// at the end of the lower slot's: a share is at least a channel long, so the
// first part is over, or nearly, when the second one is due.  No slot depends on
// another, though: both leave a mark when they reach the cut, and whoever comes
// second marches the rest.  That is the lower slot, which looks for the upper
// one's mark for up to half a millisecond first, unless the upper one's block
// was started late.  The fields pass through global memory as they do between
// two calls.
#pragma once

#include "bpm_internal.h"

namespace bpm {

constexpr int kSharePolls = 4096;  // of 100 ns and a load each

struct Share {
  int ch, z0, n;     // the piece to march: channel (-1: none left), first row, steps
  int open;          // it ends at a cut: n_steps - n steps are left for the lower slot
  long long pos;     // where the slot is on the line
};

// Starts slot `slot`.
__device__ __forceinline__ void share_begin(const MarchArgs& A, int slot, int slots, Share* s) {
  s->open = 0;
  s->pos = slot;
  if (A.per_sm) s->pos *= ((long long)A.n_ch * A.n_steps + slots - 1) / slots;
}

// Next piece of the slot; one thread calls it, after the slot's threads have met
// a barrier behind their last stores and before one in front of the next loads.
// A call, so that it leaves the march its registers.
static __device__ __noinline__ void share_next(Share* s, int slot, int slots, int n_ch, int z0, int steps,
                                        int per_sm, int* handoff) {
  s->z0 = z0;
  s->n = steps;
  if (!per_sm) {  // whole channels
    s->ch = s->pos < n_ch ? int(s->pos) : -1;
    s->pos += slots;
    return;
  }
  if (s->open) {
    const int left = s->open;
    s->open = 0;
    __threadfence();
    if (atomicExch(handoff + slot, 1) == 2) {  // the lower slot has come and gone
      handoff[slot] = 0;
      s->z0 = z0 + steps - left;
      s->n = left;
      return;
    }
  }
  const long long total = (long long)n_ch * steps, per = (total + slots - 1) / slots;
  const long long end = min((slot + 1) * per, total);
  s->ch = -1;
  if (s->pos >= end) return;
  const int ch = int(s->pos / steps);
  const long long base = (long long)ch * steps;
  const int u0 = int(s->pos - base), u1 = int(min(end - base, (long long)steps));
  s->pos = base + u1;
  if (u0 > 0) {  // cut at its lower end: the first steps
    s->n = steps - u0;
    s->open = u0;
  } else if (u1 < steps) {  // cut at its upper end: the last steps
    const volatile int* mark = handoff + slot + 1;
    for (int i = 0; i < kSharePolls && *mark != 1; ++i) __nanosleep(100);
    if (atomicExch(handoff + slot + 1, 2) != 1) return;  // the upper slot will go on
    handoff[slot + 1] = 0;
    __threadfence();
    s->z0 = z0 + steps - u1;
    s->n = u1;
  }
  s->ch = ch;
}

__device__ __forceinline__ void share_next(const MarchArgs& A, int slot, int slots, Share* s) {
  share_next(s, slot, slots, A.n_ch, A.z0, A.n_steps, A.per_sm, A.handoff);
}

}  // namespace bpm
