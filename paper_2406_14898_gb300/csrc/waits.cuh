// Tracked bounded waits on mbarriers, for kernels that wait CTA-wide and may have to give
// up (the attention kernels).
#pragma once
#include "ptx.cuh"

// Phase bookkeeping of a kernel's mbarriers (bit i: barrier i) for CTA-wide bounded waits: `done`
// the parity of the phases waited for (every thread keeps the same), `pend` marks a phase armed by
// the issuing warp (a copy's expect_tx or an MMA commit) and not yet waited for.  After a wait gave
// up, the issuing thread drains: it waits (bounded again) for what it armed, so that no
// copy or product is still writing the CTA's shared memory or TMEM when it leaves.
struct BarTracks {
  uint32_t done = 0, pend = 0;
  FL_DEV uint32_t parity(int i) const { return (done >> i) & 1; }
  FL_DEV void arm(int i) { pend |= 1u << i; }
  FL_DEV void waited(int i) {
    done ^= 1u << i;
    pend &= ~(1u << i);
  }
};
FL_DEV bool track_wait_all(uint64_t* bars, int i, BarTracks& t) {
  const bool ok = __syncthreads_and(mbar_wait(bars + i, t.parity(i)));
  if (ok) t.waited(i);
  return ok;
}
FL_DEV void track_drain(uint64_t* bars, int n, const BarTracks& t) {
  for (int i = 0; i < n; ++i)
    if ((t.pend >> i) & 1) mbar_wait(bars + i, t.parity(i));
}
