// Full barriers of a shared-memory ring that two consumer groups take in turn
// (fill k goes into buffer k mod stages and is read by group k mod 2).
//
// mbarrier waits name a phase by its parity alone: a wait for parity P passes
// whenever the phase in progress has the other parity.  That is the wanted
// phase only for a thread that waits for every phase of the barrier in turn.
// With an even number of buffers a buffer belongs to one group for good.  With an
// odd one the groups alternate on it, and with one barrier per buffer each
// would wait for every second phase: a group that is ahead passes while the
// other group's copy into the buffer is still on its way, reads what is not
// there and hands the buffer back early.  So an odd ring has two full barriers
// per buffer, one for each group's fills.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define PVS_RING_FN __host__ __device__ __forceinline__
#else
#define PVS_RING_FN inline
#endif

namespace pvs {

// Full barriers of a ring of `stages` buffers (always even).
PVS_RING_FN constexpr int turn_bars(int stages) { return stages % 2 == 0 ? stages : 2 * stages; }
// Of fill k: its barrier, that barrier's parity, and its buffer.
PVS_RING_FN int turn_bar(int k, int stages) { return k % turn_bars(stages); }
PVS_RING_FN uint32_t turn_parity(int k, int stages) {
    return (uint32_t)(k / turn_bars(stages)) & 1u;
}
PVS_RING_FN int turn_buffer(int bar, int stages) { return bar < stages ? bar : bar - stages; }

}  // namespace pvs
