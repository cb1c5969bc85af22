// The order in which a step on host weights in parts is queued, and what happens when queuing fails half-way.  Plain
// C++ over an object that queues, so that every failure can be played through on the CPU.
//
//   op.copy_in(k)    part k's weights to the device, on a stream of their own, and a mark behind them
//   op.step(k)       the caller's stream waits for that mark and steps the part
//   op.copy_out(k)   the part's reconstructed weights to the host, on a third stream, behind its step
//   op.clear()       empties the look-back words and counters in the workspace, behind what has been queued
//   op.join()        the caller's stream waits for the other two
// Each returns 0 or an error; the first error is returned.
//
// * All weights are on their way before anything is stepped: a host range that cannot be copied leaves caches, messages
//   and workspace as they were.
// * A part that cannot be launched ends the step.  The words that the parts before it left in the workspace, which only
//   the last part would have emptied, are emptied here, or the next call would take them for its own.
// * A range that cannot be copied out ends nothing: the step on the device is completed, as without parts.
#pragma once

#include <stdint.h>

namespace ciera {

template <class Ops>
int run_host_parts(Ops& op, uint32_t parts) {
    int rc = 0;
    for (uint32_t k = 0; k < parts && rc == 0; ++k) rc = op.copy_in(k);
    if (rc == 0) {
        int rc_out = 0;
        for (uint32_t k = 0; k < parts && rc == 0; ++k) {
            rc = op.step(k);
            if (rc != 0) {
                op.clear();
            } else {
                const int r = op.copy_out(k);
                if (rc_out == 0) rc_out = r;
            }
        }
        if (rc == 0) rc = rc_out;
    }
    const int r = op.join();  // whatever happened
    return rc != 0 ? rc : r;
}

}  // namespace ciera
