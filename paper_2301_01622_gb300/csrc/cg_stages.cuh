// Staging schedule of the two-component pair kernel (cg_pair.cuh).
//
// Every step of a work item waits for one group of TMA boxes; groups are numbered
// through all items of a CTA and alternate between two mbarriers.  The first two steps'
// groups are staged when the item begins, that of step s + 2 when step s has been waited
// for and read, so at the wait of step s two groups are in flight, and one at the item's
// last step.
#pragma once

namespace llb {
namespace cg {

struct Stages {
    static constexpr int kBars = 2;
    __host__ __device__ static unsigned bar(unsigned n) { return n % kBars; }
    // parity of the phase of its barrier that group n completes
    __host__ __device__ static unsigned parity(unsigned n) { return n / kBars & 1; }
    // end of the range of groups in flight at the wait for group n in step s of an item whose last step is `last`
    __host__ __device__ static unsigned in_flight_end(unsigned n, int s, int last) { return n + (s < last ? 2 : 1); }
};

}  // namespace cg
}  // namespace llb
