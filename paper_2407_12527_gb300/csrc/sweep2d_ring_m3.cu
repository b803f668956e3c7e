// sweep2d_ring_m3.cu -- the ring-staged one-row X-Y sweep (sweep2d_ring.cuh), diamond
// difference, linear-kernel mode (three source and flux moments).
#include "sweep2d_ring.cuh"

namespace romk {

cudaError_t launch_sweep2d_ring_m3(const SweepArgs &a, int n_items, int C, int G, bool homog,
                                     cudaStream_t st)
{
    if (homog) return ring_launch<3, 0, true>(a, n_items, C, G, st);
    return ring_launch<3, 0, false>(a, n_items, C, G, st);
}

}  // namespace romk
