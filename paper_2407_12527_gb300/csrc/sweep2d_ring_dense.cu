// sweep2d_ring_dense.cu -- the ring-staged one-row X-Y sweep (sweep2d_ring.cuh) in the dense
// operator mode: one source per ordinate in, psi of every ordinate out (FP32, or split BF16
// for the tensor-core contraction), both schemes.
#include "sweep2d_ring.cuh"

namespace romk {

cudaError_t launch_sweep2d_ring_dense(const SweepArgs &a, int n_items, int C, int G, int scheme,
                                      bool homog, cudaStream_t st)
{
    if (scheme == 1) {
        if (homog) return ring_launch<0, 1, true>(a, n_items, C, G, st);
        return ring_launch<0, 1, false>(a, n_items, C, G, st);
    }
    if (homog) return ring_launch<0, 0, true>(a, n_items, C, G, st);
    return ring_launch<0, 0, false>(a, n_items, C, G, st);
}

}  // namespace romk
