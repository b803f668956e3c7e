// sweep2d_ring.cu -- the ring-staged one-row X-Y sweep (sweep2d_ring.cuh): the diamond-
// difference isotropic mode here, and the dispatch to the other translation units
// (sweep2d_ring_step.cu: step scheme; sweep2d_ring_m3.cu, sweep2d_ring_m3_step.cu:
// linear-kernel moments; sweep2d_ring_dense.cu: the dense operator mode), which build in
// parallel.
#include "sweep2d_ring.cuh"

namespace romk {

cudaError_t launch_sweep2d_ring_step(const SweepArgs &a, int n_items, int C, int G, bool homog,
                                     cudaStream_t st);
cudaError_t launch_sweep2d_ring_m3(const SweepArgs &a, int n_items, int C, int G, bool homog,
                                   cudaStream_t st);
cudaError_t launch_sweep2d_ring_m3_step(const SweepArgs &a, int n_items, int C, int G, bool homog,
                                        cudaStream_t st);

cudaError_t launch_sweep2d_ring_dense(const SweepArgs &a, int n_items, int C, int G, int scheme,
                                      bool homog, cudaStream_t st);

namespace {

// Cells per lane.  8 halve the per-step overhead per cell and the number of warps; 4 are
// faster for rows one warp covers, and where there are fewer than two items per SM to share
// the schedulers (256 x 256, 128 items of 2 ordinates: 34.9 us per sweep against 42.8; 256
// items of 4: 53.2 against 56.9; 1024 items of 4: 133 against 92).
int cells_per_lane(int I, int n_items) { return I > 128 && n_items >= 2 * 152 ? 8 : 4; }

bool fits(int I, int mom, bool homog, int C)
{
    const int nw = (I + 32 * C - 1) / (32 * C);
    return nw <= 8 && ring_bytes(mom, homog, nw, kMaxG, C) <= 227 * 1024;
}

}  // namespace

bool sweep2d_ring_fits(int I, int mom, bool homog)
{
    return (mom == 0 || mom == 1 || mom == 3) && fits(I, mom, homog, I > 128 ? 8 : 4);
}

cudaError_t launch_sweep2d_ring(const SweepArgs &a, int n_items, int G, int scheme, bool homog,
                                int mom, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    if (!sweep2d_ring_fits(a.I, mom, homog) || (G != 1 && G != 2 && (G != 4 || mom == 0)) ||
        (a.grids != nullptr && (homog || a.inflow != nullptr || mom == 0)) || (!homog && a.gdesc == nullptr))
        return cudaErrorInvalidValue;
    int C = cells_per_lane(a.I, n_items);
    if (!fits(a.I, mom, homog, C)) C = 8;  // wide rows: half the warps, the same rings
    if (mom == 0) return launch_sweep2d_ring_dense(a, n_items, C, G, scheme, homog, st);
    if (mom == 3)
        return scheme == 1 ? launch_sweep2d_ring_m3_step(a, n_items, C, G, homog, st)
                           : launch_sweep2d_ring_m3(a, n_items, C, G, homog, st);
    if (scheme == 1) return launch_sweep2d_ring_step(a, n_items, C, G, homog, st);
    if (homog) return ring_launch<1, 0, true>(a, n_items, C, G, st);
    return ring_launch<1, 0, false>(a, n_items, C, G, st);
}

}  // namespace romk
