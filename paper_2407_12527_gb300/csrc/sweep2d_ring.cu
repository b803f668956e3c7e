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

// Cells per lane.  8 halve the per-step overhead per cell and the number of warps; 4 take
// half the registers and rings per warp (more CTAs per SM, a smoother last wave) and round the
// width to 128 cells instead of 256.  Microseconds per sweep, 8 against 4 cells, samples of 16:
//   up to 256 wide: 8, unless there are too few items to share the schedulers (2 per SM, of
//     four ordinates 3, with inflow 4: 256 x 256, 1200 items of two 89 against 126, 128 of two
//     43 against 39; 600 of four 65 against 80; three grids up to 200 wide, 384 of four 94
//     against 64; 211 x 173 with inflow, varying sigma_T, 384 of two 76 against 66);
//   257 .. 384 (more generally where 256-cell warps round up further): 4 (320 x 256, varying
//     sigma_T, 600 of four 221 against 147), but for uniform sigma_T with two ordinates (1200
//     of two 151 against 175);
//   above: 8 (512 x 256 uniform, 1200 of two 187 against 246), but for varying sigma_T with four
//     ordinates, whose 212 registers and 64 KB of rings want many items (448 x 64, 600 items 118
//     against 107; 448 x 448, 2048 of uneven samples 946 against 1098; the line is that of an
//     earlier form of the kernel, the present one gains from about 2000 items on, 448 x 64 306
//     against 326);
//   inflow with varying sigma_T and four ordinates: 4 (1200 items on 448 x 128 316 against 289,
//     on 144 x 128 141 against 138, but on 256 x 128 156 against 165);
//   linear kernel (three rings more): 4 (320 x 128, 1200 of four 440 against 305), but for
//     uniform sigma_T on 193 .. 256 (256 x 128 172 against 205).
int cells_per_lane(const SweepArgs &a, int n_items, int G, bool homog, int mom, int sms)
{
    const int I = a.I;
    const bool inflow = a.inflow != nullptr, four = G == 4;
    if (I <= 128 || n_items < 2 * sms) return 4;
    if (mom == 0) return 8;  // (512 x 512 x 32 of 128: 1750 against 2136)
    if (mom == 3) return homog && I > 192 && I <= 256 ? 8 : 4;
    if ((I + 127) / 128 % 2 == 1) return homog && !four && n_items >= 4 * sms ? 8 : 4;
    if (n_items < (inflow ? 4 : four ? 3 : 2) * sms) return 4;
    if (!homog && four && (inflow || (I > 256 && (long long)n_items * a.J < 4000LL * sms)))
        return 4;
    return 8;
}

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
                                int mom, int sm_count, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    if (!sweep2d_ring_fits(a.I, mom, homog) || (G != 1 && G != 2 && (G != 4 || mom == 0)) ||
        (a.grids != nullptr && (homog || a.inflow != nullptr || mom == 0)) || (!homog && a.gdesc == nullptr))
        return cudaErrorInvalidValue;
    int C = cells_per_lane(a, n_items, G, homog, mom, sm_count);
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
