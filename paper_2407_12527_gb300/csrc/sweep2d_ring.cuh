// sweep2d_ring.cuh -- the X-Y transport sweep (K1) with one grid row per wavefront step and
// the cell rows staged through per-lane rings in shared memory, for the angular-moment source
// modes (isotropic, linear kernel) and the dense operator mode.
//
// Same cell equations, work items (up to G ordinates of one quadrant of one sample) and
// moment accumulators as the other X-Y sweeps.  Lanes are numbered from the inflow face;
// lane p owns the C cells (4 or 8) at distance C p .. C p + C - 1 from it in every row, and
// lane d of a warp sweeps row t - d at the warp's step t, so the x-edge flux passes one lane
// per step by a shuffle and the y-edge fluxes stay in registers.  Warp w of a wide row runs
// kLag * 8 steps behind warp w - 1 and takes the x-edges from a shared-memory ring; the
// warps meet at one CTA barrier per 8 steps.
//
// Memory.  The lanes of a warp sit on 32 different rows, so a direct access of the warp
// would touch 32 cache lines, and the L1 takes one line per cycle: 32 cycles per access and
// three accesses per step, on the four schedulers' shared L1, against ~100 cycles of
// arithmetic per warp and step.  Instead each 8-lane group copies 128 (C = 8: 256)
// contiguous bytes of one row per step (cp.async, row t + kAhead - 8 * group) into 16-row
// rings of its lanes' columns; a lane reads its own cells when its step comes and leaves the
// moments in the same slot, and the group adds them to the accumulator row by row, again 128
// contiguous bytes at a time (red.global.add.v4), once its last lane has passed.  No lane
// touches another group's columns, so the rings need no barrier (a warp-level one with C = 8,
// where the lanes of a group copy for each other to keep the 128 bytes contiguous).  In the
// dense mode the slots hold the sources of the item's two ordinates and take their psi, which
// the group stores (FP32 or split BF16) and sums into phi.
//
// Arithmetic.  With f = 2 (diamond difference) or 1 (step), a = f|c|/dx, b = f|s|/dy,
// d = sigma_T + a + b, the edge fluxes are kept scaled so that the source enters every
// ordinate of a pack with coefficient one:
//   uniform sigma_T: X = x d / f, P = b y:    t = S + P, X' = alpha X + t,
//     DD:   alpha = (a - b - sigma_T) / d, sum = X + X', P' = 2 b / d sum - P,
//     step: alpha = a / d,                 sum = X',     P' = b / d sum,
//     moment += (w / d) sum;
//   varying sigma_T: X = a x, P = b y: psi = (S + X + P) / d, X' = f a psi - X (DD) or
//     a psi, P' likewise, moment += w psi.
// The uniform case takes five packed FP32x2 operations per cell and ordinate pair and its
// upwind chain is one FMA per cell.  (DD in uniform cells of many mean free paths: X and X'
// nearly cancel, and their sum has the rounding of the edges instead of psi's.  The 4-row
// kernel's x + x' is the same: over twelve lit media without sources the flux is off by
// 8e-7 on average at sigma_T dx = 100 and 6e-6 at 1000 with either.)  The DD closure keeps -P after even steps (and the
// varying case -X at odd cells), so that every update is one FMA without a negated operand:
// P' = c - P or -P' = P - c.  (Negated operands cost the packed instructions nothing; the
// plain form measured 4% slower on the checkerboard with four ordinates per item, 7% faster
// on three mixed grids with two, the same elsewhere.)
//
// What bounds it.  A warp issues 115-125 instructions per step of 512 updates at 2.5-3
// cycles each with the one or two warps per scheduler of most solves (fixed-latency
// dependencies, three cycles of register ports per packed FMA); with two ordinates per item
// the moment reductions (134 MB at 256 x 256 x 64 samples of 16) add 6-8 of 49 us.  One
// launch, GB300, against the row kernel of sweep2d_row.cuh: 256 x 256 x 64 samples of 16
// 49 us (70), one sample of 256 35 (54), 256 samples of 16 92 (141); 100 x 100 x 16 of 36
// 18 (45); varying sigma_T 256 x 256 x 256 of 16 165 (274).  Dense mode, 512 x 512 x 32 of
// 128: 1746 us against 2640 with the 4-row kernel (8.6 GB: 73% of the copy bandwidth);
// 150 x 130 x 8 of 48 51 against 138.
#pragma once
#include <type_traits>

#include "rom_internal.cuh"

namespace romk {
namespace {

constexpr int kRows = 16;    // rows of a ring
constexpr int kAhead = 7;    // rows a group copies ahead of its first lane's step: the slot
                             // of row r - 16 is drained one step before row r is copied
constexpr int kGrp = 8;      // steps between CTA barriers; lanes of a 128-byte group
constexpr int kLag = 5;      // groups of steps a warp runs behind its upstream warp: row r
                             // leaves that warp 9 steps before it is needed, and is read
                             // one step early, so a barrier lies between
constexpr int kEdgeRows = 32;

template <int G>
struct RingPack {
    static constexpr int N = G / 2;
};
__device__ __forceinline__ float2 qfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 qmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 qadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 qsplat(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 qneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float qrcp(float a)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));  // within 1 ulp; a >= sigma_T > 0
    return r;
}
__device__ __forceinline__ void qset(float2 &a, int i, float v)
{
    if (i) a.y = v;
    else a.x = v;
}
__device__ __forceinline__ float qget(const float2 &a, int i) { return i ? a.y : a.x; }
__device__ __forceinline__ float f4(const float4 &v, int r)
{
    return r == 0 ? v.x : r == 1 ? v.y : r == 2 ? v.z : v.w;
}
__device__ __forceinline__ unsigned ring_u32(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}
// Shared- and global-memory accesses of a step, all kept in program order.  The predicated
// ones skip by a predicate, not a branch, which would split the step's instructions: a copy
// or reduction whose row is outside [0, lim) (lim = 0: a chunk without cells), a store of a
// lane without cells.
__device__ __forceinline__ float4 lds4(unsigned p)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(p));
    return v;
}
__device__ __forceinline__ void sts4(unsigned p, const float4 &v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(p), "f"(v.x), "f"(v.y), "f"(v.z),
                 "f"(v.w)
                 : "memory");
}
template <int C>
__device__ __forceinline__ void sts_cells(const unsigned *p, unsigned off, const float *v, bool on)
{
    if constexpr (C == 8)
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %10, 0;\n\t"
                     "@q st.shared.v4.f32 [%0], {%2,%3,%4,%5};\n\t"
                     "@q st.shared.v4.f32 [%1], {%6,%7,%8,%9};\n\t}" ::"r"(p[0] + off),
                     "r"(p[1] + off), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]),
                     "f"(v[5]), "f"(v[6]), "f"(v[7]), "r"((unsigned)on)
                     : "memory");
    else
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t"
                     "@q st.shared.v4.f32 [%0], {%1,%2,%3,%4};\n\t}" ::"r"(p[0] + off), "f"(v[0]),
                     "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"((unsigned)on)
                     : "memory");
}
template <int OFF>  // bytes from src to the chunk
__device__ __forceinline__ void ring_copy(unsigned dst, const float *src, int row, int lim)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %2, %3;\n\t"
                 "@q cp.async.cg.shared.global [%0], [%1+%4], 16;\n\t}" ::"r"(dst), "l"(src),
                 "r"(row), "r"(lim), "n"(OFF)
                 : "memory");
}
template <int OFF>
__device__ __forceinline__ void ring_red(float *p, const float4 &v, int row, int lim)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %5, %6;\n\t"
                 "@q red.global.add.v4.f32 [%0+%7], {%1,%2,%3,%4};\n\t}" ::"l"(p), "f"(v.x),
                 "f"(v.y), "f"(v.z), "f"(v.w), "r"(row), "r"(lim), "n"(OFF)
                 : "memory");
}
// dense mode: psi of 4 cells, FP32 at p + o, or its BF16 parts in the 32-byte sector
// [8 hi | 8 lo] of the 8 cells they belong to (st8_split's rounding)
template <int OFF>
__device__ __forceinline__ void psi_put(float *psi, uint32_t *split, long long o, const float4 &v,
                                        int row, int lim)
{
    if (split == nullptr) {
        asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %5, %6;\n\t"
                     "@q st.global.v4.f32 [%0+%7], {%1,%2,%3,%4};\n\t}" ::"l"(psi + o), "f"(v.x),
                     "f"(v.y), "f"(v.z), "f"(v.w), "r"(row), "r"(lim), "n"(OFF)
                     : "memory");
        return;
    }
    o += OFF / 4;
    uint32_t h[2], l[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float a = e ? v.z : v.x, b = e ? v.w : v.y;
        const uint32_t b0 = (__float_as_uint(a) + 0x8000u) & 0xFFFF0000u;
        const uint32_t b1 = (__float_as_uint(b) + 0x8000u) & 0xFFFF0000u;
        h[e] = __byte_perm(b0, b1, 0x7632);
        const __nv_bfloat162 lo2 =
            __floats2bfloat162_rn(a - __uint_as_float(b0), b - __uint_as_float(b1));
        l[e] = *reinterpret_cast<const uint32_t *>(&lo2);
    }
    uint32_t *q = split + (o & ~7LL) + ((o >> 1) & 2);
    asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %5, %6;\n\t"
                 "@q st.global.v2.b32 [%0], {%1,%2};\n\t"
                 "@q st.global.v2.b32 [%0+16], {%3,%4};\n\t}" ::"l"(q), "r"(h[0]), "r"(h[1]),
                 "r"(l[0]), "r"(l[1]), "r"(row), "r"(lim)
                 : "memory");
}
// test hook: a wait, bounded in time, on an mbarrier that nothing completes
__device__ __forceinline__ bool ring_never_wait(unsigned long long *b, unsigned long long budget_ns)
{
    unsigned long long t0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (;;) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(ring_u32(b)), "r"(0u)
            : "memory");
        if (__all_sync(0xffffffffu, ok != 0)) return true;
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (__any_sync(0xffffffffu, t - t0 > budget_ns)) return false;
    }
}

// Arrays copied in: the source moments, or in the dense mode the sources of the item's two
// ordinates (their slots take the flux moments, or psi), and sigma_T.
__host__ __device__ constexpr int ring_src(int mom) { return mom == 0 ? 2 : mom; }
__host__ __device__ constexpr int ring_arrays(int mom, bool homog) { return ring_src(mom) + (homog ? 0 : 1); }
// shared memory of a CTA: the warps' rings, their incoming x-edges, 16 zero bytes
__host__ __device__ constexpr int ring_bytes(int mom, bool homog, int nwarps, int G, int C)
{
    return nwarps * (ring_arrays(mom, homog) * kRows * 32 * C + kEdgeRows * G) * 4 + 16;
}

template <int C, int G, int MOM, int SCHEME, bool HOMOG, bool XNEG, bool RAGGED, bool EDGE>
__device__ __forceinline__ void ring_item(const SweepArgs &A, const GridDesc &gd,
                                          const SweepItem &it, char *smem)
{
    constexpr int N = RingPack<G>::N;
    constexpr int NS = ring_src(MOM), NA = ring_arrays(MOM, HOMOG);
    constexpr int NP = MOM == 0 ? 2 : 1;    // base pointers of the sources
    static_assert(MOM != 0 || G == 2, "the dense mode takes two ordinates per item");
    constexpr unsigned kRowB = 32 * C * 4, kArrB = kRows * kRowB;  // bytes of a ring row, a ring
    constexpr int CH = C / 4;  // 16-byte chunks of a lane's cells
    constexpr unsigned kMask = kArrB - 1;
    constexpr unsigned kEdgeB = kEdgeRows * G * 4;
    constexpr bool DD = SCHEME == 0;
    const int nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    const int w = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);  // (uniform)
    const int L = (gd.I + C - 1) / C;  // lanes that own cells
    const int p = 32 * w + lane;
    const bool on = p < L;
    const int col = on ? C * (XNEG ? L - 1 - p : p) : 0;
    const bool yneg = (it.quad >> 1) & 1;
    const int J = gd.J;
    const float fdd = DD ? 2.f : 1.f;

    // per-ordinate constants (see the head of the file); an empty slot has weight zero
    float2 kp[N];  // dense mode: psi per sum (uniform sigma_T)
    float2 k1[N], k2[N], k2n[N], km[N], kmc[N], kms[N], kc[N], ks[N], ab[N], lx[N], wl[N];
    long long ord[G];
    float inj_x[G], inj_y[G];  // boundary value -> scaled edge flux
#pragma unroll
    for (int k = 0; k < G; ++k) {
        float c = 0.f, s = 0.f, wt = 0.f;
        ord[k] = it.ord[0];
        if (k < it.n) {
            ord[k] = it.ord[k];
            c = A.oc[ord[k]];
            s = A.os[ord[k]];
            wt = A.ow[ord[k]];
        }
        const int pk = k >> 1, i = k & 1;
        const float a = fdd * fabsf(c) * gd.inv_dx, b = fdd * fabsf(s) * gd.inv_dy;
        const float st = A.sigma_t_homog;
        const float rd = HOMOG ? 1.f / (st + a + b) : 1.f;
        const float wm = HOMOG ? wt * rd : wt;
        qset(k1[pk], i, HOMOG ? (DD ? (a - b - st) * rd : a * rd) : fdd * a);
        qset(k2[pk], i, HOMOG ? fdd * b * rd : fdd * b);
        qset(ab[pk], i, a + b);
        qset(kp[pk], i, rd);
        qset(km[pk], i, MOM == 0 ? wt : wm);
        qset(kmc[pk], i, wm * c);
        qset(kms[pk], i, wm * s);
        qset(kc[pk], i, c);
        qset(ks[pk], i, s);
        // leakage in units of dx dy, which can be outside the range of FP32 where the edge terms
        // are not: w |s| dx y = dx dy (w / f) P; w |c| dy x = dx dy w a rd X, or dx dy (w / f) X
        qset(wl[pk], i, wt / fdd);
        const float lo = HOMOG ? wt * a * rd : wt / fdd;
        qset(lx[pk], i, (A.leak != nullptr && p == L - 1) ? lo : 0.f);
        inj_x[k] = HOMOG ? (st + a + b) / fdd : a;
        inj_y[k] = b;
    }
#pragma unroll
    for (int q = 0; q < N; ++q) k2n[q] = qneg(k2[q]);
    // lane 0 takes no x-edge from the shuffle
    const float2 neg1 = qsplat(-1.f), k0 = qsplat(lane == 0 ? 0.f : 1.f);
    float2 k1f[N];
#pragma unroll
    for (int q = 0; q < N; ++q) k1f[q] = qmul(k1[q], k0);
    // real[rr]: the cell at sweep position rr (column XNEG ? 3 - rr : rr) is inside the grid
    bool real[C];
#pragma unroll
    for (int rr = 0; rr < C; ++rr)
        real[rr] = !RAGGED || col + (XNEG ? C - 1 - rr : rr) < gd.I;

    // The lane's rings, all zero at first (sigma_T one): rows before the grid's first sweep
    // zeros, and so does a lane without cells.  Slots go by step: the cells of step t are in
    // slot t mod 16 of every lane; the row copied at step t is the one of the lane's step
    // t + kAhead + (lane & 7), and the row drained, 15 rows before it, sits in the next slot.
    // Of 8 cells a lane's two halves trade places on every other 4 lanes (bank conflicts).
    // The lane copies and drains CH chunks of its group's row: lane e those of the group's
    // lanes e (C = 4), or e / 2 and 4 + e / 2 (C = 8), which keeps every access of the group
    // to 128 contiguous bytes.
    const unsigned rings = ring_u32(smem) + w * NA * kArrB;
    const int sw = CH == 2 ? (lane >> 2) & 1 : 0;
    unsigned own[CH];
#pragma unroll
    for (int h = 0; h < CH; ++h) own[h] = rings + lane * C * 4 + ((h ^ sw) * 16);
    for (int m = 0; m < NA; ++m)
        for (int r = 0; r < kRows; ++r) {
            const float z = !HOMOG && m == NS ? 1.f : 0.f;
#pragma unroll
            for (int h = 0; h < CH; ++h) sts4(own[h] + m * kArrB + r * kRowB, make_float4(z, z, z, z));
        }
    __syncwarp();
    const unsigned edges = ring_u32(smem) + nw * NA * kArrB;
    if constexpr (EDGE) {
        for (int k = threadIdx.x; k < nw * kEdgeRows * G + 4; k += blockDim.x)
            ((float *)(smem + (size_t)nw * NA * kArrB))[k] = 0.f;
        __syncthreads();
    }
    // lane 0 reads the x-edges of its warp, the others the zeros after the last ring
    const unsigned edge_in = lane == 0 ? edges + w * kEdgeB : edges + nw * kEdgeB;
    const unsigned edge_sel = lane == 0 ? kEdgeB - 1 : 0;
    const unsigned edge_out = edges + (w + 1) * kEdgeB;

    const long long so =
        A.soff ? A.soff[it.sample] : (long long)it.sample * (MOM == 0 ? 1 : MOM) * gd.cells;
    const long long rs = yneg ? -(long long)gd.NXP : (long long)gd.NXP;
    const long long cells = gd.cells;
    const int grp8 = lane & ~7;  // 8 * the lane's group

    float2 P[C][N], X[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
        X[q] = qsplat(0.f);
#pragma unroll
        for (int r = 0; r < C; ++r) P[r][q] = qsplat(0.f);
    }
    double leak = 0.0;
    // With an inflow the incoming y-edges wait in P, held by zero constants (k2, and the
    // x leakage's lx), until the lane's first row: the rows before it compute numbers that
    // reach no cell of the grid.  The step of that row finds P negated if it is odd.
    bool held = false;
    float2 k2s[N], lxs[N];  // (EDGE)
    if constexpr (EDGE) {
        held = A.inflow != nullptr;
        if (held) {
#pragma unroll
            for (int r = 0; r < C; ++r)
#pragma unroll
                for (int k = 0; k < G; ++k)
                    if (on && col + r < gd.I && k < it.n) {
                        const float b = inj_y[k] * A.inflow[(long long)ord[k] * A.inflow_stride +
                                                            2 * J + (yneg ? gd.I : 0) + col + r];
                        qset(P[r][k >> 1], k & 1, DD && (lane & 1) ? -b : b);
                        leak -= (double)(qget(wl[k >> 1], k & 1) * b);
                    }
        }
#pragma unroll
        for (int q = 0; q < N; ++q) {
            k2s[q] = k2[q];
            lxs[q] = lx[q];
            if (held) k2[q] = k2n[q] = lx[q] = qsplat(0.f);
        }
    }
    // The x-edge terms, summed over the even and over the odd steps of a group, then compensated
    // (Kahan): four rows of the item's pairs per compensated add, as in the 4-row kernel.  (A sum
    // per pair has registers spilled with four ordinates: 0.5% slower over 33 solves.)
    float lk_s = 0.f, lk_c = 0.f;
    float2 lk[2] = {qsplat(0.f), qsplat(0.f)};

    // Groups of 8 steps of the warp: steps -8 .. J + 7 + 8 * (its last lanes' group); a warp
    // starts kLag groups after the one upstream.  nwl: warps that own cells (a batch's
    // narrower grid leaves some without).
    const int nwl = (L + 31) / 32;
    auto groups = [&](int lanes) { return 1 + (J + 8 + ((lanes - 1) & ~7) + kGrp - 1) / kGrp; };
    const int n_grp_l = groups(L - 32 * (nwl - 1)), n_grp_f = groups(32);
    const int n_grp_w = w >= nwl ? 0 : w == nwl - 1 ? n_grp_l : n_grp_f;
    const int n_grp = nwl == 1 ? n_grp_l
                               : max(n_grp_f + kLag * (nwl - 2), n_grp_l + kLag * (nwl - 1));
    const bool feeds = lane == 31 && w < nwl - 1;

    bool past = false;
    int t = -kGrp;
    const long long o0 = so + (yneg ? (long long)(J - 1) * gd.NXP : 0);
    int frow = t + kAhead - grp8;  // the row copied at step t
    int lim[CH];              // J, or 0 for a chunk without cells
    unsigned fd[CH];          // the slot copied into (the row drained is in the next one)
    const int dl0 = CH == 1 ? lane & 7 : (lane & 7) >> 1, half = CH == 1 ? 0 : lane & 1;
#pragma unroll
    for (int h = 0; h < CH; ++h) {
        const int dl = dl0 + 4 * h;  // the group's lane whose cells they are
        lim[h] = 32 * w + grp8 + dl < L ? J : 0;
        fd[h] = (unsigned)(t + kAhead + dl) % kRows * kRowB;
    }
    const unsigned place = rings + (grp8 + dl0) * C * 4 + half * 16;  // of the first chunk
    constexpr unsigned kPlace1 = 4 * C * 4;  // the second: 4 lanes on, halves exchanged
    const unsigned place1 = CH == 2 ? (place ^ 16) + kPlace1 : 0;
    constexpr int kChunk1 = (XNEG ? -1 : 1) * 4 * C * 4;  // bytes between the chunks' cells
    const int cd = C * (XNEG ? L - 1 - (32 * w + grp8 + dl0) : 32 * w + grp8 + dl0) + 4 * half;
    const float *src[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k)
        src[k] = A.src + (MOM == 0 ? o0 - so + ord[k] * cells : o0) + cd + frow * rs;
    const float *sig = HOMOG ? nullptr : A.sigma_t + gd.off + (o0 - so) + cd + frow * rs;
    float *acc = A.part + o0 + cd + (frow - kRows + 1) * rs;
    long long po = o0 - so + cd + (frow - kRows + 1) * rs;  // dense mode: place of psi
    unsigned cs = 0;             // slot of the step's cells (step 0: slot 0)
    unsigned eo = 0;             // offset of the x-edges of row t + 1 (and of row t - 31)

    float4 S[NA][CH];                            // the cells of the next step
    float4 E = make_float4(0.f, 0.f, 0.f, 0.f);  // its incoming x-edge (lane 0)

    auto fill = [&]() {
#pragma unroll
        for (int m = 0; m < NA; ++m) {
            const float *p = m >= NS ? sig : MOM == 0 ? src[m % NP] : src[0] + m * cells;
            ring_copy<0>(place + m * kArrB + fd[0], p, frow, lim[0]);
            if constexpr (CH == 2)
                ring_copy<kChunk1>(place1 + m * kArrB + fd[CH - 1], p, frow, lim[CH - 1]);
        }
#pragma unroll
        for (int k = 0; k < NP; ++k) src[k] += rs;
        if constexpr (!HOMOG) sig += rs;
        ++frow;
#pragma unroll
        for (int h = 0; h < CH; ++h) fd[h] = (fd[h] + kRowB) & kMask;
        asm volatile("cp.async.commit_group;" ::: "memory");
        // this step's copies and those of the five before it may still be in flight: a row
        // is read 6 copies after its own
        asm volatile("cp.async.wait_group 6;" ::: "memory");
        if constexpr (CH == 2) __syncwarp();  // (C = 4: a lane copies and drains its own cells)
    };
    auto load = [&]() {
#pragma unroll
        for (int m = 0; m < NA; ++m)
#pragma unroll
            for (int h = 0; h < CH; ++h) S[m][h] = lds4(own[h] + m * kArrB + cs);
        if constexpr (EDGE) {
            const unsigned ep = edge_in + (eo & edge_sel);
            if constexpr (N == 2) E = lds4(ep);
            else
                asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(E.x), "=f"(E.y) : "r"(ep));
        }
    };

    // One step.  EV: some lane passes its first or last row in this group of steps; ODD: P
    // holds its negative.
    //
    // Rows past the last one compute numbers that reach no cell of the grid: their source is what
    // the lane left in the slot 16 rows before, and zero constants (k2, lx) keep them out of the
    // y-edges and the leakage, as long as they are finite.  So such a row leaves nothing in its
    // slot: one that took another's moments for a source would divide by sigma_T + a + b once
    // more every 16 rows, and overflow in small units.  (Keeping P and lk by selects instead
    // measured the same on most solves, 1-2% more on the smallest.)
    auto step = [&](auto events, auto odd) {
        constexpr bool EV = decltype(events)::value;
        constexpr int par = decltype(odd)::value;
        constexpr bool ODD = DD && par;
        fill();
        // the moments of the row that the group's last lane finished at the step before
        // (fill has moved on to its slot)
        float4 D[NS][CH];
#pragma unroll
        for (int m = 0; m < NS; ++m)
#pragma unroll
            for (int h = 0; h < CH; ++h) D[m][h] = lds4((h ? place1 : place) + m * kArrB + fd[h]);
        const unsigned slot = cs;
        float4 V[NA][CH];
#pragma unroll
        for (int m = 0; m < NA; ++m)
#pragma unroll
            for (int h = 0; h < CH; ++h) V[m][h] = S[m][h];
        float2 x[C + 1][N], sm[C][N];
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const float2 e = q == 0 ? make_float2(E.x, E.y) : make_float2(E.z, E.w);
            x[0][q] = EDGE ? qfma(X[q], k0, e) : X[q];
        }
        cs = (cs + kRowB) & kMask;
        if constexpr (EDGE) eo = (eo + G * 4) & (kEdgeB - 1);
        load();
        if constexpr (EV) {
            const int row = t - lane;
            if (EDGE && held && row == 0) {  // the lane's first row: its y-edges come free
                held = false;
#pragma unroll
                for (int q = 0; q < N; ++q) {
                    k2[q] = k2s[q];
                    k2n[q] = qneg(k2s[q]);
                    lx[q] = lxs[q];
                }
            }
            if (row == J) {  // past the last row the y-edges stay and nothing counts
                past = true;
#pragma unroll
                for (int q = 0; q < N; ++q) k2[q] = k2n[q] = lx[q] = qsplat(0.f);
            }
        }
#pragma unroll
        for (int rr = 0; rr < C; ++rr) {
            const int r = XNEG ? C - 1 - rr : rr;
#pragma unroll
            for (int q = 0; q < N; ++q) {
                float2 tt;
                if constexpr (MOM == 3) {
                    const float2 s =
                        qfma(kc[q], qsplat(f4(V[MOM == 3 ? 1 : 0][r / 4], r % 4)),
                             qfma(ks[q], qsplat(f4(V[MOM == 3 ? 2 : 0][r / 4], r % 4)), qsplat(f4(V[0][r / 4], r % 4))));
                    tt = ODD ? qfma(P[r][q], neg1, s) : qadd(s, P[r][q]);
                } else {
                    const float s = f4(V[0][r / 4], r % 4);
                    const float sy = MOM == 0 ? f4(V[MOM == 0 ? 1 : 0][r / 4], r % 4) : s;
                    tt = ODD ? make_float2(s - P[r][q].x, sy - P[r][q].y)
                             : make_float2(s + P[r][q].x, sy + P[r][q].y);
                }
                const bool first = !EDGE && rr == 0;  // lane 0 takes no x-edge
                if constexpr (HOMOG) {
                    float2 xn = qfma(first ? k1f[q] : k1[q], x[rr][q], tt);
                    if (RAGGED && !real[rr]) xn = first ? qmul(x[rr][q], k0) : x[rr][q];
                    x[rr + 1][q] = xn;
                    sm[rr][q] = !DD ? xn : first ? qfma(x[rr][q], k0, xn) : qadd(x[rr][q], xn);
                } else {
                    if (first) x[0][q] = qmul(x[0][q], k0);
                    const float s = f4(V[NA - 1][r / 4], r % 4);
                    const float2 rd = make_float2(qrcp(s + ab[q].x), qrcp(s + ab[q].y));
                    // DD: x[] holds the negative at odd cells
                    const float2 num =
                        (DD && (rr & 1)) ? qfma(x[rr][q], neg1, tt) : qadd(tt, x[rr][q]);
                    const float2 psi = qmul(num, rd);
                    sm[rr][q] = psi;
                    float2 xn = DD ? qfma((rr & 1) ? k1[q] : qneg(k1[q]), psi, x[rr][q])
                                   : qmul(k1[q], psi);
                    if (RAGGED && !real[rr]) xn = DD ? qneg(x[rr][q]) : x[rr][q];
                    x[rr + 1][q] = xn;
                }
            }
        }
        // the x-edges to the next lane, and from the last lane to the next warp
#pragma unroll
        for (int q = 0; q < N; ++q) {
            X[q].x = __shfl_up_sync(0xffffffffu, x[C][q].x, 1);
            X[q].y = __shfl_up_sync(0xffffffffu, x[C][q].y, 1);
        }
        if constexpr (EDGE) {
            if constexpr (N == 2)
                asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t"
                             "@q st.shared.v4.f32 [%0], {%1,%2,%3,%4};\n\t}" ::"r"(edge_out + eo),
                             "f"(x[C][0].x), "f"(x[C][0].y), "f"(x[C][N - 1].x),
                             "f"(x[C][N - 1].y), "r"((unsigned)feeds)
                             : "memory");
            else
                asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\t"
                             "@q st.shared.v2.f32 [%0], {%1,%2};\n\t}" ::"r"(edge_out + eo),
                             "f"(x[C][0].x), "f"(x[C][0].y), "r"((unsigned)feeds)
                             : "memory");
        }
        float v[NS][C];
#pragma unroll
        for (int rr = 0; rr < C; ++rr) {
            const int r = XNEG ? C - 1 - rr : rr;
            float2 m[MOM == 0 ? 1 : MOM];
#pragma unroll
            for (int q = 0; q < N; ++q) {
                const float2 s = sm[rr][q];
                if (!RAGGED || real[rr])
                    P[r][q] = DD ? qfma(ODD ? k2[q] : k2n[q], s, P[r][q])
                                 : EV && (held || past) ? P[r][q] : qmul(k2[q], s);
                if constexpr (MOM == 0) {  // psi of the two ordinates
                    const float2 pc = HOMOG ? qmul(kp[q], s) : s;
                    v[0][r] = (!RAGGED || real[rr]) ? pc.x : 0.f;
                    v[1][r] = (!RAGGED || real[rr]) ? pc.y : 0.f;
                }
#pragma unroll
                for (int k = 0; k < MOM; ++k) {
                    const float2 kw = k == 0 ? km[q] : k == 1 ? kmc[q] : kms[q];
                    m[k] = q == 0 ? qmul(kw, s) : qfma(kw, s, m[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < MOM; ++k) v[k][r] = (!RAGGED || real[rr]) ? m[k].x + m[k].y : 0.f;
        }
#pragma unroll
        for (int k = 0; k < NS; ++k)
            sts_cells<C>(own, k * kArrB + slot, v[k], EV ? on && !past : on);
#pragma unroll
        for (int q = 0; q < N; ++q) lk[par] = qfma(lx[q], x[C][q], lk[par]);
        if constexpr (MOM == 0) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                // (an empty slot's ordinate is the first again: not stored)
                const int l0 = k < it.n ? lim[0] : 0, l1 = k < it.n ? lim[CH - 1] : 0;
                const long long o = po + ord[k] * cells;
                psi_put<0>(A.psi, A.psi_split, o, D[k][0], frow - kRows, l0);
                if constexpr (CH == 2)
                    psi_put<kChunk1>(A.psi, A.psi_split, o, D[k][CH - 1], frow - kRows, l1);
            }
            po += rs;
        }
        if constexpr (MOM == 0) {  // the two ordinates' part of phi, in the place of psi
#pragma unroll
            for (int h = 0; h < CH; ++h) {
                float4 &d = D[0][h];
                const float4 &e = D[NS - 1][h];
                d.x = fmaf(km[0].y, e.x, km[0].x * d.x);
                d.y = fmaf(km[0].y, e.y, km[0].x * d.y);
                d.z = fmaf(km[0].y, e.z, km[0].x * d.z);
                d.w = fmaf(km[0].y, e.w, km[0].x * d.w);
            }
        }
#pragma unroll
        for (int m = 0; m < (MOM == 0 ? 1 : MOM); ++m) {
            ring_red<0>(acc + m * cells, D[m][0], frow - kRows, lim[0]);
            if constexpr (CH == 2)
                ring_red<kChunk1>(acc + m * cells, D[m][CH - 1], frow - kRows, lim[CH - 1]);
        }
        acc += rs;
        ++t;
    };

    // x inflow, scaled, of rows r0 .. r0 + 7: lane e takes ordinate e % G of row r0 + e / G
    // (32 is a multiple of G: the same ordinate in every pass)
    constexpr int kPre = (kGrp * G + 31) / 32;
    float pre[kPre], ix = 0.f, lw = 0.f;
    const float *in = nullptr;
    if (EDGE && w == 0 && A.inflow != nullptr) {
#pragma unroll
        for (int kk = 0; kk < G; ++kk)
            if (kk == lane % G) {
                if (kk < it.n) {
                    ix = inj_x[kk];
                    lw = A.ow[ord[kk]] * fabsf(A.oc[ord[kk]]) * gd.inv_dx;
                }
                in = A.inflow + (long long)ord[kk] * A.inflow_stride + (XNEG ? J : 0);
            }
    }
    auto fetch = [&](int r0) {
#pragma unroll
        for (int e = 0; e < kPre; ++e) {
            const int rr = r0 + (32 * e + lane) / G;
            float b = 0.f;
            if (32 * e + lane < kGrp * G && rr >= 0 && rr < J) b = in[yneg ? J - 1 - rr : rr];
            pre[e] = ix * b;
            leak -= (double)(lw * b);
        }
    };
    if (EDGE && w == 0 && A.inflow != nullptr) fetch(1 - kGrp);
    for (int g = 0; g < n_grp; ++g) {
        const int gl = g - kLag * w;  // the warp's own group of steps
        if (gl >= 0 && gl < n_grp_w) {
            if (EDGE && w == 0 && A.inflow != nullptr) {
                // x inflow of the rows this group reads (t + 1 .. t + 8), loaded a group ago
#pragma unroll
                for (int e = 0; e < kPre; ++e)
                    if (32 * e + lane < kGrp * G)
                        ((float *)(smem + (size_t)nw * NA * kArrB))
                            [(unsigned)(t + 1 + (32 * e + lane) / G) % kEdgeRows * G +
                             (32 * e + lane) % G] = pre[e];
                __syncwarp();
                fetch(t + 1 + kGrp);
            }
            if (gl == 0) {  // the first rows on their way
#pragma unroll 1
                for (int u = 0; u < kGrp; ++u) fill();
                acc += kGrp * rs;
                po += kGrp * rs;
                t = 0;
                load();
            } else if (t + kGrp > J || (EDGE && t < 32 && A.inflow != nullptr)) {
#pragma unroll 1
                for (int u = 0; u < kGrp; u += 2) {
                    step(std::true_type{}, std::false_type{});
                    step(std::true_type{}, std::true_type{});
                }
            } else {
#pragma unroll 1
                for (int u = 0; u < kGrp; u += 2) {
                    step(std::false_type{}, std::false_type{});
                    step(std::false_type{}, std::true_type{});
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float yv = (lk[h].x + lk[h].y) - lk_c;
                const float tt = lk_s + yv;
                lk_c = (tt - lk_s) - yv;
                lk_s = tt;
                lk[h] = qsplat(0.f);
            }
        }
        if (EDGE && nw > 1) __syncthreads();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (A.leak != nullptr) {  // the outgoing y-edges; one FP64 add per warp
        float lo = 0.f;
#pragma unroll
        for (int r = 0; r < C; ++r)
            if (on && col + r < gd.I)
#pragma unroll
                for (int q = 0; q < N; ++q) lo += wl[q].x * P[r][q].x + wl[q].y * P[r][q].y;
        // (the last row's step J - 1 + lane left -P if it was even)
        leak += (double)(DD && ((J - 1 + lane) & 1) == 0 ? -lo : lo) + ((double)lk_s - (double)lk_c);
#pragma unroll
        for (int dd = 16; dd > 0; dd >>= 1) leak += __shfl_xor_sync(0xffffffffu, leak, dd);
        if (lane == 0 && leak != 0.0)
            atomicAdd(A.leak + it.sample, leak * ((double)gd.dx * (double)gd.dy));
    }
}

template <int C, int G, int MOM, int SCHEME, bool HOMOG, bool EDGE, int MAXT>
__global__ void __launch_bounds__(MAXT) sweep2d_ring_kernel(const SweepArgs A)
{
    extern __shared__ __align__(1024) char ring_smem[];
    const SweepItem it = A.items[blockIdx.x];
    if (!A.active[it.sample]) return;
    // sigma_T varying: the grid from the table, whether it holds one or several
    GridDesc gd{A.I, A.J, A.NXP, A.inv_dx, A.inv_dy, A.dx, A.dy, 0, A.cells};
    if constexpr (!HOMOG) gd = A.gdesc[it.grid];
    if (A.stall) {  // test hook: every warp waits on a barrier that nothing completes
        __shared__ unsigned long long never;
        if (threadIdx.x == 0)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(ring_u32(&never))
                         : "memory");
        __syncthreads();
        if (!ring_never_wait(&never, A.wait_ns)) {
            if ((threadIdx.x & 31) == 0) atomicOr(A.err, 1);
            return;
        }
    }
    const bool ragged = gd.I % C != 0;
    if (it.quad & 1) {
        if (ragged) ring_item<C, G, MOM, SCHEME, HOMOG, true, true, EDGE>(A, gd, it, ring_smem);
        else ring_item<C, G, MOM, SCHEME, HOMOG, true, false, EDGE>(A, gd, it, ring_smem);
    } else {
        if (ragged) ring_item<C, G, MOM, SCHEME, HOMOG, false, true, EDGE>(A, gd, it, ring_smem);
        else ring_item<C, G, MOM, SCHEME, HOMOG, false, false, EDGE>(A, gd, it, ring_smem);
    }
}

template <int C, int G, int MOM, int SCHEME, bool HOMOG, bool EDGE>
cudaError_t ring_launch_k(const SweepArgs &a, int n_items, int nwarps, cudaStream_t st)
{
    const int bytes = ring_bytes(MOM, HOMOG, nwarps, G, C);
    auto k = sweep2d_ring_kernel<C, G, MOM, SCHEME, HOMOG, EDGE, EDGE ? 256 : 64>;
    if (bytes > 48 * 1024) {
        const cudaError_t e =
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
    }
    k<<<n_items, 32 * nwarps, bytes, st>>>(a);
    return cudaGetLastError();
}

template <int MOM, int SCHEME, bool HOMOG>
cudaError_t ring_launch(const SweepArgs &a, int n_items, int C, int G, cudaStream_t st)
{
    const int nw = (a.I + 32 * C - 1) / (32 * C);
    const bool inflow = a.inflow != nullptr;
    // items of one ordinate run on the two-ordinate kernel (the empty slot has weight zero)
#define RING_K(CC, GG)                                                                            \
    return nw > 1 || inflow ? ring_launch_k<CC, GG, MOM, SCHEME, HOMOG, true>(a, n_items, nw, st) \
                            : ring_launch_k<CC, GG, MOM, SCHEME, HOMOG, false>(a, n_items, nw, st)
    if constexpr (MOM != 0) {
        if (G == 4 && C == 8) RING_K(8, 4);
        if (G == 4) RING_K(4, 4);
    }
    if (C == 8) RING_K(8, 2);
    RING_K(4, 2);
#undef RING_K
}

}  // namespace
}  // namespace romk
