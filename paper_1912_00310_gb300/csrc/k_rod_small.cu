// k_rod_small.cu -- the resident engine's row kernel for the b = 2, 4, 8 rods of the paper's ladder
// (plan kind 3).
#include <algorithm>

#include "llg_internal.h"
#include "pair.cuh"
#include "physics.cuh"
#include "reduce.cuh"
#include "sweep32.cuh"

namespace llg {
namespace {

constexpr int kMaxThreads = 768;

// ------------------------------------------------------------------------------------------
// Row kernel (the b = 2 and 4 rods: 4x12x28, 2x6x14 cells, shapes at compile time) on pairs of cells
// with the packed FP32 instructions (pair.cuh).  A thread owns one x-row (fixed y, z) of a rod, NX / 2
// pairs of x-neighbours; it keeps the row's state, predictor, torque and thermal field in registers.
// The x-neighbours come from registers, the y- and z-neighbours, whole pairs, from shared memory, which
// holds per rod NX / 2 planes of pairs for the state M and for the predictor P: (xa, xb, ya, yb) in one
// array and (za, zb) in another, 24 bytes a pair, the rows of a plane in order with a line of zeros
// before the first plane and after every plane; the y faces are 0/1 weights, so that consecutive threads
// read consecutive entries without gaps (with ghost columns in y the b = 4 rod's neighbour loads took
// twice their wavefronts and shared memory was 78 % busy).  Per step: thermal fields and the predictor of
// the row into P, barrier, corrector into M, barrier.
//
// What bounds it: the heavy FMA pipe, 61 % busy with 608 b = 4 rods (the noise's 32-bit multiplies and
// half of every packed operation), and the two barriers' chains between (three warps a scheduler).
// 608 b = 4 rods 0.83 us a step (1.03 with one cell an instruction), 1216 1.58 (1.83), four alone 0.44
// (0.71); 152 b = 2 rods 1.55 (1.77), 256 2.98.  Threads without a row go through the work on row 0's
// places with values of no meaning and store nothing: with branches around it its parts cannot be
// interleaved (608 b = 4 rods 0.86, four 0.47, 256 b = 2 rods 3.31).  Drawing the next step's noise beside the corrector: 608 b = 4 rods 0.82,
// but 1216 1.61 and 256 b = 2 rods 3.50.
// The b = 2 rod's instance has 126 registers, so that one CTA of 352 threads fits an SM; where there are more
// rods than SMs, or jobs of a batch beside them, an instance of 80 (CTAS = 2) runs two side by side: 256 rods
// 3.08 -> 2.98 us a step, 512 6.16 -> 5.81, 1024 10.76 -> 10.01, with dispersed axes (spills) 3.33 -> 3.26 and
// 6.65 -> 6.34 at 512; alone on its SM a rod takes 1.55 us with the first and 1.72 with the second.
// ------------------------------------------------------------------------------------------
// CTAS: CTAs to an SM that the registers have to allow (0: as the compiler likes).
template <int NX, int NY, int NZ, int SHAPE, bool AX, int MAXT, int CTAS>
__global__ void __launch_bounds__(MAXT, CTAS) rod_rows_kernel(KParams p, float *__restrict__ m_glob, int n_real,
                                                        int rods_per_cta, long long step0, int n_steps,
                                                        float *__restrict__ samples, int *__restrict__ status)
{
    constexpr int NXP = NX / 2;                    // pairs of a row
    constexpr int PL = (NZ + 1) * NY;              // a plane and the ghost line after it
    constexpr int ROD = NXP * PL + NY;             // entries of one buffer of one rod
    constexpr int ROWS = NY * NZ, NCELL = NX * ROWS;
    static_assert(NX % 2 == 0, "rows of pairs");
    extern __shared__ __align__(16) unsigned char rsm[];
    const int rod0 = blockIdx.x * rods_per_cta;
    const int nrod = min(rods_per_cta, n_real - rod0);
    const int tot = rods_per_cta * ROD;
    ulonglong2 *MA = reinterpret_cast<ulonglong2 *>(rsm), *PA = MA + tot;
    pair_t *MB = reinterpret_cast<pair_t *>(PA + tot), *PB = MB + tot;
    const int T = blockDim.x;
    for (int i = threadIdx.x; i < tot; i += T) {
        MA[i] = PA[i] = make_ulonglong2(0ull, 0ull);
        MB[i] = PB[i] = 0ull;
    }
    __syncthreads();
    // this thread's row
    const int t0 = threadIdx.x;
    const bool act = t0 < nrod * ROWS;
    const int rl = act ? t0 / ROWS : 0, row = act ? t0 - rl * ROWS : 0;  // rod within the CTA, row y + NY z
    const int y = row % NY;
    const int q = rl * ROD + NY + row;             // entry of the row's first pair
    const pair_t wm = both(y > 0 ? 1.f : 0.f), wp = both(y < NY - 1 ? 1.f : 0.f);
    auto load = [](const ulonglong2 *A, const pair_t *B, int i) {
        const ulonglong2 v = A[i];
        return Pair3{v.x, v.y, B[i]};
    };
    auto store = [](ulonglong2 *A, pair_t *B, int i, Pair3 v) {
        A[i] = make_ulonglong2(v.x, v.y);
        B[i] = v.z;
    };
    Pair3 m[NXP], u[NXP];
#pragma unroll
    for (int X = 0; X < NXP; ++X) {
        m[X] = u[X] = zero_p3();
        if (act) {
            const size_t c = (size_t)(rod0 + rl) * NCELL + row * NX + 2 * X;
            const float *g = m_glob + 3 * c;
            m[X] = pair3(make_float3(g[0], g[1], g[2]), make_float3(g[3], g[4], g[5]));
            store(MA, MB, q + X * PL, m[X]);
            if constexpr (AX) u[X] = pair3(xyz(__ldg(p.axis + c)), xyz(__ldg(p.axis + c + 1)));
        }
    }
    const PairCoeffs cf = pair_coeffs(p);
    const PhiloxKeys keys = philox_keys(p.seed, p.real0 + (uint32_t)(rod0 + rl));
    const unsigned long long row_m0 = (unsigned long long)kPhiloxM0 * (uint32_t)(row * NX);
    __syncthreads();

    FieldAhead<SHAPE> field;
    field.init(step0);
    float Hn = field.next(p);
    const long long se = p.sample_every;
    const bool sampling = samples && se > 0;
    long long k_next = sampling ? step0 / se + 1 : 0;
    int to_sample = sampling ? (int)(k_next * se - step0) : -1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = T >> 5;

    // x- + x+ of pair X of a row
    auto x_sum = [](const Pair3 *v, int X) {
        const float3 none = make_float3(0.f, 0.f, 0.f);
        const float3 l = X > 0 ? hi3(v[X > 0 ? X - 1 : 0]) : none, r = X + 1 < NXP ? lo3(v[X + 1 < NXP ? X + 1 : X]) : none;
        const float3 a = X > 0 ? add3(l, hi3(v[X])) : hi3(v[X]), b = X + 1 < NXP ? add3(lo3(v[X]), r) : lo3(v[X]);
        return pair3(a, b);
    };
    auto neighbour_sum = [&](const Pair3 *v, int X, const ulonglong2 *A, const pair_t *B) {
        const int i = q + X * PL;
        Pair3 nb = axpy_p3(wm, load(A, B, i - 1), x_sum(v, X));
        nb = axpy_p3(wp, load(A, B, i + 1), nb);
        nb = add_p3(nb, load(A, B, i - NY));
        return add_p3(nb, load(A, B, i + NY));
    };
    unsigned long long n = (unsigned long long)step0;
    for (int s = 0; s < n_steps; ++s, ++n) {
        const float Hn1 = field.next(p);
        Pair3 t[NXP], s0[NXP], h[NXP];
        const pair_t H0 = both(Hn), H1 = both(Hn1);
        const PhiloxStep now = philox_step(keys, n);
#pragma unroll
        for (int X = 0; X < NXP; ++X) {
            h[X] = thermal_field_p3(keys, now, row_m0 + (unsigned long long)kPhiloxM0 * (2 * X), p.sigma_bm);
            const Pair3 nb = neighbour_sum(m, X, MA, MB);
            s0[X] = llg_torque_p3(m[X], effective_field_p3<AX>(nb, m[X], h[X], cf, H0, u[X]), cf.alpha);
            t[X] = normalised_p3(axpy_p3(cf.neg_dt_g1, s0[X], m[X]));
            if (act) store(PA, PB, q + X * PL, t[X]);
        }
        __syncthreads();
#pragma unroll
        for (int X = 0; X < NXP; ++X) {
            const Pair3 nb = neighbour_sum(t, X, PA, PB);
            const Pair3 sv = llg_torque_add_p3(s0[X], t[X], effective_field_p3<AX>(nb, t[X], h[X], cf, H1, u[X]), cf.alpha);
            m[X] = normalised_p3(axpy_p3(cf.neg_hdt_g1, sv, m[X]));
            if (act) store(MA, MB, q + X * PL, m[X]);
        }
        __syncthreads();
        Hn = Hn1;
        if (--to_sample == 0) {
            // M holds the state after step n; the next phase only reads M until the barrier that
            // precedes its next write
            to_sample = (int)se;
            const long long k = k_next++;
            if (k < p.n_samples) {
                for (int r = warp; r < nrod; r += nwarps) {
                    const pair_t *B = MB + r * ROD + NY;
                    float part = 0.f;
                    for (int c = lane; c < NCELL; c += 32) {
                        const int cx = c % NX, cr = c / NX;
                        const pair_t v = B[(cx >> 1) * PL + cr];
                        part += cx & 1 ? hi2(v) : lo2(v);
                    }
                    const float mean = warp_cell_mean(part, NCELL);
                    if (lane == 0) {
                        samples[(size_t)(rod0 + r) * p.n_samples + k] = mean;
                        if (!isfinite(mean)) atomicOr(status, 1);
                    }
                }
            }
        }
    }
    if (act) {
#pragma unroll
        for (int X = 0; X < NXP; ++X) {
            const size_t c = (size_t)(rod0 + rl) * NCELL + row * NX + 2 * X;
            float *g = m_glob + 3 * c;
            const float3 a = lo3(m[X]), b = hi3(m[X]);
            g[0] = a.x;
            g[1] = a.y;
            g[2] = a.z;
            g[3] = b.x;
            g[4] = b.y;
            g[5] = b.z;
        }
    }
}

// The same for rods one cell wide (the b = 8 rod, 1x3x7 cells): a thread is a cell, there are no pairs
// of neighbours to take, and several rods share a CTA's warps.  Two rods to a packed thread measured
// slower (four alone 0.47 us a step against 0.37, 4096 0.84 against 0.85): half the warps hide less of
// the chain.  Float4 cells in the row kernel's gapless order, and no branches around the work either:
// 4096 rods 0.71 us a step (0.77 with them).
template <int NY, int NZ, int SHAPE, bool AX, int MAXT>
__global__ void __launch_bounds__(MAXT) rod_cells_kernel(KParams p, float *__restrict__ m_glob, int n_real,
                                                         int rods_per_cta, long long step0, int n_steps,
                                                         float *__restrict__ samples, int *__restrict__ status)
{
    constexpr int NCELL = NY * NZ, ROD = NCELL + 2 * NY;
    extern __shared__ __align__(16) float4 csm[];
    const int rod0 = blockIdx.x * rods_per_cta;
    const int nrod = min(rods_per_cta, n_real - rod0);
    const int tot = rods_per_cta * ROD;
    float4 *M = csm, *P = csm + tot;
    const int T = blockDim.x;
    for (int i = threadIdx.x; i < 2 * tot; i += T) csm[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    const int t0 = threadIdx.x;
    const bool act = t0 < nrod * NCELL;
    const int rl = act ? t0 / NCELL : 0, c = act ? t0 - rl * NCELL : 0;
    const int y = c % NY, q = rl * ROD + NY + c;
    const float wm = y > 0 ? 1.f : 0.f, wp = y < NY - 1 ? 1.f : 0.f;
    float *g = m_glob + ((size_t)(rod0 + rl) * NCELL + c) * 3;
    float3 m = make_float3(0.f, 0.f, 0.f), u = make_float3(0.f, 0.f, 1.f);
    if (act) {
        m = make_float3(g[0], g[1], g[2]);
        M[q] = pad4(m);
        if constexpr (AX) u = xyz(__ldg(p.axis + (size_t)(rod0 + rl) * NCELL + c));
    }
    const PhiloxKeys keys = philox_keys(p.seed, p.real0 + (uint32_t)(rod0 + rl));
    const unsigned long long cell_m0 = (unsigned long long)kPhiloxM0 * (uint32_t)c;
    __syncthreads();
    FieldAhead<SHAPE> field;
    field.init(step0);
    float Hn = field.next(p);
    const long long se = p.sample_every;
    const bool sampling = samples && se > 0;
    long long k_next = sampling ? step0 / se + 1 : 0;
    int to_sample = sampling ? (int)(k_next * se - step0) : -1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = T >> 5;
    // the neighbour sum in every engine's order (x- + x+ = 0)
    auto neighbour_sum = [&](const float4 *A) {
        const float3 l = xyz(A[q - 1]);
        float3 nb = make_float3(wm * l.x, wm * l.y, wm * l.z);
        nb = axpy(wp, xyz(A[q + 1]), nb);
        nb = add3(nb, xyz(A[q - NY]));
        return add3(nb, xyz(A[q + NY]));
    };
    unsigned long long n = (unsigned long long)step0;
    for (int s = 0; s < n_steps; ++s, ++n) {
        const float Hn1 = field.next(p);
        const float3 h = box_muller3(philox4x32_10(keys, philox_step(keys, n), cell_m0), p.sigma_bm);
        const float3 s0 = llg_torque(m, effective_field_sel<AX>(neighbour_sum(M), m, h, p, Hn, u), p.alpha);
        const float3 t = normalised(axpy(p.neg_dt_g1, s0, m));
        if (act) P[q] = pad4(t);
        __syncthreads();
        const float3 sv = llg_torque_add(s0, t, effective_field_sel<AX>(neighbour_sum(P), t, h, p, Hn1, u), p.alpha);
        m = normalised(axpy(p.neg_hdt_g1, sv, m));
        if (act) M[q] = pad4(m);
        __syncthreads();
        Hn = Hn1;
        if (--to_sample == 0) {
            to_sample = (int)se;
            const long long k = k_next++;
            if (k < p.n_samples) {
                for (int r = warp; r < nrod; r += nwarps) {
                    float part = 0.f;
                    for (int i = lane; i < NCELL; i += 32) part += M[r * ROD + NY + i].z;
                    const float mean = warp_cell_mean(part, NCELL);
                    if (lane == 0) {
                        samples[(size_t)(rod0 + r) * p.n_samples + k] = mean;
                        if (!isfinite(mean)) atomicOr(status, 1);
                    }
                }
            }
        }
    }
    if (act) {
        g[0] = m.x;
        g[1] = m.y;
        g[2] = m.z;
    }
}

// One such rod to a CTA of one warp, for ensembles that leave the SMs few warps: its barriers are the
// warp's, and each step draws the next one's noise, whose chain is as long as a half-step's, beside the
// corrector.  What bounds it is that chain: 1 to 608 rods 0.25 us a step (the kernel above 0.30 alone,
// 0.37 before it was free of branches), 1216 0.33 (0.37), 2432 0.52 (0.47).
template <int NY, int NZ, int SHAPE, bool AX>
__global__ void __launch_bounds__(32) rod_warp_kernel(KParams p, float *__restrict__ m_glob, int n_real, int rods_per_cta,
                                                      long long step0, int n_steps, float *__restrict__ samples,
                                                      int *__restrict__ status)
{
    constexpr int NCELL = NY * NZ, ROD = NCELL + 2 * NY;
    __shared__ float4 M[ROD], P[ROD];
    const int rod = blockIdx.x, lane = threadIdx.x;
    for (int i = lane; i < ROD; i += 32) M[i] = P[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
    const bool act = lane < NCELL;
    const int c = act ? lane : 0, y = c % NY, q = NY + c;
    const float wm = y > 0 ? 1.f : 0.f, wp = y < NY - 1 ? 1.f : 0.f;
    float *g = m_glob + ((size_t)rod * NCELL + c) * 3;
    float3 m = make_float3(g[0], g[1], g[2]), u = make_float3(0.f, 0.f, 1.f);
    if (act) M[q] = pad4(m);
    if constexpr (AX) u = xyz(__ldg(p.axis + (size_t)rod * NCELL + c));
    const PhiloxKeys keys = philox_keys(p.seed, p.real0 + (uint32_t)rod);
    const unsigned long long cell_m0 = (unsigned long long)kPhiloxM0 * (uint32_t)c;
    __syncwarp();
    FieldAhead<SHAPE> field;
    field.init(step0);
    float Hn = field.next(p);
    const long long se = p.sample_every;
    const bool sampling = samples && se > 0;
    long long k_next = sampling ? step0 / se + 1 : 0;
    int to_sample = sampling ? (int)(k_next * se - step0) : -1;
    auto neighbour_sum = [&](const float4 *A) {
        const float3 l = xyz(A[q - 1]);
        float3 nb = make_float3(wm * l.x, wm * l.y, wm * l.z);
        nb = axpy(wp, xyz(A[q + 1]), nb);
        nb = add3(nb, xyz(A[q - NY]));
        return add3(nb, xyz(A[q + NY]));
    };
    auto bits = [&](unsigned long long n) { return philox4x32_10(keys, philox_step(keys, n), cell_m0); };
    unsigned long long n = (unsigned long long)step0;
    float3 h = box_muller3(bits(n), p.sigma_bm);
    for (int s = 0; s < n_steps; ++s) {
        ++n;
        const float Hn1 = field.next(p);
        const float3 s0 = llg_torque(m, effective_field_sel<AX>(neighbour_sum(M), m, h, p, Hn, u), p.alpha);
        const float3 t = normalised(axpy(p.neg_dt_g1, s0, m));
        if (act) P[q] = pad4(t);
        __syncwarp();
        const float3 next = box_muller3(bits(n), p.sigma_bm);
        const float3 sv = llg_torque_add(s0, t, effective_field_sel<AX>(neighbour_sum(P), t, h, p, Hn1, u), p.alpha);
        m = normalised(axpy(p.neg_hdt_g1, sv, m));
        if (act) M[q] = pad4(m);
        __syncwarp();
        h = next;
        Hn = Hn1;
        if (--to_sample == 0) {
            to_sample = (int)se;
            const long long k = k_next++;
            if (k < p.n_samples) {
                const float mean = warp_cell_mean(act ? m.z : 0.f, NCELL);
                if (lane == 0) {
                    samples[(size_t)rod * p.n_samples + k] = mean;
                    if (!isfinite(mean)) atomicOr(status, 1);
                }
            }
        }
    }
    if (act) {
        g[0] = m.x;
        g[1] = m.y;
        g[2] = m.z;
    }
}

template <typename K>
cudaError_t launch(K kern, const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0, int n_steps,
                   float *samples, int *status, cudaStream_t st)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem_bytes);
    if (e != cudaSuccess) return e;
    kern<<<plan.ctas, plan.threads, plan.smem_bytes, st>>>(p, m, n_real, plan.rods_per_cta, step0, n_steps, samples,
                                                           status);
    return cudaGetLastError();
}

template <int NY, int NZ, int MAXT>
cudaError_t launch_cells(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0, int n_steps,
                         float *samples, int *status, cudaStream_t st)
{
    if (plan.rods_per_cta == 1) {
        if (p.axis)
            return p.shape == 1 ? launch(rod_warp_kernel<NY, NZ, 1, true>, p, plan, m, n_real, step0, n_steps, samples, status, st)
                                : launch(rod_warp_kernel<NY, NZ, 0, true>, p, plan, m, n_real, step0, n_steps, samples, status, st);
        return p.shape == 1 ? launch(rod_warp_kernel<NY, NZ, 1, false>, p, plan, m, n_real, step0, n_steps, samples, status, st)
                            : launch(rod_warp_kernel<NY, NZ, 0, false>, p, plan, m, n_real, step0, n_steps, samples, status, st);
    }
    if (p.axis)
        return p.shape == 1 ? launch(rod_cells_kernel<NY, NZ, 1, true, MAXT>, p, plan, m, n_real, step0, n_steps, samples,
                                     status, st)
                            : launch(rod_cells_kernel<NY, NZ, 0, true, MAXT>, p, plan, m, n_real, step0, n_steps, samples,
                                     status, st);
    return p.shape == 1 ? launch(rod_cells_kernel<NY, NZ, 1, false, MAXT>, p, plan, m, n_real, step0, n_steps, samples,
                                 status, st)
                        : launch(rod_cells_kernel<NY, NZ, 0, false, MAXT>, p, plan, m, n_real, step0, n_steps, samples,
                                 status, st);
}

template <int NX, int NY, int NZ, int MAXT, int CTAS>
cudaError_t launch_rows_shaped(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0,
                               int n_steps, float *samples, int *status, cudaStream_t st)
{
#define LLG_R(S, AXV) \
    launch(rod_rows_kernel<NX, NY, NZ, S, AXV, MAXT, CTAS>, p, plan, m, n_real, step0, n_steps, samples, status, st)
    if (p.axis) return p.shape == 1 ? LLG_R(1, true) : LLG_R(0, true);
    return p.shape == 1 ? LLG_R(1, false) : LLG_R(0, false);
#undef LLG_R
}

// the rows kernel's shapes: b = 2, 4, 8 rods (x-rows of 4, 2, 1 cells)
int rows_shape(const KParams &p)
{
    if (p.nx == 4 && p.ny == 12 && p.nz == 28) return 2;
    if (p.nx == 2 && p.ny == 6 && p.nz == 14) return 4;
    if (p.nx == 1 && p.ny == 3 && p.nz == 7) return 8;
    return 0;
}

}  // namespace

bool rows_supported(const KParams &p)
{
    const long long period = p.shape == 1 ? p.period : 2 * p.n_half;
    return rows_shape(p) != 0 && (p.shape == 0 || p.shape == 1) && period < (1LL << 31) &&
           p.sample_every < (1LL << 31);
}

// Largest CTA of the rows kernel: 768 threads (80 registers) for rows of 1 or 2 cells, 384 (168
// registers) for the 4-cell rows of the b = 2 rod.
int rows_max_threads(const KParams &p) { return p.nx == 4 ? 384 : kMaxThreads; }

// What a request for rods per CTA may ask for (ghost-padded float4 rows); rows_smem_bytes, less, is
// what the launch takes.
size_t rows_rod_bytes(const KParams &p)
{
    return (size_t)2 * p.nx * (p.nz + 2) * (p.ny + 2) * sizeof(float4);
}

size_t rows_smem_bytes(const KParams &p, int rods)
{
    if (p.nx == 1) return 32 * (size_t)rods * (p.nz + 2) * p.ny;
    return 48 * (size_t)rods * ((size_t)(p.nx / 2) * (p.nz + 1) * p.ny + p.ny);
}

cudaError_t rows_advance(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0, int n_steps,
                         float *samples, int *status, cudaStream_t st)
{
    switch (rows_shape(p)) {
        case 2:
            if (plan.crowded)
                return launch_rows_shaped<4, 12, 28, 384, 2>(p, plan, m, n_real, step0, n_steps, samples, status, st);
            return launch_rows_shaped<4, 12, 28, 384, 0>(p, plan, m, n_real, step0, n_steps, samples, status, st);
        case 4:
            return launch_rows_shaped<2, 6, 14, kMaxThreads, 0>(p, plan, m, n_real, step0, n_steps, samples, status, st);
        case 8:
            return launch_cells<3, 7, kMaxThreads>(p, plan, m, n_real, step0, n_steps, samples, status, st);
        default:
            return cudaErrorInvalidValue;
    }
}

// Largest CTA that a request for cpt cells per thread may ask for (the b = 4 and b = 8 rods 768 / cpt
// threads, other grids 768); what it asks for beyond that is refused.
int twophase_max_threads(const KParams &p, int cpt)
{
    const bool b4 = p.nx == 2 && p.ny == 6 && p.nz == 14, b8 = p.nx == 1 && p.ny == 3 && p.nz == 7;
    const bool shaped = (b4 || b8) && sweep_fits_32(p) && p.sample_every < (1LL << 31);
    return shaped ? kMaxThreads / cpt : kMaxThreads;
}

}  // namespace llg
