// k_rod.cu -- the resident engine: whole rods live in shared memory for an entire launch of
// thousands of Heun steps of Eq. 1, and only the sampled M(H) values reach HBM.
//
// The kernels, chosen by rod size and ensemble (rod_plan):
//
//  rod_zpairs_kernel (rods whose state and predictor state both fit), in k_rod_zpairs.cu; for the
//      b = 2, 4, 8 rods of the paper's ladder rod_rows_kernel, rod_cells_kernel and rod_warp_kernel, in
//      k_rod_small.cu.  One or several rods per CTA, two barriers a step.
//
//  rod_split_kernel (ensembles of fewer rods than SMs, where that is faster and the launch has the GPU to
//      itself), in k_rod_split.cu: a rod cut along z over a cluster of CTAs.
//
//  rod_pipelined_kernel (the b = 1 rod, 8x24x56 = 10752 cells: M alone is 129 KB, M and a full
//      predictor copy do not fit).  One rod per CTA.  Each thread owns rows along x (fixed y, z);
//      the CTA sweeps the x planes in lock step, computing the predictor at plane x and the
//      corrector at plane x-1 in the same iteration, so only two planes of predictor state are
//      ever needed (double-buffered by the parity of the plane counter).  The x-neighbours come
//      from registers, the y- and z-neighbours from shared memory.  When nx >= 3 the corrector of
//      the last plane of step n shares its iteration with the predictor of plane 0 of step n+1,
//      so every iteration does both halves of the work: nx barriers per step.
//
//  rod_pairs_kernel (k_rod_pairs.cu): the same schedule for rods eight cells wide (the b = 1 rod), on
//      pairs of x-neighbours with packed arithmetic and a balanced schedule over the SMs.
//
// The thread count of the plane-pipelined kernels balances the rows over the SM's four
// schedulers (pipelined_threads).  The dispersed-axis mode (per-cell easy axes in global memory)
// runs the AX instances: of the two-phase kernel, of the runtime-size plane-pipelined kernel and,
// for the b = 1 rod, of the pair kernel.
//
// All kernels add the neighbours in the order x-, x+, y-, y+, z-, z+ with exact zeros for
// missing ones and use the same physics.cuh arithmetic as the plain engine, so all engines
// produce bitwise-identical trajectories.  Samples use the canonical warp reduction (reduce.cuh).
#include <algorithm>
#include <cstring>

#include "llg_internal.h"
#include "physics.cuh"
#include "reduce.cuh"
#include "rod_threads.h"

namespace llg {
namespace {

// At most 768 threads per CTA leaves 85 registers per thread, enough for the per-cell Heun
// state (predictor accumulator and thermal field) of two cells or rows without spilling.
constexpr int kMaxThreads = 768;

__device__ __forceinline__ float3 zero3() { return make_float3(0.f, 0.f, 0.f); }

// ------------------------------------------------------------------------------------------
// plane-pipelined kernel
// ------------------------------------------------------------------------------------------
// Shared memory (float4 = x, y, z, 0): M[nx][PL] (state) and S[2][PL] (predictor planes),
// PL = (nz + 2) * ny: each plane holds the rows (y, z) at offset q = (z + 1) * ny + y, with zero
// ghost lines at z = -1 and z = nz; the y faces are handled by 0/1 weights.
template <int R, bool AX>
__global__ void __launch_bounds__(pipelined_max_threads(R), 1) rod_pipelined_kernel(KParams p, float *__restrict__ m_glob,
                                                               long long step0, long long n_steps,
                                                               float *__restrict__ samples,
                                                               int *__restrict__ status)
{
    extern __shared__ float4 sm4[];
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int rows = ny * nz;
    const int PL = (nz + 2) * ny;
    float4 *M = sm4;
    float4 *S = sm4 + nx * PL;
    const int T = blockDim.x;
    const int rod = blockIdx.x;
    const int ncell = p.ncells;

    for (int i = threadIdx.x; i < (nx + 2) * PL; i += T) sm4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    {
        const float *g = m_glob + (size_t)rod * ncell * 3;
        for (int c = threadIdx.x; c < ncell; c += T) {
            const int x = c % nx, rr = c / nx;
            M[x * PL + ny + rr] = make_float4(g[3 * (size_t)c], g[3 * (size_t)c + 1], g[3 * (size_t)c + 2], 0.f);
        }
    }

    int q[R];
    float wm[R], wp[R];
    bool act[R];
    uint32_t cbase[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const int r = threadIdx.x + j * T;
        act[j] = r < rows;
        const int rr = act[j] ? r : 0;
        const int y = rr % ny;
        q[j] = ny + rr;
        wm[j] = y > 0 ? 1.f : 0.f;
        wp[j] = y < ny - 1 ? 1.f : 0.f;
        cbase[j] = (uint32_t)(rr * nx);  // cell index x + nx * (y + ny * z), rr = y + ny * z
    }
    const PhiloxKeys keys = philox_keys(p.seed, p.real0 + (uint32_t)rod);
    const float4 *axr = AX ? p.axis + (size_t)rod * ncell : nullptr;  // this rod's easy axes

    // carried per row: m(x-1), m(x); m~(x-2), m~(x-1), the torque s0(x-1) and the thermal field h(x-1)
    float3 mprev[R], mcur[R], mta[R], mtb[R], s0c[R], hth[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
        mprev[j] = mcur[j] = mta[j] = mtb[j] = s0c[j] = hth[j] = zero3();
    }
    __syncthreads();

    const bool merged = nx >= 3;
    bool pa = n_steps > 0, ca = false;
    long long sp = 0, sc = 0;
    int xp = 0, xc = 0;
    Sweep fpred, fcorr;
    fpred.init(step0, p);
    fcorr.init(step0 + 1, p);
    float Hp = fpred.value(), Hc = fcorr.value();
    const long long se = p.sample_every;
    long long next_sample = (samples && se > 0) ? (step0 / se + 1) * se : -1;
    const int lane = threadIdx.x & 31;

    while (pa || ca) {
        float3 mt_new[R], s0_new[R], h_new[R], mcorr[R];
#pragma unroll
        for (int j = 0; j < R; ++j) mcorr[j] = mprev[j];  // the state at the corrector's plane
        if (pa) {
            const unsigned long long n = (unsigned long long)(step0 + sp);
            const float4 *Mp = M + xp * PL;
            float4 *Sw = S + (int)((sp * nx + xp) & 1) * PL;
            const bool has_next = xp + 1 < nx;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (!act[j]) continue;
                const int qq = q[j];
                if (xp == 0) mcur[j] = xyz(Mp[qq]);
                const float3 mnext = has_next ? xyz(Mp[qq + PL]) : zero3();
                h_new[j] = thermal_field(keys, cbase[j] + (uint32_t)xp, n, p.sigma_bm);
                float3 nb = add3(xp == 0 ? zero3() : mprev[j], mnext);
                nb = axpy(wm[j], xyz(Mp[qq - 1]), nb);
                nb = axpy(wp[j], xyz(Mp[qq + 1]), nb);
                nb = add3(nb, xyz(Mp[qq - ny]));
                nb = add3(nb, xyz(Mp[qq + ny]));
                const float3 u = AX ? xyz(__ldg(axr + cbase[j] + xp)) : zero3();
                const float3 H = effective_field_sel<AX>(nb, mcur[j], h_new[j], p, Hp, u);
                const float3 s0 = llg_torque(mcur[j], H, p.alpha);
                mt_new[j] = normalised(axpy(p.neg_dt_g1, s0, mcur[j]));
                s0_new[j] = s0;
                Sw[qq] = pad4(mt_new[j]);
                mprev[j] = mcur[j];
                mcur[j] = mnext;
            }
        }
        if (ca) {
            const float4 *Sr = S + (int)((sc * nx + xc) & 1) * PL;
            float4 *Mw = M + xc * PL;
            const bool has_next = xc + 1 < nx;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (!act[j]) continue;
                const int qq = q[j];
                const float3 tnext = has_next ? mt_new[j] : zero3();
                float3 nb = add3(mta[j], tnext);
                nb = axpy(wm[j], xyz(Sr[qq - 1]), nb);
                nb = axpy(wp[j], xyz(Sr[qq + 1]), nb);
                nb = add3(nb, xyz(Sr[qq - ny]));
                nb = add3(nb, xyz(Sr[qq + ny]));
                const float3 u = AX ? xyz(__ldg(axr + cbase[j] + xc)) : zero3();
                const float3 H = effective_field_sel<AX>(nb, mtb[j], hth[j], p, Hc, u);
                const float3 s = llg_torque_add(s0c[j], mtb[j], H, p.alpha);
                Mw[qq] = pad4(normalised(axpy(p.neg_hdt_g1, s, mcorr[j])));
            }
        }
        if (pa) {
#pragma unroll
            for (int j = 0; j < R; ++j) {
                mta[j] = xp == 0 ? zero3() : mtb[j];
                mtb[j] = mt_new[j];
                s0c[j] = s0_new[j];
                hth[j] = h_new[j];
            }
        }
        __syncthreads();
        if (ca && xc == nx - 1 && step0 + sc + 1 == next_sample) {
            const long long k = next_sample / se;
            if (k < p.n_samples && threadIdx.x < 32) {
                float part = 0.f;
                for (int c = lane; c < ncell; c += 32) part += M[(c % nx) * PL + ny + c / nx].z;
                const float mean = warp_cell_mean(part, ncell);
                if (lane == 0) {
                    samples[(size_t)rod * p.n_samples + k] = mean;
                    if (!isfinite(mean)) atomicOr(status, 1);
                }
            }
            next_sample += se;
            __syncthreads();
        }
        // advance the schedule; the corrector takes the predictor's old position
        const bool old_pa = pa;
        const long long old_sp = sp;
        const int old_xp = xp;
        if (merged) {
            if (pa && ++xp == nx) {
                xp = 0;
                ++sp;
                fpred.inc();
                Hp = fpred.value();
                pa = sp < n_steps;
            }
        } else if (pa) {
            if (++xp == nx) pa = false;  // one corrector-only iteration closes the step
        } else if (ca) {
            ++sp;
            xp = 0;
            fpred.inc();
            Hp = fpred.value();
            pa = sp < n_steps;
        }
        ca = old_pa;
        if (old_pa) {
            if (old_sp != sc) {
                sc = old_sp;
                fcorr.inc();
                Hc = fcorr.value();
            }
            xc = old_xp;
        }
    }

    {
        float *g = m_glob + (size_t)rod * ncell * 3;
        for (int c = threadIdx.x; c < ncell; c += T) {
            const float4 v = M[(c % nx) * PL + ny + c / nx];
            g[3 * (size_t)c] = v.x;
            g[3 * (size_t)c + 1] = v.y;
            g[3 * (size_t)c + 2] = v.z;
        }
    }
}

int round_warp(int n) { return (n + 31) / 32 * 32; }

}  // namespace

// Measured, us: b = 2, 4, 8 rods 1.63, 0.44, 0.25; two-phase rods of 58, 312, 819 and 1265 cells 0.36, 0.74, 1.54 and
// 2.15; the b = 1 rod 11.2; on the runtime-size pipelined kernel 5.4 for 2880 cells.
double one_sm_us(const KParams &p, int kind)
{
    if (kind == 3) return 0.29 + 0.001 * p.ncells;
    if (kind == 1) return p.ncells <= 400 ? 0.33 + 0.0014 * p.ncells : 0.42 + 0.0013 * p.ncells;
    return pairs_supported(p) ? 0.3 + 0.00101 * p.ncells : 0.00186 * p.ncells;
}

bool rod_plan(const KParams &p, int n_real, int dev, RodPlan *plan, int force_kind, int force_rods,
              int force_rows, int force_cpt, bool may_cut, bool in_batch)
{
    int smem_optin = 0, nsm = 0;
    if (cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return false;
    if (p.periodic != 0) return false;  // rods have free faces
    const size_t rod_pad = (size_t)(p.nx + 2) * (p.ny + 2) * (p.nz + 2);
    const size_t rod_bytes = rod_pad * 2 * sizeof(float4);
    const int rows = p.ny * p.nz;
    const size_t PL = (size_t)(p.nz + 2) * p.ny;
    const size_t pipe_bytes = ((size_t)p.nx + 2) * PL * sizeof(float4);
    const bool twophase_fits = rod_bytes <= (size_t)smem_optin && p.ncells <= 4 * kMaxThreads;
    const bool pipelined_fits = pipe_bytes <= (size_t)smem_optin && rows <= 4 * 672;
    // Default (measured on GB300): the b = 2, 4, 8 rods of the paper's ladder use the row kernel (four
    // b = 4 rods 0.44 us a step against 0.60 with the two-phase kernel, 608 0.82 against 1.09); other
    // rods whose pairs fit one to a thread, or two where the rod is not eight cells wide, the two-phase
    // kernel with one rod per CTA (152 rods of 5x11x23 cells 2.11 us against 3.09 with the plane-pipelined
    // one, 7x9x13 1.51 against 3.42, 9x16x20 4.28 against 6.49, 16x10x12 2.68 against 7.67; 456 rods of
    // 7x12x20 7.99 against 9.06); larger rods the plane-pipelined kernels (12x12x21 7.25 against 8.80), and
    // eight-wide rods of two pairs a thread their own (8x24x15 4.09 against 4.29, 456 rods of 8x16x20 9.55
    // against 10.95).
    int kind = force_kind;
    if (kind == 0) {
        RodPlan one{};
        // (a request for a launch shape is the kernel's that it was always made to)
        const bool few_cells = twophase_fits && p.ncells <= kMaxThreads;
        const bool few_pairs = twophase_fits && force_rods == 0 && force_rows == 0 && force_cpt == 0 &&
                               p.sample_every < (1LL << 31) && twophase_shape(p, 1, &one) &&
                               one.pairs_per_thread <= (pairs_supported(p) ? 1 : 2);
        kind = rows_supported(p) ? 3 : (few_cells || few_pairs ? 1 : (pipelined_fits ? 2 : 1));
        // few rods: several SMs to each, where that is faster than one
        if (may_cut && force_rods == 0 && force_rows == 0 && force_cpt == 0 && n_real < nsm &&
            split_plan(p, n_real, nsm, smem_optin, dev, one_sm_us(p, kind), plan))
            return true;
    }
    if (kind == 3) {
        if (!rows_supported(p)) return false;
        const int maxt = rows_max_threads(p);
        const size_t rbytes = rows_rod_bytes(p);
        const int by_smem = (int)std::max<size_t>(1, (size_t)smem_optin / rbytes);
        int rods = force_rods;
        if (rods == 0) {
            // one rod per CTA (608 b = 4 rods 0.87 us a step; 0.90, 0.98 and 1.23 with 2, 4 and 6),
            // unless that leaves over a quarter of the last warp idle (the b = 8 rod's 21 cells) and there
            // are more rods than ten to an SM: then the fewest rods that leave at most a tenth of it
            // (4096 rods 0.71 us with 3, 0.88 with 1; 2432 0.47 and 0.52; 1216 0.37 and 0.33)
            rods = 1;
            if (4 * (round_warp(rows) - rows) > round_warp(rows) && n_real > 10 * nsm)
                for (int r = 2; r * rows <= maxt && r <= by_smem; ++r)
                    if (10 * (round_warp(r * rows) - r * rows) <= round_warp(r * rows)) {
                        rods = r;
                        break;
                    }
        }
        if (rods < 1 || rods > by_smem || round_warp(rods * rows) > maxt) return false;
        plan->kind = 3;
        plan->rods_per_cta = rods;
        plan->cells_per_thread = p.nx;
        plan->threads = round_warp(rods * rows);
        plan->rows_per_thread = 1;
        plan->smem_bytes = rows_smem_bytes(p, rods);
        plan->ctas = (n_real + rods - 1) / rods;
        plan->crowded = in_batch || plan->ctas > nsm;
        return true;
    }
    if (kind == 1) {
        if (!twophase_fits || p.sample_every >= (1LL << 31)) return false;
        // cells per thread: forced, or the fewest that hold one rod in one CTA
        int cpt = force_cpt;
        if (cpt == 0) {
            cpt = 4;
            for (int c : {2, 1})
                if (round_warp((p.ncells + c - 1) / c) <= twophase_max_threads(p, c)) cpt = c;
        }
        if (cpt != 1 && cpt != 2 && cpt != 4) return false;
        const int maxt = twophase_max_threads(p, cpt);
        const int by_smem = (int)std::max<size_t>(1, (size_t)smem_optin / rod_bytes);
        int rods = 1;
        if (force_rods > 0) rods = force_rods;
        if (rods > by_smem || round_warp((rods * p.ncells + cpt - 1) / cpt) > maxt) return false;
        // what was asked for is accepted by the sizes of one cell a thread in a ghost-padded rod; the
        // pairs take less, except for several flat rods at once: then as many of them as fit
        while (rods > 1 && (rods * twophase_rod_bytes(p) > (size_t)smem_optin || !twophase_shape(p, rods, plan))) --rods;
        if (!twophase_shape(p, rods, plan)) return false;
        plan->kind = 1;
        plan->rods_per_cta = rods;
        plan->cells_per_thread = cpt;
        plan->rows_per_thread = 0;
        plan->smem_bytes = rods * twophase_rod_bytes(p);
        plan->ctas = (n_real + rods - 1) / rods;
        // small rods a cell to a thread: the chain of a step is shorter by the packed instructions' latency
        // and the second cell's noise.  Rods of 1x2x29 cells 0.36 us a step against 0.64 (one to an SM) and
        // 1.28 against 1.35 (16), 3x4x13 0.52 and 3.59 against 0.65 and 3.91, 3x4x26 0.74 against 0.89 with one to an
        // SM but 1.80 against 1.47 with three; 4x6x20 0.96 against 0.91
        if (force_rods == 0 && force_cpt == 0 && (p.ncells <= 160 || (p.ncells <= 400 && n_real <= nsm)))
            compact_shape(p, plan);
        return true;
    }
    if (!pipelined_fits) return false;
    int R = force_rows;
    if (R == 0) {
        // three rows per thread for the b = 1 rod's 1344 rows (448 threads, 128 registers):
        // measured ahead of 672 x 2 rows (which spill at 80 registers) on GB300
        R = rows <= 768 ? 1 : (rows <= 1536 ? 3 : 4);
    }
    if (R < 1 || R > 4 || (rows + R - 1) / R > pipelined_max_threads(R)) return false;
    plan->kind = 2;
    plan->rows_per_thread = R;
    plan->threads = pipelined_threads(rows, R);
    plan->rods_per_cta = 1;
    plan->cells_per_thread = 0;
    plan->smem_bytes = pipe_bytes;
    plan->ctas = n_real;
    return true;
}

template <typename K>
static cudaError_t set_smem(K kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t rod_advance(const KParams &p, const RodPlan &plan, float *m, int n_real,
                        long long step0, long long n_steps, float *samples, int *status,
                        unsigned *flags, cudaStream_t st)
{
    if (n_steps <= 0) return cudaSuccess;
    // the kernels count the steps of one launch in 32 bits: longer runs are split (the noise and
    // the field are functions of the absolute step index, so the split changes nothing)
    constexpr long long kMaxStepsPerLaunch = 1LL << 30;
    if (n_steps > kMaxStepsPerLaunch) {
        for (long long done = 0; done < n_steps; done += kMaxStepsPerLaunch) {
            const cudaError_t e = rod_advance(p, plan, m, n_real, step0 + done,
                                              std::min(kMaxStepsPerLaunch, n_steps - done), samples, status,
                                              flags, st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    cudaError_t e = cudaSuccess;
    if (plan.kind == 1) {
        e = twophase_advance(p, plan, m, n_real, step0, (int)n_steps, samples, status, st);
        if (e != cudaSuccess) return e;
    } else if (plan.kind == 4) {
        return split_advance(p, plan, m, n_real, step0, (int)n_steps, samples, status, st);
    } else if (plan.kind == 3) {
        e = rows_advance(p, plan, m, n_real, step0, (int)n_steps, samples, status, st);
        if (e != cudaSuccess) return e;
    } else if (plan.kind == 2 && pairs_supported(p) && !plan.generic) {
        return pairs_advance(p, plan, m, n_real, step0, (int)n_steps, samples, status, flags, st);
    } else if (plan.kind == 2) {
#define LLG_PIPELINED(R)                                                                        \
    case R:                                                                                     \
        if (p.axis) {                                                                           \
            e = set_smem(rod_pipelined_kernel<R, true>, plan.smem_bytes);                       \
            if (e != cudaSuccess) return e;                                                     \
            rod_pipelined_kernel<R, true><<<plan.ctas, plan.threads, plan.smem_bytes, st>>>(    \
                p, m, step0, n_steps, samples, status);                                         \
        } else {                                                                                \
            e = set_smem(rod_pipelined_kernel<R, false>, plan.smem_bytes);                      \
            if (e != cudaSuccess) return e;                                                     \
            rod_pipelined_kernel<R, false><<<plan.ctas, plan.threads, plan.smem_bytes, st>>>(   \
                p, m, step0, n_steps, samples, status);                                         \
        }                                                                                       \
        break;
        switch (plan.rows_per_thread) {
            LLG_PIPELINED(1)
            LLG_PIPELINED(2)
            LLG_PIPELINED(3)
            LLG_PIPELINED(4)
            default:
                return cudaErrorInvalidValue;
        }
#undef LLG_PIPELINED
    } else {
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace llg
