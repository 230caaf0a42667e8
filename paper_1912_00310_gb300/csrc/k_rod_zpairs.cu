// k_rod_zpairs.cu -- the resident engine's two-phase kernel (plan kind 1), for rods whose state and
// predictor state both fit in shared memory (b >= 2 in the paper's ladder: 4x12x28, 2x6x14, 1x3x7
// cells, and any other rod of at most 3072 cells), and the kernel for single-cell grids.
//
// Pairs: a thread owns P pairs of cells (x, y, z) and (x, y, z + L), L = ceil(nz / 2) -- the same place
// in the lower and the upper half of the rod -- and works on both with the packed FP32 instructions
// (pair.cuh).  Halving the rod leaves every neighbour of a pair a pair too: the x-, y- and z-neighbours
// sit at the same offsets in both halves.  Only the cut needs help: the upper half's cells below the
// cut and the lower half's above it are copied into one ghost line at each end by the threads that own
// them.  With an odd nz the last line's upper cells do not exist; they are stored as zeros.
//
// Shared memory per rod and buffer (state M, predictor P): [ghost line][L lines of pairs][ghost line]
// [zero], a line being the nx * ny places of one z and the zero standing for every neighbour beyond a
// free face (each thread keeps its pairs' neighbour positions).  (xa, xb, ya, yb) and (za, zb) lie in
// two arrays, 24 bytes a pair, without gaps, so that consecutive threads read consecutive entries.
//
// Per Heun step: the thermal field and the predictor into P, barrier, the corrector into M, barrier.
// All use the neighbour order x-, x+, y-, y+, z-, z+ and the arithmetic of physics.cuh, so the
// trajectories are bitwise those of the plain engine.
//
// What bounds it: with one rod per SM the chain of a step (field, torque, normalisation twice, the noise,
// two barriers), with several the FMA pipes (heavy pipe 60 % busy with 608 b = 4 rods).  152 rods of
// 5x11x23 cells held in a field for 1500 steps: 4.91 -> 3.19 ms, 209 thread-instructions per cell and step; the
// b = 4 rod's were 325 with one cell to a thread in a ghost-padded float4 rod and are 173 here.
#include <algorithm>

#include "llg_internal.h"
#include "pair.cuh"
#include "physics.cuh"
#include "reduce.cuh"
#include "rod_compact.cuh"
#include "sweep32.cuh"

namespace llg {
namespace {

// Extents with the pair axis last.  A grid with nz = 1 (or ny = nz = 1) is taken as (nx, 1, ny) (or (1, 1, nx)): the cells keep their numbers and the neighbour
// sum its order, since the axes without neighbours only add zeros.
struct ZDims {
    int nx, ny, nz;
    __host__ __device__ int line() const { return nx * ny; }  // pairs of a line
    __host__ __device__ int L() const { return (nz + 1) / 2; }  // lines
    __host__ __device__ int pairs() const { return line() * L(); }
    __host__ __device__ int entries() const { return pairs() + 2 * line() + 1; }
};

template <int P, bool AX, int SHAPE, bool ONE, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) rod_zpairs_kernel(KParams p, ZDims G, float *__restrict__ m_glob, int n_real,
                                                          int rods_per_cta, long long step0, int n_steps,
                                                          float *__restrict__ samples, int *__restrict__ status)
{
    // Two pairs a thread, one rod to the CTA: threads without a pair compute pair 0's again and store nothing,
    // so that a thread's two pairs are interleaved (152 rods of 9x16x20 cells 4.60 -> 4.25 us a step).  With
    // one pair that gains nothing, and with several rods two pairs spill.
    constexpr bool kBranch = !(P == 2 && ONE);
    extern __shared__ __align__(16) unsigned char zsm[];
    const int rods = ONE ? 1 : rods_per_cta;
    const int E = G.entries(), line = G.line(), npair = G.pairs(), ncell = line * G.nz, zero = E - 1;
    const int rod0 = blockIdx.x * rods;
    const int nrod = min(rods, n_real - rod0);
    const int tot = rods * E;
    ulonglong2 *MA = reinterpret_cast<ulonglong2 *>(zsm), *PA = MA + tot;
    pair_t *MB = reinterpret_cast<pair_t *>(PA + tot), *PB = MB + tot;
    const int T = blockDim.x;
    for (int i = threadIdx.x; i < tot; i += T) {
        MA[i] = PA[i] = make_ulonglong2(0ull, 0ull);
        MB[i] = PB[i] = 0ull;
    }
    __syncthreads();

    // this thread's pairs: entry, positions of the x- and y-neighbours, first cell, rod
    int e[P], xm[P], xp[P], ym[P], yp[P], ghost_lo[P], ghost_hi[P];
    bool act[P], phantom[P];
    unsigned long long cell_m0[P];
    uint32_t real[P];
    Pair3 m[P], u[P];
    const unsigned long long up_m0 = (unsigned long long)kPhiloxM0 * (uint32_t)(line * G.L());  // to the upper cell's product
#pragma unroll
    for (int k = 0; k < P; ++k) {
        const int i = (int)threadIdx.x + k * T;
        act[k] = i < nrod * npair;
        const int ii = act[k] ? i : 0;
        const int rl = ONE ? 0 : ii / npair, pr = ONE ? ii : ii - rl * npair;
        const int base = rl * E;
        const int x = pr % G.nx, y = pr / G.nx % G.ny, l = pr / line;
        e[k] = base + line + pr;
        xm[k] = x > 0 ? e[k] - 1 : base + zero;
        xp[k] = x < G.nx - 1 ? e[k] + 1 : base + zero;
        ym[k] = y > 0 ? e[k] - G.nx : base + zero;
        yp[k] = y < G.ny - 1 ? e[k] + G.nx : base + zero;
        ghost_lo[k] = l == G.L() - 1 ? base + pr - l * line : -1;              // the line below the lower one
        ghost_hi[k] = l == 0 ? base + line + npair + pr : -1;                  // the line above the upper one
        phantom[k] = (G.nz & 1) && l == G.L() - 1;                                // the upper cell does not exist
        cell_m0[k] = (unsigned long long)kPhiloxM0 * (uint32_t)pr;
        real[k] = p.real0 + (uint32_t)(rod0 + rl);
        m[k] = u[k] = zero_p3();
        {
            const size_t ca = (size_t)(rod0 + rl) * ncell + pr, cb = ca + (size_t)line * G.L();
            const float *a = m_glob + 3 * ca, *b = m_glob + 3 * cb;
            const float3 va = make_float3(a[0], a[1], a[2]);
            const float3 vb = phantom[k] ? make_float3(0.f, 0.f, 0.f) : make_float3(b[0], b[1], b[2]);
            m[k] = pair3(va, vb);
            if constexpr (AX) {
                const float3 ub = phantom[k] ? make_float3(0.f, 0.f, 1.f) : xyz(__ldg(p.axis + cb));
                u[k] = pair3(xyz(__ldg(p.axis + ca)), ub);
            }
        }
    }
    auto load = [](const ulonglong2 *A, const pair_t *B, int i) {
        const ulonglong2 v = A[i];
        return Pair3{v.x, v.y, B[i]};
    };
    // a pair's new value, and its halves beside the cut in the ghost lines
    auto store = [&](ulonglong2 *A, pair_t *B, int k, Pair3 v) {
        A[e[k]] = make_ulonglong2(v.x, v.y);
        B[e[k]] = v.z;
        if (ghost_lo[k] >= 0) {  // the lower half's last line, below the upper half's first
            A[ghost_lo[k]] = make_ulonglong2(pack2(0.f, lo2(v.x)), pack2(0.f, lo2(v.y)));
            B[ghost_lo[k]] = pack2(0.f, lo2(v.z));
        }
        if (ghost_hi[k] >= 0) {  // the upper half's first line, above the lower half's last
            A[ghost_hi[k]] = make_ulonglong2(pack2(hi2(v.x), 0.f), pack2(hi2(v.y), 0.f));
            B[ghost_hi[k]] = pack2(hi2(v.z), 0.f);
        }
    };
    // the neighbour sum in every engine's order
    auto neighbour_sum = [&](const ulonglong2 *A, const pair_t *B, int k) {
        Pair3 nb = add_p3(load(A, B, xm[k]), load(A, B, xp[k]));
        nb = add_p3(nb, load(A, B, ym[k]));
        nb = add_p3(nb, load(A, B, yp[k]));
        nb = add_p3(nb, load(A, B, e[k] - line));
        return add_p3(nb, load(A, B, e[k] + line));
    };
    // clears the half that does not exist
    auto real_cells = [&](Pair3 v, int k) {
        if (phantom[k]) v = pair3(lo3(v), make_float3(0.f, 0.f, 0.f));
        return v;
    };
#pragma unroll
    for (int k = 0; k < P; ++k)
        if (act[k]) store(MA, MB, k, m[k]);
    const PairCoeffs cf = pair_coeffs(p);
    const PhiloxKeys one_rod = philox_keys(p.seed, p.real0 + (uint32_t)rod0);
    __syncthreads();

    FieldAhead<SHAPE> field;
    field.init(step0);
    float Hn = field.next(p);
    // steps to the next sample (32-bit countdown; the host keeps sample_every below 2^31)
    const long long se = p.sample_every;
    const bool sampling = samples && se > 0;
    long long k_next = sampling ? step0 / se + 1 : 0;
    int to_sample = sampling ? (int)(k_next * se - step0) : -1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = T >> 5;

    unsigned long long n = (unsigned long long)step0;
    for (int s = 0; s < n_steps; ++s, ++n) {
        const float Hn1 = field.next(p);
        const pair_t H0 = both(Hn), H1 = both(Hn1);
        Pair3 t[P], s0[P], h[P];
#pragma unroll
        for (int k = 0; k < P; ++k) {
            if (kBranch && !act[k]) continue;
            const PhiloxKeys keys = ONE ? one_rod : philox_keys(p.seed, real[k]);
            const PhiloxStep now = philox_step(keys, n);
            h[k] = box_muller_p3(philox4x32_10(keys, now, cell_m0[k]), philox4x32_10(keys, now, cell_m0[k] + up_m0),
                                 p.sigma_bm);
            const Pair3 nb = neighbour_sum(MA, MB, k);
            s0[k] = llg_torque_p3(m[k], effective_field_p3<AX>(nb, m[k], h[k], cf, H0, u[k]), cf.alpha);
            t[k] = real_cells(normalised_p3(axpy_p3(cf.neg_dt_g1, s0[k], m[k])), k);
            if (kBranch || act[k]) store(PA, PB, k, t[k]);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < P; ++k) {
            if (kBranch && !act[k]) continue;
            const Pair3 nb = neighbour_sum(PA, PB, k);
            const Pair3 sv = llg_torque_add_p3(s0[k], t[k], effective_field_p3<AX>(nb, t[k], h[k], cf, H1, u[k]), cf.alpha);
            m[k] = real_cells(normalised_p3(axpy_p3(cf.neg_hdt_g1, sv, m[k])), k);
            if (kBranch || act[k]) store(MA, MB, k, m[k]);
        }
        __syncthreads();
        Hn = Hn1;
        if (--to_sample == 0) {
            // M now holds the state after step n; the next phase only reads M until the
            // barrier that precedes its next write, so no extra barrier is needed here.
            to_sample = (int)se;
            const long long kk = k_next++;
            if (kk < p.n_samples) {
                for (int rod = warp; rod < nrod; rod += nwarps) {
                    const pair_t *B = MB + rod * E + line;
                    float part = 0.f;
                    for (int c = lane; c < ncell; c += 32) part += c < npair ? lo2(B[c]) : hi2(B[c - npair]);
                    const float mean = warp_cell_mean(part, ncell);
                    if (lane == 0) {
                        samples[(size_t)(rod0 + rod) * p.n_samples + kk] = mean;
                        if (!isfinite(mean)) atomicOr(status, 1);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < P; ++k) {
        if (!act[k]) continue;
        const int i = (int)threadIdx.x + k * T, rl = ONE ? 0 : i / npair, pr = i - rl * npair;
        float *a = m_glob + ((size_t)(rod0 + rl) * ncell + pr) * 3, *b = a + (size_t)line * G.L() * 3;
        const float3 va = lo3(m[k]), vb = hi3(m[k]);
        a[0] = va.x;
        a[1] = va.y;
        a[2] = va.z;
        if (!phantom[k]) {
            b[0] = vb.x;
            b[1] = vb.y;
            b[2] = vb.z;
        }
    }
}

// Single-cell grids (the paper's b = 22 block): no neighbours, so a realisation is a thread and a step
// needs no shared memory and no barrier; the next step's noise and this step's chain interleave.  Bound
// by that chain until some 600 warps are in flight: 4096 blocks with dispersed axes and the sinusoid take
// 0.18 us a step (1.53 as rods of one cell, one to a 32-thread CTA), 40000 0.40.
template <bool AX, int SHAPE>
__global__ void __launch_bounds__(32) rod_single_kernel(KParams p, float *__restrict__ m_glob, int n_real, long long step0,
                                                        int n_steps, float *__restrict__ samples, int *__restrict__ status)
{
    // the last warp's idle lanes repeat its last rod (the field's lanes work together) and write nothing
    const int own = blockIdx.x * blockDim.x + threadIdx.x;
    const bool act = own < n_real;
    const int rod = act ? own : n_real - 1;
    float *g = m_glob + 3 * (size_t)rod;
    float3 m = make_float3(g[0], g[1], g[2]);
    const float3 u = AX ? xyz(__ldg(p.axis + rod)) : make_float3(0.f, 0.f, 1.f);
    const float3 none = make_float3(0.f, 0.f, 0.f);
    const PhiloxKeys keys = philox_keys(p.seed, p.real0 + (uint32_t)rod);
    FieldAhead<SHAPE> field;
    field.init(step0);
    float Hn = field.next(p);
    const long long se = p.sample_every;
    const bool sampling = samples && se > 0;
    long long k_next = sampling ? step0 / se + 1 : 0;
    int to_sample = sampling ? (int)(k_next * se - step0) : -1;
    unsigned long long n = (unsigned long long)step0;
    float3 h = box_muller3(philox4x32_10(keys, philox_step(keys, n), 0ull), p.sigma_bm);
    for (int s = 0; s < n_steps; ++s, ++n) {
        const float Hn1 = field.next(p);
        const float3 hnext = box_muller3(philox4x32_10(keys, philox_step(keys, n + 1), 0ull), p.sigma_bm);
        const float3 s0 = llg_torque(m, effective_field_sel<AX>(none, m, h, p, Hn, u), p.alpha);
        const float3 t = normalised(axpy(p.neg_dt_g1, s0, m));
        const float3 sv = llg_torque_add(s0, t, effective_field_sel<AX>(none, t, h, p, Hn1, u), p.alpha);
        m = normalised(axpy(p.neg_hdt_g1, sv, m));
        h = hnext;
        Hn = Hn1;
        if (--to_sample == 0) {
            to_sample = (int)se;
            const long long k = k_next++;
            if (act && k < p.n_samples) {
                samples[(size_t)rod * p.n_samples + k] = m.z;
                if (!isfinite(m.z)) atomicOr(status, 1);
            }
        }
    }
    if (act) {
        g[0] = m.x;
        g[1] = m.y;
        g[2] = m.z;
    }
}

// Small rods, one to a CTA, a cell to a thread: float4 cells in cell order and one zero slot for every
// neighbour beyond a free face.  No branch surrounds a cell's work, so its parts overlap, and with up to four
// warps each step draws the next one's noise, whose chain is as long as a half-step's, beside the
// corrector (1x2x29 cells 0.355 us a step, 0.374 without; with more warps the noise of one overlaps the chain of
// another anyway, and 3x4x26 cells take 0.74, 0.78 with the noise ahead).  What bounds it is that chain:
// 0.34 us a step for 2 to 32 cells (one warp, which synchronises itself only), 0.52 for 156, 0.74 for 312;
// many rods to an SM are bound by issue (2432 of 156 cells 3.59).
template <bool AX, int SHAPE, int MAXT>
__global__ void __launch_bounds__(MAXT) rod_compact_kernel(KParams p, float *__restrict__ m_glob, long long step0, int n_steps,
                                                           float *__restrict__ samples, int *__restrict__ status)
{
    constexpr bool kAhead = MAXT <= 128;
    extern __shared__ __align__(16) float4 csm[];
    const int ncell = p.ncells, S = ncell + 1;  // cells and the zero slot
    float4 *M = csm, *P = csm + S;
    const int rod = blockIdx.x, lane = threadIdx.x & 31;
    auto sync = [] {
        if constexpr (MAXT == 32)
            __syncwarp();
        else
            __syncthreads();
    };
    // a thread without a cell computes cell 0's values again and stores nothing
    const bool act = (int)threadIdx.x < ncell;
    const int c = act ? threadIdx.x : 0;
    const grad::Nbr nb = grad::neighbours(c, p.nx, p.ny, p.nz, ncell);
    float *g = m_glob + ((size_t)rod * ncell + c) * 3;
    float3 m = make_float3(g[0], g[1], g[2]), u = make_float3(0.f, 0.f, 1.f);
    if (act) M[c] = pad4(m);
    if (threadIdx.x == 0) M[ncell] = P[ncell] = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (AX) u = xyz(__ldg(p.axis + (size_t)rod * ncell + c));
    const PhiloxKeys keys = philox_keys(p.seed, p.real0 + (uint32_t)rod);
    const unsigned long long cell_m0 = (unsigned long long)kPhiloxM0 * (uint32_t)c;
    sync();
    FieldAhead<SHAPE> field;
    field.init(step0);
    float Hn = field.next(p);
    const long long se = p.sample_every;
    const bool sampling = samples && se > 0;
    long long k_next = sampling ? step0 / se + 1 : 0;
    int to_sample = sampling ? (int)(k_next * se - step0) : -1;
    auto draw = [&](unsigned long long n) { return box_muller3(philox4x32_10(keys, philox_step(keys, n), cell_m0), p.sigma_bm); };
    unsigned long long n = (unsigned long long)step0;
    float3 h = draw(n);
    for (int s = 0; s < n_steps; ++s) {
        if constexpr (!kAhead) h = draw(n);
        ++n;
        const float Hn1 = field.next(p);
        const float3 s0 = llg_torque(m, effective_field_sel<AX>(grad::neighbour_sum(M, nb), m, h, p, Hn, u), p.alpha);
        const float3 t = normalised(axpy(p.neg_dt_g1, s0, m));
        if (act) P[c] = pad4(t);
        sync();
        float3 next;
        if constexpr (kAhead) next = draw(n);
        const float3 sv =
            llg_torque_add(s0, t, effective_field_sel<AX>(grad::neighbour_sum(P, nb), t, h, p, Hn1, u), p.alpha);
        m = normalised(axpy(p.neg_hdt_g1, sv, m));
        if (act) M[c] = pad4(m);
        if constexpr (kAhead) h = next;
        sync();
        Hn = Hn1;
        if (--to_sample == 0) {
            // M holds the state after step n until the barrier in the next step's middle
            to_sample = (int)se;
            const long long k = k_next++;
            if (k < p.n_samples && threadIdx.x < 32) {
                float part = 0.f;
                for (int i = lane; i < ncell; i += 32) part += M[i].z;
                const float mean = warp_cell_mean(part, ncell);
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

ZDims pair_dims(const KParams &p)
{
    if (p.nz > 1) return ZDims{p.nx, p.ny, p.nz};
    if (p.ny > 1) return ZDims{p.nx, 1, p.ny};
    return ZDims{1, 1, p.nx};
}

int round32(int n) { return (n + 31) / 32 * 32; }

// (pairs per thread, largest CTA), in order of preference: one pair at 768 threads (80 registers), two
// at 512 (128 registers); beyond 1024 pairs two or four at 768, which spill.
struct ZShape {
    int P, maxt;
};
constexpr ZShape kShapes[] = {{1, 768}, {2, 512}, {2, 768}, {4, 768}};

template <int P, int MAXT, bool AX, int SHAPE, bool ONE>
cudaError_t launch(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0, int n_steps,
                   float *samples, int *status, cudaStream_t st)
{
    auto kern = rod_zpairs_kernel<P, AX, SHAPE, ONE, MAXT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem_bytes);
    if (e != cudaSuccess) return e;
    kern<<<plan.ctas, plan.threads, plan.smem_bytes, st>>>(p, pair_dims(p), m, n_real, plan.rods_per_cta, step0, n_steps,
                                                           samples, status);
    return cudaGetLastError();
}

// by axes and sweep shape (32-bit where its period fits), one rod per CTA or several
template <int P, int MAXT, bool ONE>
cudaError_t launch_by(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0, int n_steps,
                      float *samples, int *status, cudaStream_t st)
{
    const int shape = sweep_fits_32(p) ? (p.shape == 1 ? 1 : 0) : -1;
#define LLG_Z(AXV, S) launch<P, MAXT, AXV, S, ONE>(p, plan, m, n_real, step0, n_steps, samples, status, st)
    if constexpr (P * MAXT <= 1024) {
        if (shape == 0) return p.axis ? LLG_Z(true, 0) : LLG_Z(false, 0);
        if (shape == 1) return p.axis ? LLG_Z(true, 1) : LLG_Z(false, 1);
    }
    return p.axis ? LLG_Z(true, -1) : LLG_Z(false, -1);
#undef LLG_Z
}

}  // namespace

size_t twophase_rod_bytes(const KParams &p)
{
    const ZDims d = pair_dims(p);
    return 48 * (size_t)d.entries();
}

void compact_shape(const KParams &p, RodPlan *plan)
{
    if (p.ncells < 2 || !sweep_fits_32(p)) return;
    plan->pairs_per_thread = 0;
    plan->threads = round32(p.ncells);
    plan->smem_bytes = 2 * (size_t)(p.ncells + 1) * sizeof(float4);
}

bool twophase_shape(const KParams &p, int rods, RodPlan *plan)
{
    const ZDims d = pair_dims(p);
    const int pairs = rods * d.pairs();
    for (const ZShape &z : kShapes) {
        const int threads = round32((pairs + z.P - 1) / z.P);
        if (threads > z.maxt) continue;
        plan->pairs_per_thread = z.P;
        plan->threads = threads;
        return true;
    }
    return false;
}

cudaError_t twophase_advance(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0,
                             int n_steps, float *samples, int *status, cudaStream_t st)
{
    if (p.ncells == 1) {
        const int shape = sweep_fits_32(p) ? (p.shape == 1 ? 1 : 0) : -1;
        const int ctas = (n_real + 31) / 32;
#define LLG_S(AXV, S) rod_single_kernel<AXV, S><<<ctas, 32, 0, st>>>(p, m, n_real, step0, n_steps, samples, status)
        if (shape == 0) p.axis ? LLG_S(true, 0) : LLG_S(false, 0);
        else if (shape == 1) p.axis ? LLG_S(true, 1) : LLG_S(false, 1);
        else p.axis ? LLG_S(true, -1) : LLG_S(false, -1);
#undef LLG_S
        return cudaGetLastError();
    }
    const bool one = plan.rods_per_cta == 1;
    const int P = plan.pairs_per_thread;
    if (P == 0) {
        auto go = [&](auto kern) {
            kern<<<n_real, plan.threads, plan.smem_bytes, st>>>(p, m, step0, n_steps, samples, status);
            return cudaGetLastError();
        };
#define LLG_C(T)                                                                                              \
    (p.shape == 1 ? (p.axis ? go(rod_compact_kernel<true, 1, T>) : go(rod_compact_kernel<false, 1, T>))       \
                  : (p.axis ? go(rod_compact_kernel<true, 0, T>) : go(rod_compact_kernel<false, 0, T>)))
        if (plan.threads <= 32) return LLG_C(32);
        if (plan.threads <= 128) return LLG_C(128);
        return LLG_C(416);
#undef LLG_C
    }
#define LLG_D(P, MAXT)                                                                                 \
    (one ? launch_by<P, MAXT, true>(p, plan, m, n_real, step0, n_steps, samples, status, st)           \
         : launch_by<P, MAXT, false>(p, plan, m, n_real, step0, n_steps, samples, status, st))
    if (P == 1) return LLG_D(1, 768);
    if (P == 2 && plan.threads <= 512) return LLG_D(2, 512);
    if (P == 2) return LLG_D(2, 768);
    if (P == 4) return LLG_D(4, 768);
#undef LLG_D
    return cudaErrorInvalidValue;
}

}  // namespace llg
