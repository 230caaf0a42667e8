// k_rod_pairs.cu -- the resident engine's kernel for rods eight cells wide (the b = 1 rod, 8x24x56 =
// 10752 cells): the plane-pipelined schedule of k_rod.cu on pairs of x-neighbours.
//
// One rod per CTA, resident in shared memory for the whole launch.  A thread owns R rows along x; a
// row's eight cells are four pairs (x, x + 1), and every arithmetic step works on a pair with the
// packed FP32 instructions (pair.cuh).  The CTA sweeps the four pair planes in lock step: one
// iteration takes the predictor of plane X and the corrector of plane X - 1 of each row, so only two
// planes of predictor state exist (double-buffered by the parity of X), and the corrector of a step's
// last plane shares its iteration with the predictor of the next step's plane 0: four barriers a
// step.  The y- and z-neighbours are whole pairs in shared memory; the x-neighbours are the other
// half of the own pair and the near halves of the row's previous and next pairs, from registers.
//
// Shared memory: pairs as (xa, xb, ya, yb) in one array and (za, zb) in another, 24 bytes a pair,
// rows of a plane in order with one line of zeros before plane 0 and after every plane (a plane's
// upper ghost line is the next one's lower); the y faces are 0/1 weights.  Consecutive threads read
// consecutive entries, 6 wavefronts a pair and neighbour where padded float4 cells took 8.
//
// What bounds it: the FMA pipes and, because every plane ends in a CTA barrier, the busiest
// scheduler's share of the rows (11 of 42 row-warps).  An IMAD.WIDE of the noise holds the pipes 4
// scheduler cycles a warp, a multiply-add 1, a packed one 2; noise and step together, from registers
// alone, run at 195 cycles per warp and cell, this kernel at 276 (the heavy FMA pipe 60 % busy, 139
// instructions per warp and cell at 50 % issue, shared memory 55 %).  152 b = 1 rods take 11.1 us a
// step, 12.5 with dispersed axes; one cell an instruction (four-byte arithmetic on padded float4
// cells, eight barriers a step) took 14.7 and 23.4.  256 rods over 1000 steps: 24.87 -> 18.90 ms.
#include <algorithm>
#include <cstring>

#include "llg_internal.h"
#include "mbarrier.cuh"
#include "pair.cuh"
#include "physics.cuh"
#include "reduce.cuh"
#include "rod_threads.h"

namespace llg {
namespace {

// NXP pair planes; NY, NZ > 0: the y and z extents at compile time (the b = 1 rod), so that every
// shared-memory offset is an immediate and the thread count a constant.
template <int R, int NXP, int NY, int NZ, int SHAPE, bool AX>
struct PairRod {
    static constexpr int NX = 2 * NXP;
    static constexpr bool kFixed = NY > 0 && NZ > 0;
    static constexpr int kT = kFixed ? pipelined_threads(NY * NZ, R) : 0;
    static constexpr bool kSameY = kFixed && kT % NY == 0;  // a thread's rows all have the same y
    ulonglong2 *MA, *SA;  // (x, y) of a pair: state planes, two predictor planes
    pair_t *MB, *SB;      // z of a pair
    int ny_rt, nz_rt, ncell;
    int q0;               // entry of the first row in its plane
    unsigned long long cell0_m0;  // kPhiloxM0 times its first cell
    pair_t wm[kSameY ? 1 : R], wp[kSameY ? 1 : R];
    bool act_rt[R];

    __device__ __forceinline__ int ny() const
    {
        if constexpr (kFixed) return NY;
        return ny_rt;
    }
    __device__ __forceinline__ int nz() const
    {
        if constexpr (kFixed) return NZ;
        return nz_rt;
    }
    __device__ __forceinline__ int threads() const
    {
        if constexpr (kFixed) return kT;
        return blockDim.x;
    }
    __device__ __forceinline__ int PL() const { return (nz() + 1) * ny(); }  // entries of a plane and a ghost line
    __device__ __forceinline__ int state_entries() const { return NXP * PL() + ny(); }
    __device__ __forceinline__ int pred_entries() const { return 2 * PL() + ny(); }
    __device__ __forceinline__ int q(int j) const { return q0 + j * threads(); }
    __device__ __forceinline__ unsigned long long cell_m0(int j, int X) const
    {
        return cell0_m0 + (unsigned long long)kPhiloxM0 * (uint32_t)(j * threads() * NX + 2 * X);
    }
    __device__ __forceinline__ bool act(int j) const
    {
        if constexpr (kFixed) {
            if ((j + 1) * kT <= NY * NZ) return true;
        }
        return act_rt[j];
    }

    __device__ __forceinline__ void setup(unsigned char *sm, const KParams &p)
    {
        ny_rt = p.ny;
        nz_rt = p.nz;
        ncell = p.ncells;
        MA = reinterpret_cast<ulonglong2 *>(sm);
        SA = MA + state_entries();
        MB = reinterpret_cast<pair_t *>(SA + pred_entries());
        SB = MB + state_entries();
        for (int i = threadIdx.x; i < state_entries(); i += threads()) {
            MA[i] = make_ulonglong2(0ull, 0ull);
            MB[i] = 0ull;
        }
        for (int i = threadIdx.x; i < pred_entries(); i += threads()) {
            SA[i] = make_ulonglong2(0ull, 0ull);
            SB[i] = 0ull;
        }
        const int rows = ny() * nz();
        q0 = ny() + (int)threadIdx.x;
        cell0_m0 = (unsigned long long)kPhiloxM0 * (threadIdx.x * (uint32_t)NX);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int r = (int)threadIdx.x + j * threads();
            act_rt[j] = r < rows;
            if (j == 0 || !kSameY) {
                const int y = r % ny();
                wm[j] = both(y > 0 ? 1.f : 0.f);
                wp[j] = both(y < ny() - 1 ? 1.f : 0.f);
            }
        }
    }

    static __device__ __forceinline__ Pair3 load(const ulonglong2 *A, const pair_t *B, int i)
    {
        const ulonglong2 v = A[i];
        return Pair3{v.x, v.y, B[i]};
    }
    static __device__ __forceinline__ void store(ulonglong2 *A, pair_t *B, int i, Pair3 v)
    {
        A[i] = make_ulonglong2(v.x, v.y);
        B[i] = v.z;
    }

    // The neighbour sum in every engine's order x-, x+, y-, y+, z-, z+: xs = x- + x+.
    __device__ __forceinline__ Pair3 neighbour_sum(Pair3 xs, const ulonglong2 *A, const pair_t *B, int i, int j) const
    {
        const pair_t a = wm[kSameY ? 0 : j], b = wp[kSameY ? 0 : j];
        Pair3 nb = axpy_p3(a, load(A, B, i - 1), xs);
        nb = axpy_p3(b, load(A, B, i + 1), nb);
        nb = add_p3(nb, load(A, B, i - ny()));
        return add_p3(nb, load(A, B, i + ny()));
    }

    __device__ __forceinline__ float mz(int c) const  // m_z of cell c
    {
        const int x = c % NX, i = (x >> 1) * PL() + ny() + c / NX;
        return x & 1 ? hi2(MB[i]) : lo2(MB[i]);
    }

    // Sample k of rod `rod`: the canonical warp reduction of m_z over the cells in M, then a
    // barrier (the next iteration overwrites plane 0).
    __device__ __forceinline__ void sample(const KParams &p, int rod, long long k, float *__restrict__ samples,
                                           int *__restrict__ status)
    {
        if (k < p.n_samples && threadIdx.x < 32) {
            float part = 0.f;
            for (int c = threadIdx.x; c < ncell; c += 32) part += mz(c);
            const float mean = warp_cell_mean(part, ncell);
            if (threadIdx.x == 0) {
                samples[(size_t)rod * p.n_samples + k] = mean;
                if (!isfinite(mean)) atomicOr(status, 1);
            }
        }
        __syncthreads();
    }

    // The easy axes of row r's pair X (AX): entries in the order of the planes' rows, so that a warp's
    // loads are dense (from the per-cell array, 128 bytes apart, they took 18.0 us a step of 152 rods).
    struct AxisRod {
        const ulonglong2 *xy;
        const pair_t *z;
    };
    __device__ __forceinline__ Pair3 axes(const AxisRod &a, int X, int r) const
    {
        if constexpr (AX) {
            const int e = X * ny() * nz() + r;
            const ulonglong2 v = __ldg(a.xy + e);
            return Pair3{v.x, v.y, __ldg(a.z + e)};
        }
        return zero_p3();
    }

    // Load rod `rod` from global memory (L2, bypassing L1: another SM may have written it during
    // this launch), advance it from step s0 by ns steps, store it back.
    __device__ __forceinline__ void run(const KParams &p, float *__restrict__ m_glob, int rod, long long s0,
                                        long long ns, float *__restrict__ samples, int *__restrict__ status)
    {
        const int PL = this->PL();
        float *g = m_glob + (size_t)rod * ncell * 3;
        for (int r = threadIdx.x; r < ny() * nz(); r += threads()) {
            const float *gr = g + (size_t)r * NX * 3;
#pragma unroll
            for (int X = 0; X < NXP; ++X) {
                float v[6];
#pragma unroll
                for (int i = 0; i < 6; ++i) v[i] = __ldcg(gr + 6 * X + i);
                store(MA, MB, X * PL + ny() + r,
                      pair3(make_float3(v[0], v[1], v[2]), make_float3(v[3], v[4], v[5])));
            }
        }
        const PhiloxKeys keys = philox_keys(p.seed, p.real0 + (uint32_t)rod);
        const PairCoeffs cf = pair_coeffs(p);
        const size_t axis_entries = (size_t)NXP * ny() * nz();
        const AxisRod axr{reinterpret_cast<const ulonglong2 *>(p.axis_pairs) + (size_t)rod * axis_entries,
                          reinterpret_cast<const pair_t *>(p.axis_pairs_z) + (size_t)rod * axis_entries};
        // carried per row, for the corrector: the high half of pair X - 2's predictor state, and of pair
        // X - 1 the torque s0 and the thermal field.  What is in shared memory (the states, the predictor
        // state of pair X - 1) is read back: carried too, it spilled 400 bytes (12.2 against 11.1 us a step
        // of 152 b = 1 rods).  The noise is drawn where it is used, so that it interleaves with the row
        // before: drawn a plane ahead it was slower (11.5 to 12.0 us), also in the gap of a split
        // arrive-and-wait barrier (11.7 us).
        Pair3 s0c[R], hth[R];
        float3 tL[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            s0c[j] = hth[j] = zero_p3();
            tL[j] = make_float3(0.f, 0.f, 0.f);
        }
        __syncthreads();

        SweepOf<SHAPE> field;
        field.init(s0, p);
        float Hs = field.value();  // field at step s
        field.inc();
        float Hs1 = field.value();  // field at step s + 1
        float Hprev = Hs;           // field at step s (the end of step s - 1), for its corrector
        const long long se = p.sample_every;
        long long next_sample = (samples && se > 0) ? (s0 / se + 1) * se : -1;

        for (long long s = 0; s < ns; ++s) {
            const PhiloxStep now = philox_step(keys, (unsigned long long)(s0 + s));
#pragma unroll
            for (int X = 0; X < NXP; ++X) {
                const int XC = X > 0 ? X - 1 : NXP - 1;  // the corrector's plane
                ulonglong2 *const SWA = SA + (X & 1) * PL, *const SRA = SA + (XC & 1) * PL;
                pair_t *const SWB = SB + (X & 1) * PL, *const SRB = SB + (XC & 1) * PL;
                const pair_t Hp = both(Hs), Hc = both(X > 0 ? Hs1 : Hprev);
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    if (!act(j)) continue;
                    const int i = q(j);
                    // ---- predictor at (s, X) ----
                    const Pair3 h = thermal_field_p3(keys, now, cell_m0(j, X), p.sigma_bm);
                    const Pair3 u = axes(axr, X, i - ny());
                    const Pair3 mo = load(MA, MB, XC * PL + i);  // the state at the corrector's plane
                    const Pair3 m = load(MA, MB, X * PL + i);
                    const float3 ml = X > 0 ? hi3(mo) : make_float3(0.f, 0.f, 0.f);
                    const float3 mr = X + 1 < NXP ? lo3(load(MA, MB, (X + 1) * PL + i)) : make_float3(0.f, 0.f, 0.f);
                    Pair3 nb = neighbour_sum(pair3(add3(ml, hi3(m)), add3(lo3(m), mr)), MA + X * PL, MB + X * PL, i, j);
                    const Pair3 sv = llg_torque_p3(m, effective_field_p3<AX>(nb, m, h, cf, Hp, u), cf.alpha);
                    const Pair3 t = normalised_p3(axpy_p3(cf.neg_dt_g1, sv, m));
                    store(SWA, SWB, i, t);
                    // ---- corrector one plane behind: (s, X - 1), or (s - 1, NXP - 1) at X = 0 (the first
                    // step's is computed and dropped: a branch would part it from the predictor, 11.27 us a
                    // step for 152 b = 1 rods instead of 11.15) ----
                    const Pair3 uc = axes(axr, XC, i - ny());
                    const Pair3 tc = load(SRA, SRB, i);
                    const float3 tr = X > 0 ? lo3(t) : make_float3(0.f, 0.f, 0.f);
                    nb = neighbour_sum(pair3(add3(tL[j], hi3(tc)), add3(lo3(tc), tr)), SRA, SRB, i, j);
                    const Pair3 H = effective_field_p3<AX>(nb, tc, hth[j], cf, Hc, uc);
                    const Pair3 sc = llg_torque_add_p3(s0c[j], tc, H, cf.alpha);
                    const Pair3 mn = normalised_p3(axpy_p3(cf.neg_hdt_g1, sc, mo));
                    if (X > 0 || s > 0) store(MA, MB, XC * PL + i, mn);
                    const float3 tl = X > 0 ? hi3(tc) : make_float3(0.f, 0.f, 0.f);
                    tL[j] = tl;
                    s0c[j] = sv;
                    hth[j] = h;
                }
                __syncthreads();
                if (X == 0 && s > 0 && s0 + s == next_sample) {
                    sample(p, rod, next_sample / se, samples, status);
                    next_sample += se;
                }
            }
            Hprev = Hs1;
            Hs = Hs1;
            field.inc();
            Hs1 = field.value();
        }
        if (ns > 0) {
            // the corrector of the last plane of the last step
            constexpr int XC = NXP - 1;
            const ulonglong2 *SRA = SA + (XC & 1) * PL;
            const pair_t *SRB = SB + (XC & 1) * PL;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (!act(j)) continue;
                const int i = q(j);
                const Pair3 tc = load(SRA, SRB, i);
                const Pair3 nb = neighbour_sum(pair3(add3(tL[j], hi3(tc)), add3(lo3(tc), make_float3(0.f, 0.f, 0.f))), SRA,
                                               SRB, i, j);
                const Pair3 H = effective_field_p3<AX>(nb, tc, hth[j], cf, both(Hprev), axes(axr, XC, i - ny()));
                const Pair3 sc = llg_torque_add_p3(s0c[j], tc, H, cf.alpha);
                store(MA, MB, XC * PL + i, normalised_p3(axpy_p3(cf.neg_hdt_g1, sc, load(MA, MB, XC * PL + i))));
            }
            __syncthreads();
            if (s0 + ns == next_sample) sample(p, rod, next_sample / se, samples, status);
        }
        for (int r = threadIdx.x; r < ny() * nz(); r += threads()) {
            float *gr = g + (size_t)r * NX * 3;
#pragma unroll
            for (int X = 0; X < NXP; ++X) {
                const Pair3 v = load(MA, MB, X * PL + ny() + r);
                const float3 a = lo3(v), b = hi3(v);
                gr[6 * X] = a.x;
                gr[6 * X + 1] = a.y;
                gr[6 * X + 2] = a.z;
                gr[6 * X + 3] = b.x;
                gr[6 * X + 4] = b.y;
                gr[6 * X + 5] = b.z;
            }
        }
        __syncthreads();
    }
};

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_gpu(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Balanced schedule of one launch (McNaughton's wrap-around rule): all n_real * N rod-steps laid
// end to end and cut into gridDim.x equal slices; a rod cut at a slice boundary runs its first
// steps at the start of the next CTA's slice and its last steps at the end of this CTA's slice,
// handed off through global memory.  Up to three segments per CTA {rod, first step offset,
// steps, kind}: kind 0 whole rod, 1 first part (release flags[rod] when done), 2 last part (wait
// for flags[rod] first).  Built on the host and passed as a kernel parameter, so the segment
// fields are uniform constant-bank values: the rod index feeds the Philox round keys, which then
// stay in uniform registers (measured on GB300: a schedule read from shared memory or walked
// on the device cost 6-9 % of the b = 1 rate).
constexpr int kMaxBalancedCtas = 256;
struct BalancedSchedule {
    int4 seg[3 * kMaxBalancedCtas];
};

struct HandoffCtl {
    unsigned long long timeout_ns;  // longest wait for a producer before giving up (status bit 1)
    int withhold;                   // test hook: producers do not release (every wait runs out)
};

// balanced == 0: one rod per CTA over [step0, step0 + n_steps); balanced == 1: the segments of
// `sched` (cooperative launch: all CTAs co-resident).  A wait for a hand-off gives up after
// hc.timeout_ns: status bit 1 is set and the CTA skips its remaining segments.
template <int R, int NXP, int NY, int NZ, int SHAPE, bool AX>
__global__ void __launch_bounds__(NY > 0 && NZ > 0 ? pipelined_threads(NY * NZ, R) : pipelined_max_threads(R), 1)
    rod_pairs_kernel(KParams p, float *__restrict__ m_glob, long long step0, int n_steps, float *__restrict__ samples,
                     int *__restrict__ status, unsigned *__restrict__ flags, int balanced,
                     const __grid_constant__ BalancedSchedule sched, HandoffCtl hc)
{
    static_assert(NXP >= 3 && NXP % 2 == 0, "merged schedule with an even plane count");
    extern __shared__ __align__(16) unsigned char pair_smem[];
    PairRod<R, NXP, NY, NZ, SHAPE, AX> w;
    __shared__ int go;
    w.setup(pair_smem, p);
    __syncthreads();
    const int nseg = balanced ? 3 : 1;
    for (int i = 0; i < nseg; ++i) {
        const int4 sg = balanced ? sched.seg[3 * blockIdx.x + i] : make_int4(blockIdx.x, 0, n_steps, 0);
        if (sg.z <= 0) continue;
        if (sg.w == 2) {
            if (threadIdx.x == 0) {
                const unsigned long long t0 = timer_ns();
                int ok = 1;
                while (ld_acquire_gpu(flags + sg.x) == 0u) {
                    if (timer_ns() - t0 > hc.timeout_ns) {
                        ok = 0;
                        atomicOr(status, 2);
                        break;
                    }
                    __nanosleep(200);
                }
                __threadfence();
                go = ok;
            }
            __syncthreads();
            if (!go) break;
        }
        w.run(p, m_glob, sg.x, step0 + sg.y, sg.z, samples, status);
        if (sg.w == 1 && threadIdx.x == 0 && !hc.withhold) {
            __threadfence();
            st_release_gpu(flags + sg.x, 1u);
        }
    }
}

// Four state planes and two predictor planes of 24-byte pairs, each plane followed by a ghost line.
size_t pairs_smem_bytes(const KParams &p)
{
    const size_t plane = (size_t)(p.nz + 1) * p.ny;
    return 24 * (4 * plane + p.ny + 2 * plane + p.ny);
}

// McNaughton's wrap-around schedule of n_real rods x N steps over G co-resident CTAs; false when
// some CTA's slice would need more than three segments (more than about two waves of rods),
// in which case the launch is not balanced.
static bool balanced_schedule(int n_real, int N, int G, BalancedSchedule *sc)
{
    if (G > kMaxBalancedCtas) return false;
    std::memset(sc, 0, sizeof *sc);
    const long long W = (long long)n_real * N;
    const long long C = (W + G - 1) / G;
    for (int j = 0; j < G; ++j) {
        const long long lo = std::min((long long)j * C, W), hi = std::min(lo + C, W);
        int k = 0;
        for (long long pos = lo; pos < hi;) {
            if (k == 3) return false;
            const long long rod = pos / N, off = pos - rod * N;
            const long long len = std::min(hi, (rod + 1) * N) - pos;
            int4 &g = sc->seg[3 * j + k++];
            g.x = (int)rod;
            g.z = (int)len;
            if (off != 0) {  // first len steps, then hand off
                g.y = 0;
                g.w = 1;
            } else if (len < N) {  // last len steps, after the hand-off
                g.y = (int)(N - len);
                g.w = 2;
            } else {
                g.y = 0;
                g.w = 0;
            }
            pos += len;
        }
    }
    return true;
}

// Launch: balanced over a co-resident grid when the rods do not
// divide evenly into waves, else one rod per CTA.
template <int R, int NY, int NZ, bool AX>
static cudaError_t launch_pairs(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0,
                                int n_steps, float *samples, int *status, unsigned *flags,
                             cudaStream_t st)
{
    auto kern = p.shape == 1 ? rod_pairs_kernel<R, 4, NY, NZ, 1, AX> : rod_pairs_kernel<R, 4, NY, NZ, 0, AX>;
    const size_t smem = pairs_smem_bytes(p);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, plan.threads, smem)) != cudaSuccess)
        return e;
    const int resident = nsm * per_sm;
    BalancedSchedule sched;
    int ns = n_steps;
    HandoffCtl hc{plan.handoff_timeout_ns, plan.withhold_handoff ? 1 : 0};
    if (plan.balance && flags && resident > 0 && n_real > resident && n_real % resident != 0 &&
        balanced_schedule(n_real, ns, resident, &sched)) {
        if ((e = cudaMemsetAsync(flags, 0, sizeof(unsigned) * (size_t)n_real, st)) != cudaSuccess) return e;
        int balanced = 1;
        void *args[] = {(void *)&p, (void *)&m, (void *)&step0, (void *)&ns, (void *)&samples,
                        (void *)&status, (void *)&flags, (void *)&balanced, (void *)&sched, (void *)&hc};
        return cudaLaunchCooperativeKernel((const void *)kern, dim3(resident), dim3(plan.threads), args,
                                           smem, st);
    }
    kern<<<n_real, plan.threads, smem, st>>>(p, m, step0, ns, samples, status, flags, 0, sched, hc);
    return cudaGetLastError();
}


template <int R>
cudaError_t launch_rows(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0, int n_steps,
                        float *samples, int *status, unsigned *flags, cudaStream_t st)
{
    if constexpr (R > 1) {  // the b = 1 rod's 1344 rows need two a thread at least
        const bool b1 = p.ny == 24 && p.nz == 56;
        if (p.axis) return launch_pairs<R, 24, 56, true>(p, plan, m, n_real, step0, n_steps, samples, status, flags, st);
        if (b1) return launch_pairs<R, 24, 56, false>(p, plan, m, n_real, step0, n_steps, samples, status, flags, st);
    }
    if (p.axis) return cudaErrorInvalidValue;
    return launch_pairs<R, 0, 0, false>(p, plan, m, n_real, step0, n_steps, samples, status, flags, st);
}

// Easy axes of the pairs of every rod, (x, y) and z apart, in the order of the kernel's planes.
__global__ void axis_pairs_kernel(ulonglong2 *__restrict__ xy, pair_t *__restrict__ z, int n_real, int rows,
                                  uint32_t seed, uint32_t real0, float w_max)
{
    const long long gid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (gid >= (long long)n_real * 4 * rows) return;
    const int r = (int)(gid % rows), X = (int)(gid / rows % 4), rod = (int)(gid / (4LL * rows));
    const uint32_t c = (uint32_t)(8 * r + 2 * X);
    const Pair3 v = pair3(easy_axis(seed, real0 + (uint32_t)rod, c, w_max), easy_axis(seed, real0 + (uint32_t)rod, c + 1, w_max));
    xy[gid] = make_ulonglong2(v.x, v.y);
    z[gid] = v.z;
}

}  // namespace

size_t pairs_axis_floats(int nx, int ny, int nz, int n_real)
{
    return nx == 8 && ny == 24 && nz == 56 ? (size_t)n_real * 3 * nx * ny * nz : 0;
}

cudaError_t pairs_axis_fill(float *out, int n_real, int ny, int nz, uint32_t seed, uint32_t real0, float w_max,
                            cudaStream_t st)
{
    const long long n = (long long)n_real * 4 * ny * nz;
    axis_pairs_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(reinterpret_cast<ulonglong2 *>(out),
                                                                  reinterpret_cast<pair_t *>(out + 4 * n), n_real, ny * nz,
                                                                  seed, real0, w_max);
    return cudaGetLastError();
}

// Rods eight cells wide: any with the easy axis along z, the b = 1 rod with dispersed axes too.
bool pairs_supported(const KParams &p) { return p.nx == 8 && (!p.axis || (p.ny == 24 && p.nz == 56)); }

cudaError_t pairs_advance(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0, int n_steps,
                          float *samples, int *status, unsigned *flags, cudaStream_t st)
{
    switch (plan.rows_per_thread) {
        case 1: return launch_rows<1>(p, plan, m, n_real, step0, n_steps, samples, status, flags, st);
        case 2: return launch_rows<2>(p, plan, m, n_real, step0, n_steps, samples, status, flags, st);
        case 3: return launch_rows<3>(p, plan, m, n_real, step0, n_steps, samples, status, flags, st);
        case 4: return launch_rows<4>(p, plan, m, n_real, step0, n_steps, samples, status, flags, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace llg
