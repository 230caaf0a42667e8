// k_rod_split.cu -- the resident engine's kernel for ensembles that leave SMs idle (plan kind 4): each rod
// is cut along z into k slabs, one CTA of a cluster each.
//
// A thread owns W neighbouring pairs of x-neighbours of one row of its slab (pair.cuh; with an odd nx the
// last pair's second cell does not exist and is kept zero), with their state, predictor, torque and thermal
// field in registers; per Heun step the predictor, a barrier, the corrector, a barrier.  The state M and the
// predictor state Q lie in shared memory, one plane per pair of a row: the slab's rows in order with a ghost
// line below and above, (xa, xb, ya, yb) in one array and (za, zb) in another; the y faces are 0/1 weights.
//
// A slab's first and last lines are stored into the neighbouring CTAs' ghost lines as well, by asynchronous
// stores (st.async), and a half-step ends at a shared-memory barrier, one for the predictor and one for the
// corrector, that counts the CTA's own warps and the bytes of the neighbours' lines.  (Remote arrivals with
// release semantics in place of the stores' own count cost 650 cycles a half-step.)  A neighbour runs at most
// one half-step ahead -- it needs this slab's line of the half-step before -- so its line never arrives in a
// phase that is still open, nor overwrites a ghost line that is still being read.  Between a warp's arrival
// and its wait it draws the next step's noise, half of it in each gap, which hides the lines' way.
//
// One more warp forms the samples from snapshots of m_z that the others leave behind, in the canonical order
// (reduce.cuh): each lane's partial sum runs through the slabs from the first CTA to the last.
//
// Every wait is bounded by the hand-off limit (status bit 1); the sampler's, which spans the steps between
// two samples, from the last 32 steps that its CTA began.  Where one gives up, the rod's threads store and arrive no
// more and leave their loops, no state and no further sample is written, and no CTA leaves before the lines
// that have been sent to it have landed (abandon).  Neighbour order, noise keys and arithmetic are every other
// engine's: bitwise the same states.
//
// What bounds it: the chain of a step -- neighbour loads, field, torque, normalisation, store, the lines' way
// to the next CTA, twice -- with one or two warps a scheduler to hide it.  One b = 1 rod takes 2.06 us a step
// over 8 CTAs (11.1 on one SM; 15 rods as many), 32 rods 3.49 over 4; three b = 2 rods 0.77 over 7 (1.55).  A way
// out of the step loop for waits that give up costs b = 1 rods up to 5 % of that, the others nothing.  Tried:
// noise drawn by warps of its own into a ring (one b = 1 rod 3.2 us: the two kinds of warp wait for one
// another's pipes), whole rows to a thread (2.70), remote arrivals as above.
#include <algorithm>

#include "llg_internal.h"
#include "mbarrier.cuh"
#include "pair.cuh"
#include "physics.cuh"
#include "reduce.cuh"
#include "sweep32.cuh"

namespace llg {
namespace {

constexpr int kBars = 2 + 8;
constexpr int kBlock = 32;  // steps between two looks for a thread that gave up (0.1 ms; a limit is 1 ms at least)

// What follows the barriers in shared memory.
struct Tail {
    // after a give-up, by half-step of a step: bytes that the neighbours have sent here, arrivals of the CTA's warps
    unsigned long long inbound[2], arrived[2];
    int step_now;      // the block of steps that this CTA is at, by its first step
    unsigned gave_up;  // a wait of some CTA of the cluster ran out
};
constexpr size_t kTailBytes = kBars * sizeof(uint64_t) + sizeof(Tail);
constexpr int kMaxThreads = 384;  // 168 registers

__host__ __device__ inline int slab_start(int nz, int k, int r) { return (int)((long long)nz * r / k); }

__host__ __device__ inline int largest_slab(int nz, int k)
{
    int most = 0;
    for (int r = 0; r < k; ++r) {
        const int n = slab_start(nz, k, r + 1) - slab_start(nz, k, r);
        most = n > most ? n : most;
    }
    return most;
}

// (out of line, as abandon below: inline they cost the step loop up to 7 %)
__device__ __noinline__ bool slow_wait(uint64_t *bar, unsigned parity, unsigned long long limit_ns)
{
    return mbar_wait(bar, parity, limit_ns);
}

// The sampler's wait for the phase of `parity`, the same in all its lanes.  The steps to the next sample may take
// longer than any wait's limit: the limit runs from the beginning of the CTA's block of steps.
__device__ __forceinline__ bool sampler_wait(uint64_t *bar, unsigned parity, const Tail *tail, unsigned long long limit_ns)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const volatile Tail *now = tail;
    int at = now->step_now;
    unsigned long long t0 = timer_ns();
    while (!__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) {
        const unsigned long long t = timer_ns();
        const int step = now->step_now;
        if (step != at) {
            at = step;
            t0 = t;
        }
        if (__any_sync(0xffffffffu, t - t0 > limit_ns)) return false;
    }
    return true;
}

// After the last store of every CTA of the cluster (a cluster barrier lies between) and with inbound and
// arrived complete: wait until the neighbours' lines that are still under way to this CTA have landed.  bar is
// the barrier of one half-step of a step, warp0 the arrivals of warp 0 there, which announce `bytes` each.
// A phase ends with wp arrivals and `bytes` landed; a warp arrives for the next one only after that, and so
// do the neighbours' lines, so min(arrived / wp, inbound / bytes) phases end by themselves.  What has been
// sent into the open one is made to end it: its count of bytes is set to what was sent and the missing
// arrivals are made.
__device__ void settle(uint64_t *bar, unsigned long long arrived, unsigned long long inbound, unsigned bytes,
                       unsigned wp, unsigned long long warp0, unsigned long long limit_ns)
{
    const unsigned long long by_arrivals = arrived / wp, by_bytes = inbound / bytes;
    const unsigned long long phases = by_arrivals < by_bytes ? by_arrivals : by_bytes;
    if (phases > 0 && !mbar_wait(bar, (unsigned)(phases - 1) & 1u, limit_ns)) return;
    const unsigned sent = (unsigned)(inbound - phases * bytes), there = (unsigned)(arrived - phases * wp);
    if (sent == 0) return;
    const unsigned announced = warp0 > phases ? bytes : 0u;
    if (sent > announced) mbar_expect_bytes(bar, sent - announced);
    if (sent < announced) mbar_complete_bytes(bar, announced - sent);
    if (there < wp) mbar_arrive_many(bar, wp - there);
    mbar_wait(bar, (unsigned)phases & 1u, limit_ns);
}

// The way out of a rod after a give-up, for the physics warps of all its CTAs, when none stores into a neighbour
// any more: what has been sent lands before the CTA that it is sent to leaves.  stored: the half-steps whose values
// this thread has stored, `pairs` pairs each, below (sides bit 0) and above (bit 1) the slab.
__device__ __noinline__ void abandon(uint64_t *half, Tail *tail, unsigned stored, int pairs, int sides, int rank,
                                     unsigned line_bytes, int wp, unsigned long long limit_ns)
{
    const unsigned sent[2] = {(stored + 1) / 2, stored / 2};
    for (int b = 0; b < 2; ++b) {
        const unsigned long long bytes = 24ull * (unsigned)pairs * sent[b];
        if (sides & 1) add_cluster(in_rank(smem_u32(&tail->inbound[b]), rank - 1), bytes);
        if (sides & 2) add_cluster(in_rank(smem_u32(&tail->inbound[b]), rank + 1), bytes);
        if ((threadIdx.x & 31) == 0) atomicAdd(&tail->arrived[b], (unsigned long long)sent[b]);
    }
    __syncwarp();
    cluster_sync();
    if (threadIdx.x == 0)
        for (int b = 0; b < 2; ++b)
            settle(half + b, tail->arrived[b], tail->inbound[b], line_bytes, (unsigned)wp, sent[b], limit_ns);
}

// FULL: every segment has W pairs and every pair two cells.
template <int W, bool FULL, bool AX, int SHAPE>
__global__ void __launch_bounds__(kMaxThreads, 1) rod_split_kernel(KParams p, int k, int wp, float *__restrict__ m_glob,
                                                                   long long step0, int n_steps,
                                                                   float *__restrict__ samples, int *__restrict__ status,
                                                                   unsigned long long limit_ns, int withhold)
{
    extern __shared__ __align__(16) unsigned char ssm[];
    const int rank = (int)(blockIdx.x % (unsigned)k), rod = (int)(blockIdx.x / (unsigned)k);
    const int nx = p.nx, ny = p.ny, nz = p.nz, ncell = p.ncells;
    const int px = (nx + 1) / 2, nseg = (px + W - 1) / W;  // pairs and segments of a row
    const int z0 = slab_start(nz, k, rank), z1 = slab_start(nz, k, rank + 1);
    const int rows = (z1 - z0) * ny;
    const int cap = largest_slab(nz, k) * ny;  // rows of the largest slab: the same layout in every CTA
    const int PL = cap + 2 * ny, E = px * PL;
    const int N = px * cap;  // pairs of the largest slab
    // (x, y) and z of the pairs: state M, predictor Q
    ulonglong2 *MA = reinterpret_cast<ulonglong2 *>(ssm), *QA = MA + E;
    pair_t *MB = reinterpret_cast<pair_t *>(QA + E), *QB = MB + E;
    pair_t *snap = QB + E;                                                // [2][px][cap] m_z at the samples
    float *carry = reinterpret_cast<float *>(snap + 2 * N);    // [2][32] partial sums from the slab below
    uint64_t *half = reinterpret_cast<uint64_t *>(carry + 64);
    uint64_t *taken = half + 2, *freed = taken + 2, *chain = freed + 2, *ack = chain + 2;
    Tail *tail = reinterpret_cast<Tail *>(half + kBars);
    const int T = blockDim.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool below = rank > 0, above = rank < k - 1;
    // bytes of the neighbours' lines in a half-step
    const unsigned line_bytes = 24u * (unsigned)(px * ny) * ((below ? 1u : 0u) + (above ? 1u : 0u));

    for (int i = threadIdx.x; i < E; i += T) {
        MA[i] = QA[i] = make_ulonglong2(0ull, 0ull);
        MB[i] = QB[i] = 0ull;
    }
    if (threadIdx.x == 0) {
        *tail = Tail{};
        for (int b = 0; b < 2; ++b) {
            mbar_init(half + b, wp);
            mbar_init(taken + b, wp);
            mbar_init(freed + b, 1);
            mbar_init(chain + b, 1);
            mbar_init(ack + b, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const size_t rod_cell = (size_t)rod * ncell;
    // pair X of a row of the slab (row -1 .. -ny: the line below it) in global memory
    auto read_pair = [&](int row, int X) {
        const float *c = m_glob + 3 * (rod_cell + (size_t)((z0 * ny + row) * nx + 2 * X));
        const float3 b = 2 * X + 1 < nx ? make_float3(c[3], c[4], c[5]) : make_float3(0.f, 0.f, 0.f);
        return pair3(make_float3(c[0], c[1], c[2]), b);
    };
    for (int row = (int)threadIdx.x + (below ? -ny : 0); row < rows + (above ? ny : 0); row += T)
        for (int X = 0; X < px; ++X) {
            const Pair3 v = read_pair(row, X);
            MA[X * PL + ny + row] = make_ulonglong2(v.x, v.y);
            MB[X * PL + ny + row] = v.z;
        }
    cluster_sync();

    const long long se = p.sample_every;
    const bool sampling = samples && se > 0;
    const long long k_first = sampling ? step0 / se + 1 : 0;
    // a warp with a wait that gave up tells the cluster
    auto tell = [&] {
        if (lane == 0) {
            atomicOr(status, 2);
            for (int r = 0; r < k; ++r) st_cluster(in_rank(smem_u32(&tail->gave_up), r), 1u);
        }
    };

    if (warp < wp) {
        // thread t has segment t / rows of row t mod rows
        bool act = (int)threadIdx.x < nseg * rows;
        const int seg = act ? (int)threadIdx.x / rows : 0, row = act ? (int)threadIdx.x - seg * rows : 0;
        const int y = row % ny, X0 = seg * W, q = X0 * PL + ny + row;
        const int nw = FULL ? W : min(W, px - X0);                  // pairs of this segment
        const bool lone = !FULL && nx < 2 * px && X0 + nw == px;    // its last pair's second cell does not exist
        const bool left = X0 > 0, right = X0 + W < px;         // pairs of the row beside the segment
        const pair_t wm = both(y > 0 ? 1.f : 0.f), wq = both(y < ny - 1 ? 1.f : 0.f);
        Pair3 m[W], u[W];
        auto has = [&](int w) { return act && w < nw; };
#pragma unroll
        for (int w = 0; w < W; ++w) {
            m[w] = u[w] = zero_p3();
            if (!has(w)) continue;
            m[w] = Pair3{MA[w * PL + q].x, MA[w * PL + q].y, MB[w * PL + q]};
            if constexpr (AX) {
                const size_t c = rod_cell + (size_t)((z0 * ny + row) * nx + 2 * (X0 + w));
                const float3 ua = xyz(__ldg(p.axis + c));
                u[w] = pair3(ua, 2 * (X0 + w) + 1 < nx ? xyz(__ldg(p.axis + c + 1)) : ua);
            }
        }
        // a first- or last-line segment's place in the neighbours' ghost lines of M, and their barriers
        unsigned belowA = 0, belowB = 0, aboveA = 0, aboveB = 0, bar_below = 0, bar_above = 0;
        const bool to_below = below && act && row < ny && !withhold, to_above = above && act && row >= rows - ny;
        if (to_below) {
            const int r = X0 * PL + ny + (z0 - slab_start(nz, k, rank - 1)) * ny + row;
            belowA = in_rank(smem_u32(MA + r), rank - 1);
            belowB = in_rank(smem_u32(MB + r), rank - 1);
            bar_below = in_rank(smem_u32(half), rank - 1);
        }
        if (to_above) {
            const int r = X0 * PL + row - (rows - ny);
            aboveA = in_rank(smem_u32(MA + r), rank + 1);
            aboveB = in_rank(smem_u32(MB + r), rank + 1);
            bar_above = in_rank(smem_u32(half), rank + 1);
        }
        auto load = [](const ulonglong2 *A, const pair_t *B, int i) {
            const ulonglong2 v = A[i];
            return Pair3{v.x, v.y, B[i]};
        };
        // half-step b's value of pair w into its buffer (0 predictor, 1 state), here and beside the slab
        auto put = [&](int b, int w, Pair3 v) {
            if (!has(w)) return;
            (b ? MA : QA)[w * PL + q] = make_ulonglong2(v.x, v.y);
            (b ? MB : QB)[w * PL + q] = v.z;
            const unsigned offA = (unsigned)((b ? 0 : E) + w * PL) * 16u, offB = (unsigned)((b ? 0 : E) + w * PL) * 8u;
            if (belowA) {
                st_async(belowA + offA, v.x, v.y, bar_below + 8u * b);
                st_async(belowB + offB, v.z, bar_below + 8u * b);
            }
            if (aboveA) {
                st_async(aboveA + offA, v.x, v.y, bar_above + 8u * b);
                st_async(aboveB + offB, v.z, bar_above + 8u * b);
            }
        };
        // the halves of the row's pairs beside the segment
        const float3 none = make_float3(0.f, 0.f, 0.f);
        auto beside_left = [&](const ulonglong2 *A, const pair_t *B) { return left ? hi3(load(A, B, q - PL)) : none; };
        auto beside_right = [&](const ulonglong2 *A, const pair_t *B) { return right ? lo3(load(A, B, q + W * PL)) : none; };
        // every engine's order; x- + x+ is the far half of the own pair and the near half beside it
        auto sum = [&](const Pair3 *v, int w, float3 l, float3 r, const ulonglong2 *A, const pair_t *B) {
            const float3 a = add3(w > 0 ? hi3(v[w > 0 ? w - 1 : 0]) : l, hi3(v[w]));
            const float3 b = add3(lo3(v[w]), w + 1 < W ? lo3(v[w + 1 < W ? w + 1 : w]) : r);
            const int i = (!FULL && w >= nw ? 0 : w) * PL + q;  // (a pair that does not exist reads the first)
            Pair3 nb = axpy_p3(wm, load(A, B, i - 1), pair3(a, b));
            nb = axpy_p3(wq, load(A, B, i + 1), nb);
            nb = add_p3(nb, load(A, B, i - ny));
            return add_p3(nb, load(A, B, i + ny));
        };
        // keeps cells that do not exist at zero: a lone pair's second, and a short segment's last pairs
        auto real_cells = [&](Pair3 v, int w) {
            if (FULL) return v;
            if (w >= nw) return zero_p3();
            return lone && w == nw - 1 ? pair3(lo3(v), none) : v;
        };
        // A thread whose wait ran out stores and arrives no more, here or beside the slab, and its warp leaves the
        // loop within a block of steps (a vote in every wait cost up to 13 % of a step).  What starves it starves the
        // cluster within a few half-steps, so that all of it gives up at about the same time.
        bool alive = true;
        unsigned stored = 0;  // the half-steps whose values it had stored
        auto arrive = [&](int b) {
            __syncwarp();
            if (lane == 0 && alive) {
                // (one instruction for both: three b = 2 rods 0.80 -> 0.77 us a step, b = 1 rods of two pairs a
                // thread 2.12 -> 2.06, but of four 3.49 -> 3.84)
                if constexpr (W < 4)
                    mbar_arrive_expect(half + b, warp == 0 ? line_bytes : 0u);
                else if (threadIdx.x == 0)
                    mbar_arrive_expect(half + b, line_bytes);
                else
                    mbar_arrive(half + b);
            }
        };
        auto wait = [&](uint64_t *bar, unsigned parity, unsigned so_far) {
            if (!alive) return;
            if (!mbar_try_wait(bar, parity) && !slow_wait(bar, parity, limit_ns)) {
                stored = so_far;
                alive = act = false;
            }
        };
        const PairCoeffs cf = pair_coeffs(p);
        const PhiloxKeys keys = philox_keys(p.seed, p.real0 + (uint32_t)rod);
        const unsigned long long row_m0 = (unsigned long long)kPhiloxM0 * (uint32_t)((z0 * ny + row) * nx + 2 * X0);
        auto draw = [&](const PhiloxStep &now, int w) {
            return thermal_field_p3(keys, now, row_m0 + (unsigned long long)kPhiloxM0 * (2 * w), p.sigma_bm);
        };
        Pair3 hn[W];
        {
            const PhiloxStep now = philox_step(keys, (unsigned long long)step0);
#pragma unroll
            for (int w = 0; w < W; ++w) hn[w] = draw(now, w);
        }
        FieldAhead<SHAPE> field;
        field.init(step0);
        float Hn = field.next(p);
        int to_sample = sampling ? (int)(k_first * se - step0) : -1;
        unsigned n_snap = 0;
        int s = 0;
        while (s < n_steps && __all_sync(0xffffffffu, alive)) {
            const int until = min(n_steps, s + kBlock);
            if (threadIdx.x == 0) *(volatile int *)&tail->step_now = s;
            for (; s < until; ++s) {
                const float Hn1 = field.next(p);
                const PhiloxStep next = philox_step(keys, (unsigned long long)(step0 + s + 1));
                const pair_t H0 = both(Hn), H1 = both(Hn1);
                Pair3 t[W], s0[W], h[W];
                float3 l = beside_left(MA, MB), r = beside_right(MA, MB);
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    h[w] = hn[w];
                    s0[w] = llg_torque_p3(m[w], effective_field_p3<AX>(sum(m, w, l, r, MA, MB), m[w], h[w], cf, H0, u[w]), cf.alpha);
                    t[w] = real_cells(normalised_p3(axpy_p3(cf.neg_dt_g1, s0[w], m[w])), w);
                }
#pragma unroll
                for (int w = 0; w < W; ++w) put(0, w, t[w]);
                arrive(0);
#pragma unroll
                for (int w = 0; w < (W + 1) / 2; ++w) hn[w] = draw(next, w);
                wait(half, (unsigned)s & 1u, 2u * s + 1u);
                l = beside_left(QA, QB), r = beside_right(QA, QB);
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const Pair3 H = effective_field_p3<AX>(sum(t, w, l, r, QA, QB), t[w], h[w], cf, H1, u[w]);
                    const Pair3 sv = llg_torque_add_p3(s0[w], t[w], H, cf.alpha);
                    m[w] = real_cells(normalised_p3(axpy_p3(cf.neg_hdt_g1, sv, m[w])), w);
                }
#pragma unroll
                for (int w = 0; w < W; ++w) put(1, w, m[w]);
                arrive(1);
#pragma unroll
                for (int w = (W + 1) / 2; w < W; ++w) hn[w] = draw(next, w);
                wait(half + 1, (unsigned)s & 1u, 2u * s + 2u);
                Hn = Hn1;
                if (--to_sample == 0) {
                    to_sample = (int)se;
                    const unsigned b = n_snap & 1u;
                    wait(freed + b, ((n_snap >> 1) & 1u) ^ 1u, 2u * s + 2u);  // the sampler is done with the buffer's last use
#pragma unroll
                    for (int w = 0; w < W; ++w)
                        if (has(w)) snap[(b * px + X0 + w) * cap + row] = m[w].z;
                    __syncwarp();
                    if (lane == 0 && alive) mbar_arrive(taken + b);
                    ++n_snap;
                }
            }
        }
        if (__any_sync(0xffffffffu, !alive)) tell();
        if (alive) stored = 2u * s;
        __syncwarp();
        cluster_sync();  // no CTA stores into a neighbour any more
        if (*(volatile unsigned *)&tail->gave_up) {  // the state stays what it was
            abandon(half, tail, stored, nw, (to_below ? 1 : 0) | (to_above ? 2 : 0), rank, line_bytes, wp, limit_ns);
            return;
        }
        if (act) {
#pragma unroll
            for (int w = 0; w < W; ++w) {
                if (!has(w)) continue;
                float *o = m_glob + 3 * (rod_cell + (size_t)((z0 * ny + row) * nx + 2 * (X0 + w)));
                const float3 a = lo3(m[w]), b = hi3(m[w]);
                o[0] = a.x;
                o[1] = a.y;
                o[2] = a.z;
                if (2 * (X0 + w) + 1 < nx) {
                    o[3] = b.x;
                    o[4] = b.y;
                    o[5] = b.z;
                }
            }
        }
        return;
    }
    if (sampling) {
        const int first = z0 * ny * nx, count = rows * nx;  // the slab's cells
        const int o = first & 31;                           // the lane of the first
        unsigned chain_up = 0, carry_up = 0, ack_down = 0;
        if (below) ack_down = in_rank(smem_u32(ack), rank - 1);
        if (above) {
            chain_up = in_rank(smem_u32(chain), rank + 1);
            carry_up = in_rank(smem_u32(carry + lane), rank + 1);
        }
        auto wait = [&](uint64_t *bar, unsigned parity) { return sampler_wait(bar, parity, tail, limit_ns); };
        const long long k_last = (step0 + n_steps) / se;
        unsigned n = 0;
        bool ok = true;
        for (long long kk = k_first; kk <= k_last; ++kk, ++n) {
            const unsigned b = n & 1u, use = (n >> 1) & 1u;
            if (!(ok = wait(taken + b, use))) break;
            float part = 0.f;
            if (below) {
                if (!(ok = wait(chain + b, use))) break;
                part = carry[b * 32 + lane];
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(ack_down + 8u * b);
            }
            for (int i = (lane - o) & 31; i < count; i += 32) {
                const int row = i / nx, x = i - row * nx;
                const pair_t v = snap[(b * px + (x >> 1)) * cap + row];
                part += x & 1 ? hi2(v) : lo2(v);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(freed + b);
            if (above) {
                if (!(ok = wait(ack + b, use ^ 1u))) break;  // the slab above has read the carry's last use
                st_cluster(carry_up + b * 128u, part);
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(chain_up + 8u * b);
            } else if (kk < p.n_samples) {
                const float mean = warp_cell_mean(part, ncell);
                if (lane == 0) {
                    samples[(size_t)rod * p.n_samples + kk] = mean;
                    if (!isfinite(mean)) atomicOr(status, 1);
                }
            }
        }
        if (!ok) tell();  // and no sample after it
    }
    __syncwarp();
    cluster_sync();
    if (*(volatile unsigned *)&tail->gave_up) cluster_sync();
}

// A kernel of the plan's shape and the launch that it takes; cfg's one attribute is *at.
template <typename K>
cudaError_t configure(K kern, const RodPlan &plan, int n_real, cudaStream_t st, cudaLaunchConfig_t *cfg, cudaLaunchAttribute *at)
{
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3((unsigned)(n_real * plan.split));
    cfg->blockDim = dim3((unsigned)plan.threads);
    cfg->dynamicSmemBytes = plan.smem_bytes;
    cfg->stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)plan.split;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem_bytes);
}

// use(kernel) with the instance for this grid and plan.
template <typename F>
cudaError_t with_kernel(const KParams &p, const RodPlan &plan, F use)
{
    const bool full = p.nx % (2 * plan.pairs_per_thread) == 0;
#define LLG_S(W, FULLV, AXV) (p.shape == 1 ? use(rod_split_kernel<W, FULLV, AXV, 1>) : use(rod_split_kernel<W, FULLV, AXV, 0>))
#define LLG_W(W)                                                                            \
    (full ? (p.axis ? LLG_S(W, true, true) : LLG_S(W, true, false))                         \
          : (p.axis ? LLG_S(W, false, true) : LLG_S(W, false, false)))
    switch (plan.pairs_per_thread) {
        case 1: return LLG_W(1);
        case 2: return LLG_W(2);
        case 4: return LLG_W(4);
        default: return cudaErrorInvalidValue;
    }
#undef LLG_W
#undef LLG_S
}

}  // namespace

// How k CTAs per rod would run: W the fewest pairs per thread that fit a CTA.
static bool split_shape(const KParams &p, int k, int smem_optin, RodPlan *plan)
{
    if (k < 1 || k > p.nz || !sweep_fits_32(p) || p.sample_every >= (1LL << 31)) return false;
    const int px = (p.nx + 1) / 2;
    const long long cap = (long long)largest_slab(p.nz, k) * p.ny;
    if (cap > kMaxThreads) return false;
    int W = 0, wp = 0;
    for (int w : {1, 2, 4}) {
        wp = (int)(((px + w - 1) / w * cap + 31) / 32);
        if (wp < kMaxThreads / 32) {
            W = w;
            break;
        }
    }
    if (W == 0) return false;
    const size_t E = (size_t)px * (size_t)(cap + 2 * p.ny), N = (size_t)px * (size_t)cap;
    const size_t smem = 48 * E + 16 * N + 64 * sizeof(float) + kTailBytes;
    if (smem + 1024 > (size_t)smem_optin) return false;
    plan->kind = 4;
    plan->split = k;
    plan->physics_warps = wp;
    plan->pairs_per_thread = W;
    plan->threads = 32 * (wp + 1);
    plan->smem_bytes = smem;
    plan->rods_per_cta = 1;
    plan->rows_per_thread = plan->cells_per_thread = 0;
    return true;
}

int split_clusters_at_once(const KParams &p, const RodPlan &plan, int dev)
{
    int prev = -1, n = 0;
    if (cudaGetDevice(&prev) != cudaSuccess || (prev != dev && cudaSetDevice(dev) != cudaSuccess)) {
        cudaGetLastError();
        return 0;
    }
    const cudaError_t e = with_kernel(p, plan, [&](auto kern) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at;
        const cudaError_t c = configure(kern, plan, 1, nullptr, &cfg, &at);
        return c != cudaSuccess ? c : cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
    });
    if (prev != dev) cudaSetDevice(prev);
    if (e == cudaSuccess) return n;
    cudaGetLastError();
    return 0;
}

// Whether cutting the rods beats one rod per SM, which takes base_us a step, and over how many CTAs.  A
// step of a slab of c pairs takes about 0.72 us + 2 ns c, with four pairs to a thread 2.1 ns where they fill
// their rows and 3.2 where not: measured 2.06 us at 672 pairs (b = 1 over 8 CTAs), 3.5 at 1344 (over 4),
// 0.77, 0.98 and 1.24 at 96, 168 and 336 (b = 2 over 8, 4 and 2), 0.84 and 1.12 at 99 and 198 (5x11x23 cells
// over 8 and 4), 3.03 at 720 (6x16x30 over 2).  Clusters run side by side as far as the GPCs hold them, the
// rest in further waves: kAtOnce is what a GB300 of 152 SMs holds at one CTA to an SM; the device at hand is asked
// about the choice (one call, not one for each k) and has the last word where it holds fewer, or none: that
// choice is made again without it, down to one rod per SM.
bool split_plan(const KParams &p, int n_real, int nsm, int smem_optin, int dev, double base_us, RodPlan *plan,
                int (*clusters_at_once)(const KParams &, const RodPlan &, int))
{
    int at_once[9] = {0, 152, 76, 48, 36, 28, 23, 15, 15};
    bool asked[9] = {};
    for (int k = 2; k <= 8; ++k) at_once[k] = std::max(1, nsm * at_once[k] / 152);
    for (;;) {
        double best = 0.9 * base_us;
        RodPlan choice{};
        for (int k = 2; k <= 8; ++k) {
            RodPlan t{};
            if (at_once[k] < 1 || !split_shape(p, k, smem_optin, &t)) continue;
            const int waves = (n_real + at_once[k] - 1) / at_once[k];
            const double c = (double)largest_slab(p.nz, k) * p.ny * ((p.nx + 1) / 2);
            const double ns = t.pairs_per_thread < 4 ? 2.0 : (p.nx % (2 * t.pairs_per_thread) == 0 ? 2.1 : 3.2);
            const double us = waves * (0.72 + 1e-3 * ns * c);
            if (us < best) {
                best = us;
                choice = t;
            }
        }
        const int k = choice.split;
        if (k == 0) return false;
        if (!asked[k]) {
            asked[k] = true;
            const int n = clusters_at_once(p, choice, dev);
            if (n < at_once[k]) {
                at_once[k] = n;
                continue;
            }
        }
        *plan = choice;
        plan->ctas = n_real * plan->split;
        return true;
    }
}

cudaError_t split_advance(const KParams &p, const RodPlan &plan, float *m, int n_real, long long step0, int n_steps,
                          float *samples, int *status, cudaStream_t st)
{
    return with_kernel(p, plan, [&](auto kern) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at;
        const cudaError_t e = configure(kern, plan, n_real, st, &cfg, &at);
        if (e != cudaSuccess) return e;
        return cudaLaunchKernelEx(&cfg, kern, p, plan.split, plan.physics_warps, m, step0, n_steps, samples, status,
                                  plan.handoff_timeout_ns, plan.withhold_handoff ? 1 : 0);
    });
}

}  // namespace llg
