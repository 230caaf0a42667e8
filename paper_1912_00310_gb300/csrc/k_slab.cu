// k_slab.cu -- the streaming engine: grids larger than shared memory (the 512x512x56 periodic
// slab) stream through shared memory once per Heun step of Eq. 1.
//
// One launch = one fused Heun step.  The state lives in HBM as float4 (x, y, z, 0) in two
// ping-pong buffers laid out [realisation][z][NY + 4][NX + 4]: every z-plane carries a two-cell
// frame holding the periodic images of the opposite faces (zeros on a free face).  So the
// halo-2 neighbourhood of any (x, y) tile of a plane is one dense rectangle of the padded plane,
// which the Tensor Memory Accelerator copies into shared memory with one instruction (a 5-D
// tiled box: float component, x, y, z, realisation) -- no per-thread staging, no index wrapping.
//
// Each CTA owns an (x, y) tile of columns and sweeps z, or a part of it with one more predictor
// plane on either side (films of few columns, slab_plan).  At iteration z it computes, column by
// column, the predictor of plane z and then the corrector of plane z-1 of the same column (the
// corrector needs the predictor of its z+ neighbour, which is that column's value just
// computed), and the predictor of a one-cell ring around the tile (the lateral neighbours the
// corrector needs next iteration).  One elected thread keeps two planes of state in flight: the
// copy of plane z+2 is issued at the start of iteration z into a three-slot ring, each slot with
// an mbarrier that completes when the copy's bytes land; every thread waits on the barrier of the
// plane it reads (with a time limit: a wait that runs out sets a status bit and the CTA stops).
// Three predictor slots rotate with z, so the corrector reads its own and its z- neighbour's
// predictor values from shared memory.  One CTA barrier per plane orders the predictor writes
// before the next plane's corrector reads and frees a state slot before it is refilled.  The
// corrector writes the new state straight to the output buffer, and the cells within two of a
// periodic face also to their images in the frame, so the next step's copies see a complete
// frame.  The three slots rotate in registers and the planes with nothing missing (no free face, no
// end of a part) run an instance of the plane without those questions: unrolling the loop by three
// instead, for compile-time slots, made it 50 KB long (458x338x45 cells 123 us a step, now 109).
//
// The arithmetic, the neighbour order (x-, x+, y-, y+, z-, z+) and the noise keys are those of
// every other engine, so the trajectory is bitwise that of the plain engine on the same grid.
//
// What bounds it: 512x512x56 takes 187 us a step on a GB300 (205 before: the noise's first rounds,
// which depend on the step only, are made once per launch; shorter noise and torque arithmetic; the
// next launch's set-up runs under the tail of this one; the shorter loop).  The state alone is 470 MB
// there and back, 70 us at the copy rate; the rest is instructions: 256 a warp-cell with the ring's
// second predictor, issued at 0.58 a cycle by the 16 warps that 128 registers leave an SM, which wait
// on fixed latencies (1.4 cycles an instruction) and on the barrier of every plane (0.9).  Tried: 20
// warps with three columns a thread at 96 registers issue at 0.64 but need a tenth more instructions
// (192 us before the shorter loop, 254 with it, from spills); noise drawn between arriving at the
// barrier and waiting for it 187; pairs of columns with packed arithmetic 266 (spills).  With
// dispersed axes 285 us (304): their loads' latency is exposed, so each plane asks L2 for the next.
#include <cuda.h>  // CUtensorMap and its enums; the encoder is fetched from the driver at run time

#include <algorithm>
#include <cmath>
#include <cstring>

#include "llg_internal.h"
#include "mbarrier.cuh"
#include "physics.cuh"

namespace llg {
namespace {

constexpr int kSlabThreads = 512;
// With one column a thread: the ring's cells then have warps of their own, so that no warp makes two
// predictors in a row (201x139x17 cells, two films: 24.0 -> 22.8 us a step; 64x64x20 8.5 -> 8.0).
constexpr int kSlabThreads1 = 576;
constexpr int kFixedThreads = 512, kFixedRows = kFixedThreads / 64;  // tiles of 64 columns in x, four a thread
constexpr int kFixedPitch = 64 + 4, kFixedBoxRows = 27 + 4;
constexpr unsigned long long kStageWaitNs = 2000000000ull;  // longest wait for a staged plane

__device__ __forceinline__ float3 zero3s() { return make_float3(0.f, 0.f, 0.f); }

// One box of the padded state: coordinates (float component, x, y, z, realisation).
__device__ __forceinline__ void tma_load_plane(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, int z,
                                               int r)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_u32(dst)),
        "l"((unsigned long long)map), "r"(0), "r"(x), "r"(y), "r"(z), "r"(r), "r"(smem_u32(bar))
        : "memory");
}

struct SlabGeom {
    int NX, NY, NZ;
    int NXp, NYp;        // padded extents NX + 4, NY + 4
    int tiles_x, tiles_y, parts;  // parts: CTAs along z
    int TXmax, TYmax;
    int pitch, rows;     // copied box: (TXmax + 4) x (TYmax + 4) float4
    int slot;            // float4 entries per state slot (box rounded up to 128 bytes)
    int tslot;           // float4 entries per predictor slot (two rows fewer)
    unsigned box_bytes;  // bytes of one copied box
};

__host__ __device__ constexpr int slot_of(int pitch, int rows) { return (pitch * rows + 7) / 8 * 8; }

// Per-CTA state of the z sweep.  PITCH, ROWS > 0: the slots' geometry at compile time.  FIXED: tiles of
// exactly PITCH - 4 = 64 columns in x and kFixedThreads threads -- then the columns of a thread share
// their x and lie kFixedRows rows apart, so their positions are strides from the first column's (kept in
// registers for one column only).  Every film of a multiple of 64 cells in x whose tiles are 25 to 27
// rows high runs it (the box may have fewer rows than its slot).
template <int CPT, int PITCH, int ROWS, bool AX, bool FIXED = false>
struct SlabSweep {
    static constexpr bool kFixed = FIXED;
    float4 *Mb, *Tb;     // [3][slot] state planes; [3][tslot] predictor planes (Tb one row early)
    uint64_t *bar;       // [3] one mbarrier per state slot
    int pitch_rt, slot_rt;
    // the CTA's part of z: planes [za, zb) get their corrector, [zs, ze) their predictor (one more on either
    // side), [l0, l1) are staged (one more again)
    int za, zb, zs, ze, l0, l1;
    bool lead;           // the thread that issues the copies
    int tile_x, tile_y, real;
    const CUtensorMap *tin;
    float4 *dst;         // this realisation's output state
    int plane_p;         // float4 entries per padded plane
    uint32_t plane_c;    // cells per interior plane
    PhiloxKeys keys;
    PhiloxStep now;      // the noise's first rounds for this step
    const float4 *axr;
    float Hn, Hn1;
    int *status;
    // columns of this thread (kFixed: only [0] is kept; column k is [0] plus k row strides)
    int q_[kFixed ? 1 : CPT];          // position in a staged plane
    uint32_t cell_[kFixed ? 1 : CPT];  // interior cell index in plane 0 (+ plane_c per plane)
    int gofs_[kFixed ? 1 : CPT];       // padded position in a plane
    unsigned actm;       // bit k: column k lies in the tile
    unsigned ghost;      // bit k: column k lies within two cells of a periodic face
    __device__ __forceinline__ int q(int k) const
    {
        if constexpr (kFixed) return q_[0] + k * kFixedRows * PITCH;
        return q_[k];
    }
    __device__ __forceinline__ uint32_t cell(int k) const
    {
        if constexpr (kFixed) return cell_[0] + (uint32_t)(k * kFixedRows * NX);
        return cell_[k];
    }
    __device__ __forceinline__ int gofs(int k) const
    {
        if constexpr (kFixed) return gofs_[0] + k * kFixedRows * NXp;
        return gofs_[k];
    }
    __device__ __forceinline__ int nthreads() const { return FIXED ? kFixedThreads : (int)blockDim.x; }
    __device__ __forceinline__ bool act(int k) const { return (actm >> k) & 1u; }
    // ring cell of this thread (predictor only)
    int rpos;
    uint32_t rcell;
    bool ract, rin;
    int NX, NY, NXp;
    bool perx, pery;
    // registers carried along z: the own state of plane z-1 (its slot is refilled before the
    // predictor of plane z reads it; the own state of plane z is re-read from its slot) and the
    // torque of the last predictor; the thermal field the corrector
    // reuses waits in shared memory (Hs), which keeps the four-column instance in registers
    float3 Sp[CPT], A[CPT];  // own state of the previous plane, torque of the last predictor
    float3 rSp;              // the ring cell's state of the previous plane
    float4 *Hs;          // [CPT][blockDim.x] thermal field of the own columns' last predictor

    __device__ __forceinline__ int pitch() const
    {
        if constexpr (PITCH > 0) return PITCH;
        return pitch_rt;
    }
    __device__ __forceinline__ int slot() const
    {
        if constexpr (PITCH > 0) return slot_of(PITCH, ROWS);
        return slot_rt;
    }
    // predictor slots hold only the tile and its one-cell ring: two rows fewer than a state slot,
    // addressed with the state slots' positions through a base one row back (Tb = start - pitch)
    __device__ __forceinline__ int tslot() const
    {
        if constexpr (PITCH > 0) return slot_of(PITCH, ROWS - 2);
        return tslot_rt;
    }
    int tslot_rt;

    unsigned box_bytes;
    int s0, sm1, sp1;  // slots of planes z, z-1, z+1 (and z-2)
    unsigned par_next;  // parity of plane z+1's use of its slot
    int last_issued;  // lead thread: the last plane whose copy was issued

    __device__ __forceinline__ float3 noise(const KParams &p, uint32_t c) const
    {
        return box_muller3(philox4x32_10(keys, now, (unsigned long long)kPhiloxM0 * c), p.sigma_bm);
    }

    __device__ __forceinline__ void issue(int z, int s)
    {
        mbar_arrive_expect(bar + s, box_bytes);
        tma_load_plane(Mb + s * slot(), tin, bar + s, tile_x, tile_y, z, real);
        last_issued = z;
    }

    // After a staging wait gave up: let the copies still in flight land before the CTA's shared
    // memory is released (each wait bounded).  The CTA's t-th plane (t = z - l0) uses slot t mod 3 for the
    // (t / 3)-th time.
    __device__ void drain()
    {
        for (int t = max(0, last_issued - l0 - 2); t <= last_issued - l0; ++t)
            mbar_wait<false>(bar + t % 3, (unsigned)((t / 3) & 1), kStageWaitNs);
    }

    // A column's new state goes to its padded position and, near a periodic face, to the images
    // of that position in the frame (x image, y image, corner image).
    __device__ __forceinline__ void store(int k, int zc, float4 v)
    {
        float4 *o = dst + (size_t)zc * plane_p;
        o[gofs(k)] = v;
        if ((ghost >> k) & 1u) {
            const int X = (int)(cell(k) % (uint32_t)NX), Y = (int)(cell(k) / (uint32_t)NX);
            const int gx = (perx && X < 2) ? X + NX + 2 : ((perx && X >= NX - 2) ? X - NX + 2 : -1);
            const int gy = (pery && Y < 2) ? Y + NY + 2 : ((pery && Y >= NY - 2) ? Y - NY + 2 : -1);
            if (gx >= 0) o[(Y + 2) * NXp + gx] = v;
            if (gy >= 0) o[gy * NXp + X + 2] = v;
            if (gx >= 0 && gy >= 0) o[gy * NXp + gx] = v;
        }
    }

    // Iteration z of the sweep: predictor of plane z and corrector of plane z - 1, where they belong to the CTA's
    // part (a first plane staged only for the predictor above it is just
    // remembered).  Ends in a CTA barrier; returns true (in every thread) when some thread's staging wait
    // gave up.
    template <bool INNER>
    __device__ __forceinline__ bool iteration(const KParams &p, int z)
    {
        const int P = pitch();
        const bool pred = INNER || (z >= zs && z < ze), corr = INNER || z > za;
        const bool has_next = INNER || z + 1 < l1;
        int fail = 0;
        // plane z+1, issued an iteration ago
        if (has_next && !mbar_wait<false>(bar + sp1, par_next, kStageWaitNs)) {
            atomicOr(status, 4);
            fail = 1;
        }
        // plane z+2 into the slot plane z-1 left (freed by the previous iteration's barrier)
        if (lead && z + 2 < l1) issue(z + 2, sm1);
        const float4 *Mz = Mb + s0 * slot(), *Mn = Mb + sp1 * slot();
        float4 *Tw = Tb + s0 * tslot();
        const float4 *Tr = Tb + sm1 * tslot(), *Tp = Tb + sp1 * tslot();
        const uint32_t zoff = plane_c * (uint32_t)z, zcoff = plane_c * (uint32_t)(z - 1);
#pragma unroll
        for (int k = 0; k < CPT; ++k) {
            if (!act(k)) continue;
            const int c = q(k);
            float3 tnew = zero3s(), h = zero3s(), anew = zero3s();
            const float3 mcorr = Sp[k];  // the state of plane z-1, which the corrector starts from
            float4 *hs = Hs + k * nthreads() + threadIdx.x;
            if (pred) {
                const float3 mcur = xyz(Mz[c]);
                const float3 mnext = has_next ? xyz(Mn[c]) : zero3s();
                h = noise(p, cell(k) + zoff);
                float3 nb = add3(xyz(Mz[c - 1]), xyz(Mz[c + 1]));
                nb = add3(nb, xyz(Mz[c - P]));
                nb = add3(nb, xyz(Mz[c + P]));
                nb = add3(nb, Sp[k]);
                nb = add3(nb, mnext);
                Sp[k] = mcur;
                const float3 u = AX ? xyz(__ldg(axr + cell(k) + zoff)) : zero3s();
                const float3 H = effective_field_sel<AX>(nb, mcur, h, p, Hn, u);
                anew = llg_torque(mcur, H, p.alpha);
                tnew = normalised(axpy(p.neg_dt_g1, anew, mcur));
                Tw[c] = pad4(tnew);
            }
            if (corr) {
                const float3 tself = xyz(Tr[c]);
                const float3 tprev = INNER || z >= 2 ? xyz(Tp[c]) : zero3s();
                float3 nb = add3(xyz(Tr[c - 1]), xyz(Tr[c + 1]));
                nb = add3(nb, xyz(Tr[c - P]));
                nb = add3(nb, xyz(Tr[c + P]));
                nb = add3(nb, tprev);
                nb = add3(nb, pred ? tnew : zero3s());
                const float3 u = AX ? xyz(__ldg(axr + cell(k) + zcoff)) : zero3s();
                const float3 H = effective_field_sel<AX>(nb, tself, xyz(*hs), p, Hn1, u);
                const float3 sv = llg_torque_add(A[k], tself, H, p.alpha);
                store(k, z - 1, pad4(normalised(axpy(p.neg_hdt_g1, sv, mcorr))));
            }
            if (pred) {
                *hs = pad4(h);  // after the corrector read the previous plane's
                A[k] = anew;
            }
        }
        if (AX && z + 1 < ze) {  // the next plane's axes on their way to L2 (their loads' latency is exposed)
#pragma unroll
            for (int k = 0; k < CPT; ++k)
                if (act(k)) asm volatile("prefetch.global.L2 [%0];" ::"l"(axr + cell(k) + zoff + plane_c));
        }
        if (!INNER && z < zs) {
#pragma unroll
            for (int k = 0; k < CPT; ++k)
                if (act(k)) Sp[k] = xyz(Mz[q(k)]);
            if (rin) rSp = xyz(Mz[rpos]);
        }
        if (pred && ract) {
            float3 rt = zero3s();
            if (rin) {
                const float3 rcur = xyz(Mz[rpos]);
                const float3 rnext = has_next ? xyz(Mn[rpos]) : zero3s();
                const float3 h = noise(p, rcell + zoff);
                float3 nb = add3(xyz(Mz[rpos - 1]), xyz(Mz[rpos + 1]));
                nb = add3(nb, xyz(Mz[rpos - P]));
                nb = add3(nb, xyz(Mz[rpos + P]));
                nb = add3(nb, rSp);
                nb = add3(nb, rnext);
                const float3 u = AX ? xyz(__ldg(axr + rcell + zoff)) : zero3s();
                const float3 H = effective_field_sel<AX>(nb, rcur, h, p, Hn, u);
                rt = normalised(axpy(p.neg_dt_g1, llg_torque(rcur, H, p.alpha), rcur));
                rSp = rcur;
            }
            Tw[rpos] = pad4(rt);
        }
        return __syncthreads_or(fail) != 0;
    }
};

template <int CPT, int PITCH, int ROWS, bool AX, bool FIXED = false>
__global__ void __launch_bounds__(FIXED ? kFixedThreads : CPT == 1 ? kSlabThreads1 : kSlabThreads, 1) slab_step_kernel(KParams p, SlabGeom G,
                                                                    const __grid_constant__ CUtensorMap tin,
                                                                    float4 *__restrict__ mout, unsigned long long n,
                                                                    int *__restrict__ status)
{
    extern __shared__ __align__(128) float4 sm4[];
    // the copies need a 128-byte aligned destination; refuse (status bit) rather than fault
    if (smem_u32(sm4) & 127u) {
        if (threadIdx.x == 0) atomicOr(status, 4);
        return;
    }
    SlabSweep<CPT, PITCH, ROWS, AX, FIXED> w;
    w.pitch_rt = G.pitch;
    w.slot_rt = G.slot;
    w.tslot_rt = G.tslot;
    const int slot = w.slot(), tslot = w.tslot();
    w.Mb = sm4;
    w.Tb = sm4 + 3 * slot - w.pitch();  // row 0 of a predictor slot is row 1 of the box
    w.Hs = sm4 + 3 * slot + 3 * tslot;
    w.bar = reinterpret_cast<uint64_t *>(w.Hs + CPT * blockDim.x);
    w.NX = G.NX;
    w.NY = G.NY;
    w.NXp = G.NXp;
    w.perx = p.periodic & 1u;
    w.pery = p.periodic & 2u;
    w.lead = threadIdx.x == 0;
    w.tin = &tin;
    w.box_bytes = G.box_bytes;
    w.status = status;
    const int tx = blockIdx.x, ty = blockIdx.y, real = blockIdx.z / G.parts, part = blockIdx.z % G.parts;
    w.za = (int)((long long)part * G.NZ / G.parts);
    w.zb = (int)((long long)(part + 1) * G.NZ / G.parts);
    w.zs = max(0, w.za - 1);
    w.ze = min(G.NZ, w.zb + 1);
    w.l0 = max(0, w.zs - 1);
    w.l1 = min(G.NZ, w.ze + 1);
    const int x0 = (int)((long long)tx * G.NX / G.tiles_x), x1 = (int)((long long)(tx + 1) * G.NX / G.tiles_x);
    const int y0 = (int)((long long)ty * G.NY / G.tiles_y), y1 = (int)((long long)(ty + 1) * G.NY / G.tiles_y);
    const int TX = x1 - x0, TY = y1 - y0;
    // the box starts two cells before the tile: padded coordinates (x0, y0)
    w.tile_x = x0;
    w.tile_y = y0;
    w.real = real;
    w.plane_p = G.NXp * G.NYp;
    w.plane_c = (uint32_t)G.NX * (uint32_t)G.NY;
    w.dst = mout + (size_t)real * (size_t)w.plane_p * G.NZ;
    w.keys = philox_keys(p.seed, p.real0 + (uint32_t)real);
    w.now = philox_step(w.keys, n);
    w.axr = AX ? p.axis + (size_t)real * w.plane_c * G.NZ : nullptr;
    {
        Sweep sw;
        sw.init((long long)n, p);
        w.Hn = sw.value();
        sw.inc();
        w.Hn1 = sw.value();
    }
    const int P = w.pitch();
    w.ghost = 0u;
    w.actm = 0u;
#pragma unroll
    for (int k = 0; k < CPT; ++k) {
        const int c = threadIdx.x + k * w.nthreads();
        const bool a = c < TX * TY;
        const int cc = a ? c : (int)threadIdx.x;  // an idle slot keeps the first column's position
        const int lx = cc % TX, ly = cc / TX;
        const int X = x0 + lx, Y = y0 + ly;
        if (k == 0 || !w.kFixed) {
            w.q_[w.kFixed ? 0 : k] = (ly + 2) * P + (lx + 2);
            w.cell_[w.kFixed ? 0 : k] = (uint32_t)(X + G.NX * Y);
            w.gofs_[w.kFixed ? 0 : k] = (Y + 2) * G.NXp + (X + 2);
        }
        const bool near = (w.perx && (X < 2 || X >= G.NX - 2)) || (w.pery && (Y < 2 || Y >= G.NY - 2));
        if (a) w.actm |= 1u << k;
        if (a && near) w.ghost |= 1u << k;
    }
    // ring cell (predictor only), counted from the last thread down: the last threads own the
    // fewest interior columns.  Order: the y- row, the y+ row, then x- / x+ pairs by row.
    {
        const int nring = 2 * TX + 2 * TY;
        const int ridx = (int)blockDim.x - 1 - (int)threadIdx.x;
        w.ract = ridx < nring;
        const int i = w.ract ? ridx : 0;
        int lx, ly;
        if (i < 2 * TX) {
            lx = i % TX;
            ly = i < TX ? -1 : TY;
        } else {
            const int j = i - 2 * TX;
            lx = (j & 1) ? TX : -1;
            ly = j >> 1;
        }
        w.rpos = (ly + 2) * P + (lx + 2);
        int gx = x0 + lx, gy = y0 + ly;
        bool in = true;
        if (gx < 0 || gx >= G.NX) {
            in = in && w.perx;
            gx = (gx % G.NX + G.NX) % G.NX;
        }
        if (gy < 0 || gy >= G.NY) {
            in = in && w.pery;
            gy = (gy % G.NY + G.NY) % G.NY;
        }
        w.rin = w.ract && in;
        w.rcell = (uint32_t)(gx + G.NX * gy);
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < 3; ++s) mbar_init(w.bar + s, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    w.last_issued = -1;
    // Everything above is this launch's own; the state that the previous step writes, and the buffer that it
    // still reads, are touched from here on.  The next step's CTAs may set themselves up meanwhile (its wait
    // is for this whole launch).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (w.lead) {
        asm volatile("fence.proxy.async;" ::: "memory");  // the copies read what the step before wrote
        w.issue(w.l0, 0);
        if (w.l0 + 1 < w.l1) w.issue(w.l0 + 1, 1);
    }
    // the first plane before the sweep starts
    int fail = 0;
    if (!mbar_wait<false>(w.bar, 0u, kStageWaitNs)) {
        atomicOr(status, 4);
        fail = 1;
    }
#pragma unroll
    for (int k = 0; k < CPT; ++k) w.Sp[k] = w.A[k] = zero3s();  // plane -1 of a first part: the free z face
    w.rSp = zero3s();
    bool aborted = __syncthreads_or(fail) != 0;
    w.s0 = 0;
    w.sp1 = 1;
    w.sm1 = 2;
    w.par_next = 0u;
    // from a part's second corrector plane to its last predictor plane but one nothing is missing
    const int inner0 = max(w.za + 1, 2), inner1 = min(w.ze, w.l1 - 1);
    for (int z = w.l0; z <= w.zb && !aborted; ++z) {
        aborted = z >= inner0 && z < inner1 ? w.template iteration<true>(p, z) : w.template iteration<false>(p, z);
        const int s = w.s0;
        w.s0 = w.sp1;
        w.sp1 = w.sm1;
        w.sm1 = s;
        if (w.sp1 == 0) w.par_next ^= 1u;
    }
    if (aborted && w.lead) w.drain();
}

// Pack the AoS float3 state into the padded float4 layout (frame = periodic images or zeros),
// and back.
// (I: the index type, 32 bits wherever the padded state has fewer entries -- three 64-bit divisions an entry
// otherwise took as long as the copy.)
template <typename I>
__global__ void pack_padded_kernel(const float *__restrict__ m, float4 *__restrict__ out, int NX, int NY, int NZ,
                                   unsigned periodic, I total)
{
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const I NXp = NX + 4, NYp = NY + 4;
    const int xp = (int)(i % NXp);
    const I t = i / NXp;
    const int yp = (int)(t % NYp);
    const I t2 = t / NYp;
    const int z = (int)(t2 % (I)NZ);
    const I r = t2 / (I)NZ;
    int x = xp - 2, y = yp - 2;
    bool in = true;
    if (x < 0 || x >= NX) {
        in = in && (periodic & 1u);
        x = (x % NX + NX) % NX;
    }
    if (y < 0 || y >= NY) {
        in = in && (periodic & 2u);
        y = (y % NY + NY) % NY;
    }
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (in) {
        const float *src = m + 3 * ((size_t)r * NX * NY * NZ + (size_t)x + (size_t)NX * (y + (size_t)NY * z));
        v = make_float4(src[0], src[1], src[2], 0.f);
    }
    out[i] = v;
}

template <typename I>
__global__ void unpack_padded_kernel(const float4 *__restrict__ in, float *__restrict__ m, int NX, int NY, int NZ, I total)
{
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const I t = i / (I)NX, t2 = t / (I)NY;
    const int x = (int)(i - t * (I)NX), y = (int)(t - t2 * (I)NY), z = (int)(t2 % (I)NZ);
    const I r = t2 / (I)NZ;
    const float4 v = in[(size_t)r * (NX + 4) * (NY + 4) * NZ + ((size_t)z * (NY + 4) + (y + 2)) * (NX + 4) + (x + 2)];
    float *o = m + 3 * (size_t)i;
    o[0] = v.x;
    o[1] = v.y;
    o[2] = v.z;
}

// Deterministic two-pass mean of m_z per realisation: pass 1 sums fixed contiguous chunks of the
// interior cell index (strided per thread, then a fixed shuffle/shared-memory tree), pass 2 sums
// the chunk partials in order with one warp.
constexpr int kRedBlocks = 256, kRedThreads = 256;

__global__ void slab_partial_kernel(const float4 *__restrict__ m, int NX, int NY, int NZ, float *__restrict__ partial)
{
    const int real = blockIdx.y;
    const long long ncells = (long long)NX * NY * NZ;
    const float4 *mr = m + (size_t)real * (NX + 4) * (NY + 4) * NZ;
    const long long chunk = (ncells + gridDim.x - 1) / gridDim.x;
    const long long a = blockIdx.x * chunk, b = min(ncells, a + chunk);
    float s = 0.f;
    for (long long i = a + threadIdx.x; i < b; i += blockDim.x) {
        const int x = (int)(i % NX), y = (int)((i / NX) % NY), z = (int)(i / ((long long)NX * NY));
        s += mr[((size_t)z * (NY + 4) + (y + 2)) * (NX + 4) + (x + 2)].z;
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    __shared__ float ws[kRedThreads / 32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < kRedThreads / 32; ++w) t += ws[w];
        partial[(size_t)real * gridDim.x + blockIdx.x] = t;
    }
}

__global__ void slab_sample_kernel(const float *__restrict__ partial, int nparts, long long ncells,
                                   long long k, long long n_samples, float *__restrict__ samples,
                                   int *__restrict__ status)
{
    const int real = blockIdx.x;
    float s = 0.f;
    for (int i = threadIdx.x; i < nparts; i += 32) s += partial[(size_t)real * nparts + i];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (threadIdx.x == 0) {
        const float mean = (float)((double)s / (double)ncells);
        samples[(size_t)real * n_samples + k] = mean;
        if (!isfinite(mean)) atomicOr(status, 1);
    }
}

// cuTensorMapEncodeTiled from the driver (no link-time dependency on libcuda).
using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder()
{
    static EncodeTiled fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
        else
            cudaGetLastError();
    }
    return fn;
}

// Tensor map of a padded state buffer: dims (4 floats, NX + 4, NY + 4, NZ, n_real), box
// (4, pitch, rows, 1, 1); out-of-range elements (past the last tile's box) read as zero.
bool encode_state_map(CUtensorMap *map, float4 *base, const SlabGeom &G, int n_real)
{
    EncodeTiled fn = encoder();
    if (!fn) return false;
    const cuuint64_t dims[5] = {4, (cuuint64_t)G.NXp, (cuuint64_t)G.NYp, (cuuint64_t)G.NZ, (cuuint64_t)n_real};
    const cuuint64_t strides[4] = {16, 16ull * G.NXp, 16ull * G.NXp * G.NYp, 16ull * G.NXp * G.NYp * G.NZ};
    const cuuint32_t box[5] = {4, (cuuint32_t)G.pitch, (cuuint32_t)G.rows, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int C, bool AX>
cudaError_t launch_step(const KParams &p, const SlabGeom &G, const SlabPlan &plan, const CUtensorMap &map,
                        float4 *out, int n_real, unsigned long long n, int *status, cudaStream_t st)
{
    const dim3 grid(G.tiles_x, G.tiles_y, n_real * G.parts);
    auto go = [&](auto kern) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem_bytes);
        if (e != cudaSuccess) return e;
        // a step may be launched while the one before it drains (griddepcontrol in the kernel)
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = dim3(plan.threads);
        cfg.dynamicSmemBytes = plan.smem_bytes;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kern, p, G, map, out, n, status);
    };
    if constexpr (C == 4)
        if (plan.fixed) return go(slab_step_kernel<4, kFixedPitch, kFixedBoxRows, AX, true>);
    if constexpr (C == 4)
        if (G.pitch == kFixedPitch && G.rows == kFixedBoxRows)
            return go(slab_step_kernel<4, kFixedPitch, kFixedBoxRows, AX>);
    return go(slab_step_kernel<C, 0, 0, AX>);
}

}  // namespace

bool slab_plan(const KParams &p, int n_real, int dev, SlabPlan *plan)
{
    if (p.periodic & 4u) return false;  // free z faces only
    // a periodic axis needs at least four cells, so that each cell has at most one image per axis
    // in the two-cell frame
    if (((p.periodic & 1u) && p.nx < 4) || ((p.periodic & 2u) && p.ny < 4)) return false;
    if (!encoder()) return false;
    int smem_optin = 0, nsm = 0;
    if (cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return false;
    const int tiles_x = (p.nx + 63) / 64;
    const int TXmax = (p.nx + tiles_x - 1) / tiles_x;
    // three state slots, three predictor slots, the thermal-field store of every column slot of the
    // CTA, three mbarriers
    auto fixed = [&](int ty) { return p.nx % 64 == 0 && 64 * ty > 3 * kSlabThreads && ty + 4 <= kFixedBoxRows; };
    auto threads_of = [&](int ty) {
        if (fixed(ty)) return +kFixedThreads;
        const int cols = (TXmax * ty + 31) / 32 * 32, ring = (2 * TXmax + 2 * ty + 31) / 32 * 32;
        if (cols <= kSlabThreads && cols + ring <= kSlabThreads1) return cols + ring;
        return std::min(+kSlabThreads, std::max(cols, ring));
    };
    auto cpt_of = [&](int ty) { return fixed(ty) ? 4 : (TXmax * ty + kSlabThreads - 1) / kSlabThreads; };
    auto smem_of = [&](int ty) {
        const int rows = fixed(ty) ? kFixedBoxRows : ty + 4;
        return (size_t)3 * (slot_of(TXmax + 4, rows) + slot_of(TXmax + 4, rows - 2)) * sizeof(float4) +
               (size_t)cpt_of(ty) * threads_of(ty) * sizeof(float4) + 3 * sizeof(uint64_t);
    };
    auto holds = [&](int ty) {
        return TXmax * ty <= 4 * kSlabThreads && smem_of(ty) <= (size_t)smem_optin && TXmax + 4 <= 256 && ty + 4 <= 256 &&
               2 * TXmax + 2 * ty <= threads_of(ty);
    };
    // The tiles and the parts of z, by the step time that fits the measured ones within a fifth: 1 us of launch,
    // and for every plane that a CTA sweeps (its part, two more predictor planes where z is cut, one more for
    // the corrector's lag) 0.63 us of latency -- copy, predictor, corrector, barrier -- and 0.05 us for every 32
    // columns (the ring's predictor counts 0.6).  A film of few columns leaves SMs idle or its CTAs with few
    // warps, so cutting z pays: 131x72x39 cells 40.9 -> 13.5 us a step (3x6 tiles, 8 parts), 64x64x20
    // 24.7 -> 8.5, 30x450x50 51.3 -> 18.1 (of which 2.5 to 4.5 us come from the overlapped launch);
    // 512x512x56 (8x19 tiles) stays whole (208.9 in two parts where it took 198.7).
    double best = 0.0;
    bool found = false;
    auto consider = [&](int tiles_y, int parts) {
        tiles_y = std::max(1, std::min(p.ny, tiles_y));
        int ty = (p.ny + tiles_y - 1) / tiles_y;
        while (ty > 1 && !holds(ty)) {
            ++tiles_y;
            ty = (p.ny + tiles_y - 1) / tiles_y;
        }
        if (!holds(ty) || (parts > 1 && (long long)n_real * parts > 65535)) return;  // the grid's z extent
        const double ctas = (double)tiles_x * tiles_y * parts * n_real;
        const int planes = (p.nz + parts - 1) / parts + 1 + (parts > 1 ? 2 : 0);
        const double warps = (TXmax * ty + 0.6 * (2 * TXmax + 2 * ty)) / 32.0;
        const double us = 1.0 + std::ceil(ctas / nsm) * planes * (0.63 + 0.05 * warps);
        if (found && us > 0.95 * best) return;
        best = us;
        found = true;
        plan->tiles_x = tiles_x;
        plan->tiles_y = tiles_y;
        plan->parts = parts;
        plan->TXmax = TXmax;
        plan->TYmax = ty;
        plan->fixed = fixed(ty);
        plan->cols_per_thread = cpt_of(ty);
        plan->threads = threads_of(ty);
        plan->smem_bytes = smem_of(ty);
    };
    consider(nsm / tiles_x, 1);
    for (int parts = 1; parts <= 8 && 3 * parts <= std::max(3, p.nz); ++parts)
        for (int per_sm : {1, 2}) consider((int)(per_sm * (long long)nsm / ((long long)tiles_x * parts * n_real)), parts);
    return found;
}

size_t slab_state_float4s(const KParams &p, int n_real)
{
    return (size_t)n_real * (size_t)(p.nx + 4) * (size_t)(p.ny + 4) * (size_t)p.nz;
}

cudaError_t slab_advance(const KParams &p, const SlabPlan &plan, float *m, int n_real, long long step0,
                         long long n_steps, float *samples, int *status, float4 *buf_a, float4 *buf_b,
                         float *partial, cudaStream_t st, long long *launches)
{
    SlabGeom G{};
    G.NX = p.nx;
    G.NY = p.ny;
    G.NZ = p.nz;
    G.NXp = p.nx + 4;
    G.NYp = p.ny + 4;
    G.tiles_x = plan.tiles_x;
    G.tiles_y = plan.tiles_y;
    G.parts = plan.parts;
    G.TXmax = plan.TXmax;
    G.TYmax = plan.TYmax;
    G.pitch = plan.TXmax + 4;
    G.rows = plan.TYmax + 4;
    G.slot = slot_of(G.pitch, plan.fixed ? kFixedBoxRows : G.rows);
    G.tslot = slot_of(G.pitch, (plan.fixed ? kFixedBoxRows : G.rows) - 2);
    G.box_bytes = (unsigned)(G.pitch * G.rows * sizeof(float4));
    CUtensorMap map_a, map_b;
    if (!encode_state_map(&map_a, buf_a, G, n_real) || !encode_state_map(&map_b, buf_b, G, n_real))
        return cudaErrorInvalidValue;
    const long long padded = (long long)slab_state_float4s(p, n_real);
    const long long total = (long long)p.ncells * n_real;
    const bool narrow = padded < (1LL << 31) && total < (1LL << 31);
    auto pack = [&](float4 *out) {
        const unsigned blocks = (unsigned)((padded + 255) / 256);
        if (narrow)
            pack_padded_kernel<unsigned><<<blocks, 256, 0, st>>>(m, out, p.nx, p.ny, p.nz, p.periodic, (unsigned)padded);
        else
            pack_padded_kernel<long long><<<blocks, 256, 0, st>>>(m, out, p.nx, p.ny, p.nz, p.periodic, padded);
    };
    pack(buf_a);
    // the output buffer's frame: its periodic images are rewritten every step, but a free face's zeros must
    // be there from the start
    const bool framed = (p.periodic & 3u) == 3u;
    if (!framed) pack(buf_b);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    float4 *a = buf_a, *b = buf_b;
    const CUtensorMap *ma = &map_a, *mb = &map_b;
    long long count = framed ? 1 : 2;
    for (long long s = 0; s < n_steps; ++s) {
        const unsigned long long n = (unsigned long long)(step0 + s);
        switch (plan.cols_per_thread) {
            case 1:
                e = p.axis ? launch_step<1, true>(p, G, plan, *ma, b, n_real, n, status, st)
                           : launch_step<1, false>(p, G, plan, *ma, b, n_real, n, status, st);
                break;
            case 2:
                e = p.axis ? launch_step<2, true>(p, G, plan, *ma, b, n_real, n, status, st)
                           : launch_step<2, false>(p, G, plan, *ma, b, n_real, n, status, st);
                break;
            case 3:
                e = p.axis ? launch_step<3, true>(p, G, plan, *ma, b, n_real, n, status, st)
                           : launch_step<3, false>(p, G, plan, *ma, b, n_real, n, status, st);
                break;
            case 4:
                e = p.axis ? launch_step<4, true>(p, G, plan, *ma, b, n_real, n, status, st)
                           : launch_step<4, false>(p, G, plan, *ma, b, n_real, n, status, st);
                break;
            default:
                return cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
        ++count;
        std::swap(a, b);
        std::swap(ma, mb);
        const long long done = (long long)n + 1;
        if (samples && p.sample_every > 0 && done % p.sample_every == 0 && done / p.sample_every < p.n_samples) {
            slab_partial_kernel<<<dim3(kRedBlocks, n_real), kRedThreads, 0, st>>>(a, p.nx, p.ny, p.nz, partial);
            slab_sample_kernel<<<n_real, 32, 0, st>>>(partial, kRedBlocks, p.ncells, done / p.sample_every,
                                                      p.n_samples, samples, status);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            count += 2;
        }
    }
    const unsigned blocks = (unsigned)((total + 255) / 256);
    if (narrow)
        unpack_padded_kernel<unsigned><<<blocks, 256, 0, st>>>(a, m, p.nx, p.ny, p.nz, (unsigned)total);
    else
        unpack_padded_kernel<long long><<<blocks, 256, 0, st>>>(a, m, p.nx, p.ny, p.nz, total);
    ++count;
    if (launches) *launches += count;
    return cudaGetLastError();
}

size_t slab_partial_floats(int n_real) { return (size_t)kRedBlocks * n_real; }

}  // namespace llg
