// Device helpers shared by the forward kernel (idm_sim.cu) and the adjoint
// kernels (idm_adjoint.cuh): work distribution, compensated sums, cp.async,
// warp groups (segments run by several warps of one block), vehicle loads.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "idm_device.cuh"
#include "idm_internal.h"

namespace idm {

// ---------------------------------------------------------------------------
// Helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ int next_segment(int *work, int lane)
{
    int s = 0;
    if (lane == 0) s = atomicAdd(work, 1);
    return __shfl_sync(FULL, s, 0);
}

// Kahan-compensated float accumulation.
__device__ __forceinline__ void kahan_add(float &sum, float &comp, float x)
{
    float y = __fsub_rn(x, comp);
    float t = __fadd_rn(sum, y);
    comp = __fsub_rn(__fsub_rn(t, sum), y);
    sum = t;
}

__device__ __forceinline__ double warp_sum_double(double x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
    return x;
}

// Asynchronous 4-byte global->shared copies (cp.async, completion tracked
// per thread in commit groups).
__device__ __forceinline__ void cp_async4(float *smem_dst, const float *gsrc)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void cp_async16(float *smem_dst, const float *gsrc)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gsrc) : "memory");
}

// Offset of pair p from the lane's first slot.
template <bool CONSEC>
__device__ __forceinline__ constexpr int pair_off(int p)
{
    return CONSEC ? 2 * p : 64 * p;
}

// Copy this lane's occupied slots (mask) of one row: dst and src point at the
// lane's first slot.  vec: all 2 NP slots are occupied and consecutive and the
// source is 16-byte aligned.
template <int NP, bool CONSEC>
__device__ __forceinline__ void prefetch_row(float *dst, const float *src, const int (&mask)[NP][2], bool vec)
{
    if (CONSEC && NP >= 2 && vec) {
#pragma unroll
        for (int c = 0; c < 2 * NP; c += 4) cp_async16(dst + c, src + c);
    } else {
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (mask[p][c]) cp_async4(dst + pair_off<CONSEC>(p) + c, src + pair_off<CONSEC>(p) + c);
    }
}

// ---------------------------------------------------------------------------
// Warp groups.  A segment of up to 32*VPT*G vehicles is run by G warps of
// one block (G = 1: a single warp, no barrier).  Warp w of the group holds
// slots [w*32*VPT, (w+1)*32*VPT).  Per step, the leader value of each warp's
// first slot and (in the adjoint) the follower terms of each warp's last
// slot cross warp boundaries through double-buffered shared cells and one
// named barrier (bar.sync id, 32*G) per exchange.
// ---------------------------------------------------------------------------
struct Grp {
    int G;       // warps per segment
    int w;       // warp index in the group
    int lane;
    int bar;     // named barrier id (1 + group index in the block)
    int *cell;   // [2] work-item broadcast
    // exchange cells, double-buffered by parity (xp, fp: 0 or G + 1): warp w
    // writes its last slot's speed and compensation to cell w + 1 of xl and
    // reads cell w; writes its first slot's follower terms to cell w of xf and
    // reads cell w + 1.  Cells 0 of xl and G of xf stay 0 (no neighbour).
    float2 *xl, *xf;
};

// Shared floats of one group's control area (cells + exchange cells).
__host__ __device__ __forceinline__ int grp_ctrl_floats(int G) { return (2 + 8 * (G + 1) + 3) & ~3; }

__device__ __forceinline__ void grp_sync(const Grp &g)
{
    if (g.G > 1)
        asm volatile("bar.sync %0, %1;" ::"r"(g.bar), "r"(32 * g.G) : "memory");
    else
        __syncwarp();
}

__device__ __forceinline__ Grp make_grp(int G, float *ctrl)
{
    Grp g;
    g.G = G;
    const int warp = threadIdx.x >> 5;
    g.w = warp % G;
    g.lane = threadIdx.x & 31;
    g.bar = 1 + warp / G;
    g.cell = reinterpret_cast<int *>(ctrl);
    g.xl = reinterpret_cast<float2 *>(ctrl + 2);
    g.xf = g.xl + 2 * (G + 1);
    if (G > 1 && g.lane < 2) {  // every warp writes the zeros that it may read
        g.xl[g.lane * (G + 1)] = make_float2(0.0f, 0.0f);
        g.xf[g.lane * (G + 1) + G] = make_float2(0.0f, 0.0f);
    }
    __syncwarp();
    return g;
}

__device__ __forceinline__ int grp_next(const Grp &g, int *work, int &par)
{
    if (g.G == 1) return next_segment(work, g.lane);
    if (g.w == 0 && g.lane == 0) g.cell[par] = atomicAdd(work, 1);
    grp_sync(g);
    const int s = g.cell[par];
    par ^= 1;
    return s;
}

// Leader speed and speed compensation of this warp's first slot (0 for the
// group's first warp); last is this lane's pair of the warp's last slot
// (used by lane 31).
__device__ __forceinline__ float2 grp_lead_in(const Grp &g, float2 last, int &xp)
{
    if (g.G == 1) return make_float2(0.0f, 0.0f);
    float2 *c = g.xl + xp + g.w;
    if (g.lane == 31) c[1] = last;
    grp_sync(g);
    xp = g.G + 1 - xp;
    return c[0];
}

// Follower terms (of position and speed) arriving at this warp's last slot (0
// for the last warp); first: this lane's of the warp's first slot (used by
// lane 0).
__device__ __forceinline__ float2 grp_follow_in(const Grp &g, float2 first, int &fp)
{
    if (g.G == 1) return make_float2(0.0f, 0.0f);
    float2 *c = g.xf + fp + g.w;
    if (g.lane == 0) c[0] = first;
    grp_sync(g);
    fp = g.G + 1 - fp;
    return c[1];
}

// Speed and compensation differences to the leaders (by shuffle; across warps
// through the group's cells).
template <int NP, bool CONSEC>
__device__ __forceinline__ void leader_diffs(const Grp &g, const State2 (&st)[NP], f2 (&dv)[NP], f2 (&dvc)[NP], int &xp)
{
    f2 vcur[NP], ccur[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        vcur[p] = st[p].v;
        ccur[p] = st[p].vc;
    }
    const float2 lead_in = grp_lead_in(g, make_float2(vcur[NP - 1].y, ccur[NP - 1].y), xp);
    minus_leader2<NP, CONSEC>(vcur, dv, g.lane, lead_in.x);
    minus_leader2<NP, CONSEC>(ccur, dvc, g.lane, lead_in.y);
}

// One Euler step (Eq. 1-3 with the Sec. III-C bounds) of this thread's
// vehicle pairs.
template <int NP, bool D4, bool CONSEC>
__device__ __forceinline__ void step_pairs(const Grp &g, State2 (&st)[NP], const VehConst2 (&kc)[NP],
                                           const ScenDesc &sc, int &xp)
{
    f2 dv[NP], dvc[NP];
    leader_diffs<NP, CONSEC>(g, st, dv, dvc, xp);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const f2 as = accel_star2<D4>(st[p].v, st[p].gap, dv[p], kc[p], sc.inv_dt, sc.a_min);
        euler2(st[p], as, dv[p], dvc[p], sc.dt);
    }
}

template <int NP, bool CONSEC>
__device__ __forceinline__ void load_vehicles(const SimArgs &a, const Seg &sg, int lane, int wb, VehConst2 (&kc)[NP],
                                              State2 (&st)[NP], bool (&vx)[NP], bool (&vy)[NP])
{
#pragma unroll
    for (int p = 0; p < NP; ++p) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int q = wb + pair_slot<NP, CONSEC>(p, lane) + c;
            const bool ok = q < sg.n_veh;
            float inv_v0 = 1.0f, T = 0.0f, s0 = 0.0f, am = 1.0f, cc = 0.5f, dl = 4.0f;  // ghost slot
            float ph = 0.0f, v = 0.0f, gap = INFINITY;
            if (ok) {
                const int gi = sg.veh_begin + q;
                inv_v0 = __frcp_rn(a.v0[gi]);
                T = a.T[gi];
                s0 = a.s0[gi];
                am = a.am[gi];
                cc = c_of(am, a.b[gi]);
                dl = a.delta[gi];
                ph = a.p_init[gi];
                v = a.v_init[gi];
                gap = a.g0[gi];
            }
            if (c == 0) {
                vx[p] = ok;
                kc[p].inv_v0.x = inv_v0; kc[p].T.x = T; kc[p].s0.x = s0; kc[p].am.x = am; kc[p].c.x = cc;
                kc[p].delta.x = dl;
                st[p].ph.x = ph; st[p].pl.x = 0.0f; st[p].v.x = v; st[p].gap.x = gap; st[p].vc.x = 0.0f;
            } else {
                vy[p] = ok;
                kc[p].inv_v0.y = inv_v0; kc[p].T.y = T; kc[p].s0.y = s0; kc[p].am.y = am; kc[p].c.y = cc;
                kc[p].delta.y = dl;
                st[p].ph.y = ph; st[p].pl.y = 0.0f; st[p].v.y = v; st[p].gap.y = gap; st[p].vc.y = 0.0f;
            }
        }
    }
}

// True when every occupied slot of the warp has delta == 4, so the step body
// can use the squaring form of (v/v0)^delta with no branch.  (Both variants
// execute the same sequence of group barriers.)
template <int NP>
__device__ __forceinline__ bool segment_is_d4(const VehConst2 (&kc)[NP], const bool (&vx)[NP], const bool (&vy)[NP])
{
    bool ok = true;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        if (vx[p] && kc[p].delta.x != 4.0f) ok = false;
        if (vy[p] && kc[p].delta.y != 4.0f) ok = false;
    }
    return __all_sync(FULL, ok);
}

// Store one pair to a scalar array at slot offset q (two 4-byte stores:
// the pair's global index need not be 8-byte aligned).
__device__ __forceinline__ void store_pair(float *base, int q, f2 x, bool vx, bool vy)
{
    if (vx) base[q] = x.x;
    if (vy) base[q + 1] = x.y;
}

__device__ __forceinline__ f2 load_pair(const float *base, int q, bool vx, bool vy)
{
    return make_float2(vx ? base[q] : 0.0f, vy ? base[q + 1] : 0.0f);
}


// This lane's pairs of a shared row (consecutive ones 16 bytes at a time).
template <int NP, bool CONSEC>
__device__ __forceinline__ void lds_row(const float *r, f2 (&x)[NP])
{
    if (NP == 1 || !CONSEC) {
#pragma unroll
        for (int p = 0; p < NP; ++p) x[p] = *reinterpret_cast<const f2 *>(r + pair_off<CONSEC>(p));
    } else {
#pragma unroll
        for (int p = 0; p + 1 < NP; p += 2) {
            const float4 v = *reinterpret_cast<const float4 *>(r + 2 * p);
            x[p] = make_float2(v.x, v.y);
            x[p + 1] = make_float2(v.z, v.w);
        }
    }
}
template <int NP, bool CONSEC>
__device__ __forceinline__ void sts_row(float *r, const f2 (&x)[NP])
{
    if (NP == 1 || !CONSEC) {
#pragma unroll
        for (int p = 0; p < NP; ++p) *reinterpret_cast<f2 *>(r + pair_off<CONSEC>(p)) = x[p];
    } else {
#pragma unroll
        for (int p = 0; p + 1 < NP; p += 2)
            *reinterpret_cast<float4 *>(r + 2 * p) = make_float4(x[p].x, x[p].y, x[p + 1].x, x[p + 1].y);
    }
}

// Shared floats of one adjoint group: tapes of speeds, frd and targets (dense
// seeds) turned seeds, [T][G*SL] each, a state stage [STATE_ROWS][G*SL] laid
// over the first two (the targets start at row bwd_target_row), and the control
// area; T is the tape depth (the checkpoint interval, or less when
// blocks restart from sub-checkpoints).  With prefetch the target tape is
// doubled and the state stage apart, and the next block's rows and starting
// state are copied (cp.async) while the current block runs (the state stage is
// free as soon as the block has loaded its own).
__host__ __device__ __forceinline__ int bwd_target_row(int T, bool pf)
{
    return pf || 2 * T > STATE_ROWS ? 2 * T : STATE_ROWS;
}
__host__ __device__ __forceinline__ int bwd_group_floats(int vpt, int T, int G, bool pf)
{
    const int rows = bwd_target_row(T, pf) + (pf ? 2 * T + STATE_ROWS : T);
    return rows * 32 * vpt * G + grp_ctrl_floats(G);
}

}  // namespace idm
