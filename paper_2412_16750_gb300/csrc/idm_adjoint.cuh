// Adjoint kernel templates; each idm_shape_v<VPT>_g<G>.cu instantiates the
// variants of one kernel shape (so they compile in parallel).
#pragma once
#include <limits.h>

#include "idm_gemm_tc.cuh"
#include "idm_sim_common.cuh"

namespace idm {

// ---------------------------------------------------------------------------
// Adjoint.  Per segment of C steps (last first): cp.async the observed
// targets of the C steps into the seed tape, reload the checkpoint,
// recompute the C steps, recording each step's speed, seed and reverse-step
// coefficients, then run the reverse recurrences
//   lp_k = seed_k + lp_{k+1} + mu A_p + mu_f A_ph(f)
//   lv_k = dt lp_{k+1} + lv_{k+1} + mu A_v + mu_f A_vh(f)
// with mu = dt lv_{k+1}; the follower's terms arrive by one warp shuffle
// (and across warps through the group's exchange cells).  The six factored
// gradient sums of each slot accumulate in registers and are folded into
// compensated totals about every FOLD_STEPS steps.
//
// The coefficients come out of the recompute's own model evaluation, whose
// softplus, reciprocal and power terms they share.  Four of them per
// vehicle go to tensor memory: private to the thread that reads them back, 64
// KB per SM quarter that a kernel without matrix products leaves idle, and
// beside the shared memory that the tape of speeds, seeds and the fifth
// coefficient, and the next run's copies, fill to the last resident block.
// Bound by issue and dependent latency (ncu on 400,000 vehicles x 256 steps:
// 57 % of the issue slots, FMA pipe 46 % of its cycles, 3.31 warp-instructions
// per vehicle and step).  Measured on GB300 with the same packing, against a
// second evaluation in the reverse sweep: loss + gradient of 10,000 uneven lanes
// over 301 steps 2.35 -> 2.2 ms, of 1,500 lanes of 100 over 300 steps 542 -> 432
// us; a 50-iteration fit of 1,000 vehicles 3.08 -> 2.82 ms.
// ---------------------------------------------------------------------------
// Compensated gradient sums.  Within a fold window of max(1, FOLD_STEPS / C)
// checkpoint segments (counted from the last) the six factored sums of a slot
// accumulate in FP32 registers; at the end of each window they are added to
// the slot's running totals, kept in a.gsum as unevaluated float pairs
// hi + lo, by Knuth's TwoSum, which returns the rounding error of the
// addition exactly.  The error of a slot's sum then stays that of one
// window's FP32 accumulation, whatever the horizon.  The totals of segment
// s_idx occupy 6 x (capacity / 2) float4 (hi.x, hi.y, lo.x, lo.y) per vehicle
// pair, each written and read back by the thread that owns the pair.
// ---------------------------------------------------------------------------
constexpr int FOLD_STEPS = GSUM_FOLD_STEPS;

// Checkpoint segments per fold.  Without totals the sums stay in registers: a
// call whose horizons are within FOLD_STEPS has none, although such a horizon can
// have more segments than a window (251-256 steps at interval 50: six of them,
// five to a window).
__device__ __forceinline__ int folds_every(const SimArgs &a)
{
    return a.gsum ? max(1, FOLD_STEPS / a.C) : INT_MAX;
}

// ---------------------------------------------------------------------------
// The tape's tensor-memory part: per step TAPE_WORDS * VPT 32-bit columns of
// this thread's lane, one tcgen05.st / tcgen05.ld of a whole step at a time.
// A warp reaches the 32 lanes of its quarter (warp index mod 4) only, so the
// warps w, w + 4, ... of a block use consecutive column ranges.
// ---------------------------------------------------------------------------
// Tensor memory of the block's tapes: `cols` columns (a power of two >= 32) and,
// for two steps more than the 8 that 128 columns hold with 4 vehicles per thread,
// `more` of them; allocated and freed by warp 0, every thread of the block calls
// both.  A block keeps the permit to allocate until it has both parts, so one that
// waits for its second waits for blocks that hold all of theirs.  Three blocks of
// 160 columns fit an SM; as one power of two each would take 256.
struct TapeMem {
    uint32_t at;    // first column
    uint32_t jump;  // from the end of the first part to the second
};
__device__ __forceinline__ TapeMem tape_alloc(int cols, int more)
{
    __shared__ uint32_t slot[2];
    if (threadIdx.x < 32) {
        tc::tmem_alloc_part((uint32_t)__cvta_generic_to_shared(slot), (uint32_t)cols);
        if (more > 0) tc::tmem_alloc_part((uint32_t)__cvta_generic_to_shared(slot + 1), (uint32_t)more);
        tc::tmem_alloc_done();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    return TapeMem{slot[0], more > 0 ? slot[1] - slot[0] - (uint32_t)cols : 0u};
}
__device__ __forceinline__ void tape_free(TapeMem m, int cols, int more)
{
    tc::fence_before_sync();
    __syncthreads();
    if (threadIdx.x < 32) {
        tc::fence_after_sync();
        if (more > 0) tc::tmem_dealloc(m.at + (uint32_t)cols + m.jump, (uint32_t)more);
        tc::tmem_dealloc(m.at, (uint32_t)cols);
    }
}
// This warp's columns: `words` per warp, quarter warp mod 4 of the lanes.
__device__ __forceinline__ TapeMem tape_base(TapeMem m, int warp, int words)
{
    return TapeMem{m.at + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * words), m.jump};
}

__device__ __forceinline__ void tape_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tape_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tape_st(uint32_t at, const float (&r)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(at), "f"(r[0]),
                 "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7])
                 : "memory");
}
__device__ __forceinline__ void tape_st(uint32_t at, const float (&r)[16])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15, %16};" ::"r"(at),
                 "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]), "f"(r[8]),
                 "f"(r[9]), "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15])
                 : "memory");
}
__device__ __forceinline__ void tape_st(uint32_t at, const float (&r)[32])
{
    const float (&lo)[16] = reinterpret_cast<const float (&)[16]>(r[0]), (&hi)[16] = reinterpret_cast<const float (&)[16]>(r[16]);
    tape_st(at, lo);
    tape_st(at + 16u, hi);
}
// The loaded values are valid after tape_wait_ld.
__device__ __forceinline__ void tape_ld(uint32_t at, float (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                 : "r"(at)
                 : "memory");
}
__device__ __forceinline__ void tape_ld(uint32_t at, float (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15}, [%16];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
                   "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
                 : "r"(at)
                 : "memory");
}
__device__ __forceinline__ void tape_ld(uint32_t at, float (&r)[32])
{
    tape_ld(at, reinterpret_cast<float (&)[16]>(r[0]));
    tape_ld(at + 16u, reinterpret_cast<float (&)[16]>(r[16]));
}

template <int NP, bool WD>
__device__ __forceinline__ void fold_sums(const SimArgs &a, int s_idx, const Grp &g, f2 (&sacc)[6][NP], bool have,
                                          bool last)
{
    const int pairs = 32 * NP * g.G;  // vehicle pairs of a segment
    float4 *base = reinterpret_cast<float4 *>(a.gsum) + (size_t)s_idx * 6 * pairs + g.w * 32 * NP + g.lane;
#pragma unroll
    for (int q = 0; q < (WD ? 6 : 5); ++q) {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float4 *t = base + (size_t)q * pairs + 32 * p;
            f2 hi = F2(0.0f), lo = F2(0.0f);
            if (have) {
                const float4 v = *t;
                hi = make_float2(v.x, v.y);
                lo = make_float2(v.z, v.w);
            }
            const f2 x = sacc[q][p];
            const f2 sum = add2(hi, x);  // TwoSum: sum + e == hi + x exactly
            const f2 bb = sub2(sum, hi);
            const f2 e = add2(sub2(hi, sub2(sum, bb)), sub2(x, bb));
            lo = add2(lo, e);
            if (last) {
                sacc[q][p] = add2(sum, lo);
            } else {
                *t = make_float4(sum.x, sum.y, lo.x, lo.y);
                sacc[q][p] = F2(0.0f);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Epilogue of a segment: the parameter gradients from the six factored
// sums, then either their output or (fit) the Adam update with the box
// projection in place.  Adam is taken in the reordered form of Kingma & Ba
// (2015, Sec. 2): with alpha_t = lr sqrt(1 - beta2^t) / (1 - beta1^t) and
// eps_t = eps sqrt(1 - beta2^t), theta -= alpha_t m / (sqrt(v) + eps_t) is
// the bias-corrected step with its per-iteration factors computed once per
// thread.  Every load of a slot is issued before the slot's stores: the
// parameter and moment arrays may alias as far as the compiler knows, so a
// store would otherwise hold back each later load for a full memory round
// trip (this epilogue was half of a short-horizon fit iteration).
template <int NP, bool ADAM, bool WD, bool D4, bool CONSEC>
__device__ __forceinline__ void segment_epilogue(const SimArgs &a, const Seg &sg, int at0, const int (&mask)[NP][2],
                                                 const VehConst2 (&kc)[NP], const f2 (&sacc)[6][NP],
                                                 const f2 (&lp)[NP], const f2 (&lv)[NP])
{
    float step_t = 0.0f, eps_t = 0.0f;
    if (ADAM) {
        const int it = a.iter;
        const float lr = a.n_iter > 1 ? a.lr0 + (a.lr1 - a.lr0) * (float)it / (float)(a.n_iter - 1) : a.lr0;
        const float bc1 = 1.0f - powf(0.9f, (float)(it + 1)), bc2 = 1.0f - powf(0.999f, (float)(it + 1));
        const float sb2 = sqrtf(bc2);
        step_t = lr * sb2 / bc1;
        eps_t = 1e-8f * sb2;
    }
    float *const th[5] = {const_cast<float *>(a.v0), const_cast<float *>(a.T), const_cast<float *>(a.s0),
                          const_cast<float *>(a.am), const_cast<float *>(a.b)};
    bool bad = false;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (!mask[p][c]) continue;
            const int gi = sg.veh_begin + at0 + pair_off<CONSEC>(p) + c;
            // this slot's loads, all ahead of its stores
            float tv[5], mm[5], vm[5];
            if (ADAM) {
#pragma unroll
                for (int r = 0; r < 5; ++r) {
                    const size_t mi = (size_t)r * a.N_total + gi;
                    tv[r] = th[r][gi];
                    mm[r] = a.adam_m[mi];
                    vm[r] = a.adam_v[mi];
                }
            } else {
                tv[0] = a.v0[gi];
                tv[4] = a.b[gi];
            }
            const float v0 = tv[0], b = tv[4];
            const float am = c ? kc[p].am.y : kc[p].am.x, cc = c ? kc[p].c.y : kc[p].c.x;
            const float dl = D4 ? 4.0f : (c ? kc[p].delta.y : kc[p].delta.x);
            const float A0 = c ? sacc[0][p].y : sacc[0][p].x, A1 = c ? sacc[1][p].y : sacc[1][p].x;
            const float A2 = c ? sacc[2][p].y : sacc[2][p].x, A3 = c ? sacc[3][p].y : sacc[3][p].x;
            const float A4 = c ? sacc[4][p].y : sacc[4][p].x, A5 = c ? sacc[5][p].y : sacc[5][p].x;
            float gr[6];
            gr[0] = am * dl * A4 / v0;                 // v0
            gr[1] = -A1;                               // T
            gr[2] = -A0;                               // s0
            gr[3] = A3 + A2 * cc / (2.0f * am);        // a_max
            gr[4] = A2 * cc / (2.0f * b);              // b
            gr[5] = -am * A5;                          // delta
#pragma unroll
            for (int r = 0; r < 6; ++r) bad |= !isfinite(gr[r]);
            if (ADAM) {
#pragma unroll
                for (int r = 0; r < 5; ++r) {
                    const size_t mi = (size_t)r * a.N_total + gi;
                    const float m = 0.9f * mm[r] + 0.1f * gr[r];
                    const float vv = 0.999f * vm[r] + 0.001f * gr[r] * gr[r];
                    a.adam_m[mi] = m;
                    a.adam_v[mi] = vv;
                    const float x = tv[r] - step_t * m / (sqrtf(vv) + eps_t);
                    th[r][gi] = fminf(fmaxf(x, a.lo[r]), a.hi[r]);
                }
            } else {
                if (a.g_v0) a.g_v0[gi] = gr[0];
                if (a.g_T) a.g_T[gi] = gr[1];
                if (a.g_s0) a.g_s0[gi] = gr[2];
                if (a.g_am) a.g_am[gi] = gr[3];
                if (a.g_b) a.g_b[gi] = gr[4];
                if (a.g_delta) a.g_delta[gi] = WD ? gr[5] : 0.0f;
                if (a.g_p_init) a.g_p_init[gi] = c ? lp[p].y : lp[p].x;
                if (a.g_v_init) a.g_v_init[gi] = c ? lv[p].y : lv[p].x;
            }
        }
    }
    if (__any_sync(FULL, bad) && (threadIdx.x & 31) == 0) atomicOr(a.status, IDM_STATUS_NONFINITE);
}

// ---------------------------------------------------------------------------
// The adjoint of one segment by one warp of its group.  A run covers n <= T
// steps: the shared tape holds, per step, a row of speeds, a row of frd and a
// row of targets or dense seeds that becomes the seeds (each [SLG] floats, the
// lane's 2 NP slots adjacent), the tensor memory the other coefficients.
// ---------------------------------------------------------------------------
template <int NP, bool DENSE, bool WD, bool D4, bool CONSEC, bool JUMP>
struct Sweep {
    const SimArgs &a;
    const ScenDesc &sc;
    Grp &g;
    const VehConst2 (&kc)[NP];
    State2 (&st)[NP];
    const int SLG;        // slots of the group
    const int wb;         // this warp's first slot in the group
    const int at0;        // this lane's first slot in the group
    const int wl;         // scenario-local index of this lane's first slot
    const int TS;         // floats of T tape rows
    float *const tv;      // this lane's slots of the speed row 0; frd rows TS after
    const TapeMem tape;   // tensor memory of the recorded steps
    f2 lp[NP], lv[NP];    // adjoints of position and speed
    f2 sacc[6][NP];       // the six factored gradient sums, over all steps
    f2 qc[NP];            // 4 a_max / v0 (D4)
    int mask[NP][2];      // all ones for an occupied slot
    float lsum = 0.0f, lcomp = 0.0f;  // squared residuals (MSE): Kahan over runs
    int xp = 0, fp = 0;   // parities of the exchange cells

    __device__ __forceinline__ Sweep(const SimArgs &a_, const ScenDesc &sc_, const Seg &sg, int lb, Grp &g_, float *base,
                                     TapeMem tape_, int T, const VehConst2 (&kc_)[NP], State2 (&st_)[NP])
        : a(a_), sc(sc_), g(g_), kc(kc_), st(st_), SLG(64 * NP * g_.G), wb(g_.w * 64 * NP),
          at0(g_.w * 64 * NP + pair_slot<NP, CONSEC>(0, g_.lane)), wl(lb + at0), TS(T * 64 * NP * g_.G),
          tv(base + at0), tape(tape_)
    {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            qc[p] = D4 ? mul2(mul2(kc[p].am, F2(4.0f)), kc[p].inv_v0) : F2(0.0f);
            lp[p] = F2(0.0f);
            lv[p] = F2(0.0f);
            mask[p][0] = at0 + pair_off<CONSEC>(p) < sg.n_veh ? -1 : 0;
            mask[p][1] = at0 + pair_off<CONSEC>(p) + 1 < sg.n_veh ? -1 : 0;
#pragma unroll
            for (int q = 0; q < 6; ++q) sacc[q][p] = F2(0.0f);
        }
    }

    // Tensor-memory column of recorded step s from its column in one part (JUMP:
    // from the ninth step on in the second; the others skip the arithmetic, which
    // costs 2 %).
    __device__ __forceinline__ uint32_t column(uint32_t at, int s) const
    {
        return JUMP ? at + (uint32_t)(s >> 3) * tape.jump : at;
    }

    // The copies fill occupied slots only, so empty ones of the dense seeds' rows
    // are set to 0 (a target row's become 0 when its seeds are recorded).
    __device__ __forceinline__ void clear_empty(float *tr, int rows) const
    {
        if (!DENSE) return;
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (!mask[p][c])
                    for (int s = 0; s < rows; ++s) tr[s * SLG + pair_off<CONSEC>(p) + c] = 0.0f;
    }

    // First observed step >= max(c0, 1).
    __device__ __forceinline__ int first_obs(int c0) const
    {
        return max((c0 + sc.obs_stride - 1) / sc.obs_stride, 1) * sc.obs_stride;
    }

    // cp.async of the rows of steps [c0, c0 + n) into tr (observed targets, or
    // the dense seeds of every step) and of a state's rows at base into ck;
    // each thread copies its own slots.
    __device__ __forceinline__ void prefetch(float *tr, float *ck, int c0, int n, const float *base, size_t stride) const
    {
        const int step = DENSE ? 1 : sc.obs_stride;
        const int k0 = DENSE ? c0 : first_obs(c0);
        const float *row = DENSE ? a.gP + sc.traj_off + (size_t)k0 * sc.n_veh + wl
                                 : a.targets + sc.tgt_off + (size_t)(k0 / step - 1) * sc.n_veh + wl;
        const bool full = mask[NP - 1][1] != 0;  // (consecutive slots: the last one)
        const bool vec = full && ((reinterpret_cast<uintptr_t>(row) | (size_t)sc.n_veh * sizeof(float)) & 15) == 0;
        for (int k = k0; k < c0 + n; k += step, row += sc.n_veh)
            prefetch_row<NP, CONSEC>(tr + (k - c0) * SLG, row, mask, vec);
        const bool cvec = full && ((reinterpret_cast<uintptr_t>(base) | stride * sizeof(float)) & 15) == 0;
#pragma unroll
        for (int f = 0; f < STATE_ROWS; ++f)
            prefetch_row<NP, CONSEC>(ck + f * SLG, base + (size_t)f * stride, mask, cvec);
        cp_async_commit();
    }

    // The state of an empty slot: at rest at 0 with a free road ahead.
    __device__ __forceinline__ void load_state(const float *ck)
    {
        f2 r[STATE_ROWS][NP];
#pragma unroll
        for (int f = 0; f < STATE_ROWS; ++f) lds_row<NP, CONSEC>(ck + f * SLG, r[f]);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const bool x = mask[p][0] != 0, y = mask[p][1] != 0;
            st[p].ph = make_float2(x ? r[0][p].x : 0.0f, y ? r[0][p].y : 0.0f);
            st[p].pl = make_float2(x ? r[1][p].x : 0.0f, y ? r[1][p].y : 0.0f);
            st[p].v = make_float2(x ? r[2][p].x : 0.0f, y ? r[2][p].y : 0.0f);
            st[p].gap = make_float2(x ? r[3][p].x : INFINITY, y ? r[3][p].y : INFINITY);
            st[p].vc = make_float2(x ? r[4][p].x : 0.0f, y ? r[4][p].y : 0.0f);
        }
    }

    // One recomputed step: its speeds, residuals (as seeds) and coefficients to
    // the tape, then (advance) the state update.  The observation handling has
    // no branch: an unobserved step's residual, read from a row the copies did
    // not fill, is masked to 0.
    __device__ __forceinline__ void record(bool advance, bool obs, float *rv, float *rr, uint32_t at, f2 scale, f2 &lseg)
    {
        f2 v[NP], dv[NP], dvc[NP], frd[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) v[p] = st[p].v;
        sts_row<NP, CONSEC>(rv, v);
        if constexpr (!DENSE) {
            const int om = obs ? -1 : 0;
            f2 y[NP];
            lds_row<NP, CONSEC>(rr, y);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                f2 r = residual2(st[p], y[p]);
                r.x = __int_as_float(__float_as_int(r.x) & mask[p][0] & om);
                r.y = __int_as_float(__float_as_int(r.y) & mask[p][1] & om);
                y[p] = mul2(scale, r);
                lseg = fma2(r, r, lseg);
            }
            sts_row<NP, CONSEC>(rr, y);
        }
        leader_diffs<NP, CONSEC>(g, st, dv, dvc, xp);
        float w[8 * NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            StepJac2 J;
            const f2 as = accel_jac2<D4>(v[p], st[p].gap, dv[p], kc[p], sc.inv_dt, sc.a_min, qc[p], J);
            w[8 * p] = J.Aph.x;
            w[8 * p + 1] = J.Aph.y;
            w[8 * p + 2] = J.Avn.x;
            w[8 * p + 3] = J.Avn.y;
            w[8 * p + 4] = J.w0n.x;
            w[8 * p + 5] = J.w0n.y;
            w[8 * p + 6] = J.fa.x;
            w[8 * p + 7] = J.fa.y;
            frd[p] = J.frd;
            if (advance) euler2(st[p], as, dv[p], dvc[p], sc.dt);
        }
        sts_row<NP, CONSEC>(rv + TS, frd);
        tape_st(at, w);
    }

    // What a reverse step reads back of its recorded step.
    struct Rec {
        f2 v[NP], dv[NP], frd[NP], Aph[NP], Avn[NP], w0n[NP], fa[NP];
    };
    __device__ __forceinline__ void read(const float *rv, uint32_t at, Rec &t) const
    {
        float w[8 * NP];
        tape_ld(at, w);
        lds_row<NP, CONSEC>(rv, t.v);
        lds_row<NP, CONSEC>(rv + TS, t.frd);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            // the leader's speed of the pair's first slot
            const float h = CONSEC && p > 0 ? t.v[p - 1].y : (p > 0 || at0 > 0 ? rv[pair_off<CONSEC>(p) - 1] : 0.0f);
            t.dv[p] = make_float2(__fsub_rn(t.v[p].x, h), __fsub_rn(t.v[p].y, t.v[p].x));
        }
        tape_wait_ld();
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            t.Aph[p] = make_float2(w[8 * p], w[8 * p + 1]);
            t.Avn[p] = make_float2(w[8 * p + 2], w[8 * p + 3]);
            t.w0n[p] = make_float2(w[8 * p + 4], w[8 * p + 5]);
            t.fa[p] = make_float2(w[8 * p + 6], w[8 * p + 7]);
        }
    }

    // One reverse step (seeds rr, step k); the record of the step before is
    // read inside it (NEXT) for every step but a run's first.
    template <bool NEXT>
    __device__ __forceinline__ void reverse(Rec &J, const float *rr, int k, const float *rv_next, uint32_t at_next)
    {
        const float dt = sc.dt;
        f2 to_lp[NP], to_lv[NP], t1[NP], nlv[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const f2 mu = mul2(F2(dt), lv[p]);
            const f2 w0nv = mul2(J.w0n[p], J.v[p]);
            to_lp[p] = mul2(mu, J.Aph[p]);
            to_lv[p] = mul2(mu, mul2(mul2(J.w0n[p], kc[p].c), J.v[p]));
            t1[p] = sub2(lp[p], to_lp[p]);                                   // lp + mu A_p
            nlv[p] = fma2(neg2(mu), J.Avn[p], fma2(F2(dt), lp[p], lv[p]));  // dt lp + lv + mu A_v
            sacc[0][p] = fma2(mu, J.w0n[p], sacc[0][p]);
            sacc[1][p] = fma2(mu, w0nv, sacc[1][p]);
            sacc[2][p] = fma2(mu, mul2(w0nv, J.dv[p]), sacc[2][p]);
            sacc[3][p] = fma2(mu, J.fa[p], sacc[3][p]);
            sacc[4][p] = fma2(mu, J.frd[p], sacc[4][p]);
            if (WD) sacc[5][p] = fma2(mu, delta_factor2<D4>(J.v[p], J.frd[p], kc[p]), sacc[5][p]);
        }
        f2 sd[NP];
        lds_row<NP, CONSEC>(rr, sd);
        if (NEXT) read(rv_next, at_next, J);
        const float2 in = grp_follow_in(g, make_float2(to_lp[0].x, to_lv[0].x), fp);
        add_follower2<NP, CONSEC>(t1, to_lp, g.lane, in.x);
        add_follower2<NP, CONSEC>(nlv, to_lv, g.lane, in.y);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            lp[p] = add2(t1[p], sd[p]);
            lv[p] = nlv[p];
        }
        if (DENSE && a.gV) add_gV(k);
    }
    __device__ __forceinline__ void add_gV(int k)
    {
        const float *r = a.gV + sc.traj_off + (size_t)k * sc.n_veh + wl;
#pragma unroll
        for (int p = 0; p < NP; ++p) lv[p] = add2(lv[p], load_pair(r, pair_off<CONSEC>(p), mask[p][0] != 0, mask[p][1] != 0));
    }

    // Steps [c0, c0 + n): recompute from the state st, then reverse.  The last
    // recomputed step is peeled off: the state after it is needed only at the
    // end of the horizon (the seed of step K).
    __device__ __forceinline__ void run(int c0, int n, float *tr)
    {
        const bool end = c0 + n == sc.K;
        const f2 scale = F2(2.0f * sc.inv_nobs);
        f2 lseg = F2(0.0f), lfirst = F2(0.0f);
        const int split = a.loss_split;
        {
            int obs_k = first_obs(c0), k = c0;
            float *rv = tv, *rr = tr;
            uint32_t at = tape.at;
            for (int s = 0; s + 1 < n; ++s, ++k, rv += SLG, rr += SLG, at += TAPE_WORDS * 2 * NP) {
                const bool obs = k == obs_k;
                if (!DENSE && k == split) {
                    lfirst = lseg;
                    lseg = F2(0.0f);
                }
                record(true, obs, rv, rr, column(at, s), scale, lseg);
                obs_k += obs ? sc.obs_stride : 0;
            }
            if (!DENSE && k == split) {
                lfirst = lseg;
                lseg = F2(0.0f);
            }
            record(end, k == obs_k, rv, rr, column(at, n - 1), scale, lseg);
        }
        if (end) {  // the state is now at step K: seed of the final step
            if (DENSE) {
                const float *r = a.gP + sc.traj_off + (size_t)sc.K * sc.n_veh + wl;
#pragma unroll
                for (int p = 0; p < NP; ++p) lp[p] = load_pair(r, pair_off<CONSEC>(p), mask[p][0] != 0, mask[p][1] != 0);
                if (a.gV) add_gV(sc.K);
            } else if (sc.n_obs > 0 && sc.K % sc.obs_stride == 0) {
                const float *y = a.targets + sc.tgt_off + (size_t)(sc.K / sc.obs_stride - 1) * sc.n_veh + wl;
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    f2 r = residual2(st[p], load_pair(y, pair_off<CONSEC>(p), mask[p][0] != 0, mask[p][1] != 0));
                    r.x = mask[p][0] ? r.x : 0.0f;
                    r.y = mask[p][1] ? r.y : 0.0f;
                    lp[p] = mul2(scale, r);
                    lseg = fma2(r, r, lseg);
                }
            }
        }
        kahan_add(lsum, lcomp, __fadd_rn(lseg.x, lseg.y));
        if (!DENSE && split > 0) kahan_add(lsum, lcomp, __fadd_rn(lfirst.x, lfirst.y));
        tape_wait_st();
        grp_sync(g);  // the whole group's tape is written
        Rec J;
        const float *rv = tv + (n - 1) * SLG, *rr = tr + (n - 1) * SLG;
        uint32_t at = tape.at + (uint32_t)((n - 1) * TAPE_WORDS * 2 * NP);
        read(rv, column(at, n - 1), J);
        int k = c0 + n - 1;
        for (int s = n - 1; s >= 1; --s, --k, rr -= SLG) {
            rv -= SLG;
            at -= TAPE_WORDS * 2 * NP;
            reverse<true>(J, rr, k, rv, column(at, s - 1));
        }
        reverse<false>(J, rr, k, rv, at);
    }

    template <bool ADAM>
    __device__ __forceinline__ void finish(const Seg &sg, int s_idx)
    {
        segment_epilogue<NP, ADAM, WD, D4, CONSEC>(a, sg, at0, mask, kc, sacc, lp, lv);
        if (!DENSE) {
            const double part = warp_sum_double((double)lsum - (double)lcomp) * (double)sc.inv_nobs;
            if (g.lane == 0) a.loss_part[(size_t)s_idx * g.G + g.w] = part;
        }
    }
};

// The tape is as deep as the checkpoint interval: one run per checkpoint
// segment, last first.
template <int NP, bool DENSE, bool ADAM, bool WD, bool D4, bool CONSEC>
__device__ __forceinline__ void backward_segment(const SimArgs &a, const ScenDesc &sc, const Seg &sg, int s_idx, int lb,
                                                 Grp &g, float *base, TapeMem tape, const VehConst2 (&kc)[NP],
                                                 State2 (&st)[NP])
{
    Sweep<NP, DENSE, WD, D4, CONSEC, false> w(a, sc, sg, lb, g, base, tape, a.C, kc, st);
    const int nb = a.bwd_pf ? 2 : 1;                     // stages (two with prefetch)
    float *trb = w.tv + bwd_target_row(a.C, nb > 1) * w.SLG;  // nb target tapes
    float *ckb = nb > 1 ? trb + nb * w.TS : w.tv;        // checkpoint stage [STATE_ROWS][SLG] (without prefetch over the tape)
    w.clear_empty(trb, nb * a.C);
    auto prefetch = [&](int cs) {
        const int par = nb > 1 ? cs & 1 : 0, c0 = cs * a.C;
        w.prefetch(trb + par * w.TS, ckb, c0, min(a.C, sc.K - c0),
                   a.ckpt + sc.ckpt_off + (size_t)cs * STATE_ROWS * sc.n_veh + w.wl, (size_t)sc.n_veh);
    };
    const int n_ck = (sc.K + a.C - 1) / a.C;
    const int fold_every = folds_every(a);
    if (nb > 1) prefetch(n_ck - 1);
    for (int cs = n_ck - 1; cs >= 0; --cs) {
        const int par = nb > 1 ? cs & 1 : 0, c0 = cs * a.C;
        if (nb == 1) prefetch(cs);
        cp_async_wait<0>();  // this segment's rows and checkpoint (this thread's own slots)
        w.load_state(ckb);
        if (nb > 1 && cs > 0) prefetch(cs - 1);  // lands while this segment runs
        w.run(c0, min(a.C, sc.K - c0), trb + par * w.TS);
        // a fold window is fold_every checkpoint segments, counted from the last
        if (cs > 0 && (n_ck - cs) % fold_every == 0)
            fold_sums<NP, WD>(a, s_idx, g, w.sacc, n_ck - cs > fold_every, false);
        grp_sync(g);  // the tape may be overwritten by the next segment
    }
    if (n_ck > fold_every) fold_sums<NP, WD>(a, s_idx, g, w.sacc, true, true);
    w.template finish<ADAM>(sg, s_idx);
}

// The same adjoint when the tape is shallower than the checkpoint interval, or
// has a second part of tensor memory (an interval of 9 or 10 steps in one run):
// each checkpoint segment is first run forward once writing sub-checkpoints
// every T steps (global scratch, this thread's own slots), then processed as
// tape blocks of T steps, last first.
template <int NP, bool DENSE, bool ADAM, bool WD, bool D4, bool CONSEC>
__device__ __forceinline__ void backward_segment_blocks(const SimArgs &a, const ScenDesc &sc, const Seg &sg, int s_idx,
                                                        int lb, Grp &g, float *base, TapeMem tape,
                                                        const VehConst2 (&kc)[NP], State2 (&st)[NP])
{
    const int T = a.tape_T;
    Sweep<NP, DENSE, WD, D4, CONSEC, NP == 2> w(a, sc, sg, lb, g, base, tape, T, kc, st);
    const int nb = a.bwd_pf ? 2 : 1;
    float *trb = w.tv + bwd_target_row(T, nb > 1) * w.SLG;
    float *ckb = nb > 1 ? trb + nb * w.TS : w.tv;
    w.clear_empty(trb, nb * T);
    // Block j > 0 of a checkpoint segment starts from sub-checkpoint row j - 1,
    // block 0 from the checkpoint.  With several vehicle pairs per thread (tapes
    // of 8 or 10 steps) the first block takes the remainder: the forward pass then
    // ends where the last full block begins (42 steps of 50 instead of 48 with
    // tapes of 8: two iterations of 2M x 1,000 31.13 -> 30.89 ms).
    constexpr bool SHORT_FIRST = NP >= 2;
    auto seg_len = [&](int cs) { return min(a.C, sc.K - cs * a.C); };
    auto n_sub = [&](int cs) { return (seg_len(cs) + T - 1) / T; };
    auto first_len = [&](int cs) { return SHORT_FIRST ? seg_len(cs) - (n_sub(cs) - 1) * T : min(T, seg_len(cs)); };
    auto blk_at = [&](int cs, int j) { return j == 0 ? 0 : first_len(cs) + (j - 1) * T; };
    auto blk_len = [&](int cs, int j) { return j == 0 ? first_len(cs) : min(T, seg_len(cs) - blk_at(cs, j)); };
    auto sub_row = [&](int j) { return a.sub_ckpt + (size_t)(j - 1) * STATE_ROWS * a.N_total + sg.veh_begin + w.at0; };
    auto ckpt_row = [&](int cs) { return a.ckpt + sc.ckpt_off + (size_t)cs * STATE_ROWS * sc.n_veh + w.wl; };
    auto prefetch = [&](int cs, int j, int par) {
        w.prefetch(trb + par * w.TS, ckb, cs * a.C + blk_at(cs, j), blk_len(cs, j),
                   j == 0 ? ckpt_row(cs) : sub_row(j), j == 0 ? (size_t)sc.n_veh : (size_t)a.N_total);
    };
    const int n_ck = (sc.K + a.C - 1) / a.C;
    const int fold_every = folds_every(a);
    int par = 0;
    bool have_next = false;  // the next block's stage is already being filled
    if (nb > 1 && n_sub(n_ck - 1) == 1) {
        prefetch(n_ck - 1, 0, 0);
        have_next = true;
    }
    for (int cs = n_ck - 1; cs >= 0; --cs) {
        const int nsub = n_sub(cs);
        if (nsub > 1) {  // forward pass over the segment writing the sub-checkpoints
            const float *b = ckpt_row(cs);
            const size_t n = (size_t)sc.n_veh;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const bool x = w.mask[p][0] != 0, y = w.mask[p][1] != 0;
                const int o = pair_off<CONSEC>(p);
                st[p].ph = load_pair(b, o, x, y);
                st[p].pl = load_pair(b + n, o, x, y);
                st[p].v = load_pair(b + 2 * n, o, x, y);
                const f2 gp = load_pair(b + 3 * n, o, x, y);
                st[p].gap = make_float2(x ? gp.x : INFINITY, y ? gp.y : INFINITY);
                st[p].vc = load_pair(b + 4 * n, o, x, y);
            }
            for (int j = 1; j < nsub; ++j) {
                for (int s = 0, n_s = blk_len(cs, j - 1); s < n_s; ++s) step_pairs<NP, D4, CONSEC>(g, st, kc, sc, w.xp);
                float *row = sub_row(j);
                const size_t m = (size_t)a.N_total;
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const bool x = w.mask[p][0] != 0, y = w.mask[p][1] != 0;
                    const int o = pair_off<CONSEC>(p);
                    store_pair(row, o, st[p].ph, x, y);
                    store_pair(row + m, o, st[p].pl, x, y);
                    store_pair(row + 2 * m, o, st[p].v, x, y);
                    store_pair(row + 3 * m, o, st[p].gap, x, y);
                    store_pair(row + 4 * m, o, st[p].vc, x, y);
                }
            }
            __threadfence_block();  // the rows are read back below (this thread's own slots)
        }
        for (int j = nsub - 1; j >= 0; --j) {
            if (!have_next) prefetch(cs, j, par);
            cp_async_wait<0>();  // this block's rows and starting state (this thread's own slots)
            w.load_state(ckb);
            // start filling the other stage with the next block when its state exists
            have_next = nb > 1 && (j > 0 || (cs > 0 && n_sub(cs - 1) == 1));
            if (have_next) prefetch(j > 0 ? cs : cs - 1, j > 0 ? j - 1 : 0, par ^ 1);
            w.run(cs * a.C + blk_at(cs, j), blk_len(cs, j), trb + par * w.TS);
            grp_sync(g);  // the tape may be overwritten by the next block
            if (nb > 1) par ^= 1;
        }
        if (cs > 0 && (n_ck - cs) % fold_every == 0)
            fold_sums<NP, WD>(a, s_idx, g, w.sacc, n_ck - cs > fold_every, false);
    }
    if (n_ck > fold_every) fold_sums<NP, WD>(a, s_idx, g, w.sacc, true, true);
    w.template finish<ADAM>(sg, s_idx);
}

// Register budgets: 2 vehicles per thread fit 128 registers (2 blocks of 8 warps
// per SM); 4 per thread take 168, so their blocks are 4 warps (3 blocks per SM)
// unless the segment has 8 warps (256 threads, one block per SM); 8 per thread use
// up to 255.  Some of what stays live across a step's barriers spills: up to 36
// bytes with 4 per thread, up to 200 with 8 (the delta gradient with tape blocks).
// The same loops bounded to one block of twelve warps (as many registers) came
// out 2 to 4 % slower.
template <int VPT, int GW>
struct BwdBounds {
    static constexpr bool narrow = VPT == 4 && GW < 8;
    static constexpr int threads = narrow ? 128 : 256;
    static constexpr int blocks = VPT == 2 ? 2 : (narrow ? 3 : 1);
};

// The warps per segment GW are a compile-time constant of each kernel: the
// group exchange, its barriers and every slot offset of the shared tape then
// fold into immediates (measured on GB300 at 4 vehicles x 4 warps: 7 % fewer
// instructions and an 11 % shorter adjoint than with GW read from SimArgs).
template <int VPT, int GW, bool DENSE, bool ADAM, bool WD, bool SUB, bool CONSEC>
__global__ void __launch_bounds__(BwdBounds<VPT, GW>::threads, BwdBounds<VPT, GW>::blocks)
backward_kernel(SimArgs a)
{
    constexpr int NP = VPT / 2;
    constexpr int G = GW;
    extern __shared__ __align__(16) float smem[];
    const int warp = threadIdx.x >> 5;
    float *gbase = smem + (warp / G) * bwd_group_floats(VPT, a.tape_T, G, a.bwd_pf != 0);
    float *ctrl = gbase + bwd_group_floats(VPT, a.tape_T, G, a.bwd_pf != 0) - grp_ctrl_floats(G);
    Grp g = make_grp(G, ctrl);
    const TapeMem tmem = tape_alloc(a.tape_cols, VPT == 4 && SUB ? a.tape_more : 0);
    const TapeMem tape = tape_base(tmem, warp, TAPE_WORDS * VPT * a.tape_T);
    int par = 0;
    for (;;) {
        const int s_idx = grp_next(g, a.work, par);
        if (s_idx >= *a.n_seg) break;
        const Seg sg = a.seg[s_idx];
        const ScenDesc sc = a.scen_tab ? a.scen_tab[sg.scen] : a.scen0;
        const int lb = sg.veh_begin - sc.veh_begin;
        VehConst2 kc[NP];
        State2 st[NP];
        bool vx[NP], vy[NP];
        load_vehicles<NP, CONSEC>(a, sg, g.lane, g.w * 64 * NP, kc, st, vx, vy);
        if constexpr (SUB) {
            if (segment_is_d4<NP>(kc, vx, vy))
                backward_segment_blocks<NP, DENSE, ADAM, WD, true, CONSEC>(a, sc, sg, s_idx, lb, g, gbase, tape, kc, st);
            else
                backward_segment_blocks<NP, DENSE, ADAM, WD, false, CONSEC>(a, sc, sg, s_idx, lb, g, gbase, tape, kc, st);
        } else {
            if (segment_is_d4<NP>(kc, vx, vy))
                backward_segment<NP, DENSE, ADAM, WD, true, CONSEC>(a, sc, sg, s_idx, lb, g, gbase, tape, kc, st);
            else
                backward_segment<NP, DENSE, ADAM, WD, false, CONSEC>(a, sc, sg, s_idx, lb, g, gbase, tape, kc, st);
        }
    }
    tape_free(tmem, a.tape_cols, VPT == 4 && SUB ? a.tape_more : 0);
}

// Kernel variants of one (vehicles per thread, warps per segment) shape:
// seeds from dense gradients or from targets, fused Adam or gradient output,
// with or without the delta gradient, tape blocks (SUB), and the slot mapping
// (consecutive with dense seeds and, with Adam and 4 vehicles per thread, where
// the caller says so; the two are one with 2, and the consecutive code then
// serves Adam).
template <int VPT, int GW, bool SUB>
inline void *backward_fn_t(bool dense, bool adam, bool wd, bool consec)
{
    if (dense)
        return wd ? (void *)backward_kernel<VPT, GW, true, false, true, SUB, true>
                  : (void *)backward_kernel<VPT, GW, true, false, false, SUB, true>;
    if (adam)
        return VPT != 4 || !consec ? (void *)backward_kernel<VPT, GW, false, true, false, SUB, VPT == 2>
                                   : (void *)backward_kernel<VPT, GW, false, true, false, SUB, VPT <= 4>;
    return wd ? (void *)backward_kernel<VPT, GW, false, false, true, SUB, false>
              : (void *)backward_kernel<VPT, GW, false, false, false, SUB, false>;
}

}  // namespace idm
