// Simulation kernels of libidm for sm_103a: initial gaps, lane packing into
// segments, the fused forward (Eq. 1-3 with the Sec. III-C bounds,
// checkpoints, optional trajectory output) and the launch / dispatch code of
// the reverse-time adjoint, whose kernels live in idm_adjoint.cuh
// (arXiv 2412.16750, Sec. III and IV-A).
//
// Mapping.  Vehicles are ordered lane by lane, head first.  Whole lanes are
// packed into segments of at most 32*VPT*G vehicles, each run by G warps of
// one block.  Thread l of a warp holds pairs of adjacent slots (pair p:
// slots 64p + 2l and 64p + 2l + 1), so the leader of a pair's second slot is
// in the same register pair and the leader of its first slot is one warp
// shuffle away; across warps the value goes through shared cells and one
// named barrier per step.  Groups take segments from a global atomic counter
// (persistent grid).
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "idm_forward.cuh"

namespace idm {

// ---------------------------------------------------------------------------
// Initial gaps g0[i] = p_init[i-1] - p_init[i] - length[i-1] (Sec. III-A),
// +inf for lane heads.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float initial_gap(const float *p_init, const float *length, int i)
{
    if (i == 0) return INFINITY;
    return (float)((double)p_init[i - 1] - (double)p_init[i] - (double)length[i - 1]);
}

__device__ __forceinline__ bool bad_lane(int l, int a, int e, int n_lanes, int N)
{
    return e < a || a < 0 || e > N || (l == 0 && a != 0) || (l == n_lanes - 1 && e != N);
}

__global__ void gap_kernel(const float *p_init, const float *length, int N, float *g0)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) g0[i] = initial_gap(p_init, length, i);
}

__global__ void head_kernel(const int *lane_off, int n_lanes, int N, float *g0, unsigned *status)
{
    int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= n_lanes) return;
    int a = lane_off[l], e = lane_off[l + 1];
    if (bad_lane(l, a, e, n_lanes, N)) { atomicOr(status, IDM_STATUS_BAD_LANE_OFF); return; }
    if (a < e) g0[a] = INFINITY;
}

cudaError_t launch_prep_gap(const int *lane_off, int n_lanes, const float *p_init, const float *length,
                            int N, float *g0, unsigned *status, cudaStream_t st)
{
    if (N > 0) gap_kernel<<<(N + 255) / 256, 256, 0, st>>>(p_init, length, N, g0);
    if (n_lanes > 0) head_kernel<<<(n_lanes + 255) / 256, 256, 0, st>>>(lane_off, n_lanes, N, g0, status);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Lane packing: each thread packs a contiguous chunk of `per` lanes
// greedily into segments of at most `cap` vehicles; a block scan places the
// chunks' segments.  A lane longer than cap is skipped and flagged.
//
// A chunk's last segment is half empty on average, so a chunk holds about 32
// segments' vehicles (with 1,024 chunks whatever the scene, 2,000 lanes of 100
// made 1,000 segments of 2 lanes in 512 slots instead of 400 of 5, and the
// simulation of such a scene took 1.4 to 2.3 times as long).  Scenes of short
// lanes (under 16 vehicles), and those whose lanes fit one wave as segments of
// their own (one_wave), keep 1,024 chunks.
//
// A thread that walked its chunk lane by lane would take ~25 us for 150 lanes.
// So the chunks are spread over a cluster of PACK_BLOCKS blocks (scenes of up to
// 4,096 lanes: the one block that prep_kernel has for it), each with the offsets
// of its chunks in shared memory; all threads find every lane's successor (the
// first lane that no longer fits a segment starting there, or the chunk's end)
// with doubling strides, one thread per chunk jumps from segment to segment, and
// all threads write the segments.  One forward step of 40,000 lanes of 16,
// preparation included, took 220 us with one block whose 40 threads walked 1,024
// lanes each and takes 41; loss and gradient of 32,768 lanes of which 101 hold a
// vehicle took 7.2 ms with the successors searched lane by lane and take 64 us.
// ---------------------------------------------------------------------------
constexpr int BUILD_THREADS = SEG_BUILD_CHUNKS;
constexpr int PACK_BLOCKS = 8;         // a portable cluster
constexpr int STAGED_LANES = 32768;    // lanes whose offsets one block's shared memory holds

__host__ __device__ inline size_t staged_bytes(int n_lanes) { return (size_t)(n_lanes + 1) * 6 + 16; }

// One chunk lane by lane: more lanes than the staging holds, or lanes that are
// malformed or longer than cap.
template <bool EMIT>
__device__ int pack_lanes(const int *lane_off, int l0, int l1, int cap, int N, Seg *out, unsigned *status)
{
    int cnt = 0, fill = 0, seg_begin = 0;
    for (int l = l0; l < l1; ++l) {
        const int a = lane_off[l], e = lane_off[l + 1], n = e - a;
        const bool bad = a < 0 || e > N || n < 0;  // malformed: never read outside [0, N)
        const bool skip = bad || n > cap;
        if (skip && EMIT) atomicOr(status, bad ? IDM_STATUS_BAD_LANE_OFF : IDM_STATUS_LANE_TOO_LONG);
        if (fill > 0 && (skip || fill + n > cap)) {
            if (EMIT) out[cnt] = Seg{seg_begin, fill, 0, 0};
            ++cnt;
            fill = 0;
        }
        if (skip || n == 0) continue;
        if (fill == 0) seg_begin = a;
        fill += n;
    }
    if (fill > 0) {
        if (EMIT) out[cnt] = Seg{seg_begin, fill, 0, 0};
        ++cnt;
    }
    return cnt;
}

// The chunks of block `rank` of `ranks` (a cluster, or one block alone).
__device__ __forceinline__ void build_segments(const int *lane_off, int n_lanes, int cap, int N, int per, bool staged,
                                               Seg *seg, int *n_seg, unsigned *status, int *off, int *sc, int rank,
                                               int ranks)
{
    const int t = threadIdx.x;
    const int chunks = (n_lanes + per - 1) / per, own = (chunks + ranks - 1) / ranks;  // own <= BUILD_THREADS
    const int b0 = (int)min((long long)n_lanes, (long long)rank * own * per);
    const int b1 = (int)min((long long)n_lanes, (long long)(rank + 1) * own * per);    // this block's lanes
    const int l0 = (int)min((long long)b1, b0 + (long long)t * per), l1 = (int)min((long long)b1, (long long)l0 + per);
    const int n = b1 - b0;
    unsigned short *jump = reinterpret_cast<unsigned short *>(off + n + 1);  // lanes of the segment from a lane
    if (staged) {
        for (int l = t; l <= n; l += BUILD_THREADS) off[l] = lane_off[b0 + l];
        __syncthreads();
        bool odd = false;
        for (int l = t; l < n; l += BUILD_THREADS) {
            const int a = off[l], e = off[l + 1];
            odd |= a < 0 || e > N || e < a || e - a > cap;
        }
        staged = !__syncthreads_or(odd);
    }
    if (staged) {  // successors of this thread's share of the lanes, each within its chunk
        const int share = (n + BUILD_THREADS - 1) / BUILD_THREADS;
        const int s0 = min(n, t * share), s1 = min(n, s0 + share);
        int m = s0, end = s0 / per * per;  // end of the lane's chunk
        for (int l = s0; l < s1; ++l) {
            if (l == end || l == s0) end = min(n, end + per);
            const int lim = off[l] + cap;
            m = max(m, l);  // lanes [l, m) fit: forward by doubling strides, then by halving ones
            int d = 1;
            for (; m + d <= end && off[m + d] <= lim; d <<= 1) m += d;
            while ((d >>= 1) > 0)
                if (m + d <= end && off[m + d] <= lim) m += d;
            jump[l] = (unsigned short)(m - l);
        }
        __syncthreads();
    }
    int cnt = 0;
    if (staged) {  // this chunk by jumps; its segments' first lanes over the jumps already taken
        unsigned short *first = jump + (l0 - b0);
        for (int l = l0 - b0; l < l1 - b0;) {
            const int m = l + (int)jump[l];
            if (off[m] > off[l]) first[cnt++] = (unsigned short)l;
            l = m;
        }
    } else {
        cnt = pack_lanes<false>(lane_off, l0, l1, cap, N, nullptr, status);
    }
    sc[t] = cnt;
    __syncthreads();
    for (int o = 1; o < own; o <<= 1) {  // inclusive Hillis-Steele scan
        const int v = t >= o ? sc[t - o] : 0;
        __syncthreads();
        sc[t] += v;
        __syncthreads();
    }
    const int total = own > 0 ? sc[own - 1] : 0;
    int before = 0;  // segments of the blocks before this one
    if (ranks > 1) {
        auto cluster = cooperative_groups::this_cluster();
        cluster.sync();
        for (int r = 0; r < rank; ++r) before += cluster.map_shared_rank(sc, r)[own - 1];
        cluster.sync();  // every block's totals have been read
    }
    if (staged) {  // as many threads per chunk as there are
        int per_chunk = 1;
        while (2 * per_chunk * own <= BUILD_THREADS) per_chunk <<= 1;
        const int c = t / per_chunk;
        if (c < own) {
            const int k0 = c > 0 ? sc[c - 1] : 0, k1 = sc[c], c0 = min(n, c * per), c1 = min(n, c0 + per);
            const unsigned short *first = jump + c0;
            for (int k = k0 + t % per_chunk; k < k1; k += per_chunk) {
                const int l = first[k - k0], e = k + 1 < k1 ? (int)first[k - k0 + 1] : c1;  // (empty lanes may follow)
                seg[before + k] = Seg{off[l], off[e] - off[l], 0, 0};
            }
        }
    } else {
        pack_lanes<true>(lane_off, l0, l1, cap, N, seg + before + (sc[t] - cnt), status);
    }
    // (malformed offsets, flagged, can make more segments than their users size
    // buffers for)
    if (t == 0 && rank == ranks - 1) *n_seg = (int)min((long long)(before + total), segment_bound(N, n_lanes, cap));
}

__global__ void __cluster_dims__(PACK_BLOCKS, 1, 1) __launch_bounds__(BUILD_THREADS)
build_segments_kernel(const int *lane_off, int n_lanes, int cap, int N, int per, bool staged, Seg *seg, int *n_seg,
                      int *work_f, int *work_b, unsigned *status)
{
    extern __shared__ int off[];  // offsets of the block's lanes when staged, and the jumps
    __shared__ int sc[BUILD_THREADS];
    if (blockIdx.x == 0 && threadIdx.x == 0) *work_f = *work_b = 0;
    build_segments(lane_off, n_lanes, cap, N, per, staged, seg, n_seg, status, off, sc, blockIdx.x, PACK_BLOCKS);
}

// The whole preparation in one launch, for scenes whose staged offsets leave
// room for other blocks: block 0 clears the work counters, checks the lanes and
// packs them; the others compute the initial gaps of 1,024 vehicles each, the
// lane heads among them found in one pass over the offsets.  (A clear and three
// kernels of 3-4 us each before a small scene's 75 us of simulation otherwise.)
constexpr int FUSED_PREP_LANES = 4096;

__global__ void __launch_bounds__(BUILD_THREADS)
prep_kernel(const int *lane_off, int n_lanes, const float *p_init, const float *length, int N, float *g0, int cap, int per,
            Seg *seg, int *ctl_nseg, int *work_f, int *work_b, unsigned *status)
{
    extern __shared__ int off[];
    __shared__ int sc[BUILD_THREADS];
    const int t = threadIdx.x;
    if (blockIdx.x == 0) {
        if (t == 0) *work_f = *work_b = 0;
        for (int l = t; l < n_lanes; l += BUILD_THREADS)
            if (bad_lane(l, lane_off[l], lane_off[l + 1], n_lanes, N)) atomicOr(status, IDM_STATUS_BAD_LANE_OFF);
        build_segments(lane_off, n_lanes, cap, N, per, true, seg, ctl_nseg, status, off, sc, 0, 1);
        return;
    }
    const int first = ((int)blockIdx.x - 1) * BUILD_THREADS, i = first + t;
    sc[t] = 0;  // 1: a lane's head
    __syncthreads();
    for (int l = t; l < n_lanes; l += BUILD_THREADS) {
        const int a = lane_off[l], e = lane_off[l + 1];
        if (a < e && a >= first && a < first + BUILD_THREADS && !bad_lane(l, a, e, n_lanes, N)) sc[a - first] = 1;
    }
    __syncthreads();
    if (i < N) g0[i] = sc[t] ? INFINITY : initial_gap(p_init, length, i);
}

// Lanes per chunk of the packing.
static int lanes_per_chunk(int n_lanes, int cap, int N, bool one_wave)
{
    // 32 segments of as many whole lanes of the mean length as fit
    const long long mean = N > 0 ? ((long long)N + n_lanes - 1) / n_lanes : 1;
    const long long full = 32 * (mean < cap ? cap / mean : 1), least = ((long long)n_lanes + BUILD_THREADS - 1) / BUILD_THREADS;
    const bool short_lanes = (long long)N < 16LL * n_lanes;
    return (int)(one_wave || short_lanes || full < least ? least : full);
}

cudaError_t launch_prep(const int *lane_off, int n_lanes, const float *p_init, const float *length, int N, float *g0, int cap,
                        bool one_wave, Seg *seg, int *n_seg, int *work_f, int *work_b, unsigned *status, cudaStream_t st)
{
    cudaError_t e;
    if (n_lanes <= FUSED_PREP_LANES) {
        const int blocks = 1 + (N + BUILD_THREADS - 1) / BUILD_THREADS;
        prep_kernel<<<blocks, BUILD_THREADS, staged_bytes(n_lanes), st>>>(lane_off, n_lanes, p_init, length, N, g0, cap,
                                                                          lanes_per_chunk(n_lanes, cap, N, one_wave), seg,
                                                                          n_seg, work_f, work_b, status);
        return cudaGetLastError();
    }
    if ((e = launch_prep_gap(lane_off, n_lanes, p_init, length, N, g0, status, st)) != cudaSuccess) return e;
    int per = lanes_per_chunk(n_lanes, cap, N, one_wave);
    const int least = (n_lanes + BUILD_THREADS - 1) / BUILD_THREADS;
    auto block_lanes = [&] { return (long long)(((n_lanes + per - 1) / per + PACK_BLOCKS - 1) / PACK_BLOCKS) * per; };
    // more lanes than the blocks' shared memory holds: as many threads as can walk
    const bool staged = block_lanes() <= STAGED_LANES;
    if (!staged) per = least;
    const size_t smem = staged ? staged_bytes((int)block_lanes()) : 0;
    e = cudaFuncSetAttribute(build_segments_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)staged_bytes(STAGED_LANES));
    if (e != cudaSuccess) return e;
    build_segments_kernel<<<PACK_BLOCKS, BUILD_THREADS, smem, st>>>(lane_off, n_lanes, cap, N, per, staged, seg, n_seg,
                                                                    work_f, work_b, status);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Deterministic loss reduction over segments (fixed order).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024)
loss_finalize_kernel(const double *part, const int *n_seg, int per_seg, double *out)
{
    __shared__ double sh[1024];
    const int n = *n_seg * per_seg;
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0 && out) *out = sh[0];
}

cudaError_t launch_loss_finalize(const double *loss_part, const int *n_seg, int per_seg, long long max_part, double *out,
                                 cudaStream_t st)
{
    // a power of two of threads that covers the partials gives the sum of 1,024
    // (whose other terms are zeros) with fewer barriers
    int threads = 32;
    while (threads < 1024 && threads < max_part) threads <<= 1;
    loss_finalize_kernel<<<1, threads, 0, st>>>(loss_part, n_seg, per_seg, out);
    return cudaGetLastError();
}

// The losses of all iterations of a single-launch fit: block it sums the
// partials of iteration it in the order of loss_finalize_kernel, so each
// value equals that of the per-iteration reduction.
__global__ void __launch_bounds__(1024)
loss_finalize_iters_kernel(const double *part, long long stride, const int *n_seg, int per_seg, double *out)
{
    __shared__ double sh[1024];
    const long long n = (long long)*n_seg * per_seg;
    if (n > stride) {  // flagged by the fit kernel
        if (threadIdx.x == 0) out[blockIdx.x] = __longlong_as_double(0x7ff8000000000000LL);
        return;
    }
    const double *pi = part + (size_t)blockIdx.x * (size_t)stride;
    double s = 0.0;
    for (long long i = threadIdx.x; i < n; i += blockDim.x) s += pi[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sh[0];
}

cudaError_t launch_loss_finalize_iters(const double *loss_part, long long stride, const int *n_seg, int per_seg,
                                       int n_iter, double *out, cudaStream_t st)
{
    if (n_iter < 1) return cudaSuccess;
    loss_finalize_iters_kernel<<<n_iter, 1024, 0, st>>>(loss_part, stride, n_seg, per_seg, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Dispatch
// ---------------------------------------------------------------------------
// Forward kernels of every shape live in idm_shape_v<V>_g<G>.cu (COUNT: the
// variant that also counts gap-floor and kink-band events).
static void *forward_fn_v(int vpt, int G, bool count)
{
#define IDM_PICK(V, GW) \
    if (vpt == V && G == GW) return forward_fn_v##V##_g##GW(count);
    IDM_SHAPES(IDM_PICK)
#undef IDM_PICK
    return nullptr;
}

cudaError_t launch_forward(int vpt, int G, bool traj, bool vtraj, bool ckpt, const SimArgs &a, int grid, int wpb,
                           cudaStream_t st)
{
    FwdFlags f{traj, vtraj, ckpt, a.eval_targets != nullptr && a.eval_part != nullptr};
    void *fn = forward_fn_v(vpt, G, a.events != nullptr);
    if (!fn) return cudaErrorInvalidValue;
    const size_t smem = forward_smem_bytes(vpt, G, wpb);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    SimArgs args = a;
    args.G = G;
    void *params[] = {&args, &f};
    return cudaLaunchKernel(fn, dim3(grid), dim3(32 * wpb), params, smem, st);
}

size_t backward_smem_bytes(int vpt, int T, int G, int wpb, bool prefetch)
{
    return (size_t)bwd_group_floats(vpt, T, G, prefetch) * (wpb / G) * sizeof(float);
}

size_t forward_smem_bytes(int vpt, int G, int wpb)
{
    (void)vpt;
    return (size_t)grp_ctrl_floats(G) * (wpb / G) * sizeof(float);
}

// The slot mapping of a fit's adjoint.  Interleaved, but for a scene's long
// horizons with 4 vehicles per thread, whose tape rows are one 16-byte access
// when a thread's vehicles follow one another (2M x 1,000 at interval 50: 15.45
// -> 15.22 ms per iteration); its loads and stores of vehicles, checkpoints and
// moments then touch four times the sectors, which short horizons do not earn
// back (40 iterations of 20,000 lanes of 100 over 9 steps: 9.86 ms consecutive,
// 9.18 interleaved; 200 steps 7.53 and 7.63 per three), and with 8 vehicles per
// thread no horizon does (three of 700 lanes of 2,000 over 200 steps at interval
// 50: 9.83 and 8.13 ms, 40 over 9 steps 11.1 and 7.96).  A batch's losses are
// reported per scenario, and a scenario's FP32 partial sums by thread keep their
// grouping; loss and gradient without Adam stay interleaved too (10,000 lanes of
// 2-200 vehicles, 301 steps: 2.23 ms against 2.31).
constexpr int CONSEC_MIN_STEPS = 256;
static bool consecutive_slots(int vpt, const SimArgs &a)
{
    return vpt == 4 && a.scen_tab == nullptr && a.scen0.K >= CONSEC_MIN_STEPS;
}

// The kernels with tape blocks: for a tape shallower than the interval, and for
// one with a second part.
static bool tape_blocks(const SimArgs &a) { return a.tape_T < a.C || a.tape_more > 0; }

// Adjoint variants of every shape live in idm_shape_v<V>_g<G>.cu (with
// 4 vehicles per thread, segments of up to 4 warps run in 4-warp blocks and
// 8-warp segments in 8-warp blocks); SUB: tape shallower than the checkpoint
// interval.
static void *backward_fn_v(int vpt, int G, bool dense, bool adam, bool wd, bool sub, bool consec)
{
#define IDM_PICK(V, GW) \
    if (vpt == V && G == GW) return backward_fn_v##V##_g##GW(dense, adam, wd, sub, consec);
    IDM_SHAPES(IDM_PICK)
#undef IDM_PICK
    return nullptr;
}

// Resident blocks per SM of a kernel that allocates `cols` tensor-memory
// columns per block, from its registers, shared memory and columns (the
// runtime's occupancy query answers 1 for any kernel that allocates tensor
// memory).  A block waits for its columns, so no more than fit are launched.
static int adjoint_blocks_per_sm(const void *fn, int G, int wpb, size_t smem, int cols)
{
    cudaFuncAttributes at;
    if (cudaFuncGetAttributes(&at, fn) != cudaSuccess) return 1;
    const int regs = (at.numRegs + 7) / 8 * 8 * 32 * wpb;
    const size_t sh = (smem + at.sharedSizeBytes + 127) / 128 * 128 + 1024;
    int n = 65536 / regs;
    n = n < (int)(228 * 1024 / sh) ? n : (int)(228 * 1024 / sh);
    n = n < TMEM_COLS / cols ? n : TMEM_COLS / cols;
    // 64 named barriers per SM, 16 per block where groups have them (their ids are run-time values)
    if (G > 1) n = n < 4 ? n : 4;
    n = n < 64 / wpb ? n : 64 / wpb;
    n = n < 32 ? n : 32;
    return n > 1 ? n : 1;
}

int backward_blocks_per_sm(int vpt, int G, bool dense, bool adam, bool want_delta, int wpb, size_t smem, bool sub, int cols)
{
    void *fn = backward_fn_v(vpt, G, dense, adam, want_delta && !adam, sub, true);
    return fn ? adjoint_blocks_per_sm(fn, G, wpb, smem, cols) : 1;
}

bool backward_narrow(int vpt, int G) { return vpt == 4 && G <= 4; }

int backward_max_warps(int vpt, int G) { return backward_narrow(vpt, G) ? 4 : 8; }

int backward_resident_warps(int vpt, int G)
{
    if (vpt == 2) return 16;
    if (backward_narrow(vpt, G)) return 12;
    return 8;
}

cudaError_t launch_backward(int vpt, int G, bool dense_seed, bool adam, bool want_delta, const SimArgs &a, int grid,
                            int wpb, cudaStream_t st)
{
    if (dense_seed && adam) return cudaErrorInvalidValue;
    if (wpb > backward_max_warps(vpt, G) || wpb % G || a.tape_cols + a.tape_more > TMEM_COLS) return cudaErrorInvalidValue;
    void *fn = backward_fn_v(vpt, G, dense_seed, adam, want_delta && !adam, tape_blocks(a), consecutive_slots(vpt, a));
    if (!fn) return cudaErrorInvalidValue;
    size_t smem = backward_smem_bytes(vpt, a.tape_T, G, wpb, a.bwd_pf != 0);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    SimArgs args = a;
    args.G = G;
    void *params[] = {&args};
    return cudaLaunchKernel(fn, dim3(grid), dim3(32 * wpb), params, smem, st);
}

// Single-launch fit kernels of every shape live in idm_shape_v<V>_g<G>.cu.
static void *fused_fn_v(int vpt, int G, bool sub, bool consec)
{
#define IDM_PICK(V, GW) \
    if (vpt == V && G == GW) return fused_fn_v##V##_g##GW(sub, consec);
    IDM_SHAPES(IDM_PICK)
#undef IDM_PICK
    return nullptr;
}

cudaError_t launch_fit_fused(int vpt, int G, const SimArgs &a, long long part_stride, int grid, int wpb,
                             cudaStream_t st)
{
    if (wpb > backward_max_warps(vpt, G) || wpb % G || a.tape_cols + a.tape_more > TMEM_COLS) return cudaErrorInvalidValue;
    void *fn = fused_fn_v(vpt, G, tape_blocks(a), consecutive_slots(vpt, a));
    if (!fn) return cudaErrorInvalidValue;
    const size_t smem = backward_smem_bytes(vpt, a.tape_T, G, wpb, a.bwd_pf != 0);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, n_sm = 1;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const int cap = n_sm * adjoint_blocks_per_sm(fn, G, wpb, smem, a.tape_cols + a.tape_more);
    SimArgs args = a;
    args.G = G;
    long long stride = part_stride;
    void *params[] = {&args, &stride};
    return cudaLaunchKernel(fn, dim3(grid < cap ? grid : cap), dim3(32 * wpb), params, smem, st);
}

int forward_blocks_per_sm(int vpt, int G, int wpb)
{
    void *fn = forward_fn_v(vpt, G, false);
    if (!fn) return 1;
    const size_t smem = forward_smem_bytes(vpt, G, wpb);
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, 32 * wpb, smem) != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}

}  // namespace idm
