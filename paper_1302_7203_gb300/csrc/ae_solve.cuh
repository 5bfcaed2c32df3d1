// ae_solve.cuh -- the pipeline after the reduction, as templates over the
// problem kind: the fixed-point passes of ae_fast.cuh (far poles' moments, FP32
// opening, evaluation, step, further evaluations, the FP64 solver for what they
// leave), or k_eig, the FP64 solver for all eigenpairs, a warp each (Algorithm 1's
// shift, Algorithm 2's inverse with b by Theorem 6 under Algorithm 5's gate,
// Algorithm 3's bisection or the bracketed Newton finish); then the remedies of
// Theorem C1 and Remarks 1-2, output placement and the columns.  ae_arrow.cu
// instantiates it for the arrowhead itself;
// each other kind has a translation unit of its own (ae_solve_*.cu), so that
// the kinds compile in parallel.
#pragma once

#include <cuda_runtime.h>

#include "ae_fast.cuh"
#include "ae_internal.h"
#include "ae_pipeline.cuh"

namespace ae {

// ---------------------------------------------------------------------------
// eigenpairs
// ---------------------------------------------------------------------------
// The FP64 solver for all eigenpairs, a warp each: callers that bring no
// memory for the fixed-point path (arrow_eig_noalloc), and options it does not
// serve.
template <Kind K>
__global__ void __launch_bounds__(256, 3) k_eig(Scratch S, SolveOpts o) {
    const int lane = threadIdx.x & 31;
    const int m = S.cnt[C_M];
    const auto R = PolesOf<K>::make(S, m);
    const WarpTeam T{lane};
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    double2 *buf = S.wbuf ? S.wbuf + gw * S.wstride : nullptr;
    // a part also solves the eigenpair on each side of its range (Algorithm
    // 1's solve only, the same bits its owner computes): the remedy decision
    // of Eq. (K0) needs both neighbours.  Its tickets start at its first such
    // eigenpair (k_part sets the counter); the range is re-read per item
    // rather than held in registers across the solve.
    const int k_hi = S.cnt[C_PART] ? S.cnt[C_KHI] : m + 1;
    for (;;) {
        int k = 0;
        if (lane == 0) k = atomicAdd(S.cnt + C_WORK, 1);
        k = __shfl_sync(FULL, k, 0);
        if (k >= k_hi) break;
        eig_item<K>(R, T, S, k, o, buf);
    }
}

// Remedy decisions: one thread per eigenpair (of the part).  k_ffix takes
// them up: the solves on a DPR1 inverse (Remarks 1, 2(b)), which add a
// double-double pass, are listed from the front of the n-entry list and the
// others from its back, so that the remedy kernel deals the costlier ones out
// first, one per SM in turn.
static __global__ void k_fix_decide(Kind kind, Scratch S, double knu_max) {
    after_previous();
    const PartRange P = part_range(S);
    const int k = P.k0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (k < P.k1) fix_decide_item(kind, S, k, knu_max);
}

// remedy w of the list k_ffix wrote (front part first, then the back)
__device__ __forceinline__ int fix_at(const Scratch &S, long long w, int n) {
    const int nf = S.cnt[C_NFIX];
    return w < nf ? S.fixlist[w] : S.fixlist[n - 1 - (int)(w - nf)];
}

// Remedy solves by teams of NW warps (NW = 8, 4 or 2) that share their CTA:
// team g of CTA b takes remedies w = g * grid + b, then w + teams, ... (so that
// consecutive remedies land on different SMs), each on the stored-pair slice
// of the team's first warp (the grid never exceeds k_eig's, so the slices
// exist).
template <Kind K, int NW>
__device__ __forceinline__ void fix_solve_teams(const Scratch &S, const SolveOpts &o, int n,
                                                int nfix, double *red) {
    constexpr int TPC = 8 / NW;                  // teams per CTA of 8 warps
    const int m = S.cnt[C_M];
    const auto R = PolesOf<K>::make(S, m);
    const int g = (int)(threadIdx.x >> 5) / NW;
    const CtaTeam<NW> T{(int)threadIdx.x - g * 32 * NW, red + 2 * NW * g, NW == 8 ? 0 : 1 + g};
    const long long w0 = (long long)blockIdx.x * 8 + (long long)g * NW;
    double2 *buf = S.wbuf ? S.wbuf + w0 * S.wstride : nullptr;
    for (long long w = (long long)g * gridDim.x + blockIdx.x; w < nfix;
         w += (long long)TPC * gridDim.x) {
        fix_solve_item<K>(R, T, S, fix_at(S, w, n), o, buf);
        T.sync();                                // before buf and red are reused
    }
}

// Remedy solves.  The team size is the largest of 8, 4, 2 warps that still
// gives every listed eigenpair a team of its own (one wave over the grid);
// with more remedies than half the grid's warps, one warp each, remedy w on
// warp w / CTAs of CTA w mod CTAs: spread over all SMs.
template <Kind K>
__global__ void __launch_bounds__(256) k_fix_solve(Scratch S, SolveOpts o, int n) {
    after_previous();
    __shared__ double red[16];
    const int nfix = S.cnt[C_NFIX] + S.cnt[C_NFIX2];
    const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
    if (nfix == 0) return;
    if (nwarps / 8 >= nfix) {
        fix_solve_teams<K, 8>(S, o, n, nfix, red);
    } else if (nwarps / 4 >= nfix) {
        fix_solve_teams<K, 4>(S, o, n, nfix, red);
    } else if (nwarps / 2 >= nfix) {
        fix_solve_teams<K, 2>(S, o, n, nfix, red);
    } else {
        const int m = S.cnt[C_M];
        const auto R = PolesOf<K>::make(S, m);
        const int lane = threadIdx.x & 31;
        const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
        double2 *buf = S.wbuf ? S.wbuf + gw * S.wstride : nullptr;
        // (tickets would hand consecutive remedies to the warps of the first
        // CTAs to arrive, on a few SMs)
        const int wi = threadIdx.x >> 5;
        for (long long w = (long long)wi * gridDim.x + blockIdx.x; w < nfix;
             w += (long long)(blockDim.x >> 5) * gridDim.x) {
            fix_solve_item<K>(R, WarpTeam{lane}, S, fix_at(S, w, n), o, buf);
            __syncwarp();
        }
    }
}

// ---------------------------------------------------------------------------
// host orchestration
// ---------------------------------------------------------------------------
static int sm_count() {
    static int cached = 0;
    if (!cached) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&cached, cudaDevAttrMultiProcessorCount, dev);
        if (cached <= 0) cached = 1;
    }
    return cached;
}

// A kernel that begins with after_previous(), set up while the one before it on the
// stream drains: some 15 to 22 short kernels make up a small solve, ~2 us each
// between them (us plainly / so: n = 64 100 / 72, n = 1000 182 / 137, n = 1500
// 218 / 170).  No kernel lets the next one start before its own end: waiting CTAs
// then sit on the SMs and the few busy CTAs of the kernels between crowd together
// (n = 64 76, n = 1000 274, DPR1 n = 8192 502 -> 620).
template <class... P, class... A>
static void launch_after(void (*k)(P...), dim3 grid, int block, cudaStream_t st, A... a) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3(block);
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, k, P(a)...);
}

// Segments of the poles (rows) that k_feval (k_fcols) CTAs of a unit of 8 (32)
// eigenpairs take: enough for 8 waves of 3 CTAs an SM, so that the last one is at
// most an eighth of the time (n = 8192 alone is 2.25 waves of 8), but no less than
// a tile each.
static int segments(int units, int rows, int tile) {
    const int want = (24 * sm_count() + units - 1) / units;
    const int tiles = (rows + tile - 1) / tile;
    return want < 1 ? 1 : want < tiles ? want : tiles < 1 ? 1 : tiles;
}

// K: the arrowhead the kernels solve; VK: the kind of the vector epilogue
// (Hermitian and non-symmetric inputs solve the real arrowhead of their moduli).
// grid: k_eig's CTAs, no more than the stored-pair slices allocated (8 a CTA).
template <Kind K, Kind VK>
static void launch_pipeline(int n, int grid, Scratch S, const SolveOpts &so,
                            const RunOpts &ro, const VecArgs &va, cudaStream_t st) {
    const int sms = sm_count();
    const int gt = (n + 63) / 64, gm = n < 2 * sms ? n : 2 * sms, g8 = (n + 7) / 8, g32 = (n + 31) / 32;
    const SrcOne src{S, va};
    if (ro.ev[1]) cudaEventRecord(ro.ev[1], st);
    if (S.f.p) {
        const int diag = va.out.dg_b || va.out.dg_Kb || va.out.dg_flags;
        // (one unit more for a part that starts inside a group, and unit 0)
        if (va.n1 >= kFarFrom) launch_after(k_fgroup<K, SrcOne>, g32 + 2, 256, st, src);
        launch_after(k_fopen<K, SrcOne>, g32 + 2, 256, st, src, so);
        launch_after(k_feval<SrcOne>,
                     dim3(g8 + 1, segments(g8, va.n1 < 2 * kTile ? va.n1 : 2 * kTile, kTile)), 256,
                     st, src);
        launch_after(k_fstep<K, SrcOne>, gt, 64, st, src, so, diag);
        launch_after(k_fmore<K, SrcOne>, gm, 32 * kMoreWarps, st, src, so, 0, diag);
        launch_after(k_fold<K, SrcOne>, grid, 256, st, src, so);
        if (diag) launch_after(k_fdiag<K, SrcOne>, g8, 256, st, src, so);
    } else {
        k_eig<K><<<grid, 256, 0, st>>>(S, so);
    }
    if (ro.ev[2]) cudaEventRecord(ro.ev[2], st);
    if (ro.fixup) {
        launch_after(k_fix_decide, (n + 255) / 256, 256, st, K, S, ro.knu_max);
        launch_after(k_ffix<K, SrcOne>, gt, 64, st, src);
        if (S.f.p) launch_after(k_fmore<K, SrcOne>, gm, 32 * kMoreWarps, st, src, so, 1, 0);
        // every CTA resident at once (the remedies are assigned statically)
        static int fix_per_sm = 0;
        if (!fix_per_sm) {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fix_per_sm, k_fix_solve<K>, 256, 0);
            if (fix_per_sm <= 0) fix_per_sm = 1;
        }
        int fgrid = sms * fix_per_sm;
        fgrid = fgrid < grid ? fgrid : grid;
        fgrid = n < fgrid ? n : fgrid;
        launch_after(k_fix_solve<K>, fgrid, 256, st, S, so, n);
    }
    if (ro.ev[3]) cudaEventRecord(ro.ev[3], st);
    launch_after(k_fout<VK, SrcOne>, gt, 64, st, src);
    if (va.out.V) {
        if (S.f.p)
            launch_after(k_fcols<VK, SrcOne>,
                         dim3(g32 + 1, segments(g32 + 1, va.n1, col_rows(va.n1))), 256, st, src);
        launch_after(k_vectors<VK, SrcOne>, n < 4 * sms ? n : 4 * sms, 256, st, src);
    }
}

// The pipeline for each kind other than the arrowhead, one translation unit
// each (ae_solve_dpr1.cu, ae_solve_svd.cu, ae_solve_herm.cu, ae_solve_nsym.cu).
void launch_pipeline_dpr1(int n, int grid, Scratch S, const SolveOpts &so, const RunOpts &ro,
                          const VecArgs &va, cudaStream_t st);
void launch_pipeline_tsvd(int n, int grid, Scratch S, const SolveOpts &so, const RunOpts &ro,
                          const VecArgs &va, cudaStream_t st);
void launch_pipeline_herm(int n, int grid, Scratch S, const SolveOpts &so, const RunOpts &ro,
                          const VecArgs &va, cudaStream_t st);
void launch_pipeline_nsym(int n, int grid, Scratch S, const SolveOpts &so, const RunOpts &ro,
                          const VecArgs &va, cudaStream_t st);

}  // namespace ae
