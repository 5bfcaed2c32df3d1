// ae_arrow.cu -- the eigen-solver pipeline on one stream, for the problem
// kinds that reduce to a real symmetric arrowhead (the kernels after the
// reduction are in ae_solve.cuh; this unit instantiates them for the
// arrowhead, ae_solve_*.cu for the other kinds):
//   ARROW  A = [diag(d) z; z^T alpha]                       (Sec. 1)
//   DPR1   M = diag(d) + rho u u^T, via A = L^{-1} M L        (Sec. 6.3)
//   SVD    B = [diag(d) z; 0 alpha], via A = B^T B            (Sec. 6.2)
//
// Preparation (ae_prep.cuh): k_prep, or k_check, k_rank, k_order, k_heads,
// k_reduce, k_kind, k_post, k_forms over the rows.  Eigenpairs, remedies and
// columns: ae_fast.cuh, launched by ae_solve.cuh.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "ae_internal.h"
#include "ae_pipeline.cuh"
#include "ae_prep.cuh"
#include "ae_solve.cuh"

namespace ae {

// ---------------------------------------------------------------------------
// checks, order, reduction, forms: over the rows by a grid (ae_prep.cuh)
// ---------------------------------------------------------------------------
template <Kind K>
__global__ void __launch_bounds__(256) k_check(PrepArgs A, Scratch S) {
    after_previous();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    int flags = 0;
    if (r < A.n1) {
        flags = check_item<K>(A, S, r);
        S.spos[r] = 0;                              // (k_rank counts there)
    }
    flags = __reduce_or_sync(FULL, flags);
    if ((threadIdx.x & 31) == 0 && flags) atomicOr(S.cnt + C_FLAGS, flags);
}

// Sorted input without zero spikes: reduced as it stands.  Else the rows' ranks
// (descending, ties by lower row), each CTA counting 256 rows against one tile
// of 1024 keys (blockIdx.y).
__global__ void __launch_bounds__(256) k_rank(int n1, const double *__restrict__ key,
                                              const double *__restrict__ spk, Scratch S) {
    after_previous();
    __shared__ unsigned long long tile[1024];
    const int flags = S.cnt[C_FLAGS];
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (!(flags & CF_UNSORTED)) {
        if (blockIdx.y) return;
        if (flags & CF_ZERO) {
            if (r < n1) S.spos[r] = r;
            return;
        }
        if (r < n1) identity_row(S, key, spk, r);
        if (r == 0) {
            S.cnt[C_M] = n1;
            S.cnt[C_ND] = 0;
        }
        return;
    }
    const int base = blockIdx.y * 1024, lim = min(1024, n1 - base);
    for (int t = threadIdx.x; t < lim; t += 256) tile[t] = order_key(key[base + t]);
    __syncthreads();
    if (r >= n1) return;
    const unsigned long long kr = order_key(key[r]);
    int rank = 0;
#pragma unroll 4
    for (int t = 0; t < lim; ++t) {
        const unsigned long long q = tile[t];
        rank += (q > kr) || (q == kr && base + t < r);
    }
    if (rank) atomicAdd(S.spos + r, rank);
}

__global__ void __launch_bounds__(256) k_order(int n1, Scratch S) {
    after_previous();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n1 && (S.cnt[C_FLAGS] & (CF_UNSORTED | CF_ZERO))) S.perm[S.spos[r]] = r;
}

// heads of runs in each CTA's 256 sorted positions (counted in fixlist, which
// nothing uses before the remedies)
__global__ void __launch_bounds__(256) k_heads(int n1, const double *__restrict__ key,
                                               const double *__restrict__ spk, Scratch S) {
    after_previous();
    if (!(S.cnt[C_FLAGS] & (CF_UNSORTED | CF_ZERO))) return;
    const int s = blockIdx.x * 256 + threadIdx.x;
    const bool head = s < n1 && is_head(key, spk, S.perm, s);
    const int c = __syncthreads_count(head);
    if (threadIdx.x == 0) S.fixlist[blockIdx.x] = c;
}

__global__ void __launch_bounds__(256) k_reduce(int n1, const double *__restrict__ key,
                                                const double *__restrict__ spk, Scratch S) {
    after_previous();
    __shared__ int wh[8], before;
    if (!(S.cnt[C_FLAGS] & (CF_UNSORTED | CF_ZERO))) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // heads before this CTA's positions, then before this thread's
    if (wid == 0) {
        int c = 0;
        for (int b = lane; b < (int)blockIdx.x; b += 32) c += S.fixlist[b];
        c = __reduce_add_sync(FULL, c);
        if (lane == 0) before = c;
    }
    const int s = blockIdx.x * 256 + threadIdx.x;
    const bool in = s < n1, head = in && is_head(key, spk, S.perm, s);
    const unsigned bal = __ballot_sync(FULL, head);
    if (lane == 0) wh[wid] = __popc(bal);
    __syncthreads();
    int jk = before + __popc(bal & ((1u << lane) - 1u));
    for (int w = 0; w < wid; ++w) jk += wh[w];
    if (in) reduce_item(S, key, spk, n1, s, head, jk, s - jk);
    if (s == n1 - 1) {
        S.cnt[C_M] = jk + (head ? 1 : 0);
        S.cnt[C_ND] = n1 - S.cnt[C_M];
    }
}

template <Kind K>
__global__ void __launch_bounds__(kChunk) k_kind(PrepArgs A, Scratch S) {
    after_previous();
    __shared__ PoleShare sh[kChunk / 32];
    kind_chunk<K>(A, S, S.cnt[C_M], blockIdx.x, threadIdx.x, sh, 0);
}
template <Kind K>
__global__ void __launch_bounds__(32) k_post(PrepArgs A, Scratch S) {
    after_previous();
    prep_finish<K>(A, S, threadIdx.x);
}
template <Kind K>
__global__ void __launch_bounds__(256) k_forms(Scratch S, VecArgs va) {
    after_previous();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < va.n1) forms_item<K>(S, va, t);
}

// all of it by one CTA
template <Kind K>
__global__ void __launch_bounds__(1024) k_prep(PrepArgs A, Scratch S, VecArgs va) {
    after_previous();
    prep_block<K>(A, S, va);
}

// Up to this many rows one CTA prepares an instance (one launch instead of ten
// operations on the stream).  A whole solve, one CTA against the grid kernels
// (launched plainly):
// n = 64 99 / 120 us, n = 400 115 / 135 (rows in no order: 175 / 184),
// n = 1000 163 / 177 (226 / 204), n = 1500 222 / 231 (581 / 430).
constexpr int kPrepRows = 640;

template <Kind K>
static cudaError_t launch_prep(const PrepArgs &A, const Scratch &S, const VecArgs &va,
                               cudaStream_t st) {
    if (A.n1 <= kPrepRows) {
        k_prep<K><<<1, 1024, 0, st>>>(A, S, va);
        return cudaSuccess;
    }
    cudaError_t e = cudaMemsetAsync(S.cnt, 0, sizeof(int) * C_COUNT, st);
    if (!e) e = cudaMemsetAsync(S.cnt64, 0, sizeof(unsigned long long) * C64_COUNT, st);
    if (e) return e;
    const int n1 = A.n1, g = (n1 + 255) / 256;
    k_check<K><<<g, 256, 0, st>>>(A, S);
    launch_after(k_rank, dim3(g, (n1 + 1023) / 1024), 256, st, n1, va.key, va.spk, S);
    launch_after(k_order, g, 256, st, n1, S);
    launch_after(k_heads, g, 256, st, n1, va.key, va.spk, S);
    launch_after(k_reduce, g, 256, st, n1, va.key, va.spk, S);
    launch_after(k_kind<K>, g, kChunk, st, A, S);
    launch_after(k_post<K>, 1, 32, st, A, S);
    launch_after(k_forms<K>, g, 256, st, S, va);
    return cudaSuccess;
}

// One part of a split solve: its eigenpair range (an even split of the m + 1
// computed eigenpairs), its deflated rows and its first output position.
__global__ void k_part(Scratch S, int part, int nparts) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int nd = S.cnt[C_ND], ncomp = S.cnt[C_M] + 1;
    const int k0 = (int)((long long)part * ncomp / nparts);
    const int k1 = (int)((long long)(part + 1) * ncomp / nparts);
    // deflated values (non-increasing) in [p_{k1-1}, p_{k0-1})
    const int u0 = k0 == 0 ? 0 : count_ge(S.dval, nd, S.pv[k0 - 1], false);
    const int u1 = k1 == ncomp ? nd : (k1 == 0 ? 0 : count_ge(S.dval, nd, S.pv[k1 - 1], false));
    S.cnt[C_K0] = k0;
    S.cnt[C_K1] = k1;
    S.cnt[C_U0] = u0;
    S.cnt[C_U1] = u1 > u0 ? u1 : u0;
    S.cnt[C_POS0] = k0 + u0;
    S.cnt[C_WORK] = k0 > 0 ? k0 - 1 : 0;             // k_eig's first ticket
    S.cnt[C_KHI] = k1 < ncomp ? k1 + 1 : ncomp;
    S.cnt[C_PART] = 1;
}

__global__ void k_debug_rcp(int n, const double *x, double *y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = rcp(x[i]);
}

// The FP64 finish (newton_finish) on the shifted inverse's Pick function
// F(x) = (b - x) - c (sum_j cj_j / (1 - x delta_j) - 1/x), kappa = -1, from a
// caller's bracket, start and F' estimate; one thread.  out: nu (the right end
// of the final bracket), the FP64 evaluations, those with F'.
__global__ void k_debug_newton(int m, const double *__restrict__ delta,
                               const double *__restrict__ cj, DebugNewton a, double *out) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    auto FD = [&](double x, bool need_d, double &dF, double &err) {
        double S = 0.0, Sd = 0.0;
        for (int j = 0; j < m; ++j) {
            const double t = rcp(fma(-x, delta[j], 1.0));
            const double q = cj[j] * t;
            S += q;
            if (need_d) Sd = fma(q * delta[j], t, Sd);
        }
        const double rx = rcp(x);
        if (need_d) dF = -1.0 - a.c * fma(rx, rx, Sd);
        err = 0x1p-52 * (fabs(a.b) + fabs(x) + a.c * (fabs(S) + fabs(rx)));
        return (a.b - x) - a.c * (S - rx);
    };
    double left = a.left, right = a.right;
    bool fb;
    int itd = 0;
    const int it = newton_finish(FD, a.side, a.pole, -1.0, left, right, true, true, a.max_iter,
                                 left, right, fb, a.dF0, &itd, a.x0, a.c, a.xdF0, a.rel0);
    out[0] = right;
    out[1] = (double)it;
    out[2] = (double)itd;
}

// ---------------------------------------------------------------------------
// scratch layout
// ---------------------------------------------------------------------------
// One layout routine serves both sizing and carving, so they cannot disagree:
// every array starts on a 256-byte boundary.
static size_t layout(uintptr_t base, int n, Scratch *S) {
    const size_t n1 = n > 1 ? (size_t)n : 1;     // rows: n - 1 (arrowhead) or n (DPR1)
    const size_t nn = (size_t)n;
    uintptr_t p = (base + 255) & ~(uintptr_t)255;
    const uintptr_t start = base;
    auto take = [&](size_t bytes) {
        uintptr_t q = p;
        p += (bytes + 255) & ~(size_t)255;
        return (void *)q;
    };
    Scratch T;
    T.cnt = (int *)take(sizeof(int) * C_COUNT);
    T.cnt64 = (unsigned long long *)take(sizeof(unsigned long long) * C64_COUNT);
    T.prm = (double *)take(sizeof(double) * P_COUNT);
    T.perm = (int *)take(sizeof(int) * n1);
    T.spos = (int *)take(sizeof(int) * n1);
    T.kind = (int *)take(sizeof(int) * n1);
    T.run_s0 = (int *)take(sizeof(int) * n1);
    T.run_R = (double *)take(sizeof(double) * 2 * n1);
    T.key = (double *)take(sizeof(double) * n1);
    T.spk = (double *)take(sizeof(double) * n1);
    T.pd = (double *)take(sizeof(double) * n1);
    T.pz = (double *)take(sizeof(double) * n1);
    T.pz2 = (double *)take(sizeof(double) * n1);
    T.pz2lo = (double *)take(sizeof(double) * n1);
    T.pv = (double *)take(sizeof(double) * n1);
    T.pdh = (float *)take(sizeof(float) * n1);
    T.pdl = (float *)take(sizeof(float) * n1);
    T.pz2f = (float *)take(sizeof(float) * n1);
    T.prow = (int *)take(sizeof(int) * n1);
    T.drow = (int *)take(sizeof(int) * n1);
    T.dval = (double *)take(sizeof(double) * n1);
    T.es_sigma = (double *)take(sizeof(double) * nn);
    T.es_mu = (double *)take(sizeof(double) * nn);
    T.es_lam = (double *)take(sizeof(double) * nn);
    T.es_b = (double *)take(sizeof(double) * nn);
    T.es_Kb = (double *)take(sizeof(double) * nn);
    T.es_Knu = (double *)take(sizeof(double) * nn);
    T.es_fixshift = (double *)take(sizeof(double) * nn);
    T.es_pole = (int *)take(sizeof(int) * nn);
    T.es_iters = (int *)take(sizeof(int) * nn);
    T.es_flags = (int *)take(sizeof(int) * nn);
    T.es_fixpole = (int *)take(sizeof(int) * nn);
    T.fixlist = (int *)take(sizeof(int) * nn);
    T.pos = (int *)take(sizeof(int) * nn);
    T.cols = (int *)take(sizeof(int) * nn);
    T.wbuf = nullptr;
    T.wstride = 0;
    T.f = FastPtrs{};
    if (S) *S = T;
    return (size_t)(p - start);
}

// bytes to request: the layout from a 256-aligned base, plus room to align
// (fixed-point path, carved the same way from its own block)
static size_t fast_layout(uintptr_t base, int n, FastPtrs *F) {
    const size_t n1 = n > 1 ? (size_t)n : 1, nn = (size_t)n;
    uintptr_t p = (base + 255) & ~(uintptr_t)255;
    auto take = [&](size_t bytes) {
        uintptr_t q = p;
        p += (bytes + 255) & ~(size_t)255;
        return (void *)q;
    };
    using u64 = unsigned long long;
    FastPtrs T;
    T.grp = (GroupData *)take(sizeof(GroupData) * (nn / kGroup + 2));
    T.p = (double *)take(8 * n1);
    T.plo = (double *)take(8 * n1);
    T.P = (u64 *)take(8 * n1);
    T.P2 = (u64 *)take(8 * n1);
    T.z = (u64 *)take(8 * n1);
    T.zh = (u64 *)take(8 * n1);
    T.zl = (u64 *)take(8 * n1);
    T.ez = (int *)take(4 * n1);
    T.rp = (double *)take(8 * n1);
    T.rP = (u64 *)take(8 * n1);
    T.mu = (double *)take(8 * nn);
    T.mulo = (double *)take(8 * nn);
    T.lhi = (double *)take(8 * nn);
    T.llo = (double *)take(8 * nn);
    T.N = (double *)take(8 * nn);
    T.Nlo = (double *)take(8 * nn);
    T.M2u = (double *)take(8 * nn);
    T.lmod = (u64 *)take(8 * nn);
    T.lmod2 = (u64 *)take(8 * nn);
    T.cm = (u64 *)take(8 * nn);
    T.cm2 = (u64 *)take(8 * nn);
    T.ce = (int *)take(4 * nn);
    T.ce2 = (int *)take(4 * nn);
    T.l32 = (int *)take(4 * nn);
    T.K1 = (int *)take(4 * nn);
    T.K2 = (int *)take(4 * nn);
    T.er = (int *)take(4 * nn);
    T.s1 = (long long *)take(8 * nn);
    T.s3 = (long long *)take(8 * nn);
    T.s5 = (long long *)take(8 * nn);
    T.s2 = (u64 *)take(8 * nn);
    T.s4 = (u64 *)take(8 * nn);
    T.l1 = (long long *)take(8 * nn);
    T.l2 = (u64 *)take(8 * nn);
    T.st = (int *)take(4 * nn);
    T.old = (int *)take(4 * nn);
    T.more = (int *)take(4 * nn);
    if (F) *F = T;
    return (size_t)(p - base);
}

size_t fast_bytes(int n) { return fast_layout(0, n, nullptr) + 256; }

FastPtrs carve_fast(void *base, int n) {
    FastPtrs F;
    fast_layout((uintptr_t)base, n, &F);
    return F;
}

size_t arrow_scratch_bytes(int n) { return layout(0, n, nullptr) + 256; }

Scratch carve_scratch(void *base, int n) {
    Scratch S;
    layout((uintptr_t)base, n, &S);
    return S;
}

// ---------------------------------------------------------------------------
// host orchestration
// ---------------------------------------------------------------------------
// CTAs of k_eig: enough for every eigenpair, at most what stays resident
// (every kind's k_eig has the same launch bounds, so the arrowhead's
// occupancy holds for all; the stored-pair slices are allocated for this grid)
static int eig_grid(int n) {
    static int per_sm = 0;
    if (!per_sm) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_eig<KIND_ARROW>, 256, 0);
        if (per_sm <= 0) per_sm = 1;
    }
    const int want = (n + 7) / 8;
    const int cap = sm_count() * per_sm;
    return want < cap ? want : cap;
}

int eig_grid_warps(int n) { return eig_grid(n) * 8; }

cudaError_t launch_solve(Kind kind, int n, const double *d, const double *z, double alpha,
                         double rho, const Outputs &out, const RunOpts &ro, Scratch S,
                         cudaStream_t st, const double *zrow) {
    const int n1 = kind == KIND_DPR1 ? n : n - 1;
    const double sgn = (kind == KIND_DPR1 && rho < 0.0) ? -1.0 : 1.0;
    const double *key = (kind == KIND_DPR1 && sgn < 0.0) ? S.key : d;
    const bool rho0 = kind == KIND_DPR1 && rho == 0.0;   // M = D: every row deflates
    const bool own_spk = kind == KIND_TSVD || kind == KIND_HERM || kind == KIND_NSYM || rho0;
    const double *spk = own_spk ? S.spk : z;
    if (ro.max_iter < kMinIterCap) S.f = FastPtrs{};
    const SolveOpts so{ro.max_iter, ro.precision, ro.finish, ro.bgate, ro.kb_max};
    const VecArgs va{n, n1, key, spk, z, zrow, kind == KIND_DPR1 ? rho : alpha, sgn, out};
    const PrepArgs A{n1, d, z, zrow, alpha, rho, sgn};
    const int grid = eig_grid(n);
    cudaError_t e = cudaSuccess;
    if (ro.ev[0]) cudaEventRecord(ro.ev[0], st);
    switch (kind) {
        case KIND_ARROW:
            e = launch_prep<KIND_ARROW>(A, S, va, st);
            if (!e) launch_pipeline<KIND_ARROW, KIND_ARROW>(n, grid, S, so, ro, va, st);
            break;
        case KIND_DPR1:
            e = launch_prep<KIND_DPR1>(A, S, va, st);
            if (!e) launch_pipeline_dpr1(n, grid, S, so, ro, va, st);
            break;
        case KIND_TSVD:
            e = launch_prep<KIND_TSVD>(A, S, va, st);
            if (!e) launch_pipeline_tsvd(n, grid, S, so, ro, va, st);
            break;
        case KIND_HERM:
            e = launch_prep<KIND_HERM>(A, S, va, st);
            if (!e) launch_pipeline_herm(n, grid, S, so, ro, va, st);
            break;
        case KIND_NSYM:
            e = launch_prep<KIND_NSYM>(A, S, va, st);
            if (!e) launch_pipeline_nsym(n, grid, S, so, ro, va, st);
            break;
    }
    if (e) return e;
    if (ro.ev[4]) cudaEventRecord(ro.ev[4], st);
    return cudaGetLastError();
}

cudaError_t launch_arrow_part(int n, const double *d, const double *z, double alpha, int part,
                              int nparts, int cap, const Outputs &out, const RunOpts &ro,
                              Scratch S, cudaStream_t st, int *pos0, int *count) {
    const int n1 = n - 1;
    if (ro.max_iter < kMinIterCap) S.f = FastPtrs{};
    const VecArgs va{n, n1, d, z, z, nullptr, alpha, 1.0, out};
    if (ro.ev[0]) cudaEventRecord(ro.ev[0], st);
    cudaError_t e =
        launch_prep<KIND_ARROW>(PrepArgs{n1, d, z, nullptr, alpha, 0.0, 1.0}, S, va, st);
    if (e) return e;
    k_part<<<1, 32, 0, st>>>(S, part, nparts);
    int h[C_COUNT];
    e = cudaMemcpyAsync(h, S.cnt, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (!e) e = cudaStreamSynchronize(st);
    if (e) return e;
    *pos0 = h[C_POS0];
    *count = (h[C_K1] - h[C_K0]) + (h[C_U1] - h[C_U0]);
    if (!out.lambda || *count > cap) return cudaSuccess;   // size query, or no room
    const SolveOpts so{ro.max_iter, ro.precision, ro.finish, ro.bgate, ro.kb_max};
    launch_pipeline<KIND_ARROW, KIND_ARROW>(n, eig_grid(n), S, so, ro, va, st);
    if (ro.ev[4]) cudaEventRecord(ro.ev[4], st);
    return cudaGetLastError();
}

cudaError_t launch_debug_rcp(int n, const double *x, double *y, cudaStream_t st) {
    if (n > 0) k_debug_rcp<<<(n + 255) / 256, 256, 0, st>>>(n, x, y);
    return cudaGetLastError();
}

cudaError_t launch_debug_newton(int m, const double *delta, const double *cj,
                                const DebugNewton &a, double *out, cudaStream_t st) {
    k_debug_newton<<<1, 32, 0, st>>>(m, delta, cj, a, out);
    return cudaGetLastError();
}

}  // namespace ae
