// ae_pipeline.cuh -- the per-instance and per-eigenpair bodies of the solver
// pipeline, shared by the single-instance kernels (ae_arrow.cu) and the
// batched, persistent ones (ae_batch.cu).  Each function states which threads
// call it: a whole CTA of 1024 threads (the *_block functions), one thread, one
// warp, or one team.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "ae_internal.h"
#include "ae_solver.cuh"

namespace ae {

// block-wide exclusive scan of one int per thread (blockDim = 1024)
__device__ __forceinline__ int block_exscan(int v, int *warp_tot, int &total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int t = warp_tot[lane];
        int u = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(FULL, u, o);
            if (lane >= o) u += y;
        }
        warp_tot[lane] = u - t;       // exclusive prefix of warp totals
        if (lane == 31) warp_tot[32] = u;
    }
    __syncthreads();
    const int res = warp_tot[wid] + x - v;
    total = warp_tot[32];
    __syncthreads();
    return res;
}

template <Kind K>
struct PolesOf;
template <>
struct PolesOf<KIND_ARROW> {
    using type = ArrowPoles;
    __device__ static ArrowPoles make(const Scratch &S, int m) {
        return {m,      S.pd,  S.pz,  S.pz2,          S.pz2lo,        S.prm[P_ALPHA_HI],
                S.prm[P_ALPHA_LO], S.pdh, S.pdl,      S.pz2f,         S.prm[P_DS],
                S.prm[P_ZS],       S.prm[P_ZSUM]};
    }
};
template <>
struct PolesOf<KIND_DPR1> : PolesOf<KIND_ARROW> {};
template <>
struct PolesOf<KIND_HERM> : PolesOf<KIND_ARROW> {};
template <>
struct PolesOf<KIND_NSYM> : PolesOf<KIND_ARROW> {};
template <>
struct PolesOf<KIND_TSVD> {
    using type = TsvdPoles;
    __device__ static TsvdPoles make(const Scratch &S, int m) {
        return {m,     S.pd,     S.pv,              S.pz,  S.pz2, S.pz2lo,
                S.prm[P_ALPHA_HI], S.prm[P_ALPHA_LO], S.pdh, S.pdl, S.pz2f,
                S.prm[P_DS],       S.prm[P_ZS],       S.prm[P_ZSUM]};
    }
};

__device__ __forceinline__ void store_result(const Scratch &S, int k, const EigResult &r) {
    S.es_sigma[k] = r.sigma;
    S.es_mu[k] = r.mu;
    S.es_lam[k] = r.lam;
    S.es_b[k] = r.b;
    S.es_Kb[k] = r.Kb;
    S.es_pole[k] = r.pole;
    S.es_iters[k] = r.iters;
}

__device__ __forceinline__ void record_stats(const Scratch &S, const EigResult &r,
                                             bool fix = false) {
    atomicAdd(S.cnt64 + C64_ITERS, (unsigned long long)r.iters);
    if (r.iters_d && !fix) atomicAdd(S.cnt64 + C64_DERIV, (unsigned long long)r.iters_d);
    if (fix) atomicAdd(S.cnt64 + C64_ITERS_FIX, (unsigned long long)r.iters);
    if (r.f32p) atomicAdd(S.cnt64 + C64_F32, (unsigned long long)r.f32p);
    if (r.dfp) atomicAdd(S.cnt64 + C64_DF, (unsigned long long)r.dfp);
    atomicMax(S.cnt + C_MAXIT, r.iters);
    if (r.flags & AE_FLAG_CAPPED) atomicAdd(S.cnt + C_CAPPED, 1);
    if (r.flags & AE_FLAG_FP32_FALLBACK) atomicAdd(S.cnt + C_FP32FB, 1);
    if (r.flags & AE_FLAG_DDB) atomicAdd(S.cnt + C_DDB, 1);
    if (r.flags & AE_FLAG_MID64) atomicAdd(S.cnt + C_MID64, 1);
    if (isfinite(r.Kb)) atomic_max_nonneg(S.cnt64 + C64_MAXKB, r.Kb);
}

// Eigenpair k of the reduced arrowhead by one team; the team's rank-0 thread
// stores the result.
template <Kind K, class Team>
__device__ __forceinline__ void eig_item(const typename PolesOf<K>::type &R, const Team &T,
                                         const Scratch &S, int k, const SolveOpts &o,
                                         double2 *buf = nullptr) {
    const int m = R.m;
    EigResult res;
    if (m == 0) {
        const double a = S.prm[P_ALPHA_HI];
        res = {a, S.prm[P_ALPHA_LO], a, NAN, 0.0, -1, 0, 0};
    } else {
        int i, side;
        bool ran32 = false;
        const bool mid64 = select_shift(R, T, k, i, side, o.precision == 1, &ran32);
        res = solve_shifted(R, T, i, side, o, buf);
        if (mid64) res.flags |= AE_FLAG_MID64;
        if (ran32) ++res.f32p;
    }
    if (T.rank == 0) {
        store_result(S, k, res);
        S.es_flags[k] = res.flags;
        S.es_Knu[k] = 1.0;
        record_stats(S, res);
    }
}

// Remedy decision for eigenpair k; returns the AE_FLAG_* remedy (0: none).
static __device__ int fix_decide_item(Kind kind, const Scratch &S, int k, double knu_max) {
    const int m = S.cnt[C_M];
    if (k > m || m <= 0) return 0;
    const double lam = S.es_lam[k], sig = S.es_sigma[k], mu = S.es_mu[k];
    const int i = S.es_pole[k];
    const double q = (fabs(sig) + fabs(mu)) / fabs(lam);
    int remedy = 0;
    double knu = 1.0;
    if (kind == KIND_DPR1 && k == m &&
        fabs(lam - S.prm[P_PLAST]) < fabs(mu)) {
        // DPR1: the last eigenvalue lies between the last arrowhead pole and
        // the DPR1's last pole p_last, which is not a pole of the arrowhead; when
        // it is nearer p_last, re-solve from (A - p_last I)^{-1} so that
        // lambda - p_last (and the vector's last component) keep relative accuracy.
        S.es_fixshift[k] = S.prm[P_PLAST];
        remedy = AE_FLAG_DPR1SHIFT;
    } else if (q > 3.0 && !(S.cnt[C_FLAGS] & CF_ZEROPOLE)) {
        // Theorem C1 bounds the quotient by 3 except in the special cases
        // (a)-(c); Remark 1 needs D nonsingular.
        remedy = AE_FLAG_NEARZERO;
    } else if (i >= 0) {
        // K_nu = |mu| / min(|mu|, |mu_o|), mu_o from the eigenvalue on the other
        // side of the shift pole
        const int kn = mu > 0.0 ? k + 1 : k - 1;
        if (kn >= 0 && kn <= m) {
            const double muo = (S.es_sigma[kn] - sig) + S.es_mu[kn];
            knu = fmax(1.0, fabs(mu) / fabs(muo));
        }
        if (knu > knu_max) {
            // Remark 2(a): the other pole of lambda's interval, if its K_nu is small
            const int io = mu > 0.0 ? i - 1 : i + 1;
            const int kn2 = mu > 0.0 ? k - 1 : k + 1;
            if (io >= 0 && io < m) {
                const double po = S.pv[io];
                const double mu2 = lam - po;
                double k2 = 1.0;
                if (kn2 >= 0 && kn2 <= m) {
                    const double muo2 = (S.es_sigma[kn2] - po) + S.es_mu[kn2];
                    k2 = fmax(1.0, fabs(mu2) / fabs(muo2));
                }
                if (k2 <= knu_max) {
                    remedy = AE_FLAG_OTHERPOLE;
                    S.es_fixpole[k] = io;
                }
            }
            if (!remedy) {
                // Remark 2(b): shift near lambda, inside its interval, not a pole
                double sh = lam;
                const double lo = k < m ? S.pv[k] : -INFINITY;
                const double hi = k > 0 ? S.pv[k - 1] : INFINITY;
                if (!(sh > lo)) sh = nextafter(lo, INFINITY);
                if (!(sh < hi)) sh = nextafter(hi, -INFINITY);
                S.es_fixshift[k] = sh;
                remedy = AE_FLAG_DPR1SHIFT;
            }
        }
    }
    S.es_Knu[k] = knu;
    atomic_max_nonneg(S.cnt64 + C64_MAXKNU, knu);
    if (remedy) {
        S.es_flags[k] |= remedy;
        atomicAdd(S.cnt + (remedy == AE_FLAG_NEARZERO ? C_NEARZERO
                           : remedy == AE_FLAG_OTHERPOLE ? C_OTHERPOLE : C_DPR1), 1);
    }
    return remedy;
}

// Remedy solve of eigenpair k by a team (a CTA in the single-instance pipeline,
// a warp in the batched one); all of its threads call it.
// buf: the team's slice of stored pairs (or null).
template <Kind K, class Team>
__device__ void fix_solve_item(const typename PolesOf<K>::type &R, const Team &T, const Scratch &S,
                               int k, const SolveOpts &o, double2 *buf = nullptr) {
    const int m = S.cnt[C_M];
    const int f = S.es_flags[k];
    EigResult res;
    if (f & AE_FLAG_NEARZERO) {
        res = solve_dpr1_shift(R, T, 0.0, o, buf);
    } else if (f & AE_FLAG_OTHERPOLE) {
        const int io = S.es_fixpole[k];
        const int side = io < S.es_pole[k] ? -1 : +1;   // other pole above -> lambda below it
        res = solve_shifted(R, T, io, side, o, buf);
    } else {
        res = solve_dpr1_shift(R, T, S.es_fixshift[k], o, buf);
    }
    // the result must stay in the eigenvalue's interlacing interval
    const double lo = k < m ? R.pole(k) : (K == KIND_DPR1 ? S.prm[P_PLAST] : -INFINITY);
    const double hi = k > 0 ? R.pole(k - 1) : INFINITY;
    const bool ok = (res.lam >= lo && res.lam <= hi) && isfinite(res.lam);
    if (T.rank == 0) {
        if (ok) {
            // b and K_b stay those of Algorithm 1's shift pole
            res.b = S.es_b[k];
            res.Kb = S.es_Kb[k];
            store_result(S, k, res);
            S.es_flags[k] = f | res.flags;
            record_stats(S, res, true);
        } else {
            S.es_flags[k] = f & ~(AE_FLAG_NEARZERO | AE_FLAG_OTHERPOLE | AE_FLAG_DPR1SHIFT);
        }
    }
}

// The items a solve writes: all of them, or one part of a split solve --
// computed eigenpairs [k0, k1) and the deflated rows [u0, u1) whose values
// lie in [p_{k1-1}, p_{k0-1}), which together hold the output positions
// [pos0, pos0 + (k1 - k0) + (u1 - u0)) of the whole decomposition.
struct PartRange {
    int k0, k1, u0, u1, pos0;
};

__device__ __forceinline__ PartRange part_range(const Scratch &S) {
    if (!S.cnt[C_PART]) return {0, S.cnt[C_M] + 1, 0, S.cnt[C_ND], 0};
    return {S.cnt[C_K0], S.cnt[C_K1], S.cnt[C_U0], S.cnt[C_U1], S.cnt[C_POS0]};
}

// number of entries of a non-increasing array that are >= x (or > x)
__device__ __forceinline__ int count_ge(const double *a, int len, double x, bool strict) {
    int lo = 0, hi = len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const bool in = strict ? (a[mid] > x) : (a[mid] >= x);
        if (in) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// output position of item t (computed eigenpairs first, then deflated rows).
// A deflated row's value v lies in its part's interval [p_{k1-1}, p_{k0-1}),
// so every computed eigenvalue before k0 exceeds it and none from k1 on does:
// only the part's own eigenvalues need comparing.
static __device__ void place_item(const Scratch &S, int t) {
    const int m = S.cnt[C_M], nd = S.cnt[C_ND];
    const int ncomp = m + 1;
    if (t < ncomp) {
        S.pos[t] = nd ? t + count_ge(S.dval, nd, S.es_lam[t], false) : t;
    } else if (t < ncomp + nd) {
        const int u = t - ncomp;
        const PartRange P = part_range(S);
        S.pos[t] = u + P.k0 + count_ge(S.es_lam + P.k0, P.k1 - P.k0, S.dval[u], true);
    }
}

// Helmert-type vector of a run-folded row:
// (-s_q sum_{l<m} s_l e_l + R_{m-1}^2 e_q) / (R_{m-1} R_m) with the run's spikes s
template <int STRIDE = 32>
__device__ __forceinline__ void run_column(const Scratch &S, const double *spk, int row, int lane,
                                           double *col, double sign) {
    const double Rm1 = S.run_R[2 * row], Rm = S.run_R[2 * row + 1];
    const double zq = spk[row];
    const double den = Rm1 * Rm;
    const int s0 = S.run_s0[row], s1 = S.spos[row];
    for (int s = s0 + lane; s < s1; s += STRIDE) {
        const int rq = S.perm[s];
        const double zl = spk[rq];
        if (zl != 0.0) col[rq] = sign * (-(zq * zl) / den);
    }
    if (lane == 0) col[row] = sign * (Rm1 / Rm);
}

// output position of item `item` in the caller's arrays (a part's own block;
// -M's order reversed for a DPR1 with rho < 0).  Inside the block also where an
// eigenvalue is NaN (input that is rejected when the caller asks): no write may
// leave the arrays meanwhile.
template <Kind K>
__device__ __forceinline__ int out_pos(const Scratch &S, int n, double sgn, int item) {
    int pos = S.pos[item];
    if (S.cnt[C_PART]) {
        const PartRange P = part_range(S);
        pos = min(max(pos - P.pos0, 0), (P.k1 - P.k0) + (P.u1 - P.u0) - 1);
    }
    return K == KIND_DPR1 && sgn < 0.0 ? n - 1 - pos : pos;
}

// SVD: the singular value of computed eigenpair k, from lambda = d_i^2 + mu
// (pole shift) or sigma + mu in double-double
__device__ __forceinline__ double sv_of(const Scratch &S, int k) {
    const int pi = S.es_pole[k];
    const double mu = S.es_mu[k];
    dd l2;
    if (pi >= 0) {
        const double di = S.pd[pi];
        l2 = dd_add(two_prod(di, di), dd{mu, 0.0});
    } else {
        l2 = two_sum(S.es_sigma[k], mu);
    }
    return dd_sqrt(l2).hi;
}

// Scalar outputs of item `item` (a computed eigenpair, or a deflated row) by
// one thread: the value, optional shift / mu, diagnostics.
template <Kind K>
__device__ void scalar_item(int n, const double *__restrict__ key, double sgn, const Scratch &S,
                            const Outputs &out, int item) {
    const int ncomp = S.cnt[C_M] + 1;
    const int pos = out_pos<K>(S, n, sgn, item);
    if (item < ncomp) {
        const int k = item;
        const double sig = S.es_sigma[k], mu = S.es_mu[k];
        double value = S.es_lam[k];
        if (K == KIND_TSVD) value = sv_of(S, k);
        else if (K == KIND_DPR1) value = sgn * value;
        out.lambda[pos] = value;
        if (out.shift) out.shift[pos] = K == KIND_DPR1 ? sgn * sig : sig;
        if (out.mu) out.mu[pos] = K == KIND_DPR1 ? sgn * mu : mu;
        if (out.dg_b) out.dg_b[pos] = S.es_b[k];
        if (out.dg_Kb) out.dg_Kb[pos] = S.es_Kb[k];
        if (out.dg_Knu) out.dg_Knu[pos] = S.es_Knu[k];
        if (out.dg_iters) out.dg_iters[pos] = S.es_iters[k];
        if (out.dg_flags) out.dg_flags[pos] = S.es_flags[k];
    } else {
        const double kv = key[S.drow[item - ncomp]];
        const double value = K == KIND_DPR1 ? sgn * kv : kv;
        out.lambda[pos] = value;
        if (out.shift) out.shift[pos] = value;
        if (out.mu) out.mu[pos] = 0.0;
        if (out.dg_b) out.dg_b[pos] = NAN;
        if (out.dg_Kb) out.dg_Kb[pos] = 0.0;
        if (out.dg_Knu) out.dg_Knu[pos] = 1.0;
        if (out.dg_iters) out.dg_iters[pos] = 0;
        if (out.dg_flags) out.dg_flags[pos] = AE_FLAG_DEFLATED;
    }
}

// Column(s) of item `item` by one team in FP64: deflated rows, and eigenpairs
// the FP64 solver took.  stage: room for the column (two doubles a row for HERM)
// that pass 1 fills instead of the column itself, which may lie in host memory.  `key`/`spk` are the transformed inputs the reduction
// saw; z is the caller's spike array (SVD: for the left vectors; HERM: the
// complex spikes; NSYM: the column spikes, zrow the row spikes).
// HERM writes U = Phi V (Sec. 6.1) as complex columns, row r at doubles 2r,
// 2r+1: u_r = zeta_r t_r / ||x|| with t_r = 1/((d_r - sigma) - mu), since
// Phi_r |zeta_r| = zeta_r.  NSYM writes the right vectors X = Psi V into V and
// the left ones Y = Psi^{-1} V into U: x_r = zc_r t_r / ||x||, y_r = zr_r t_r
// / ||x||, since Psi_r sqrt(zc_r zr_r) = zc_r; then y^T x = 1.
template <Kind K, class Team>
__device__ void vector_item(int n, int n1, const double *__restrict__ key,
                            const double *__restrict__ spk, const double *__restrict__ z,
                            const double *__restrict__ zrow, double alpha, double sgn,
                            const Scratch &S, const Outputs &out, int item, const Team &T,
                            double *stage = nullptr) {
    const int lane = T.rank;
    constexpr bool CPLX = K == KIND_HERM;
    constexpr bool TWO = K == KIND_NSYM;
    constexpr int RS = CPLX ? 2 : 1;           // doubles per row
    const int m = S.cnt[C_M];
    const int ncomp = m + 1;
    const bool last_row = K != KIND_DPR1;     // arrowhead rows have the x_n = -1 entry
    const int pos = out_pos<K>(S, n, sgn, item);
    double *col = out.V ? out.V + (size_t)pos * out.ldv : nullptr;
    double *ucol = ((K == KIND_TSVD || TWO) && out.U) ? out.U + (size_t)pos * out.ldu : nullptr;
    if (!col) return;
    if (item < ncomp) {
        const int k = item;
        const double sig = S.es_sigma[k], mu = S.es_mu[k];
        const int pi = S.es_pole[k];
        const double sv = K == KIND_TSVD ? sv_of(S, k) : 0.0;   // the singular value
        // 1/(shifted difference of row r - mu); 0 for a zero spike
        const double unit = unit_reg();
        auto recip = [&](int r) {
            if (spk[r] == 0.0) return 0.0;
            double del;
            if (K == KIND_TSVD) {
                const double dr = key[r];
                if (pi >= 0) {
                    const double di = S.pd[pi];
                    del = (dr - di) * (dr + di);
                } else {
                    del = fma(dr, dr, -sig);
                }
            } else {
                del = key[r] - sig;
            }
            return rcp_o(del - mu, unit);
        };
        // component of row r of x = [(D - lambda I)^{-1} spikes; -1]
        auto comp = [&](int r) { return spk[r] * recip(r); };
        // Pass 1 stores x (HERM, NSYM: the reciprocal t) and sums x^2 in sorted
        // order (so the norm does not depend on the order of the input rows);
        // pass 2 scales.
        double *keep = stage ? stage : col;      // pass-1 values, RS doubles a row
        // two rows a lane at a time, two independent sums (the same order for
        // every kind, so that real spikes give the real solver's bits)
        auto one = [&](int r, double &acc) {
            if (CPLX || TWO) {
                const double t = recip(r);
                keep[RS * r] = t;
                const double x = spk[r] * t;
                acc = fma(x, x, acc);
            } else {
                const double x = comp(r);
                keep[r] = x;
                acc = fma(x, x, acc);
            }
        };
        double s = 0.0, s1 = 0.0;
        int q0 = lane;
        for (; q0 + Team::size < n1; q0 += 2 * Team::size) {
            one(S.perm[q0], s);
            one(S.perm[q0 + Team::size], s1);
        }
        if (q0 < n1) one(S.perm[q0], s);
        s += s1;
        s = T.sum(s) + (last_row ? 1.0 : 0.0);
        double inv, scale = 1.0;
        bool stored = true;
        if (isfinite(s) && s > 0x1p-960) {
            inv = 1.0 / sqrt(s);
        } else {
            // rescale by the largest component to avoid overflow/underflow
            stored = false;
            double xm = last_row ? 1.0 : 0.0;
            for (int r = lane; r < n1; r += Team::size) xm = fmax(xm, fabs(comp(r)));
            xm = T.max(xm);
            scale = 1.0 / xm;
            double s2 = 0.0;
            for (int q = lane; q < n1; q += Team::size) {
                const double x = comp(S.perm[q]) * scale;
                s2 = fma(x, x, s2);
            }
            s2 = T.sum(s2) + (last_row ? scale * scale : 0.0);
            inv = 1.0 / sqrt(s2);
        }
        // DPR1 with rho < 0 solved -M: q ~ (D - lambda)^{-1} u needs a sign flip
        const double vs = (K == KIND_DPR1 && sgn < 0.0) ? -1.0 : 1.0;
        T.sync();
        int r0 = lane;
        if (stored && !CPLX && !TWO) {
            // the common case, four rows a lane at a time so that four loads of
            // the pass-1 values are in flight (vs = +-1, so x (vs inv) is
            // bitwise vs x inv)
            const double f = vs * inv;
            constexpr int ST = Team::size;
            for (; r0 + 3 * ST < n1; r0 += 4 * ST) {
                const double x0 = keep[r0], x1 = keep[r0 + ST], x2 = keep[r0 + 2 * ST],
                             x3 = keep[r0 + 3 * ST];
                const double v0 = x0 * f, v1 = x1 * f, v2 = x2 * f, v3 = x3 * f;
                col[r0] = v0;
                col[r0 + ST] = v1;
                col[r0 + 2 * ST] = v2;
                col[r0 + 3 * ST] = v3;
                if (ucol) {
                    ucol[r0] = sv * v0 / key[r0];
                    ucol[r0 + ST] = sv * v1 / key[r0 + ST];
                    ucol[r0 + 2 * ST] = sv * v2 / key[r0 + 2 * ST];
                    ucol[r0 + 3 * ST] = sv * v3 / key[r0 + 3 * ST];
                }
            }
        }
        for (int r = r0; r < n1; r += Team::size) {
            if (CPLX) {
                const double t = (stored ? keep[2 * r] : recip(r) * scale) * inv;
                col[2 * r] = z[2 * r] * t;
                col[2 * r + 1] = z[2 * r + 1] * t;
            } else if (TWO) {
                const double t = (stored ? keep[r] : recip(r) * scale) * inv;
                col[r] = z[r] * t;
                if (ucol) ucol[r] = zrow[r] * t;
            } else {
                const double x = stored ? keep[r] : comp(r) * scale;
                const double v = vs * x * inv;
                col[r] = v;
                if (ucol) ucol[r] = sv * v / key[r];      // u_j = s v_j / d_j
            }
        }
        if (last_row && lane == 0) {
            const double vn = -scale * inv;
            col[RS * n1] = vn;
            if (CPLX) col[RS * n1 + 1] = 0.0;
            if (ucol) ucol[n1] = K == KIND_TSVD ? alpha * vn / sv : vn;   // SVD: u_n = alpha v_n / s
        }
    } else {
        const int u = item - ncomp;
        const int row = S.drow[u];
        for (int r = lane; r < RS * n; r += Team::size) col[r] = 0.0;
        if (TWO && ucol)
            for (int r = lane; r < n; r += Team::size) ucol[r] = 0.0;
        T.sync();
        if (S.kind[row] == 1) {
            if (lane == 0) {
                col[RS * row] = 1.0;
                if (TWO && ucol) ucol[row] = 1.0;
            }
        } else if (CPLX || TWO) {
            // Phi (resp. Psi, Psi^{-1}) times the real Helmert-type vector of
            // the moduli: rows l before `row` in its run get -|zeta_q| s_l /
            // (R_{m-1} R_m), the row itself (s_q / |zeta_q|) R_{m-1} / R_m, with
            // s the caller's spike (zeta, zc or zr)
            const double Rm1 = S.run_R[2 * row], Rm = S.run_R[2 * row + 1];
            const double zq = spk[row];
            const double f = -zq / (Rm1 * Rm);
            const int s0 = S.run_s0[row], s1 = S.spos[row];
            for (int q = s0 + lane; q < s1; q += Team::size) {
                const int rq = S.perm[q];
                if (spk[rq] == 0.0) continue;
                if (CPLX) {
                    col[2 * rq] = f * z[2 * rq];
                    col[2 * rq + 1] = f * z[2 * rq + 1];
                } else {
                    col[rq] = f * z[rq];
                    if (ucol) ucol[rq] = f * zrow[rq];
                }
            }
            if (lane == 0) {
                const double g = Rm1 / (Rm * zq);
                if (CPLX) {
                    col[2 * row] = g * z[2 * row];
                    col[2 * row + 1] = g * z[2 * row + 1];
                } else {
                    col[row] = g * z[row];
                    if (ucol) ucol[row] = g * zrow[row];
                }
            }
        } else {
            run_column<Team::size>(S, spk, row, lane, col, 1.0);
        }
        if (K == KIND_TSVD && ucol) {
            // B v = d_r v for a deflated right vector (its last entry is 0)
            T.sync();
            for (int r = lane; r < n; r += Team::size) ucol[r] = col[r];
        }
    }
}

}  // namespace ae
