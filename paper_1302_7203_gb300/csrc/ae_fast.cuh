// ae_fast.cuh -- all eigenpairs of a reduced arrowhead by a few O(n) passes in
// fixed point (ae_fixed.cuh), one thread per eigenpair for everything scalar.
//
// The secular function f(lambda) = alpha - lambda - sum_j zeta_j^2 / (p_j - lambda)
// (the shifted inverse's Pick function F of Algorithm 3 is f divided by
// zeta_i^2 / mu^2 up to sign) is evaluated at lambda = p_i + mu with every
// difference exact and every term good to ~2^-59, against 2^-53 a rounding in
// FP64: that covers what the paper's doubled-precision b buys wherever the
// terms' cancellation against the pole's own term stays below 2^7 (kErrTerm).
// Beyond it f is summed in 128 bits (~2^-80), and wherever a range test fails
// the eigenpair takes the FP64 / double-double solver (k_fold, ae_solver.cuh).
//
//   k_fprep   poles, spikes and rows in scaled and fixed-point form
//   k_fgroup  the poles far from 32 consecutive eigenvalues as 20 moments about
//             their middle, in fixed point: O(n) work a group instead of an
//             eigenpair
//   k_fopen   FP32: midpoint test (Algorithm 1), K_b (Algorithm 5's gate
//             counters), model steps to |error| < 2^-16 of the distance to the
//             nearest pole; a warp holds 4 eigenpairs, so that a pole read
//             from L1/L2 serves 4
//   k_feval   fixed point: f and its next four derivatives' sums over the near
//             poles in one pass
//   k_fstep   one thread per eigenpair: the zero from the quartic expansion
//             (relative error eps^4 at a step eps of the pole distance), the
//             vector's norm from the same sums, else a model step
//   k_fmore   the few (1-4 %) whose opening was too far off or whose terms
//             cancel too much, and the outermost two: further evaluations, a
//             CTA each, with f summed in 128 bits
//   k_fold    the FP64 solver for what is left, a warp or a CTA per eigenpair
//   k_ffix    remedies (Remarks 1, 2): the zero is already known beyond double
//             precision, so moving it to the remedy's shift is a subtraction;
//             checked, else k_fmore evaluates f at the zero in 128 bits first,
//             and what that does not settle is left to k_fix_solve
//   k_fcols   columns: one difference (for rows far from a group without FP64),
//             one reciprocal and two products a component, normalised in the
//             same step and written once
#pragma once
#include <type_traits>

#include "ae_fixed.cuh"
#include "ae_pipeline.cuh"

namespace ae {

// states of a computed eigenpair in the fast path
enum { FST_EVAL = 0, FST_DONE = 1, FST_OLD = 2, FST_MORE = 3 };

// A zero's offset mu is taken from an evaluation whose error is below 2^-52 of
// it (2^-54 as a rule: the bounds below are worst cases).  Two errors count, both over f' |mu|: the terms' and sums', 2^-59 (in
// 128 bits 2^-80) of sum |zeta^2/(p - lambda)|, and that of the differences'
// unit, 2^-105 of sum zeta^2/(p - lambda)^2 (the differences formed in
// double-double left out).  Hence the weights of the two sums against f' |mu|:
constexpr double kErrTerm = 0x1p-7, kErrTermWide = 0x1p-25, kErrUnit = 0x1p-50;
// largest step, relative to the distance to the nearest pole, that the quartic
// expansion closes: (2^-14)^4 = 2^-56
constexpr double kStepMax = 0x1p-14;
constexpr int kMoreRounds = 4;
// iteration caps below this are meant to stop a solve: the FP64 solver takes them
constexpr int kMinIterCap = 100;

__device__ __forceinline__ unsigned long long shr64(unsigned long long v, unsigned s) {
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));   // 0 from 64 on
    return r;
}
// the 32 bits below the last place of v >> s (s up to 95)
__device__ __forceinline__ unsigned low32(unsigned long long v, unsigned s) {
    unsigned long long r;
    unsigned q;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(64u - s));          // 0 from s = 65 on
    asm("shr.u32 %0, %1, %2;" : "=r"(q) : "r"((unsigned)(v >> 32)), "r"(s - 64u));   // up to 63
    return (unsigned)(r >> 32) | q;
}
__device__ __forceinline__ int sar32(int v, unsigned s) {
    int r;
    asm("shr.s32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));   // the sign from 32 on
    return r;
}
__device__ __forceinline__ unsigned hi32(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ unsigned bexp(double x) { return (hi32(x) << 1) >> 21; }

// ---------------------------------------------------------------------------
// where the kernels find their instances
// ---------------------------------------------------------------------------
struct SrcOne {          // one instance, by value
    Scratch S;
    VecArgs va;
    __device__ bool unit(long long u, int per, int &i, int &first) const {
        i = 0;
        first = (int)u * per;
        return true;
    }
    __device__ bool item(long long t, int &i, int &idx) const {
        i = 0;
        idx = (int)t;
        return t < va.n;
    }
    __device__ const Scratch &scr(int) const { return S; }
    __device__ const VecArgs &vec(int) const { return va; }
    __device__ void push_old(int, int k) const { S.f.old[atomicAdd(S.cnt + C_NOLD, 1)] = k; }
    __device__ int old_count() const { return S.cnt[C_NOLD]; }
    __device__ int2 old_at(int w) const { return make_int2(0, S.f.old[w]); }
    __device__ int *old_ticket(int ph) const { return S.cnt + (ph ? C_OLDTK2 : C_OLDTK); }
    // eigenpairs for k_fmore: phase 0 after k_fstep, phase 1 after k_ffix (the
    // list of phase 0 is done with by then)
    __device__ void push_more(int ph, int, int k) const {
        S.f.more[atomicAdd(S.cnt + C_NMORE + ph, 1)] = k;
    }
    __device__ int more_count(int ph) const { return S.cnt[C_NMORE + ph]; }
    __device__ int2 more_at(int w) const { return make_int2(0, S.f.more[w]); }
    // columns for k_vectors
    __device__ void push_col(int, int item) const {
        S.cols[atomicAdd(S.cnt + C_NCOL, 1)] = item;
    }
    __device__ int col_count() const { return S.cnt[C_NCOL]; }
    __device__ int2 col_at(int w) const { return make_int2(0, S.cols[w]); }
    __device__ void push_fix(int, int k, bool front, int n) const {
        if (front) S.fixlist[atomicAdd(S.cnt + C_NFIX, 1)] = k;
        else S.fixlist[n - 1 - atomicAdd(S.cnt + C_NFIX2, 1)] = k;
    }
    __device__ double2 *slice(long long w) const {
        return S.wbuf ? S.wbuf + w * S.wstride : nullptr;
    }
};

// eigenpairs [lo, hi) of the reduced arrowhead that this solve computes (a
// part also solves the eigenpair on each side of its range)
__device__ __forceinline__ void fast_range(const Scratch &S, int &lo, int &hi) {
    lo = 0;
    hi = S.cnt[C_M] + 1;
    if (S.cnt[C_PART]) {
        lo = S.cnt[C_K0] > 0 ? S.cnt[C_K0] - 1 : 0;
        hi = S.cnt[C_KHI];
    }
}

// Groups of 32 eigenpairs start at multiples of 32 whatever a part's range, so
// that a part forms the sums the whole solve forms.
constexpr int kGroup = 32;

// power of two that scales the poles below 1/2 (see k_fprep)
template <Kind K>
__device__ __forceinline__ int fast_scale(const Scratch &S) {
    const int e = ilogb(S.prm[P_DS]);
    return K == KIND_TSVD ? 2 * e - 3 : e - 2;
}

__device__ __forceinline__ double pow2(int e) {          // 2^e, -1022 <= e <= 1023
    return __longlong_as_double((long long)(1023 + e) << 52);
}
__device__ __forceinline__ double pow2_or(int e) {       // any e
    return e >= -1022 && e <= 1023 ? pow2(e) : ldexp(1.0, e);
}
// x 2^e for |e| <= 2000 (two products, where ldexp takes some twenty operations)
__device__ __forceinline__ double scalb2(double x, int e) {
    const int h = e >> 1;
    return x * pow2(h) * pow2(e - h);
}

// ---------------------------------------------------------------------------
// k_fprep
// ---------------------------------------------------------------------------
// pole (or row) value in scaled double-double: d, or d^2 for the SVD
template <Kind K>
__device__ __forceinline__ dd fast_pole(double d, int es) {
    if (K == KIND_TSVD) {
        const double s = d * pow2((es + 3) / 2);
        const dd q = two_prod(s, s);
        return dd{q.hi * 0.125, q.lo * 0.125};
    }
    return dd{d * pow2(es), 0.0};
}

// One thread per pole and row.  Whatever falls outside the ranges the fixed-
// point passes are made for sets CF_NOFAST, and the whole instance is solved
// by the FP64 solver.
template <Kind K>
__device__ __forceinline__ void fprep_item(const Scratch &S, const VecArgs &va, int t) {
    const int m = S.cnt[C_M];
    bool bad = false;
    const int es = fast_scale<K>(S);
    const int e0 = K == KIND_TSVD ? (es + 3) / 2 : es;
    if (m < 2 || es < -480 || es > 480 || e0 < -480 || e0 > 480) {
        if (t == 0) atomicOr(S.cnt + C_FLAGS, CF_NOFAST);
        return;
    }
    if (t < m) {
        const dd p = fast_pole<K>(S.pd[t], es);
        S.f.p[t] = p.hi;
        S.f.plo[t] = p.lo;
        S.f.P[t] = fix_mod(p.hi) + fix_mod(p.lo);
        S.f.P2[t] = fix_mod<kFixFrac2>(p.hi) + fix_mod<kFixFrac2>(p.lo);
        bad |= !(fabs(p.hi) < 0.5) || (p.hi != 0.0 && fabs(p.hi) < 0x1p-900);
        // zeta^2 as a 64-bit significand and z2's exponent (scaled by 4^es)
        const double z2 = S.pz2[t], zl = S.pz2lo[t];
        const int e = (int)bexp(z2) - 1023;
        bad |= !(e > -900 && e < 900);
        if (!bad) {
            const unsigned long long b = (unsigned long long)__double_as_longlong(z2);
            S.f.z[t] = fix_mant(z2, __double2ll_rn(zl * pow2(63 - e)));
            // and in 128 bits
            const unsigned __int128 W =
                ((unsigned __int128)((b & 0xfffffffffffffull) | 0x10000000000000ull) << 75) +
                (unsigned __int128)((__int128)(long long)(zl * pow2(115 - e)) << 12);
            S.f.zh[t] = (unsigned long long)(W >> 64);
            S.f.zl[t] = (unsigned long long)W;
            S.f.ez[t] = e + 2 * es;
        }
    }
    if (t < va.n1) {
        const dd p = fast_pole<K>(va.key[t], es);
        S.f.rp[t] = p.hi;
        if (K == KIND_TSVD) S.f.rP[t] = fix_mod(p.hi) + fix_mod(p.lo);
    }
    if (t == 0) bad |= !(fabs(S.prm[P_ALPHA_HI] * pow2(es)) < 0x1p300);
    if (bad) atomicOr(S.cnt + C_FLAGS, CF_NOFAST);
}

// ---------------------------------------------------------------------------
// the evaluation point of an eigenpair
// ---------------------------------------------------------------------------
// lambda = sigma + mu as its rounded value and its fixed-point form.  Beyond
// |lambda| = 5/2 (an outermost eigenvalue far from all poles) the rounded
// value IS the point, mu absorbs the difference, and no tails are taken.
__device__ __forceinline__ bool set_point(const Scratch &S, int k, dd sg, dd mu) {
    dd l = two_sum(sg.hi, mu.hi);
    l.lo += sg.lo + mu.lo;
    l = fast_two_sum(l.hi, l.lo);
    const bool notail = !(fabs(l.hi) < 2.5);
    if (notail) {
        mu = dd_add(dd{l.hi, 0.0}, dd_neg(sg));
        l.lo = 0.0;
    }
    S.f.mu[k] = mu.hi;
    S.f.mulo[k] = mu.lo;
    S.f.lhi[k] = l.hi;
    S.f.llo[k] = l.lo;
    S.f.lmod[k] = fix_mod(l.hi) + fix_mod(l.lo);
    S.f.lmod2[k] = fix_mod<kFixFrac2>(l.hi) + fix_mod<kFixFrac2>(l.lo);
    return isfinite(l.hi);
}

// Differences whose biased exponent lies in [lo, lo + span) are formed as
// fl(p - lambda) with the modular tail (tails != 0) or without one (a point
// beyond 5/2); the others as (p - sigma) - mu in double-double: those small
// against lambda or the unit, and a DPR1's last pole, which is no pole of the
// arrowhead and may lie far outside the others or next to such a point.
struct DiffRange {
    unsigned lo, span;
    unsigned lo0;         // lo without the unit's limit
    int tails;            // mask of the tail
};
__device__ __forceinline__ DiffRange diff_range(double lhi) {
    const unsigned e = bexp(lhi);
    const unsigned a = e > kTailSpan ? e - kTailSpan : 0u;
    if (!(fabs(lhi) < 2.5)) return {a, 4096u, a, 0};
    const unsigned lo = a > kFixMinExp2 ? a : kFixMinExp2;
    return {lo, 1025u - lo, a, -1};
}

// (p - sigma) - mu in double-double: exact but for roundings of the low parts
// (the differences do not cancel: |p - lambda| is at least half of |p - sigma|
// or of |mu|)
__device__ __forceinline__ dd near_diff(dd p, dd sg, dd mu) {
    const dd d = two_sum(p.hi, -sg.hi);
    const dd D = two_sum(d.hi, -mu.hi);
    return fast_two_sum(D.hi, D.lo + (d.lo + ((p.lo - sg.lo) - mu.lo)));
}
// its tail along |D.hi|, in 2^-7 of D's last place
__device__ __forceinline__ int near_tail(dd D) {
    const double t = (D.hi < 0.0 ? -D.lo : D.lo) * pow2(7 + 1075 - (int)bexp(D.hi));
    return __double2int_rd(t);
}

// sigma (the shift pole, or another shift) in scaled double-double
template <Kind K>
__device__ __forceinline__ dd fast_sigma(const Scratch &S, int k, int es) {
    const int i = S.es_pole[k];
    if (i >= 0) return dd{S.f.p[i], S.f.plo[i]};
    return dd{S.es_sigma[k] * pow2(es), 0.0};
}

__device__ __forceinline__ float sqrt_f32(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ dd dd_of_ll(long long v) {
    const double h = (double)v;
    return fast_two_sum(h, (double)(v - (long long)h));
}

// ---------------------------------------------------------------------------
// k_fgroup: far poles as moments
// ---------------------------------------------------------------------------
// For the eigenvalues of a group, all inside an interval with middle c and half
// length r, a pole with |p - c| >= 8 r contributes
//     zeta^2 / (p - lambda) = sum_q t^q zeta^2 / (p - c)^(q+1),   t = lambda - c,
// with |t / (p - c)| <= 1/8: 20 terms leave 8^-20 = 2^-60 of it.  The moments
// A_q = sum zeta^2 / (p - c)^(q+1) are summed in fixed point as k_feval's sums
// are (order q needs 60 - 3 q bits: 62-bit products up to q = 9, 32-bit ones
// beyond; the bits below the last place, whose loss is a bias of n / 2 last
// places, up to q = 4), ~250 instructions a pole for 32 eigenpairs, where opening and
// evaluating at each pole takes 32 x 250.  8 balances the two parts: the near
// poles (~ 8 groups' worth, 256) and the moments (n / 32 a pair).
// Stored per group: A_q 2^(q e) with 2^e <= 8 r, the first three as
// double-doubles; the opening's FP32 copies; the indices [jlo, jhi) of the
// poles left to the passes (all of them where fewer than kMinFar would go).
// Bound by issue slots.  Graded n = 16384: 0.17 ms here; opening 0.72 -> 0.07,
// k_feval 1.81 -> 0.08 ms.  DPR1 n = 8192: 0.05 here; 0.27 -> 0.04, 0.47 -> 0.03.
// Fewer than kFarFrom poles form no groups, and their outermost eigenpairs are
// opened by a warp like the others: one solve (kernels launched plainly) at n = 64
// / 256 / 1000 takes 97 / 109 / 179 us so, and 116 / 126 / 184 us with groups and an opening by CTA
// (two latencies more); at 1500 it is 225 against 219, and a batch, bound by
// issue slots, gains from about 700 on.
constexpr int kMoments = 20, kMomWide = 10, kMom32 = 10, kMomLow = 5;
constexpr int kMinFar = 256, kFarFrom = 768;

struct GroupData {
    double A[kMoments], Al[3];
    double c, r8;           // the middle, and 8 r (infinite: no interval)
    float fa[kMom32];       // A_q 2^(q e) in the opening's units
    float T, W;             // sum |zeta^2/(p-c)|, sum |zeta/(p-c)| in those units
    float ku;               // t 2^-e = tau0 + u ku for an offset u in those units
    int e, jlo, jhi;
};

// sum A_q tau^q and its derivative by u, in the opening's units
__device__ __forceinline__ float far32(const GroupData &G, float tau, float &d) {
    float v = 0.f, w = 0.f;
#pragma unroll
    for (int q = kMom32 - 1; q >= 0; --q) {
        w = fmaf(w, tau, v);
        v = fmaf(v, tau, G.fa[q]);
    }
    d = w * G.ku;
    return v;
}

// |x| as a float from the high word of a double x with 2^-120 < |x| < 2
__device__ __forceinline__ float f32_of_bits(unsigned h) {
    return __uint_as_float(((h & 0x7fffffffu) - (896u << 20)) << 3);
}

template <Kind K, class Src>
__global__ void __launch_bounds__(256, 2) k_fgroup(const __grid_constant__ Src src) {
    after_previous();
    __shared__ float rt[8], rw[8];
    __shared__ int jb[2];
    __shared__ unsigned long long acc[8][kMoments + kMomLow];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inst, first;
    if (!src.unit(blockIdx.x, kGroup, inst, first) || first == 0) return;
    const Scratch &S = src.scr(inst);
    const int m = S.cnt[C_M];
    int klo, khi;
    fast_range(S, klo, khi);
    const int k0 = (klo & ~(kGroup - 1)) + first - kGroup;
    if (k0 >= khi || (S.cnt[C_FLAGS] & CF_NOFAST) || m < kFarFrom) return;
    GroupData &G = S.f.grp[k0 / kGroup];
    // the group's interior eigenvalues lie between these poles (k0 = m: none)
    const int ka = k0 > 1 ? k0 : 1, kb = min(k0 + kGroup - 1, m - 1);
    const double top = S.f.p[min(ka - 1, m - 1)], bot = S.f.p[max(kb, 0)];
    const double c = 0.5 * (top + bot), r = fmax(top - c, c - bot);
    const int e = (int)bexp(8.0 * r) - 1023;
    if (threadIdx.x < 2) {
        // poles >= c + 8 r, poles > c - 8 r
        const double x = threadIdx.x ? c - 8.0 * r : c + 8.0 * r;
        int lo = 0, hi = m;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            const double p = S.f.p[mid];
            if (threadIdx.x ? p > x : p >= x) lo = mid + 1;
            else hi = mid;
        }
        jb[threadIdx.x] = lo;
    }
    __syncthreads();
    const int jlo = jb[0] & ~31, jhi = min((jb[1] + 31) & ~31, m);
    const bool none = kb < ka || !(r > 0.0) || e < -100;
    if (threadIdx.x == 0) {
        G.c = c;
        G.e = e;
        G.r8 = none ? INFINITY : 8.0 * r;
    }
    if (none || m - (jhi - jlo) < kMinFar) {
        if (threadIdx.x == 0) {
            G.jlo = 0;
            G.jhi = m;
        }
        return;
    }
    const double one = unit_reg();
    // bound of the sums, and the Gershgorin share, in FP32
    float T = 0.f, Wf = 0.f;
    for (int j = threadIdx.x; j < m; j += 256) {
        if (j >= jlo && j < jhi) continue;
        const float q = rcp_f32(f32_of_bits(hi32(fma(S.f.p[j], one, -c))));
        const float z = S.pz2f[j];
        T = fmaf(z, q, T);
        Wf = fmaf(sqrt_f32(z), q, Wf);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        T += __shfl_xor_sync(FULL, T, o);
        Wf += __shfl_xor_sync(FULL, Wf, o);
    }
    if (lane == 0) {
        rt[wid] = T;
        rw[wid] = Wf;
    }
    __syncthreads();
    T = rt[0];
    Wf = rw[0];
    for (int w = 1; w < 8; ++w) {
        T += rt[w];
        Wf += rw[w];
    }
    const int es = fast_scale<K>(S), ezs = ilogb(S.prm[P_ZS]);
    const int eL = K == KIND_TSVD ? 2 * ilogb(S.prm[P_DS]) : ilogb(S.prm[P_DS]);
    const int K0 = T > 0.f ? ilogbf(T * 1.02f) + 1 + 2 * es - ezs : 0;
    const DiffRange dr = diff_range(c);
    const unsigned long long L = fix_mod(c), L2 = fix_mod<kFixFrac2>(c);
    const int c1 = K0 + 1 - 1023, cs = 1 - e - 1023;
    unsigned long long a[kMoments], l[kMomLow];
#pragma unroll
    for (int q = 0; q < kMoments; ++q) a[q] = 0;
#pragma unroll
    for (int q = 0; q < kMomLow; ++q) l[q] = 0;
    auto add = [&](int j) {
        const double p = S.f.p[j];
        double D = fma(p, one, -c);
        int tl;
        unsigned dh = hi32(D), dl = (unsigned)__double2loint(D);
        unsigned eb = (dh << 1) >> 21;
        if (eb - dr.lo >= dr.span) {
            const dd Dd = near_diff(dd{p, S.f.plo[j]}, dd{c, 0.0}, dd{0.0, 0.0});
            D = Dd.hi;
            tl = near_tail(Dd);
            dh = hi32(D);
            dl = (unsigned)__double2loint(D);
            eb = (dh << 1) >> 21;
        } else if (eb < kFixMinExp && dr.tails) {
            tl = tail_of<kFixFrac2>(S.f.P2[j] - L2, dh, dl, eb);
        } else {
            tl = tail_of(S.f.P[j] - L, dh, dl, eb) & dr.tails;
        }
        const unsigned seed = hi32(rcp_seed(__hiloint2double(
            (int)((dh & 0xfffffu) | 0x3ff00000u), 0)));
        // (2^64 / m, so that a product keeps its place: 2^63 of the term)
        unsigned long long R = recip63<true>(dh, dl, tl, seed);
        R = R >> 63 ? ~0ull : R + R;
        unsigned long long q = mul_hi3(S.f.z[j], R);
        unsigned s = (unsigned)(c1 + (int)eb - S.f.ez[j]);
        a[0] += shr64(q, s);
        l[0] += low32(q, s);
#pragma unroll
        for (int i = 1; i < kMoments; ++i) {
            q = i < kMomWide ? mul_hi3(q, R)
                             : (unsigned long long)(unsigned)(q >> 32) * (unsigned)(R >> 32);
            s += eb + cs;
            a[i] += shr64(q, s);
            if (i < kMomLow) l[i] += low32(q, s);
        }
    };
    for (int j = threadIdx.x; j < jlo; j += 256) add(j);
    // (odd powers change sign below c)
#pragma unroll
    for (int q = 0; q < kMoments; q += 2) a[q] = 0ull - a[q];
#pragma unroll
    for (int q = 0; q < kMomLow; q += 2) l[q] = 0ull - l[q];
    for (int j = jhi + threadIdx.x; j < m; j += 256) add(j);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int q = 0; q < kMoments; ++q) a[q] += __shfl_xor_sync(FULL, a[q], o);
#pragma unroll
        for (int q = 0; q < kMomLow; ++q) l[q] += __shfl_xor_sync(FULL, l[q], o);
    }
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < kMoments; ++q) acc[wid][q] = a[q];
#pragma unroll
        for (int q = 0; q < kMomLow; ++q) acc[wid][kMoments + q] = l[q];
    }
    __syncthreads();
    if (threadIdx.x < kMoments) {
        const int q = threadIdx.x;
        unsigned long long v = 0, y = 0;
        for (int w = 0; w < 8; ++w) {
            v += acc[w][q];
            if (q < kMomLow) y += acc[w][kMoments + q];
        }
        // A_q 2^(q e): the unit of order q is 2^(K0 - q e - (62 - q))
        dd x = dd_of_ll((long long)v);
        if (q < kMomLow) x = dd_add(x, dd{(double)(long long)y * 0x1p-32, 0.0});
        const double u = scalb2(q & 1 ? 1.0 : -1.0, K0 - 62 + q);
        G.A[q] = x.hi * u;
        if (q < 3) G.Al[q] = x.lo * u;
        if (q < kMom32) G.fa[q] = (float)scalb2(x.hi * u, ezs - eL - es);
    }
    if (threadIdx.x == 0) {
        const float f = (float)pow2(es - eL) * (8.f / 7.f);
        G.T = T * f;
        G.W = Wf * f;
        G.ku = (float)pow2(es - eL - e);
        G.jlo = jlo;
        G.jhi = jhi;
    }
}

// ---------------------------------------------------------------------------
// k_fopen
// ---------------------------------------------------------------------------
// Sums over the warp of four values, one per eigenpair: lane group g = lane/8
// ends with the sum of v[g] (6 shuffles instead of 20).
__device__ __forceinline__ float reduce4(const float (&v)[4], int lane) {
    const bool h = lane & 16, q = lane & 8;
    float a = h ? v[2] : v[0], b = h ? v[3] : v[1];
    const float sa = h ? v[0] : v[2], sb = h ? v[1] : v[3];
    a += __shfl_xor_sync(FULL, sa, 16);
    b += __shfl_xor_sync(FULL, sb, 16);
    float k = q ? b : a;
    const float s = q ? a : b;
    k += __shfl_xor_sync(FULL, s, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(FULL, k, o);
    return k;
}
__device__ __forceinline__ float reduce4max(const float (&v)[4], int lane) {
    const bool h = lane & 16, q = lane & 8;
    float a = h ? v[2] : v[0], b = h ? v[3] : v[1];
    const float sa = h ? v[0] : v[2], sb = h ? v[1] : v[3];
    a = fmaxf(a, __shfl_xor_sync(FULL, sa, 16));
    b = fmaxf(b, __shfl_xor_sync(FULL, sb, 16));
    float k = q ? b : a;
    const float s = q ? a : b;
    k = fmaxf(k, __shfl_xor_sync(FULL, s, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) k = fmaxf(k, __shfl_xor_sync(FULL, k, o));
    return k;
}

// Zero of the model Phi(mu) ~ A + B / (dn - mu) = w / mu fitted to (Phi, Phi')
// at u, as |mu|: with e = |dn| the distance to the interval's other pole (0:
// none, then Phi is linear), s the side, everything scaled by a power of two
// so that squares stay in range.  (The one-pole model of the Newton finish,
// written in mu = 1/x.)
__device__ __forceinline__ float model_root(float s, float Phi, float dPhi, float u, float e,
                                            float w) {
    const float mu = fabsf(u);
    if (e > 0.f) {
        const float g = e - mu;
        float B = dPhi * g * g;
        float A = s * Phi - dPhi * g;
        float X = fmaf(A, e, B);
        const float big = fmaxf(fmaxf(fabsf(X), B), w);
        const float c = __uint_as_float((254u << 23) - (__float_as_uint(big) & 0x7f800000u));
        X *= c; B *= c; A *= c; w *= c;
        const float b = X + w;
        const float h = X - w;
        const float rt = sqrt_f32(fmaf(4.f * w, B, h * h));
        return b >= 0.f ? __fdividef(2.f * w * e, b + rt) : __fdividef(b - rt, 2.f * A);
    }
    const float A = s * Phi - dPhi * mu;             // A + B m = w / m
    const float B = dPhi;
    const float rt = sqrt_f32(fmaf(4.f * B, w, A * A));
    return A >= 0.f ? __fdividef(2.f * w, A + rt) : __fdividef(rt - A, 2.f * B);
}

// An outermost eigenvalue beyond its pole, |mu| = x: s Phi = -s Af + gam x - R
// with the other poles' R (dR its slope) at offset x.  Own pole plus R's tangent,
// and one pole c / (x + dl) fitted to the whole sum, both lie below the sum, so
// that the larger zero is the better one; far from the pole the tangent alone
// creeps (of 336 such eigenvalues, n = 5 to 3000, 2 to 32 steps; both: at most 7).
__device__ __forceinline__ float model_root_outer(float A, float gam, float R, float dR, float x,
                                                  float w) {
    const float lin = model_root(1.f, A + gam * x - R, gam + dR, x, 0.f, w);
    const float q = __fdividef(w, x), S = q + R, dS = __fdividef(q, x) + dR;
    const float h = __fdividef(S, dS), dl = h - x, c = S * h;
    const float b = fmaf(gam, dl, A), a = fmaf(-gam, dl, A);
    const float rt = sqrt_f32(fmaf(4.f * gam, c, a * a));
    const float m = b < 0.f ? __fdividef(rt - b, 2.f * gam)
                            : __fdividef(2.f * (c - A * dl), b + rt);
    return dS < 1e36f && m > lin && m < 1e36f ? m : lin;
}

// NW warps share 4 eigenpairs (kc: eigenpair of this lane group, or some valid
// one where have is false), each over its share of the poles [jlo, jhi); G: the
// far poles' moments, or null.  red: 4 NW floats.
template <Kind K, int NW, class Src>
__device__ __forceinline__ void open_items(const Src &src, int inst, const Scratch &S,
                                           const SolveOpts &o, int kc, bool have, int jlo,
                                           int jhi, const GroupData *G, float *red) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int m = S.cnt[C_M], k = kc;
    const int js = jlo + lane + (NW > 1 ? 32 * wid : 0);
    constexpr int JS = 32 * NW;
    // a lane group's sum (maximum) over the team, from its warp's
    auto team = [&](float v, bool mx) {
        if (NW == 1) return v;
        __syncthreads();
        if ((lane & 7) == 0) red[wid * 4 + (lane >> 3)] = v;
        __syncthreads();
        float r = red[lane >> 3];
        for (int w = 1; w < NW; ++w) {
            const float x = red[w * 4 + (lane >> 3)];
            r = mx ? fmaxf(r, x) : r + x;
        }
        return r;
    };
    const int es = fast_scale<K>(S);
    const auto R = PolesOf<K>::make(S, m);
    const bool lowx = kc == 0, upx = kc == m;         // outermost eigenvalues
    const double Ld = R.f32_scale();
    const double g1 = R.zs / Ld;                      // scales f to the FP32 sums
    const float gam = (float)(g1 / Ld);
    float sh, sl, mf, tf[4], af[4], bf[4], df[4];
    // ---- the sign of f at the midpoint of the eigenvalue's interval ----
    int i = lowx ? 0 : upx ? m - 1 : kc, side = lowx ? +1 : -1;
    const double sk = R.pole(i);
    const double middle = (lowx || upx) ? 0.0 : 0.5 * R.shifted(kc - 1, sk, kc);
    R.f32_shift(sk, i, sh, sl);
    mf = (float)(middle * Ld);
    float tm, am, bm, dm;
    {
        float she[4], sle[4], mfe[4];
        bool bad[4] = {false, false, false, false};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            she[e] = __shfl_sync(FULL, sh, 8 * e);
            sle[e] = __shfl_sync(FULL, sl, 8 * e);
            mfe[e] = __shfl_sync(FULL, mf, 8 * e);
            tf[e] = af[e] = bf[e] = df[e] = 0.f;
        }
        for (int j = js; j < jhi; j += JS) {
            const float z = R.z2f(j);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float gg;
                const float D = R.shifted_f32_mag(j, she[e], sle[e], gg) - mfe[e];
                bad[e] |= !(fabsf(D) >= fmaf(gg, 0x1p-20f, 0x1p-100f));
                const float r = rcp_f32(D);
                const float t = z * r;
                tf[e] += t;
                af[e] += fabsf(t);
                bf[e] += fabsf(r);
                df[e] = fmaf(t, r, df[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (bad[e]) bf[e] = INFINITY;
        tm = team(reduce4(tf, lane), false);
        am = team(reduce4(af, lane), false);
        bm = team(reduce4(bf, lane), false);
        dm = team(reduce4(df, lane), false);
    }
    // far poles: their sum at this lane group's pole + u
    float tau0 = 0.f;
    auto far = [&](float u, float &d) { return far32(*G, fmaf(u, G->ku, tau0), d); };
    auto set_tau = [&](int i) { tau0 = (float)((S.f.p[i] - G->c) * pow2(-G->e)); };
    if (G) {
        set_tau(i);
        float d;
        tm += far(mf, d);
        dm += d;
        am += G->T;
    }
    bool ok = true, mid64 = false;
    int passes = 0;
    if (!lowx && !upx) {
        // (the bound is select_shift's)
        const double a = R.a_dd(sk, i).hi - middle;
        const double f = Ld / R.zs;
        const double L = (double)((m + 31) / 32);
        const double F32 = a - f * (double)tm;
        const double ET = 2.0 * (L + 24.0) * 0x1p-24 * (2.0 * (double)am) +
                          0x1p-148 * ((double)bm + (double)m);
        const double M = f * ET * (1.0 + 0x1p-20) + (L + 16.0) * 0x1p-52 * fabs(a);
        mid64 = !(isfinite(F32) && fabs(F32) > M * (1.0 + 0x1p-40));
        // (left open: either side serves -- the zero is moved to the nearer
        // pole once it is known, k_fstep)
        if (F32 < 0.0) side = +1;
        else { i = kc - 1; side = -1; }
        ++passes;
        // poles that FP32 pairs cannot tell apart here
        ok &= middle > 0x1p-32 * fabs(sk);
    }
    // ---- the chosen pole: model steps ----
    const double sig = R.pole(i);
    R.f32_shift(sig, i, sh, sl);
    if (G) set_tau(i);
    const int jn = side > 0 ? i - 1 : i + 1;          // the interval's other pole
    const float en = (jn >= 0 && jn < m) ? (float)(fabs(R.shifted(jn, sig, i)) * Ld) : 0.f;
    const double a64 = R.a_dd(sig, i).hi;
    const float Af = (float)(a64 * g1);
    const float w = R.z2f(i);
    const float s = (float)side;
    const int jb = side > 0 ? i + 1 : i - 1;          // the pole behind it
    bool close = en < 0x1p-100f && jn >= 0 && jn < m;   // poles closer than FP32's range?
    if (jb >= 0 && jb < m) {
        const double gap = fabs(R.shifted(jb, sig, i));
        ok &= gap > 0x1p-32 * fabs(sig);
        close |= gap * Ld < 0x1p-100;
    }
    close = __any_sync(FULL, close);
    ok &= lowx || upx || en > 0x1p-100f;              // (0: below FP32's range)
    ok &= w > 0x1p-100f && fabsf(Af) < 0x1p100f && gam < 0x1p60f;
    float rm = 0.f;
    if (!lowx && !upx) {
        // from the midpoint: own term taken out (|mf| from either pole)
        const float um = s * mf;
        const float to = -w / um;                     // w / (0 - um)
        const float Phi = -Af + gam * um + (tm - to);
        const float dPhi = gam + fmaxf(dm - w / (mf * mf), 0.f);
        rm = model_root(s, Phi, dPhi, um, en, w);
    }
    float u = 0.f, ul = 0.f, wsum = 0.f, wmax = 0.f, num = 0.f, Tabs = 0.f, dsum = 0.f;
    bool done = false;
    const bool gersh = o.finish == 0;
    // At the pole itself closer terms are left out: their squares overflow.  Beyond
    // the outermost pole, crowded ones nearby would start the steps where the models
    // drown in rounding.
    const float cut = lowx || upx ? 0x1p-30f : 0x1p-60f;
    // (3 to 5 passes nearly always; one eigenpair in some thousands takes over 9,
    // and one that ran out of passes costs the FP64 solver's 220 us)
    for (int it = 0; it < 24; ++it) {
        float she[4], sle[4], ue[4], wi[4], sd[4], ws[4], wx[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            she[e] = __shfl_sync(FULL, sh, 8 * e);
            sle[e] = __shfl_sync(FULL, sl, 8 * e);
            ue[e] = __shfl_sync(FULL, u, 8 * e);
            tf[e] = af[e] = df[e] = 0.f;
        }
        // tf, af, df over the poles j for which skip(j, e, D) is false
        auto sums = [&](auto skip) {
            for (int j = js; j < jhi; j += JS) {
                const float z = R.z2f(j);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float D = R.shifted_f32(j, she[e], sle[e]);
                    const float rr = rcp_f32(D - ue[e]);
                    const float r = skip(j, e, D) ? 0.f : rr;
                    const float t = z * r;
                    tf[e] += t;
                    af[e] += fabsf(t);
                    df[e] = fmaf(t, r, df[e]);
                }
            }
        };
        float ce[4];
        if (it == 0) {
#pragma unroll
            for (int e = 0; e < 4; ++e) ce[e] = __shfl_sync(FULL, cut, 8 * e);
        }
        if (it == 0 && gersh) {
            // with Algorithm 3's bracket: sum and extreme of the Gershgorin
            // quantities |w_j| = zeta_j / (|delta_j| zeta_i)
            const float iw = rcp_f32(sqrt_f32(w));
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                wi[e] = __shfl_sync(FULL, iw, 8 * e);
                sd[e] = __shfl_sync(FULL, s, 8 * e);
                ws[e] = wx[e] = 0.f;
            }
            for (int j = js; j < jhi; j += JS) {
                const float z = R.z2f(j), q = sqrt_f32(z);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float D = R.shifted_f32(j, she[e], sle[e]);
                    const float r = fabsf(D) < ce[e] ? 0.f : rcp_f32(D);
                    const float t = z * r;
                    tf[e] += t;
                    af[e] += fabsf(t);
                    df[e] = fmaf(t, r, df[e]);
                    const float aw = q * fabsf(r) * wi[e];
                    ws[e] += aw;
                    wx[e] = fmaxf(wx[e], fmaf(sd[e], r, aw));
                }
            }
            wsum = team(reduce4(ws, lane), false);
            wmax = team(reduce4max(wx, lane), true);
            if (G) wsum = fmaf(G->W, iw, wsum);
        } else if (it == 0) {
            sums([&](int, int e, float D) { return fabsf(D) < ce[e]; });
        } else if (!close) {
            sums([](int, int, float D) { return D == 0.f; });     // the shift pole's own
        } else {
            // (poles closer to it than FP32's range have D = 0 too, and count)
            int ie[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) ie[e] = __shfl_sync(FULL, i, 8 * e);
            sums([&](int j, int e, float) { return j == ie[e]; });
        }
        float t = team(reduce4(tf, lane), false);
        float a = team(reduce4(af, lane), false);
        float d = team(reduce4(df, lane), false);
        if (G) {
            float fd;
            t += far(u, fd);
            d += fd;
            a += G->T;
        }
        if (!done) {
            ++passes;
            const float Phi = -Af + gam * u + t, dPhi = gam + d;
            if (it == 0) {
                num = Phi;
                Tabs = a;
                dsum = d;
                // between the zeros of the models at the pole and at the midpoint
                const float r0 = model_root(s, Phi, dPhi, 0.f, en, w);
                u = (!lowx && !upx) ? s * 0.5f * (r0 + rm) : s * r0;
            } else {
                const float mo = fabsf(u);
                const float mn = lowx || upx ? model_root_outer(-s * Af, gam, -s * t, d, mo, w)
                                             : model_root(s, Phi, dPhi, u, en, w);
                const float rho = en > 0.f ? fminf(mn, en - mn) : mn;
                if (!(mn > 0.f) || (en > 0.f && !(mn < en))) { ok = false; done = true; }
                else if (fabsf(mn - mo) <= 0x1p-8f * rho) {
                    ul = s * mn;
                    Tabs = a + __fdividef(w, mn);     // (num keeps the pole's own sums)
                    dsum = d;
                    done = true;
                }
                u = s * mn;
            }
        }
        if (it == 0) {
            // Algorithm 5's gate quantities, for its counters (Eq. K2: P + Q over |P - Q|)
            float kb = __fdividef(Tabs + fabsf(Af), fabsf(num));
            bm = kb;
            am = wsum;
            tm = wmax;
        }
        if (__all_sync(FULL, done || !ok)) break;
    }
    ok &= done && isfinite(ul) && ul != 0.f && isfinite(Tabs) && Tabs > 0.f && isfinite(dsum);
    if (!have || (lane & 7) != 0 || (NW > 1 && wid != 0)) return;
    int flags = 0;
    if (o.precision == 1) {
        atomicAdd(S.cnt64 + C64_F32, (unsigned long long)passes);
        if (mid64) flags |= AE_FLAG_MID64;             // (counted when solved)
    }
    if (o.bgate) {
        const double zi = R.zabs(i);
        if (R.zsum - zi > (double)(m + 1) * zi && !((double)bm <= o.kb_max)) {
            flags |= AE_FLAG_DDB;
        }
    }
    S.es_flags[k] = flags;
    S.es_pole[k] = i;
    S.es_Knu[k] = 1.0;
    S.es_b[k] = (double)num / (double)w * R.f32_scale();
    S.es_Kb[k] = (double)bm;
    S.es_iters[k] = 0;
    const int eL = ilogb(Ld), ezs = ilogb(R.zs);
    const double mu = scalb2((double)ul, es - eL);
    if (gersh) {
        // steps of Algorithm 3 from its Gershgorin bracket (1/mu inside it) to
        // the width 2 eps |1/mu|; after an FP32 bracket, from that one's width
        const float iw = rcp_f32(sqrt_f32(w));
        const float b = s * num / w;                   // (in units of 1/D)
        const float left = en > 0.f ? rcp_f32(en) : 0.f;
        const float wz = iw * sqrt_f32(gam);           // 1/zeta_i
        const float right = fmaxf(fmaxf(tm, wz), b + am + wz);
        const float W = (right - left) * fabsf(ul);
        int N = isfinite(W) && W > 0.f ? (int)ceilf(log2f(W) + 51.f) : 62;
        N = N < 1 ? 1 : N;
        if (o.precision == 1 && N > 32) N = 32;
        S.es_iters[k] = N;
    }
    const dd sg = {S.f.p[i], S.f.plo[i]};
    ok &= set_point(S, k, sg, dd{mu, 0.0});
    // bounds of the sums: sum |t| < 2^K1, sum zeta^2/D^2 < 2^K2 (the pole's own
    // term by its exponent: it can exceed FP32's range), |D| >= 2^er
    const float mn = fabsf(ul);
    S.f.K1[k] = ilogbf(Tabs * 1.02f) + 1 + eL + es - ezs;
    S.f.K2[k] = max(dsum > 0.f ? ilogbf(dsum * 1.04f) + 1 : -200,
                    ilogbf(__fdividef(w, mn) * 1.04f) + 1 - ilogbf(mn)) + 1 + 2 * eL - ezs;
    S.f.er[k] = ilogbf(0.98f * (en > 0.f ? fminf(mn, en - mn) : mn)) + es - eL;
    S.f.s1[k] = S.f.s3[k] = S.f.s5[k] = 0;
    S.f.s2[k] = S.f.s4[k] = 0;
    S.f.l1[k] = 0;
    S.f.l2[k] = 0;
    // (the outermost ones, which no group holds, are evaluated by k_fmore)
    S.f.st[k] = !ok ? FST_OLD : NW > 1 ? FST_MORE : FST_EVAL;
    if (!ok) src.push_old(inst, k);
    else if (NW > 1) src.push_more(0, inst, k);
}

template <Kind K, class Src>
__global__ void __launch_bounds__(256) k_fopen(const __grid_constant__ Src src, SolveOpts o) {
    after_previous();
    __shared__ float red[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inst, first;
    if (!src.unit(blockIdx.x, kGroup, inst, first)) return;
    const Scratch &S = src.scr(inst);
    const int m = S.cnt[C_M];
    int klo, khi;
    fast_range(S, klo, khi);
    if ((S.cnt[C_FLAGS] & CF_NOFAST) || m < 2) {
        const int k = (klo & ~(kGroup - 1)) + first - kGroup + lane;
        if (first && wid == 0 && k >= klo && k < khi) {
            S.f.st[k] = FST_OLD;
            src.push_old(inst, k);
        }
        return;
    }
    const int g = lane >> 3;                          // this lane group's eigenpair
    const bool groups = m >= kFarFrom;
    if (first == 0) {
        // poles that open_items refuses as shifts, about: spikes below 2^-50 of the
        // largest, gaps below 2^-31 (2^21 last places; for k_fold's teams)
        int hard = 0;
        for (int t = threadIdx.x; t < m; t += 256) {
            bool h = !(S.pz2f[t] > 0x1p-100f);
            if (t + 1 < m) {
                const unsigned long long a = __double_as_longlong(S.pd[t]);
                const unsigned long long b = __double_as_longlong(S.pd[t + 1]);
                h |= (a > b ? a - b : b - a) <= 1ull << 21;
            }
            hard += h;
        }
        hard = __reduce_add_sync(FULL, hard);
        if (lane == 0 && hard) atomicAdd(S.cnt + C_HARD, hard);
        if (!groups) return;
        // the instance's outermost eigenpairs: all poles, by the CTA
        const int k = g == 0 ? 0 : m;
        const bool have = g < 2 && k >= klo && k < khi;
        if (__syncthreads_or(have))
            open_items<K, 8>(src, inst, S, o, k, have, 0, m, nullptr, red);
        return;
    }
    const int k0 = (klo & ~(kGroup - 1)) + first - kGroup, k = k0 + 4 * wid + g;
    const int x = groups ? 1 : 0;                     // (unit 0 has the outermost ones)
    const bool have = k >= klo && k < khi && k >= x && k <= m - x;
    if (!__any_sync(FULL, have)) return;
    const GroupData *G = groups ? S.f.grp + k0 / kGroup : nullptr;
    const int jlo = groups ? G->jlo : 0, jhi = groups ? G->jhi : m;
    open_items<K, 1>(src, inst, S, o, min(max(k, x), m - x), have, jlo, jhi,
                     jhi - jlo < m ? G : nullptr, red);
}

// ---------------------------------------------------------------------------
// k_feval
// ---------------------------------------------------------------------------
// Five sums over the poles at each eigenpair's point: zeta^2/(p - lambda)^r for
// r = 1..5, over the poles near its group, a warp per eigenpair (and segment of
// the poles, blockIdx.y: the sums are integers, so that segments add up in any
// order), the 8 warps of a CTA sharing tiles of poles in shared memory.  Bound
// by issue slots: ~90 a term (FP64: one subtraction, 64 clocks of that pipe,
// behind them); the r = 4, 5 sums are skipped, warp by warp, where no lane's
// term reaches 2^-44 of their bound.
constexpr int kTile = 256;

template <class Src>
__global__ void __launch_bounds__(256, 3) k_feval(const __grid_constant__ Src src) {
    after_previous();
    __shared__ double tp[2][kTile];
    __shared__ unsigned long long tP[2][kTile], tz[2][kTile];
    __shared__ int te[2][kTile];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inst, first;
    if (!src.unit(blockIdx.x, 8, inst, first)) return;
    const Scratch &S = src.scr(inst);
    int klo, khi;
    fast_range(S, klo, khi);
    const int kf = (klo & ~7) + first;               // (8 eigenpairs of one group)
    if (kf >= khi) return;
    const int k = kf + wid;
    const bool act = k >= klo && k < khi && S.f.st[k] == FST_EVAL;
    if (!__syncthreads_or(act)) return;
    const int ka = act ? k : kf >= klo ? kf : klo;
    int jlo = 0, m = S.cnt[C_M];                     // the near poles: [jlo, m)
    if (m >= kFarFrom) {
        const GroupData &G = S.f.grp[kf / kGroup];
        jlo = G.jlo;
        m = G.jhi;
    }
    const double lhi = S.f.lhi[ka];
    const unsigned long long L = S.f.lmod[ka];
    const DiffRange dr = diff_range(lhi);
    const int K1 = S.f.K1[ka], K2 = S.f.K2[ka], er = S.f.er[ka];
    const int c1 = K1 - 1023, c2 = K2 - K1 + 1 - 1023, c3 = 2 - er - 1023, c4 = 1 - er - 1023;
    const double one = unit_reg();
    unsigned long long a1 = 0, a2 = 0, a3 = 0, a4 = 0, a5 = 0;
    unsigned long long l1 = 0, l2 = 0;       // 32 bits below a1, a2 (summed apart)
    // this segment's poles: whole tiles
    const int all_tiles = (m - jlo + kTile - 1) / kTile;
    const int t0 = (int)((long long)blockIdx.y * all_tiles / gridDim.y);
    const int tiles = (int)((long long)(blockIdx.y + 1) * all_tiles / gridDim.y);
    bool flip = k >= jlo + t0 * kTile;
    auto load = [&](int t, double &p, unsigned long long &P, unsigned long long &z, int &e) {
        const int j = jlo + t * kTile + threadIdx.x;
        p = 4.0; P = 0; z = 0; e = -8192;               // padding: terms of 0
        if (j < m) {
            p = S.f.p[j];
            P = S.f.P[j];
            z = S.f.z[j];
            e = S.f.ez[j];
        }
    };
    double lp;
    unsigned long long lP, lz;
    int le;
    load(t0, lp, lP, lz, le);
    for (int t = t0; t < tiles; ++t) {
        const int bsel = t & 1;
        tp[bsel][threadIdx.x] = lp;
        tP[bsel][threadIdx.x] = lP;
        tz[bsel][threadIdx.x] = lz;
        te[bsel][threadIdx.x] = le;
        __syncthreads();
        if (t + 1 < tiles) load(t + 1, lp, lP, lz, le);
        if (!act) continue;
        const int left = m - jlo - t * kTile;
        const int nc = left >= kTile ? kTile / 32 : (left + 31) / 32;
#pragma unroll 1
        for (int c = 0; c < nc; ++c) {
            const int x = c * 32 + lane;
            const int j0 = jlo + t * kTile + c * 32;
            double D = fma(tp[bsel][x], one, -lhi);    // (an FMA: 2.0 lanes a clock, DADD 1.7)
            int tl;
            unsigned dh = hi32(D), dl = (unsigned)__double2loint(D);
            unsigned eb = (dh << 1) >> 21;
            const int j = j0 + lane;
            if (eb - dr.lo >= dr.span && j < m) {
                const dd pj = {tp[bsel][x], S.f.plo[j]};
                const int i = S.es_pole[ka];
                const dd sg = {S.f.p[i], S.f.plo[i]};
                const dd Dd = near_diff(pj, sg, dd{S.f.mu[ka], S.f.mulo[ka]});
                D = Dd.hi;
                tl = near_tail(Dd);
                dh = hi32(D);
                dl = (unsigned)__double2loint(D);
                eb = (dh << 1) >> 21;
            } else if (eb < kFixMinExp && dr.tails) {
                tl = tail_of<kFixFrac2>(S.f.P2[j < m ? j : 0] - S.f.lmod2[ka], dh, dl, eb);
            } else {
                tl = tail_of(tP[bsel][x] - L, dh, dl, eb) & dr.tails;
            }
            const unsigned seed = hi32(rcp_seed(__hiloint2double(
                (int)((dh & 0xfffffu) | 0x3ff00000u), 0)));
            const unsigned long long Rr = recip63<true>(dh, dl, tl, seed);
            unsigned long long q = mul_hi3(tz[bsel][x], Rr);       // 2^62 of the term
            const unsigned s1 = (unsigned)(c1 + (int)eb - te[bsel][x]);
            unsigned long long v1 = shr64(q, s1);
            unsigned long long w1 = low32(q, s1);
            q = mul_hi3(q, Rr);
            const unsigned s2 = s1 + eb + c2;
            a2 += shr64(q, s2);
            l2 += low32(q, s2);
            q = mul_hi3(q, Rr);
            const unsigned s3 = s2 + eb + c3;
            unsigned long long v3 = shr64(q, s3);
            unsigned long long v5 = 0;
            const unsigned s4 = s3 + eb + c4;
            if (__any_sync(FULL, (int)s4 < 44)) {
                q = (unsigned long long)(unsigned)(q >> 32) * (unsigned)(Rr >> 32);
                a4 += shr64(q, s4);
                const unsigned s5 = s4 + eb + c4;
                q = (unsigned long long)(unsigned)(q >> 32) * (unsigned)(Rr >> 32);
                v5 = shr64(q, s5);
            }
            if (k >= j0 && k < j0 + 32) {
                // the poles change sides of lambda in this chunk: sums of odd
                // order end as (below) - (above)
                const bool above = j < k;
                a1 = (above ? 0ull - v1 : v1) - a1;
                a3 = (above ? 0ull - v3 : v3) - a3;
                a5 = (above ? 0ull - v5 : v5) - a5;
                l1 = (above ? 0ull - w1 : w1) - l1;
                flip = false;
            } else {
                a1 += v1;
                a3 += v3;
                a5 += v5;
                l1 += w1;
            }
        }
    }
    if (!act) return;
    if (flip) {
        a1 = 0ull - a1;
        a3 = 0ull - a3;
        a5 = 0ull - a5;
        l1 = 0ull - l1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a1 += __shfl_xor_sync(FULL, a1, o);
        a2 += __shfl_xor_sync(FULL, a2, o);
        a3 += __shfl_xor_sync(FULL, a3, o);
        a4 += __shfl_xor_sync(FULL, a4, o);
        a5 += __shfl_xor_sync(FULL, a5, o);
        l1 += __shfl_xor_sync(FULL, l1, o);
        l2 += __shfl_xor_sync(FULL, l2, o);
    }
    if (lane == 0) {
        atomicAdd((unsigned long long *)S.f.s1 + k, a1);
        atomicAdd(S.f.s2 + k, a2);
        atomicAdd((unsigned long long *)S.f.s3 + k, a3);
        atomicAdd(S.f.s4 + k, a4);
        atomicAdd((unsigned long long *)S.f.s5 + k, a5);
        atomicAdd((unsigned long long *)S.f.l1 + k, l1);
        atomicAdd(S.f.l2 + k, l2);
    }
}

// ---------------------------------------------------------------------------
// k_fstep
// ---------------------------------------------------------------------------
// M2 from its fixed-point sum and the 32 bits a term below
__device__ __forceinline__ dd sum2(unsigned long long a, unsigned long long l, int K2) {
    const double h = (double)a;
    const double r = (double)(long long)(a - (unsigned long long)h) + (double)l * 0x1p-32;
    const dd v = fast_two_sum(h, r);
    const double u = scalb2(1.0, K2 - 60);
    return dd{v.hi * u, v.lo * u};
}

// the counters of a solved eigenpair, added up over the warp's lanes that
// share its instance
__device__ __forceinline__ void fast_stats(const Scratch &S, int inst, int iters, int deriv,
                                           double Kb, bool ddb, bool any) {
    const unsigned act = __ballot_sync(FULL, any);
    if (!any) return;
    const unsigned grp = __match_any_sync(act, inst);
    const int it = __reduce_add_sync(grp, iters);
    const int de = __reduce_add_sync(grp, deriv);
    const int mx = __reduce_max_sync(grp, iters);
    const int dd_ = __reduce_add_sync(grp, ddb ? 1 : 0);
    const unsigned kb = __reduce_max_sync(grp, isfinite(Kb) && Kb >= 0.0
                                                  ? __float_as_uint((float)Kb) : 0u);
    if ((threadIdx.x & 31) == __ffs(grp) - 1) {
        atomicAdd(S.cnt64 + C64_ITERS, (unsigned long long)it);
        if (de) atomicAdd(S.cnt64 + C64_DERIV, (unsigned long long)de);
        atomicMax(S.cnt + C_MAXIT, mx);
        if (dd_) atomicAdd(S.cnt + C_DDB, dd_);
        atomic_max_nonneg(S.cnt64 + C64_MAXKB, (double)__uint_as_float(kb));
    }
}

// Sums of an evaluation at sigma + mu: M1 = (below - above), M_r = sum zeta^2 /
// (p - lambda)^r for r >= 2, in scaled units.
struct FastSums {
    dd M1, M2;
    double M3, M4, M5;
};

// The far poles' share at lambda = c + t: the moments' polynomial and its Taylor
// coefficients (order 0 to more than double: the first three moments in
// double-double, the rest weighs at most 8^-3).
__device__ __forceinline__ void add_far(const GroupData &G, dd t, FastSums &s) {
    const double sc = pow2(-G.e);
    const dd x = {t.hi * sc, t.lo * sc};
    double b0 = 0.0, b1 = 0.0, b2 = 0.0, b3 = 0.0, b4 = 0.0, p3 = 0.0;
#pragma unroll
    for (int q = kMoments - 1; q >= 0; --q) {
        b4 = fma(b4, x.hi, b3);
        b3 = fma(b3, x.hi, b2);
        b2 = fma(b2, x.hi, b1);
        b1 = fma(b1, x.hi, b0);
        b0 = fma(b0, x.hi, G.A[q]);
        if (q == 3) p3 = b0;
    }
    dd v = dd_add(dd{G.A[2], G.Al[2]}, two_prod(x.hi, p3));
    v = dd_add(dd{G.A[1], G.Al[1]}, dd_mul(x, v));
    v = dd_add(dd{G.A[0], G.Al[0]}, dd_mul(x, v));
    s.M1 = dd_add(s.M1, dd_neg(v));
    s.M2 = dd_add(s.M2, dd{b1 * sc, 0.0});
    s.M3 += b2 * sc * sc;
    s.M4 += b3 * sc * sc * sc;
    s.M5 += (b4 * sc) * sc * (sc * sc);
}

// The zero from an evaluation, by one thread.  cterm: the weight of the terms'
// error (kErrTerm...); M2u: the sum the unit's error counts over (negative:
// M2 less the pole's own term, always formed in double-double when small).
// Returns FST_DONE with
// the result stored (when no round is left FST_OLD), or FST_MORE with the next
// point set: the model's zero, or the zero found where only its accuracy is
// wanting (unit_bad: for the differences' unit alone).
template <Kind K>
__device__ int fast_advance(const Scratch &S, int k, const FastSums &q, double cterm, double M2u,
                            bool &unit_bad) {
    unit_bad = false;
    const int m = S.cnt[C_M];
    const int es = fast_scale<K>(S);
    int i = S.es_pole[k];
    const dd sg = {S.f.p[i], S.f.plo[i]};
    const dd mu = {S.f.mu[k], S.f.mulo[k]};
    const int K1 = S.f.K1[k], K2 = S.f.K2[k];
    const dd N2 = dd_add(q.M2, dd{1.0, 0.0});
    const double N = N2.hi;
    // f = (alpha - sigma - mu) + (sum below - sum above)
    const double sc = pow2(es);
    dd a = dd{S.prm[P_ALPHA_HI] * sc, S.prm[P_ALPHA_LO] * sc};
    a = dd_add(a, dd_neg(sg));
    a = dd_add(a, dd_neg(mu));
    const double f = dd_add(a, q.M1).hi;
    // distances to the interval's poles
    const bool up = mu.hi > 0.0;
    const int jn = up ? i - 1 : i + 1;
    const bool other = jn >= 0 && jn < m;
    dd dn = {0.0, 0.0};
    double rho = fabs(mu.hi);
    if (other) {
        dn = dd_add(dd{S.f.p[jn], S.f.plo[jn]}, dd_neg(sg));
        rho = fmin(rho, fabs(dn.hi - mu.hi));
    }
    const double iN = rcp(N);
    double d = f * iN;
    if (!(isfinite(d) && N >= 1.0)) return FST_OLD;
    if (fabs(d) <= kStepMax * rho) {
        // d = f / (N + M3 d + M4 d^2 + M5 d^3): each turn gains a factor |d|/rho
#pragma unroll
        for (int r = 0; r < 4; ++r) d = f * rcp(N + d * (q.M3 + d * (q.M4 + d * q.M5)));
        // f' there, to more than double: the vector's norm
        const dd Nd = dd_add(N2, dd{d * (2.0 * q.M3 + d * (3.0 * q.M4 + d * (4.0 * q.M5))), 0.0});
        const double Nf = Nd.hi;
        // lambda = sigma + mu + d
        dd mf = two_sum(mu.hi, d);
        mf.lo += mu.lo;
        mf = fast_two_sum(mf.hi, mf.lo);
        if (!(Nf >= 1.0)) return FST_OLD;
        if (M2u < 0.0) {
            const double z2 = S.pz2[i] * sc * sc;
            // (a difference with that unit is at least 2^-45: the second bound,
            // for offsets so small that the first one cancels)
            M2u = fmin(fmax(q.M2.hi - (z2 / mu.hi) / mu.hi, 0.0) + 0x1p-50 * q.M2.hi,
                       0x1p45 * pow2(K1));
        }
        if (!(pow2(K1) * cterm + M2u * kErrUnit <= Nf * fabs(mf.hi))) {
            unit_bad = M2u * kErrUnit > 0.25 * Nf * fabs(mf.hi);
            set_point(S, k, sg, mf);
            return FST_MORE;
        }
        // the nearer pole is the shift (the upper one where they tie, as the
        // midpoint test has it)
        if (other) {
            const dd alt = dd_add(mf, dd_neg(dn));
            const double x = fabs(mf.hi), y = fabs(alt.hi);
            if (y < x || (y == x && up)) {
                i = jn;
                mf = alt;
            }
        }
        if (mf.hi > 0.0 ? k != i : k != i + 1) return FST_OLD;   // outside its interval
        const double sigma = PolesOf<K>::make(S, m).pole(i);
        const double muu = mf.hi * pow2(-es);
        if (!(fabs(muu) >= 0x1p-1000)) return FST_OLD;
        S.es_pole[k] = i;
        S.es_sigma[k] = sigma;
        S.es_mu[k] = muu;
        S.es_lam[k] = sigma + muu;
        S.f.N[k] = Nf;
        S.f.Nlo[k] = Nd.lo;
        // (for a remedy's shift nearer than this one: the step d, in double, is
        // known to 2^-53 of itself)
        S.f.M2u[k] = M2u + Nf * fabs(d) / kErrUnit;
        set_point(S, k, dd{S.f.p[i], S.f.plo[i]}, mf);
        S.f.mu[k] = mf.hi;           // (set_point may have moved it to the rounded lambda)
        S.f.mulo[k] = mf.lo;
        return FST_DONE;
    }
    // the model's zero, in double; a short step is the Newton step
    double mn;
    const double s = up ? 1.0 : -1.0, x = fabs(mu.hi);
    if (fabs(d) <= 0x1p-10 * rho) {
        mn = s * (mu.hi + d);
    } else {
        const double z2 = S.pz2[i] * sc * sc, t = z2 / mu.hi;
        const double Phi = t - f, dPhi = fmax(N - t / mu.hi, 1.0);
        if (other) {
            const double e = fabs(dn.hi), g = e - x;
            const double B = dPhi * g * g, A = s * Phi - dPhi * g, X = A * e + B;
            const double b = X + z2, h = X - z2, rt = sqrt(h * h + 4.0 * z2 * B);
            mn = b >= 0.0 ? 2.0 * z2 * e / (b + rt) : (b - rt) / (2.0 * A);
        } else {
            const double A = s * Phi - dPhi * x, rt = sqrt(A * A + 4.0 * dPhi * z2);
            mn = A >= 0.0 ? 2.0 * z2 / (A + rt) : (rt - A) / (2.0 * dPhi);
        }
    }
    // at most a quarter of the distance to the nearest pole, so that the sums'
    // bounds grow by less than 4/3 and 16/9
    const double lim = 0.25 * rho;
    mn = fmin(fmax(mn, x - lim), x + lim);
    if (!(isfinite(mn) && mn > 0.0) || !set_point(S, k, sg, dd{s * mn, 0.0})) return FST_OLD;
    S.f.K1[k] = K1 + 1;
    S.f.K2[k] = K2 + 1;
    S.f.er[k] -= 1;
    return FST_MORE;
}

// Eigenpair k moved to its remedy's shift (other pole, the eigenvalue itself,
// 0, or a DPR1's last pole) when the zero is known well enough for what that
// shift is meant to keep: the error of f over f' against |lambda|, the
// distance to the nearest pole and the new offset.  False: not moved.
template <Kind K>
__device__ bool fast_remedy(const Scratch &S, int k, double cterm) {
    const int es = fast_scale<K>(S), m = S.cnt[C_M];
    const int rem = S.es_flags[k];
    const dd sg = fast_sigma<K>(S, k, es);
    const dd mu = {S.f.mu[k], S.f.mulo[k]};
    const double sc = pow2(es);
    int i = -1;
    dd s2;
    double sv;
    if (rem & AE_FLAG_NEARZERO) {
        sv = 0.0;
        s2 = dd{0.0, 0.0};
    } else if (rem & AE_FLAG_OTHERPOLE) {
        i = S.es_fixpole[k];
        s2 = dd{S.f.p[i], S.f.plo[i]};
        sv = S.pv[i];
    } else {
        sv = S.es_fixshift[k];
        s2 = dd{sv * sc, 0.0};
    }
    const dd mu2 = dd_add(dd_add(sg, dd_neg(s2)), mu);
    const double lam = dd_add(s2, mu2).hi;
    double need = fmin(fabs(mu.hi), fabs(lam));
    for (int j = k - 1; j <= k; ++j)
        if (j >= 0 && j < m) {
            const dd dj = dd_add(sg, dd_neg(dd{S.f.p[j], S.f.plo[j]}));
            need = fmin(need, fabs(dd_add(dj, mu).hi));
        }
    // (the offset itself counts from a pole, the DPR1's last one included)
    if (i >= 0 || (K == KIND_DPR1 && sv == S.prm[P_PLAST])) need = fmin(need, fabs(mu2.hi));
    const double muu = mu2.hi * pow2(-es), l2 = sv + muu;
    const auto R = PolesOf<K>::make(S, m);
    const double lo = k < m ? R.pole(k) : (K == KIND_DPR1 ? S.prm[P_PLAST] : -INFINITY);
    const double hi = k > 0 ? R.pole(k - 1) : INFINITY;
    // (mu itself is a double-double: 2^-105 of it)
    if (!(pow2(S.f.K1[k]) * cterm + S.f.M2u[k] * kErrUnit <= S.f.N[k] * need &&
          0x1p-53 * fabs(mu.hi) <= need && isfinite(mu2.hi) && l2 >= lo && l2 <= hi &&
          (i < 0 || muu != 0.0)))
        return false;
    S.es_pole[k] = i;
    S.es_sigma[k] = sv;
    S.es_mu[k] = muu;
    S.es_lam[k] = l2;
    set_point(S, k, s2, mu2);
    S.f.mu[k] = mu2.hi;
    S.f.mulo[k] = mu2.lo;
    return true;
}

// the counters and iteration count of a solved eigenpair
__device__ __forceinline__ void fast_count(const Scratch &S, int k, const SolveOpts &o, int diag,
                                           int rounds, int &iters, int &deriv, double &Kb,
                                           bool &ddb) {
    iters = o.finish == 0 ? S.es_iters[k] : rounds;
    deriv = o.finish == 0 ? 0 : rounds;
    S.es_iters[k] = iters;
    Kb = diag ? 0.0 : S.es_Kb[k];
    ddb = !diag && (S.es_flags[k] & AE_FLAG_DDB);
    if (S.es_flags[k] & AE_FLAG_MID64) atomicAdd(S.cnt + C_MID64, 1);
}

// One thread per eigenpair: the zero from k_feval's sums, or on to k_fmore.
template <Kind K, class Src>
__global__ void __launch_bounds__(64) k_fstep(const __grid_constant__ Src src, SolveOpts o,
                                              int diag) {
    after_previous();
    int inst = 0, idx = 0, klo = 0, khi = 0, k = 0;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    bool act = src.item(t, inst, idx);
    const Scratch &S = src.scr(inst);
    if (act) {
        fast_range(S, klo, khi);
        k = klo + idx;
        act = k < khi && S.f.st[k] == FST_EVAL;
    }
    int iters = 0, deriv = 0;
    double Kb = 0.0;
    bool ddb = false, fin = false;
    if (act) {
        const int K1 = S.f.K1[k], K2 = S.f.K2[k], er = S.f.er[k];
        const int K3 = K2 - er, K4 = K3 - er, K5 = K4 - er;
        FastSums q;
        const dd v = dd_add(dd_of_ll(S.f.s1[k]), dd{(double)S.f.l1[k] * 0x1p-32, 0.0});
        const double us = scalb2(1.0, K1 - 62);
        q.M1 = dd{v.hi * us, v.lo * us};
        q.M2 = sum2(S.f.s2[k], S.f.l2[k], K2);
        q.M3 = -scalb2((double)S.f.s3[k], K3 - 57);
        q.M4 = scalb2((double)S.f.s4[k], K4 - 55);
        q.M5 = -scalb2((double)S.f.s5[k], K5 - 53);
        const GroupData &G = S.f.grp[k / kGroup];
        if (S.cnt[C_M] >= kFarFrom && G.jhi - G.jlo < S.cnt[C_M]) {
            const int i = S.es_pole[k];
            dd tt = dd_add(dd{S.f.p[i], S.f.plo[i]}, dd{-G.c, 0.0});
            tt = dd_add(tt, dd{S.f.mu[k], S.f.mulo[k]});
            add_far(G, tt, q);
        }
        bool unit_bad;
        const int st = fast_advance<K>(S, k, q, kErrTerm, -1.0, unit_bad);
        S.f.st[k] = st;
        if (st == FST_OLD) src.push_old(inst, k);
        else if (st == FST_MORE) src.push_more(0, inst, k);
        else {
            fast_count(S, k, o, diag, 1, iters, deriv, Kb, ddb);
            fin = true;
        }
    }
    fast_stats(S, inst, iters, deriv, Kb, ddb, fin);
}

// ---------------------------------------------------------------------------
// k_fmore
// ---------------------------------------------------------------------------
// |p - lambda| as its rounded value (returned) and m 2^127, m in [1, 2) the
// whole difference's significand
__device__ __forceinline__ unsigned __int128 wide_mant(double D, unsigned __int128 tail) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(D);
    const unsigned long long Dm = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    return ((unsigned __int128)Dm << 75) + tail;
}

// v >> s, 0 from 128 on
__device__ __forceinline__ unsigned __int128 shr128(unsigned __int128 v, unsigned s) {
    const unsigned long long lo = (unsigned long long)v, hi = (unsigned long long)(v >> 64);
    const unsigned t = s & 63;
    const unsigned long long h = hi >> t, x = t ? hi << (64 - t) : 0ull, l = (lo >> t) | x;
    const unsigned __int128 a = ((unsigned __int128)h << 64) | l;
    return s < 64 ? a : s < 128 ? (unsigned __int128)h : (unsigned __int128)0;
}

// high 128 bits of a b
__device__ __forceinline__ unsigned __int128 mul_hi128(unsigned __int128 a,
                                                       unsigned __int128 b) {
    const unsigned long long al = (unsigned long long)a, ah = (unsigned long long)(a >> 64);
    const unsigned long long bl = (unsigned long long)b, bh = (unsigned long long)(b >> 64);
    return (unsigned __int128)ah * bh + __umul64hi(ah, bl) + __umul64hi(al, bh);
}

// 2^127 / m for the significand m 2^127 = M, from its 63-bit reciprocal R
__device__ __forceinline__ unsigned __int128 recip127(unsigned __int128 M, unsigned long long R) {
    if (R >> 63) R = 0x7fffffffffffffffull;
    const unsigned __int128 V =
        (unsigned __int128)(unsigned long long)(M >> 64) * R + __umul64hi((unsigned long long)M, R);
    const __int128 E = (__int128)(((unsigned __int128)1 << 126) - V);      // e 2^126, |e| < 2^-58
    const __int128 c = (__int128)(long long)(E >> 5) * (__int128)(long long)R;
    return ((unsigned __int128)R << 64) + (unsigned __int128)(c >> 57);
}

__device__ __forceinline__ dd dd_of_i128(__int128 v) {
    const double a = (double)(long long)(v >> 84) * 0x1p84;
    const double b = (double)((unsigned long long)(v >> 42) & 0x3ffffffffffull) * 0x1p42;
    const double c = (double)((unsigned long long)v & 0x3ffffffffffull);
    return dd_add(two_sum(a, b), dd{c, 0.0});
}

// One CTA per listed eigenpair: evaluations with f in 128 bits (a term to
// ~2^-85, D's fixed-point unit 2^-106 permitting) and the other sums as
// k_feval forms them, until the zero is accurate enough.  A few items are bound by
// a thread's own chain of ~300 instructions a term, so a single solve gives each
// 16 warps (graded n = 16384: 584 -> 457 us for both phases, DPR1 n = 8192: 177 ->
// 116); a batch, with many short ones, 8 (84 us for a batch of 512, 153 with 16).  Phase 1 (after
// k_ffix): one evaluation at a flagged eigenpair's zero, then its remedy.
constexpr int kMoreWarps = 16;                // at most

template <Kind K, class Src>
__global__ void __launch_bounds__(32 * kMoreWarps) k_fmore(const __grid_constant__ Src src, SolveOpts o,
                                               int phase, int diag) {
    after_previous();
    constexpr int NW = kMoreWarps;
    __shared__ unsigned long long sh1[NW], sh1h[NW], sh2[NW], sh2u[NW], sh4[NW];
    __shared__ long long sh3[NW], sh5[NW];
    __shared__ unsigned long long sh2l[NW];
    __shared__ int verdict, verdict_unit;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int cnt = src.more_count(phase);
    for (int w = blockIdx.x; w < cnt; w += gridDim.x) {
        const int2 ik = src.more_at(w);
        const Scratch &S = src.scr(ik.x);
        const int k = ik.y, m = S.cnt[C_M];
        int st = FST_MORE;
        bool unit_bad = false;
        if (phase == 1) {
            // (an outermost eigenvalue's point is its rounded lambda)
            if (threadIdx.x == 0)
                set_point(S, k, dd{S.f.p[S.es_pole[k]], S.f.plo[S.es_pole[k]]},
                          dd{S.f.mu[k], S.f.mulo[k]});
            __syncthreads();
        }
        for (int round = 0; round < kMoreRounds && st == FST_MORE; ++round) {
            const double lhi = S.f.lhi[k];
            const unsigned long long L = S.f.lmod[k];
            const DiffRange dr = diff_range(lhi);
            // (a unit's error that one evaluation showed to be too large: every
            // difference in double-double)
            const bool all_dd = unit_bad && dr.tails;
            const int K1 = S.f.K1[k], K2 = S.f.K2[k], er = S.f.er[k];
            const int c1 = K1 - 1023, c2 = K2 - K1 + 1 - 1023, c3 = 2 - er - 1023,
                      c4 = 1 - er - 1023;
            __int128 a1 = 0;
            unsigned long long a2 = 0, a2u = 0, a4 = 0;
            long long a3 = 0, a5 = 0;
            unsigned long long l2 = 0;
            for (int j = threadIdx.x; j < m; j += blockDim.x) {
                const double p = S.f.p[j];
                double D = p - lhi;
                unsigned dh = hi32(D), eb = (dh << 1) >> 21;
                int tl;
                unsigned __int128 M;
                const bool dd_diff = eb - dr.lo >= dr.span || (dr.tails && eb < kFixMinExp) || all_dd;
                if (dd_diff) {
                    const int i = S.es_pole[k];
                    const dd Dd = near_diff(dd{p, S.f.plo[j]}, dd{S.f.p[i], S.f.plo[i]},
                                            dd{S.f.mu[k], S.f.mulo[k]});
                    D = Dd.hi;
                    dh = hi32(D);
                    eb = (dh << 1) >> 21;
                    const double lo = (D < 0.0 ? -Dd.lo : Dd.lo) * pow2(51 + 1075 - (int)eb);
                    const long long li = __double2ll_rd(lo);     // 2^-51 of D's last place
                    tl = (int)(li >> 44);
                    M = wide_mant(D, (unsigned __int128)((__int128)li << 24));
                } else if (dr.tails) {
                    const unsigned dl = (unsigned)__double2loint(D);
                    unsigned long long T = S.f.P[j] - L;
                    if (dh >> 31) T = 0ull - T;
                    const unsigned long long Dm =
                        ((unsigned long long)((dh & 0xfffffu) | 0x100000u) << 32) | dl;
                    const int sh = (int)eb - (1075 - kFixFrac);
                    const long long tail = (long long)(T - (Dm << (sh & 63)));
                    tl = (int)(tail >> ((sh - 7) & 63));
                    M = wide_mant(D, (unsigned __int128)((__int128)tail << (75 - sh)));
                } else {
                    tl = 0;
                    M = wide_mant(D, 0);
                }
                const unsigned seed = hi32(rcp_seed(__hiloint2double(
                    (int)((dh & 0xfffffu) | 0x3ff00000u), 0)));
                const unsigned long long R =
                    recip63<true>(dh, (unsigned)__double2loint(D), tl, seed);
                const bool above = j < k;
                const int ez = S.f.ez[j];
                // f's term: zeta^2 in double-double over the wide difference
                {
                    const unsigned __int128 Z =
                        ((unsigned __int128)S.f.zh[j] << 64) | S.f.zl[j];
                    const unsigned __int128 q = mul_hi128(Z, recip127(M, R));
                    const __int128 v =
                        (__int128)shr128(q, (unsigned)(K1 + 2 - ez + (int)eb - 1023));
                    a1 += above ? -v : v;
                }
                unsigned long long q = mul_hi3(S.f.z[j], R);
                const unsigned s2 = (unsigned)(c1 + (int)eb - ez) + eb + c2;
                q = mul_hi3(q, R);
                const unsigned long long v2 = shr64(q, s2);
                a2 += v2;
                a2u += dd_diff ? 0ull : v2;
                l2 += low32(q, s2);
                q = mul_hi3(q, R);
                const unsigned s3 = s2 + eb + c3;
                const long long v3 = (long long)shr64(q, s3);
                a3 += above ? -v3 : v3;
                const unsigned s4 = s3 + eb + c4;
                q = (unsigned long long)(unsigned)(q >> 32) * (unsigned)(R >> 32);
                a4 += shr64(q, s4);
                q = (unsigned long long)(unsigned)(q >> 32) * (unsigned)(R >> 32);
                const long long v5 = (long long)shr64(q, s4 + eb + c4);
                a5 += above ? -v5 : v5;
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) {
                const unsigned long long hl = __shfl_xor_sync(FULL, (unsigned long long)a1, s);
                const unsigned long long hh =
                    __shfl_xor_sync(FULL, (unsigned long long)((unsigned __int128)a1 >> 64), s);
                a1 += (__int128)(((unsigned __int128)hh << 64) | hl);
                a2 += __shfl_xor_sync(FULL, a2, s);
                a2u += __shfl_xor_sync(FULL, a2u, s);
                l2 += __shfl_xor_sync(FULL, l2, s);
                a3 += __shfl_xor_sync(FULL, a3, s);
                a4 += __shfl_xor_sync(FULL, a4, s);
                a5 += __shfl_xor_sync(FULL, a5, s);
            }
            __syncthreads();
            if (lane == 0) {
                sh2l[wid] = l2;
                sh1[wid] = (unsigned long long)a1;
                sh1h[wid] = (unsigned long long)((unsigned __int128)a1 >> 64);
                sh2[wid] = a2;
                sh2u[wid] = a2u;
                sh3[wid] = a3;
                sh4[wid] = a4;
                sh5[wid] = a5;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int x = 1; x < (int)(blockDim.x >> 5); ++x) {
                    a1 += (__int128)(((unsigned __int128)sh1h[x] << 64) | sh1[x]);
                    a2 += sh2[x];
                    a2u += sh2u[x];
                    l2 += sh2l[x];
                    a3 += sh3[x];
                    a4 += sh4[x];
                    a5 += sh5[x];
                }
                const int K3 = K2 - er, K4 = K3 - er, K5 = K4 - er;
                FastSums q;
                const dd v = dd_of_i128(a1);
                const double us = scalb2(1.0, K1 - 124);
                q.M1 = dd{v.hi * us, v.lo * us};
                q.M2 = sum2(a2, l2, K2);
                q.M3 = -scalb2((double)a3, K3 - 57);
                q.M4 = scalb2((double)a4, K4 - 55);
                q.M5 = -scalb2((double)a5, K5 - 53);
                const double ct = dr.tails ? kErrTermWide : kErrTerm;
                bool ub;
                int v2 = fast_advance<K>(S, k, q, ct, dr.tails ? scalb2((double)a2u, K2 - 60) : 0.0,
                                         ub);
                if (v2 == FST_MORE && round + 1 == kMoreRounds) v2 = FST_OLD;
                if (phase == 0) {
                    if (v2 == FST_DONE) {
                        int iters, deriv;
                        double Kb;
                        bool ddb;
                        fast_count(S, k, o, diag, 2 + round, iters, deriv, Kb, ddb);
                        EigResult r{};
                        r.iters = iters;
                        r.iters_d = deriv;
                        r.Kb = Kb;
                        r.flags = ddb ? AE_FLAG_DDB : 0;
                        record_stats(S, r);
                    } else if (v2 == FST_OLD) {
                        src.push_old(ik.x, k);
                    }
                    S.f.st[k] = v2;
                } else if (v2 != FST_MORE) {
                    atomicAdd(S.cnt64 + C64_ITERS, (unsigned long long)(round + 1));
                    atomicAdd(S.cnt64 + C64_ITERS_FIX, (unsigned long long)(round + 1));
                    if (v2 != FST_DONE || !fast_remedy<K>(S, k, ct)) {
                        S.f.st[k] = FST_OLD;
                        const bool op = S.es_flags[k] & AE_FLAG_OTHERPOLE;
                        src.push_fix(ik.x, k, !op, src.vec(ik.x).n);
                    }
                }
                verdict = v2;
                verdict_unit = v2 == FST_MORE && ub;
            }
            __syncthreads();
            st = verdict;
            unit_bad |= verdict_unit != 0;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// k_fold: the FP64 solver for the eigenpairs left over
// ---------------------------------------------------------------------------
// A warp each, as k_eig and k_batch_eig have it, or a CTA of 8 warps where that is
// the shorter way.  The choice is the instance's (order, form and the poles that
// k_fopen counted), never the pass's, so that an eigenpair has the same bits in a
// solve alone, a part or a merged pass.  One pass over the poles is bound by the
// SM's FP64 pipe, which a warp alone nearly fills: a CTA gains where few eigenpairs
// are left and each is long.  A whole solve, a warp / a CTA each, uniform poles, us:
// one spike of 1e-18, bisection: n = 200 553 / 605, 1000 1510 / 916, 4097 3566 /
// 1658, 8192 7204 / 3188; Newton: 200 223 / 264, 1000 369 / 396, 4097 700 / 600, 8192
// 1196 / 890.  A quarter of the poles (spikes over 20 decades), bisection: 1000 1590 /
// 1433, 4097 6233 / 4432, 8192 18473 / 14185; Newton: 1000 402 / 498, 4097 983 / 1177,
// 8192 2548 / 2676.  All (scaled by 2^500), bisection: 200 483 / 1699, 1000 1395 /
// 2557, 4097 12102 / 14579.  Three CTAs an SM, as k_eig (128 registers and two: all of
// n = 4097 12.1 ms and 2.70 by Newton instead of 11.5 and 2.42).
constexpr int kFoldCta = 768, kFoldCtaNewton = 2048;
__device__ __forceinline__ bool fold_by_cta(const Scratch &S, const SolveOpts &o) {
    const int m = S.cnt[C_M], hard = S.cnt[C_HARD];
    if (S.cnt[C_FLAGS] & CF_NOFAST) return false;
    return o.finish == 0 ? m >= kFoldCta && 2 * hard <= m : m >= kFoldCtaNewton && 64 * hard <= m;
}

template <Kind K, class Src>
__global__ void __launch_bounds__(256, 3) k_fold(const __grid_constant__ Src src, SolveOpts o) {
    after_previous();
    __shared__ double red[16];
    __shared__ int tick;
    const int cnt = src.old_count();
    if (cnt == 0) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int w = blockIdx.x; w < cnt;) {
        const int2 ik = src.old_at(w);
        const Scratch &S = src.scr(ik.x);
        if (fold_by_cta(S, o))
            eig_item<K>(PolesOf<K>::make(S, S.cnt[C_M]), CtaTeam<8>{(int)threadIdx.x, red, 0}, S,
                        ik.y, o, src.slice((long long)blockIdx.x * 8));
        __syncthreads();
        if (threadIdx.x == 0) tick = gridDim.x + atomicAdd(src.old_ticket(0), 1);
        __syncthreads();
        w = tick;
    }
    // (each warp's first one spreads them over the SMs)
    double2 *buf = src.slice((long long)blockIdx.x * 8 + wid);
    for (int w = wid * gridDim.x + blockIdx.x; w < cnt;) {
        const int2 ik = src.old_at(w);
        const Scratch &S = src.scr(ik.x);
        if (!fold_by_cta(S, o))
            eig_item<K>(PolesOf<K>::make(S, S.cnt[C_M]), WarpTeam{lane}, S, ik.y, o, buf);
        __syncwarp();
        if (lane == 0) w = 8 * gridDim.x + atomicAdd(src.old_ticket(1), 1);
        w = __shfl_sync(FULL, w, 0);
    }
}

// b and K_b of Algorithm 2 for callers that ask for the diagnostics, as the
// FP64 solver forms them (a warp per eigenpair)
template <Kind K, class Src>
__global__ void __launch_bounds__(256) k_fdiag(const __grid_constant__ Src src, SolveOpts o) {
    after_previous();
    const int lane = threadIdx.x & 31;
    const WarpTeam T{lane};
    int inst, first;
    if (!src.unit(blockIdx.x, 8, inst, first)) return;
    const Scratch &S = src.scr(inst);
    int klo, khi;
    fast_range(S, klo, khi);
    const int k = klo + first + (int)(threadIdx.x >> 5);
    if (k >= khi || S.f.st[k] != FST_DONE) return;
    const auto R = PolesOf<K>::make(S, S.cnt[C_M]);
    const int i = S.es_pole[k];
    double b, Kb;
    const bool dd2 = shifted_b(R, T, i, o, b, Kb);
    if (lane == 0) {
        S.es_b[k] = b;
        S.es_Kb[k] = Kb;
        S.es_flags[k] = (S.es_flags[k] & ~AE_FLAG_DDB) | (dd2 ? AE_FLAG_DDB : 0);
        if (dd2) atomicAdd(S.cnt + C_DDB, 1);
        if (isfinite(Kb)) atomic_max_nonneg(S.cnt64 + C64_MAXKB, Kb);
    }
}

// ---------------------------------------------------------------------------
// k_ffix: remedies
// ---------------------------------------------------------------------------
// The eigenpairs k_fix_decide flagged: moved by a subtraction where that
// serves, else on to k_fmore, or (those the FP64 solver took) to k_fix_solve.
template <Kind K, class Src>
__global__ void __launch_bounds__(64) k_ffix(const __grid_constant__ Src src) {
    after_previous();
    int inst = 0, idx = 0;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (!src.item(t, inst, idx)) return;
    const Scratch &S = src.scr(inst);
    const PartRange P = part_range(S);
    const int k = P.k0 + idx;
    if (k >= P.k1) return;
    const int rem = S.es_flags[k] & (AE_FLAG_NEARZERO | AE_FLAG_OTHERPOLE | AE_FLAG_DPR1SHIFT);
    if (!rem) return;
    if (S.f.p && S.f.st[k] == FST_DONE) {
        if (!fast_remedy<K>(S, k, kErrTerm)) src.push_more(1, inst, k);
    } else {
        src.push_fix(inst, k, !(rem & AE_FLAG_OTHERPOLE), src.vec(inst).n);
    }
}

// ---------------------------------------------------------------------------
// k_fcols
// ---------------------------------------------------------------------------
// significand (64 bits, top bit set), biased exponent and sign of a double;
// a zero has significand 0 and an exponent below all others
struct Mant {
    unsigned long long m;
    int e;                // bit 31: the sign, low bits: the biased exponent
};
__device__ __forceinline__ Mant mant_of(double x) {
    unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned sg = (unsigned)(b >> 32) & 0x80000000u;
    int e = (int)((b >> 52) & 0x7ff), off = 0;
    if (e == 0 && x != 0.0) {
        b = (unsigned long long)__double_as_longlong(x * 0x1p64);
        e = (int)((b >> 52) & 0x7ff);
        off = 64;
    }
    Mant r;
    r.m = e ? ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 11 : 0ull;
    r.e = (int)(((unsigned)(e ? e - off : -8192) & 0xffffu) | sg);
    return r;
}

// a G / 2^61 2^(be - 1023) rounded to double, a G / 2^64 in (2^58, 2^63), a's
// significand in [2^63, 2^64) or 0 with be < -1000; sgn: the sign bit.  CHECK:
// the result may lie outside the normal range.
template <bool CHECK>
__device__ __forceinline__ double pack_prod(unsigned long long a, unsigned long long G, int be,
                                            unsigned sgn) {
    const unsigned long long H0 = mul_hi3(a, G);
    const unsigned h = (unsigned)(H0 >> 32);
    const int lz = __clz(h);                            // 1..5
    const unsigned long long H = (H0 << (lz - 1)) + 0x200ull;
    const int e1 = be + 1 - lz;                         // exponent - 1
    const unsigned lo = (unsigned)(H >> 10);
    const unsigned hi = (unsigned)(H >> 42) + ((unsigned)e1 << 20);
    if (CHECK && (unsigned)e1 >= 2045u) {
        if (a == 0) return __hiloint2double((int)sgn, 0);
        // below the normal range (or above it): in FP64
        const double v = ldexp((double)(H >> 10), e1 - 1074);
        return sgn ? -v : v;
    }
    return __hiloint2double((int)(hi | sgn), (int)lo);
}

// 1 / sqrt(x) in double-double
__device__ __forceinline__ dd dd_rsqrt(dd x) {
    const double r = 1.0 / sqrt(x.hi);
    const dd t = dd_mul(two_prod(r, r), x);                    // 1 + O(eps)
    const double e = (1.0 - t.hi) - t.lo;
    return fast_two_sum(r, 0.5 * r * e);
}

// a positive double-double as a significand of 64 bits (top bit set) and an
// exponent
__device__ __forceinline__ void scale_of(dd x, unsigned long long &m, int &e) {
    const Mant h = mant_of(x.hi);
    e = h.e - 1023;
    m = h.m + (unsigned long long)__double2ll_rn(scalb2(x.lo, 63 - e));
    if (!(m >> 63)) m = h.m;                                   // (the low part crossed a power of 2)
}

// One thread per item: its output position and scalar outputs, and for an
// eigenpair the fast path solved what its column needs -- the scale 1/||x|| (and
// the second matrix's) as significand and exponent, lambda's tail.  The other
// items' columns are listed for k_vectors.
template <Kind VK, class Src>
__global__ void __launch_bounds__(64) k_fout(const __grid_constant__ Src src) {
    after_previous();
    int inst = 0, idx = 0;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (!src.item(t, inst, idx)) return;
    const Scratch &S = src.scr(inst);
    const VecArgs &va = src.vec(inst);
    const int ncomp = S.cnt[C_M] + 1;
    const PartRange P = part_range(S);
    const int nk = P.k1 - P.k0;
    if (idx >= nk + P.u1 - P.u0) return;
    const int item = idx < nk ? P.k0 + idx : ncomp + P.u0 + (idx - nk);
    place_item(S, item);
    scalar_item<VK>(va.n, va.key, va.sgn, S, va.out, item);
    if (!va.out.V) return;
    if (item >= ncomp || !S.f.p || S.f.st[item] != FST_DONE) {
        src.push_col(inst, item);
        return;
    }
    const int k = item, es = fast_scale<VK>(S);
    // the norm is sqrt(f') but for the DPR1, whose vector (without the
    // arrowhead's corner) has ||x||^2 = f' / (|rho| (lambda - p_last))
    dd nrm = {S.f.N[k], S.f.Nlo[k]};
    if (VK == KIND_DPR1) {
        const dd sg = fast_sigma<VK>(S, k, es);
        const dd pl = {S.prm[P_PLAST] * pow2(es), 0.0};
        const dd x = dd_add(dd_add(sg, dd_neg(pl)), dd{S.f.mu[k], S.f.mulo[k]});
        nrm = dd_div(nrm, dd_mul_d(x, fabs(va.alpha) * pow2(es)));   // (va.alpha is rho; u is
    }                                                                //  not scaled)
    // scaled multipliers: spikes and poles both scale by 2^es (DPR1: see nrm)
    const dd inv = dd_rsqrt(nrm);
    scale_of(inv, S.f.cm[k], S.f.ce[k]);
    if (VK != KIND_DPR1) {
        S.f.ce[k] += es;
        // the last component
        const int pos = out_pos<VK>(S, va.n, va.sgn, k);
        double *col = va.out.V + (size_t)pos * va.out.ldv;
        double *ucol = va.out.U ? va.out.U + (size_t)pos * va.out.ldu : nullptr;
        const double vn = -inv.hi;
        if (VK == KIND_HERM) {
            col[2 * va.n1] = vn;
            col[2 * va.n1 + 1] = 0.0;
        } else {
            col[va.n1] = vn;
            if (VK == KIND_TSVD && ucol) ucol[va.n1] = va.alpha * vn / sv_of(S, k);
            if (VK == KIND_NSYM && ucol) ucol[va.n1] = vn;
        }
    }
    if (VK == KIND_TSVD) {
        scale_of(dd_mul_d(inv, sv_of(S, k)), S.f.cm2[k], S.f.ce2[k]);
        S.f.ce2[k] += es;
    }
    // lambda's own tail, as an integer of 2^-30 last places of lambda
    const double lhi = S.f.lhi[k];
    if (S.cnt[C_M] >= kFarFrom) {
        // its offset from the group's middle, in 2^(e - 64) (s1 is free by now)
        const GroupData &G = S.f.grp[k / kGroup];
        if (G.r8 < 1e300) {
            const dd x = two_sum(lhi, -G.c);
            const double u = pow2(64 - G.e);
            S.f.s1[k] = __double2ll_rn(x.hi * u) + __double2ll_rn((x.lo + S.f.llo[k]) * u);
        }
    }
    S.f.l32[k] = fabs(lhi) < 2.5
                     ? (int)rint(S.f.llo[k] * pow2(min(1075 - (int)bexp(lhi) + 30, 1023)))
                     : 0;
}

// Columns of the eigenpairs the fast path solved: a CTA has a group of 32 of
// them and a segment of the rows (blockIdx.y), a warp 32 rows at a time, a lane
// one row for all columns (few rows: the warps share the columns out).
// Component a_r / ((d_r - sigma) - mu) / ||x||, for the second matrix (SVD: U,
// NSYM: Y) or the imaginary part (HERM) with its own multiplier.
// Rows whose poles are far from the group's middle c (|p - c| >= 8 r, a warp's 32
// rows all): the significand of p - c, formed once a row, less lambda - c shifted
// to its place is the difference to 2^-62 with no FP64 operation, and its
// reciprocal starts from an FP32 one: ~70 instructions an entry.  Other rows: the
// difference is fl(d_r - lambda) with lambda's tail taken into its reciprocal
// (SVD, whose poles d^2 are no doubles: the exact tail), ~115 an entry.  Either
// way a component's error is that of one subtraction and one rounding.
// Bound by issue slots and the wide multiplies' pipe (59 % and 53 % busy).  All
// entries by ~115 instructions -> now: DPR1 n = 8192 331 -> 214 us, graded n =
// 16384 1223 -> 787 us (2.7 TB/s written), a whole batch of 512 8.5 -> 7.0 ms (both
// sides in one run of the whole step; the columns alone had read 307 and 1130 us).
// rows a CTA takes at least: few rows are split further, for latency
__host__ __device__ constexpr int col_rows(int n1) { return n1 < kFarFrom ? 32 : 128; }

template <Kind VK, class Src>
__global__ void __launch_bounds__(256, 3) k_fcols(const __grid_constant__ Src src) {
    after_previous();
    constexpr bool CPLX = VK == KIND_HERM;
    constexpr bool TWO = VK == KIND_HERM || VK == KIND_NSYM || VK == KIND_TSVD;
    constexpr bool SVD = VK == KIND_TSVD;
    __shared__ ulonglong2 sA[2][kGroup];       // +-(lambda - c), scale
    struct alignas(16) Out { double *v; int e, pad; };
    __shared__ Out so[kGroup];                 // column, scale's exponent
    __shared__ double *su[TWO && !CPLX ? kGroup : 1];
    __shared__ double sl[kGroup];
    __shared__ int4 sd[kGroup];                // diff_range, l32
    __shared__ int se2[SVD ? kGroup : 1];
    __shared__ unsigned long long sm2[SVD ? kGroup : 1], sL[SVD ? kGroup : 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inst, first;
    if (!src.unit(blockIdx.x, kGroup, inst, first)) return;
    const Scratch &S = src.scr(inst);
    const VecArgs &va = src.vec(inst);
    const PartRange P = part_range(S);
    const int kf = (P.k0 & ~(kGroup - 1)) + first;
    if (!va.out.V || kf >= P.k1) return;
    // every warp looks at the columns, the first prepares them
    const int kl = kf + lane;
    const bool act = kl >= P.k0 && kl < P.k1 && S.f.st[kl] == FST_DONE;
    const unsigned cols = __ballot_sync(FULL, act);
    if (!cols) return;
    const int n1 = va.n1, m = S.cnt[C_M], es = fast_scale<VK>(S);
    const GroupData &G = S.f.grp[kf / kGroup];
    const bool groups = m >= kFarFrom && G.r8 < 1e300;
    // (the outermost eigenvalues are in no group)
    const unsigned fcol = __ballot_sync(FULL, groups && act && kl > 0 && kl < m);
    if (wid == 0 && act) {
        const int k = kl;
        const double lhi = S.f.lhi[k];
        DiffRange dr = diff_range(lhi);
        if (!SVD) {
            dr = {dr.lo0, 4096u, dr.lo0, dr.tails};        // (no unit to mind)
        } else if (dr.tails) {
            // (the rows carry the unit 2^-106 alone)
            const unsigned lo = max(dr.lo0, kFixMinExp);
            dr = {lo, 1025u - lo, dr.lo0, dr.tails};
        }
        sl[lane] = lhi;
        sd[lane] = make_int4((int)dr.lo, (int)dr.span, dr.tails, S.f.l32[k]);
        const unsigned long long t = groups ? (unsigned long long)S.f.s1[k] : 0ull;
        sA[0][lane] = make_ulonglong2(t, S.f.cm[k]);
        sA[1][lane] = make_ulonglong2(0ull - t, S.f.cm[k]);
        if (SVD) {
            sL[lane] = S.f.lmod[k];
            sm2[lane] = S.f.cm2[k];
            se2[lane] = S.f.ce2[k] + 1023;
        }
        const int pos = out_pos<VK>(S, va.n, va.sgn, k);
        double *col = va.out.V + (size_t)pos * va.out.ldv;
        double *ucol = (TWO && !CPLX && va.out.U) ? va.out.U + (size_t)pos * va.out.ldu : nullptr;
        so[lane] = Out{col, S.f.ce[k] + 1023, 0};
        if (TWO && !CPLX) su[lane] = ucol;
    }
    // the range of the scales' exponents
    const int ce = act ? S.f.ce[kl] + 1023 : 1023, ce2 = SVD && act ? S.f.ce2[kl] + 1023 : ce;
    const int emin = __reduce_min_sync(FULL, min(ce, ce2)), emax = __reduce_max_sync(FULL, max(ce, ce2));
    __syncthreads();
    const unsigned vsg = (VK == KIND_DPR1 && va.sgn < 0.0) ? 0x80000000u : 0u;
    const double one = unit_reg();
    // this segment's rows, whole tiles
    const int tile = col_rows(n1), all_tiles = (n1 + tile - 1) / tile;
    const int r0 = (int)((long long)blockIdx.y * all_tiles / gridDim.y) * tile;
    const int r1 = min((int)((long long)(blockIdx.y + 1) * all_tiles / gridDim.y) * tile, n1);
    const int nch = (r1 - r0 + 31) / 32;
    const int parts = nch >= 5 ? 1 : nch >= 3 ? 2 : nch == 2 ? 4 : 8;
    const int per = kGroup / parts, x0 = (wid % parts) * per;
    const unsigned mine = (per == 32 ? ~0u : ((1u << per) - 1u) << x0) & cols;
    for (int ch = wid / parts; ch < nch; ch += 8 / parts) {
        const int r = r0 + ch * 32 + lane;
        const bool in = r < r1;
        double p = 4.0;
        unsigned long long rP = 0;
        Mant la = {0, -8192}, lb = {0, -8192};
        if (in) {
            p = S.f.rp[r];
            if (SVD) rP = S.f.rP[r];
            if (CPLX) {
                la = mant_of(va.z[2 * r]);
                lb = mant_of(va.z[2 * r + 1]);
            } else if (VK == KIND_NSYM) {
                la = mant_of(va.z[r]);
                lb = mant_of(va.zrow[r]);
            } else if (SVD) {
                la = mant_of(va.spk[r]);
                lb = mant_of(va.z[r]);                 // u_r = s v_r / d_r, spike d_r z_r
            } else {
                la = mant_of(va.spk[r]);
            }
        }
        const int e1 = (int)(short)(la.e & 0xffff), e2 = (int)(short)(lb.e & 0xffff);
        // the entry of column x from the reciprocal R (2^63 / significand) of a
        // difference with biased exponent ed and sign bit dsg
        auto put = [&](auto chk, int x, unsigned long long cm, unsigned long long R, int ed,
                       unsigned dsg) {
            constexpr bool C = decltype(chk)::value;
            const unsigned long long Gp = mul_hi3(cm, R);
            const Out o = so[x];
            const double v = pack_prod<C>(la.m, Gp, (e1 - ed) + o.e,
                                          ((unsigned)(la.e ^ dsg) & 0x80000000u) ^ vsg);
            if (CPLX) {
                const double vi = pack_prod<C>(lb.m, Gp, (e2 - ed) + o.e,
                                               (unsigned)(lb.e ^ dsg) & 0x80000000u);
                if (in) {
                    o.v[2 * r] = v;
                    o.v[2 * r + 1] = vi;
                }
            } else {
                if (in) o.v[r] = v;
                if (TWO && su[x]) {
                    const unsigned long long G2 = SVD ? mul_hi3(sm2[x], R) : Gp;
                    const double vu = pack_prod<C>(lb.m, G2, (e2 - ed) + (SVD ? se2[x] : o.e),
                                                   (unsigned)(lb.e ^ dsg) & 0x80000000u);
                    if (in) su[x][r] = vu;
                }
            }
        };
        unsigned far = 0;
        if (groups) {
            dd D = two_sum(p, -G.c);
            if (SVD && in) D = near_diff(fast_pole<VK>(va.key[r], es), dd{G.c, 0.0}, dd{0.0, 0.0});
            if (__all_sync(FULL, fabs(D.hi) >= G.r8)) {
                far = fcol & mine;
                // |p - c| in 2^(e0 - 62)
                const int e0 = (int)bexp(D.hi);
                const unsigned long long b = (unsigned long long)__double_as_longlong(D.hi);
                const unsigned long long Dm =
                    (((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10) +
                    (unsigned long long)__double2ll_rd((D.hi < 0.0 ? -D.lo : D.lo) *
                                                       pow2(10 + 1075 - e0));
                const int sh = min(e0 - 1023 - G.e + 2, 63);
                const unsigned dsg = (unsigned)(b >> 32);
                const ulonglong2 *A = sA[dsg >> 31];
                auto entry = [&](auto chk, int x) {
                    const ulonglong2 a = A[x];
                    const unsigned long long M =
                        Dm - (unsigned long long)((long long)a.x >> sh);
                    const float y = fmaf(rcp_f32((float)(unsigned)(M >> 32)), 0x1p30f, 2.f);
                    put(chk, x, a.y, recip62(M, __float_as_uint(y) - 0x40000000u), e0 - 1, dsg);
                };
                // all of this warp's columns, no result near the ends of the range
                const int lo = min(e1, TWO ? e2 : e1) - e0 + emin,
                          hi = max(e1, TWO ? e2 : e1) - e0 + emax;
                if (far == (per == 32 ? ~0u : ((1u << per) - 1u) << x0) &&
                    __all_sync(FULL, (lo > 8 && hi < 2030) || !in)) {
#pragma unroll 4
                    for (int x = x0; x < x0 + per; ++x) entry(std::false_type{}, x);
                } else {
                    for (unsigned left = far; left; left &= left - 1)
                        entry(std::true_type{}, __ffs(left) - 1);
                }
            }
        }
        for (unsigned left = mine & ~far; left; left &= left - 1) {
            const int x = __ffs(left) - 1;
            const double lhi = sl[x];
            const int4 q = sd[x];
            double D = fma(p, one, -lhi);              // (an FMA: 2.0 lanes a clock, DADD 1.7)
            int tl;
            unsigned dh = hi32(D), dl = (unsigned)__double2loint(D);
            unsigned ed = (dh << 1) >> 21;
            if (ed - (unsigned)q.x >= (unsigned)q.y && in) {
                const int k = kf + x;
                const dd pr = fast_pole<VK>(va.key[r], es);
                const dd Dd =
                    near_diff(pr, fast_sigma<VK>(S, k, es), dd{S.f.mu[k], S.f.mulo[k]});
                D = Dd.hi;
                tl = near_tail(Dd);
                dh = hi32(D);
                dl = (unsigned)__double2loint(D);
                ed = (dh << 1) >> 21;
            } else {
                // -lambda's tail for p above, + below, in 2^-7 of D's last place
                tl = SVD ? tail_of(rP - sL[x], dh, dl, ed) & q.z
                         : sar32(q.w ^ ~((int)dh >> 31), ed - ((int)bexp(lhi) - 23));
            }
            const unsigned seed = hi32(rcp_seed(__hiloint2double(
                (int)((dh & 0xfffffu) | 0x3ff00000u), 0)));
            put(std::true_type{}, x, sA[0][x].y, recip63<false>(dh, dl, tl, seed), (int)ed, dh);
        }
    }
}

// The columns k_fcols does not write -- those of deflated rows and of eigenpairs the
// FP64 solver took.  A CTA each, staged in a slice of stored pairs, so that V, which
// may lie in host memory, is written once (arrow_eig_host, n = 4097, spikes over 20
// decades: 6.3 -> 5.2 ms).  Fewer rows: a warp each; CTAs then wait on their barriers
// (300 instances of n = 100 to 800, all columns here: 20.1 ms by CTAs, 18.6 with this
// line at 256 rows, 18.1 at 512, 17.1 at 1024, where one column of n = 1000 takes
// 25 us longer; 10000 of n = 2: 1.83 -> 1.60 ms).
constexpr int kWarpCols = 512;

template <Kind VK, class Src>
__global__ void __launch_bounds__(256) k_vectors(const __grid_constant__ Src src) {
    after_previous();
    __shared__ double red[16];
    const int cnt = src.col_count();
    for (int w = blockIdx.x; w < cnt; w += gridDim.x) {
        const int2 ik = src.col_at(w);
        const VecArgs &va = src.vec(ik.x);
        if (va.n1 < kWarpCols) continue;
        vector_item<VK>(va.n, va.n1, va.key, va.spk, va.z, va.zrow, va.alpha, va.sgn,
                        src.scr(ik.x), va.out, ik.y, CtaTeam<8>{(int)threadIdx.x, red, 0},
                        (double *)src.slice(blockIdx.x));
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    for (int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < cnt; w += 8 * gridDim.x) {
        const int2 ik = src.col_at(w);
        const VecArgs &va = src.vec(ik.x);
        if (va.n1 < kWarpCols)
            vector_item<VK>(va.n, va.n1, va.key, va.spk, va.z, va.zrow, va.alpha, va.sgn,
                            src.scr(ik.x), va.out, ik.y, WarpTeam{lane});
        __syncwarp();
    }
}

}  // namespace ae
