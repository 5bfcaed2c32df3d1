// ae_prep.cuh -- checks, order, reduction (Sec. 1) and the arrowhead's data in the
// forms the solver reads, for one instance: as grid kernels over its rows
// (ae_arrow.cu, larger orders), or by one CTA of 1024 threads (prep_block: small
// orders and each instance of a batch).  Both give the same bits: sums are
// taken per chunk of 256 poles, the chunks' sums in a fixed order.
#pragma once
#include "ae_fast.cuh"
#include "ae_pipeline.cuh"

namespace ae {

constexpr int kChunk = 256;        // poles a partial sum covers

// what the caller passed in
struct PrepArgs {
    int n1;
    const double *d, *z, *zrow;
    double alpha, rho, sgn;        // (sgn: -1 for a DPR1 with rho < 0, solved as -M)
};

// Row r: its key and spike as the reduction sees them, and CF_* flags.
// ARROW: key d, spike z.  DPR1: key sgn d, spike u (0 for rho = 0: every row
// deflates).  SVD: key d (> 0 required), spike d z.  HERM: spike |zeta_r| of the
// complex (z[2r], z[2r+1]).  NSYM: spike sqrt(zc_r zr_r) of the pair (z[r],
// zrow[r]), which must share a sign or both be zero (the Remark of Sec. 6.1).
template <Kind K>
__device__ __forceinline__ int check_item(const PrepArgs &A, const Scratch &S, int r) {
    int flags = 0;
    const double dr = A.d[r];
    const double zr = K == KIND_HERM ? A.z[2 * r] : A.z[r];
    if (!isfinite(dr) || !isfinite(zr)) flags |= CF_BAD;
    double key = dr, spk = zr;
    if (K == KIND_DPR1) {
        key = A.sgn * dr;
        S.key[r] = key;
        if (A.rho == 0.0) S.spk[r] = spk = 0.0;
    } else if (K == KIND_TSVD) {
        if (!(dr > 0.0)) flags |= CF_BAD;
        S.spk[r] = spk = dr * zr;
    } else if (K == KIND_HERM) {
        const double zi = A.z[2 * r + 1];
        if (!isfinite(zi)) flags |= CF_BAD;
        S.spk[r] = spk = hypot(zr, zi);
    } else if (K == KIND_NSYM) {
        const double zw = A.zrow[r];
        if (!isfinite(zw)) flags |= CF_BAD;
        if ((zr == 0.0) != (zw == 0.0) || (zr != 0.0 && (zr > 0.0) != (zw > 0.0)))
            flags |= CF_BAD;
        S.spk[r] = spk = sqrt(fabs(zr)) * sqrt(fabs(zw));
    }
    if (spk == 0.0) flags |= CF_ZERO;
    if (key == 0.0) flags |= CF_ZEROPOLE;
    if (r + 1 < A.n1) {
        const double kn = K == KIND_DPR1 ? A.sgn * A.d[r + 1] : A.d[r + 1];
        if (!(key > kn)) flags |= CF_UNSORTED;
    }
    return flags;
}

// A key as an integer of the same order; NaN as -inf, so that ranks always form
// a permutation (the input is rejected later, but no index may leave its array
// meanwhile).  Integer comparisons: an FP64 one costs the FP64 pipe 16 clocks a
// warp (ranks of 6000 rows: 890 us with them).
__device__ __forceinline__ unsigned long long order_key(double x) {
    if (isnan(x)) x = -INFINITY;
    const unsigned long long b = (unsigned long long)__double_as_longlong(x + 0.0);   // (-0 as 0)
    return b >> 63 ? ~b : b | 0x8000000000000000ull;
}

// A row of an input that is sorted and has no zero spikes: it is its own pole.
__device__ __forceinline__ void identity_row(const Scratch &S, const double *key,
                                             const double *spk, int r) {
    const double d = key[r], a = fabs(spk[r]), a2 = a * a;
    S.perm[r] = r;
    S.spos[r] = r;
    S.pd[r] = S.pv[r] = d;
    S.pz[r] = a;
    S.pz2[r] = a2;
    S.pz2lo[r] = fma(a, a, -a2);
    S.prow[r] = r;
    S.kind[r] = 0;
}

// Sorted position s: whether its row is the head of a run of equal poles (the
// first with a nonzero spike).
__device__ __forceinline__ bool is_head(const double *key, const double *spk, const int *perm,
                                        int s) {
    const int r = perm[s];
    const double dr = key[r];
    if (spk[r] == 0.0) return false;
    for (int q = s - 1; q >= 0; --q) {
        const int rq = perm[q];
        if (key[rq] != dr) break;
        if (spk[rq] != 0.0) return false;
    }
    return true;
}

// Sorted position s as reduced pole jk (head) or deflated row jd.
__device__ __forceinline__ void reduce_item(const Scratch &S, const double *key,
                                            const double *spk, int n1, int s, bool head, int jk,
                                            int jd) {
    const int *perm = S.perm;
    const int r = perm[s];
    const double dr = key[r], zr = spk[r];
    S.spos[r] = s;
    if (head) {
        // reduced spike: sqrt of the sum of squares over the run
        double acc = fabs(zr);
        for (int q = s + 1; q < n1; ++q) {
            const int rq = perm[q];
            if (key[rq] != dr) break;
            acc = hypot(acc, spk[rq]);
        }
        S.pd[jk] = dr;
        S.pv[jk] = dr;
        S.pz[jk] = acc;
        const double a2 = acc * acc;
        S.pz2[jk] = a2;
        S.pz2lo[jk] = fma(acc, acc, -a2);
        S.prow[jk] = r;
        S.kind[r] = 0;
        return;
    }
    S.kind[r] = zr == 0.0 ? 1 : 2;
    S.drow[jd] = r;
    S.dval[jd] = dr;
    if (zr != 0.0) {
        // Helmert-type vector data: R_{m-1} over earlier nonzero members of the
        // run, R_m including this row
        double Rm1 = 0.0;
        int q = s - 1;
        for (; q >= 0; --q) {
            const int rq = perm[q];
            if (key[rq] != dr) break;
            Rm1 = hypot(Rm1, spk[rq]);
        }
        S.run_s0[r] = q + 1;
        S.run_R[2 * r] = Rm1;
        S.run_R[2 * r + 1] = hypot(Rm1, zr);
    }
}

// Poles of the arrowhead behind m0 reduced ones: a DPR1's arrowhead has one less
// (m0 - 1 = -1: nothing to solve).
template <Kind K>
__device__ __forceinline__ int arrow_poles(int m0) {
    return K == KIND_DPR1 ? m0 - 1 : m0;
}

// Kind-specific data of reduced pole j of m0 (and row j); its share of the sums:
// w for the corner, zeta, |pole| and zeta^2 for the scales.
// DPR1 (Sec. 6.3): the arrowhead L^{-1} M L has poles p_0..p_{m0-2}, spikes
// zeta_j = u'_j sqrt(rho (p_j - p_last)) and corner p_last + rho u'^T u'.
// SVD (Sec. 6.2): B^T B has poles d_j^2, spikes d_j z_j, corner alpha^2 + z^T z
// (over all rows; runs of equal d keep their folded spike).
// HERM, NSYM: |zeta|^2 = re^2 + im^2 (Sec. 6.1), resp. zc zr (its Remark),
// exactly, as the paper asks for the moduli in doubled precision.
struct PoleShare {
    dd w;
    double z;
    unsigned long long d, z2;      // bits of nonnegative doubles
};
template <Kind K>
__device__ __forceinline__ PoleShare kind_item(const PrepArgs &A, const Scratch &S, int m0,
                                               int j) {
    PoleShare r = {{0.0, 0.0}, 0.0, 0ull, 0ull};
    const int m = arrow_poles<K>(m0);
    if (K == KIND_DPR1) {
        if (j < m0) r.w = two_prod(S.pz[j], S.pz[j]);
        if (j < m) {
            const dd z2 = dd_mul(dd_mul_d(r.w, fabs(A.rho)), two_sum(S.pd[j], -S.pd[m0 - 1]));
            S.pz2[j] = z2.hi;
            S.pz2lo[j] = z2.lo;
            S.pz[j] = dd_sqrt(z2).hi;
        }
    } else if (K == KIND_TSVD) {
        if (j < A.n1) r.w = two_prod(A.z[j], A.z[j]);
        if (j < m) {
            const double dj = S.pd[j];
            S.pv[j] = dj * dj;
            const int row = S.prow[j];
            // a single-row pole: (d_j z_j)^2 exactly in double-double
            if ((j + 1 == m || S.pd[j + 1] != dj) && S.pz[j] == fabs(S.spk[row])) {
                const dd dz = two_prod(dj, A.z[row]);
                const dd z2 = dd_mul(dz, dz);
                S.pz2[j] = z2.hi;
                S.pz2lo[j] = z2.lo;
            }
        }
        if (j < S.cnt[C_ND]) S.dval[j] = S.dval[j] * S.dval[j];
    } else if (K == KIND_HERM || K == KIND_NSYM) {
        if (j < m) {
            const int row = S.prow[j];
            if (S.pz[j] == S.spk[row]) {             // no other row was folded in
                const dd z2 = K == KIND_HERM ? dd_add(two_prod(A.z[2 * row], A.z[2 * row]),
                                                      two_prod(A.z[2 * row + 1], A.z[2 * row + 1]))
                                             : two_prod(A.z[row], A.zrow[row]);
                S.pz2[j] = z2.hi;
                S.pz2lo[j] = z2.lo;
                S.pz[j] = dd_sqrt(z2).hi;
            }
        }
    }
    if (j < m) {
        r.z = S.pz[j];
        r.d = (unsigned long long)__double_as_longlong(fabs(S.pd[j]));
        r.z2 = (unsigned long long)__double_as_longlong(S.pz2[j]);
    }
    return r;
}

__device__ __forceinline__ unsigned long long max64(unsigned long long a, unsigned long long b) {
    return a > b ? a : b;
}
// (the corner's sum for the kinds that have one: ~100 dependent FP64 operations)
template <Kind K>
constexpr bool kCorner = K == KIND_DPR1 || K == KIND_TSVD;
template <Kind K>
__device__ __forceinline__ PoleShare warp_share(PoleShare v) {
    if (kCorner<K>) v.w = warp_sum_dd(v.w);
    v.z = warp_sum(v.z);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.d = max64(v.d, __shfl_xor_sync(FULL, v.d, o));
        v.z2 = max64(v.z2, __shfl_xor_sync(FULL, v.z2, o));
    }
    return v;
}
template <Kind K>
__device__ __forceinline__ PoleShare add_share(PoleShare a, const PoleShare &b) {
    if (kCorner<K>) a.w = dd_add(a.w, b.w);
    a.z += b.z;
    a.d = max64(a.d, b.d);
    a.z2 = max64(a.z2, b.z2);
    return a;
}

// The shares of chunk `blk` (256 poles) by the 256 threads of `grp` (t their
// index, sh 8 slots of theirs, bar their barrier), kept in the eigenpair arrays
// until prep_finish reads them.
template <Kind K>
__device__ __forceinline__ void kind_chunk(const PrepArgs &A, const Scratch &S, int m0, int blk,
                                           int t, PoleShare *sh, int bar) {
    PoleShare v = warp_share<K>(kind_item<K>(A, S, m0, blk * kChunk + t));
    if ((t & 31) == 0) sh[t >> 5] = v;
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(kChunk) : "memory");
    if (t == 0) {
        for (int w = 1; w < kChunk / 32; ++w) v = add_share<K>(v, sh[w]);
        S.es_sigma[blk] = v.w.hi;
        S.es_mu[blk] = v.w.lo;
        S.es_lam[blk] = v.z;
        S.es_b[blk] = __longlong_as_double((long long)v.d);
        S.es_Kb[blk] = __longlong_as_double((long long)v.z2);
    }
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(kChunk) : "memory");
}

// The chunks' shares added up by one warp: corner, scales, number of poles.
template <Kind K>
__device__ __forceinline__ void prep_finish(const PrepArgs &A, const Scratch &S, int lane) {
    const int m0 = S.cnt[C_M];
    const int chunks = ((K == KIND_TSVD ? A.n1 : m0) + kChunk - 1) / kChunk;
    PoleShare v = {{0.0, 0.0}, 0.0, 0ull, 0ull};
    for (int b = lane; b < chunks; b += 32)
        v = add_share<K>(v, PoleShare{{S.es_sigma[b], S.es_mu[b]},
                                   S.es_lam[b],
                                   (unsigned long long)__double_as_longlong(S.es_b[b]),
                                   (unsigned long long)__double_as_longlong(S.es_Kb[b])});
    v = warp_share<K>(v);
    if (lane != 0) return;
    dd al = {A.alpha, 0.0};
    if (K == KIND_DPR1) {
        const double plast = m0 > 0 ? S.pd[m0 - 1] : 0.0;
        al = dd_add(dd{plast, 0.0}, dd_mul_d(v.w, fabs(A.rho)));
        S.prm[P_PLAST] = plast;
    } else if (K == KIND_TSVD) {
        al = dd_add(two_prod(A.alpha, A.alpha), v.w);
    }
    S.cnt[C_M] = arrow_poles<K>(m0);
    S.prm[P_ALPHA_HI] = al.hi;
    S.prm[P_ALPHA_LO] = al.lo;
    // Algorithm 5's spike ratio needs sum_j |zeta_j| over the reduced poles
    S.prm[P_ZSUM] = v.z;
    // FP32 copies: keys and spike^2 scaled by powers of two so that the
    // largest of each is O(1)
    const double mxd = __longlong_as_double((long long)v.d),
                 mxz = __longlong_as_double((long long)v.z2);
    S.prm[P_DS] = (mxd > 0.0 && isfinite(mxd)) ? pow2_or(-ilogb(mxd)) : 1.0;
    S.prm[P_ZS] = (mxz > 0.0 && isfinite(mxz)) ? pow2_or(-ilogb(mxz)) : 1.0;
}

// Pole / row t in the forms the passes read: FP32 copies, then fixed point.
template <Kind K>
__device__ __forceinline__ void forms_item(const Scratch &S, const VecArgs &va, int t) {
    if (t < S.cnt[C_M]) {
        const double v = S.pd[t] * S.prm[P_DS];
        const float h = (float)v;
        S.pdh[t] = h;
        S.pdl[t] = (float)(v - (double)h);
        S.pz2f[t] = (float)(S.pz2[t] * S.prm[P_ZS]);
    }
    if (S.f.p) fprep_item<K>(S, va, t);
}

// All of it by one CTA of 1024 threads.
template <Kind K>
__device__ __forceinline__ void prep_block(const PrepArgs &A, const Scratch &S,
                                           const VecArgs &va) {
    __shared__ unsigned long long tile[1024];
    __shared__ PoleShare sh[4][kChunk / 32];
    __shared__ int sflags, wt[33];
    const int n1 = A.n1;
    if (threadIdx.x < C_COUNT) S.cnt[threadIdx.x] = 0;
    if (threadIdx.x < C64_COUNT) S.cnt64[threadIdx.x] = 0ull;
    if (threadIdx.x == 0) sflags = 0;
    __syncthreads();
    int flags = 0;
    for (int r = threadIdx.x; r < n1; r += 1024) flags |= check_item<K>(A, S, r);
    flags = __reduce_or_sync(FULL, flags);
    if ((threadIdx.x & 31) == 0 && flags) atomicOr(&sflags, flags);
    __syncthreads();
    flags = sflags;
    if (threadIdx.x == 0) S.cnt[C_FLAGS] = flags;
    const double *key = va.key, *spk = va.spk;
    if (!(flags & (CF_UNSORTED | CF_ZERO))) {
        for (int r = threadIdx.x; r < n1; r += 1024) identity_row(S, key, spk, r);
        if (threadIdx.x == 0) {
            S.cnt[C_M] = n1;
            S.cnt[C_ND] = 0;
        }
    } else {
        // order: identity when sorted, else ranks counted against tiles of the keys
        for (int rb = 0; rb < n1; rb += 1024) {
            const int r = rb + threadIdx.x;
            if (!(flags & CF_UNSORTED)) {
                if (r < n1) S.perm[r] = r;
                continue;
            }
            const unsigned long long kr = r < n1 ? order_key(key[r]) : 0ull;
            int rank = 0;
            for (int base = 0; base < n1; base += 1024) {
                __syncthreads();
                if (base + (int)threadIdx.x < n1)
                    tile[threadIdx.x] = order_key(key[base + threadIdx.x]);
                __syncthreads();
                const int lim = min(1024, n1 - base);
                for (int t = 0; t < lim; ++t) {
                    const unsigned long long q = tile[t];
                    rank += (q > kr) || (q == kr && base + t < r);
                }
            }
            if (r < n1) S.perm[rank] = r;
        }
        __syncthreads();
        int carry_keep = 0, carry_defl = 0;
        for (int base = 0; base < n1; base += 1024) {
            const int s = base + threadIdx.x;
            const bool in = s < n1, head = in && is_head(key, spk, S.perm, s);
            int tk, td;
            const int jk = block_exscan(head ? 1 : 0, wt, tk) + carry_keep;
            const int jd = block_exscan(in && !head ? 1 : 0, wt, td) + carry_defl;
            if (in) reduce_item(S, key, spk, n1, s, head, jk, jd);
            carry_keep += tk;
            carry_defl += td;
        }
        if (threadIdx.x == 0) {
            S.cnt[C_M] = carry_keep;
            S.cnt[C_ND] = carry_defl;
        }
    }
    __syncthreads();
    const int m0 = S.cnt[C_M];
    const int chunks = ((K == KIND_TSVD ? n1 : m0) + kChunk - 1) / kChunk;
    const int grp = threadIdx.x / kChunk;
    for (int b = grp; b < chunks; b += 4)
        kind_chunk<K>(A, S, m0, b, threadIdx.x % kChunk, sh[grp], 1 + grp);
    __syncthreads();
    if (threadIdx.x < 32) prep_finish<K>(A, S, threadIdx.x);
    __syncthreads();
    for (int t = threadIdx.x; t < n1; t += 1024) forms_item<K>(S, va, t);
}

}  // namespace ae
