// ae_batch.cu -- many arrowheads of uneven order solved together.
//
// All instances go through the same pipeline as arrow_eig, but each stage is
// ONE launch over every instance:
//   k_batch_prep      one CTA per instance: checks, order, reduction, FP32 and
//                     fixed-point copies
//   k_fgroup, k_fopen, k_feval, k_fstep, k_fmore, k_fold, k_ffix, k_fcols
//                     (ae_fast.cuh) on units of 32, 8 or 1 eigenpairs of one
//                     instance (SrcMany)
//   k_batch_eig       the FP64 solver instead, for options the fixed-point path
//                     does not serve: global work queue of (instance, eigenpair)
//                     units; a unit is 32/W eigenpairs of one instance solved by
//                     W-lane teams (W = 8, 16 or 32, chosen per order bucket by
//                     the tuner)
//   k_batch_fix_*     remedy decisions over all eigenpairs, a warp per FP64 remedy
//   k_fout, k_fcols, k_vectors, k_batch_status
// A plan (ae_batch_create) owns the descriptor table and the scratch of every
// instance and captures the whole sequence in a CUDA graph that
// ae_batch_run replays.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <sys/stat.h>

#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "ae_fast.cuh"
#include "ae_pipeline.cuh"
#include "ae_prep.cuh"

namespace ae {

// ---------------------------------------------------------------------------
// sub-warp teams: W consecutive lanes of a warp share one eigenpair
// ---------------------------------------------------------------------------
template <int W>
struct SubWarpTeam {
    int rank;        // lane within the team
    unsigned mask;   // the team's lanes
    static constexpr int size = W;
    __device__ __forceinline__ double sum(double v) const {
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
        return v;
    }
    __device__ __forceinline__ float sumf(float v) const {
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
        return v;
    }
    __device__ __forceinline__ dd sum(dd v) const {
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) {
            dd w = {__shfl_xor_sync(mask, v.hi, o), __shfl_xor_sync(mask, v.lo, o)};
            v = dd_add(v, w);
        }
        return v;
    }
    __device__ __forceinline__ double max(double v) const {
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(mask, v, o));
        return v;
    }
    __device__ __forceinline__ double min(double v) const {
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(mask, v, o));
        return v;
    }
    __device__ __forceinline__ void sync() const { __syncwarp(mask); }
};

struct BatchInst {
    int n, n1;
    const double *d, *z, *alpha;   // device inputs of this instance
    Scratch S;
    VecArgs va;                    // (alpha is read from the device, not from here)
    int team;                      // eigenpair team width W
};

struct BatchCtl {
    int tick_eig, tick_fix, nfix, nold, tick_old[2], nmore[2], ncol;
};

// index i with off[i] <= t < off[i+1]
__device__ __forceinline__ int find_inst(const long long *off, int count, long long t) {
    int lo = 0, hi = count;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

// the instances of a batch, for the kernels of ae_fast.cuh
struct SrcMany {
    const BatchInst *__restrict__ I;
    int count;
    const long long *__restrict__ eoff, *__restrict__ off8, *__restrict__ off32;
    BatchCtl *ctl;
    int2 *old, *fix, *more;
    double2 *wbuf;
    long long wstride;
    __device__ bool unit(long long u, int per, int &i, int &first) const {
        const long long *off = per == 8 ? off8 : off32;
        if (u >= off[count]) return false;
        i = find_inst(off, count, u);
        first = (int)(u - off[i]) * per;
        return true;
    }
    __device__ bool item(long long t, int &i, int &idx) const {
        if (t >= eoff[count]) return false;
        i = find_inst(eoff, count, t);
        idx = (int)(t - eoff[i]);
        return true;
    }
    __device__ const Scratch &scr(int i) const { return I[i].S; }
    __device__ const VecArgs &vec(int i) const { return I[i].va; }
    __device__ void push_old(int i, int k) const {
        old[atomicAdd(&ctl->nold, 1)] = make_int2(i, k);
    }
    __device__ int old_count() const { return ctl->nold; }
    __device__ int2 old_at(int w) const { return old[w]; }
    __device__ int *old_ticket(int ph) const { return ctl->tick_old + ph; }
    __device__ void push_more(int ph, int i, int k) const {
        more[atomicAdd(&ctl->nmore[ph], 1)] = make_int2(i, k);
    }
    __device__ int more_count(int ph) const { return ctl->nmore[ph]; }
    __device__ int2 more_at(int w) const { return more[w]; }
    // (the remedy list is done with by then)
    __device__ void push_col(int i, int item) const {
        fix[atomicAdd(&ctl->ncol, 1)] = make_int2(i, item);
    }
    __device__ int col_count() const { return ctl->ncol; }
    __device__ int2 col_at(int w) const { return fix[w]; }
    __device__ void push_fix(int i, int k, bool, int) const {
        fix[atomicAdd(&ctl->nfix, 1)] = make_int2(i, k);
    }
    __device__ double2 *slice(long long w) const { return wbuf ? wbuf + w * wstride : nullptr; }
};

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_batch_prep(const BatchInst *__restrict__ I,
                                                     BatchCtl *ctl) {
    const BatchInst &B = I[blockIdx.x];
    if (blockIdx.x == 0 && threadIdx.x == 0) *ctl = BatchCtl{};
    const PrepArgs A{B.n1, B.d, B.z, nullptr, *B.alpha, 0.0, 1.0};
    prep_block<KIND_ARROW>(A, B.S, B.va);
}

// buf: this warp's 4 slices of stored (delta_j, c_j) pairs, `stride` apart
template <int W>
__device__ __forceinline__ void batch_unit(const BatchInst &B, long long unit_in_inst, int lane,
                                           const SolveOpts &o, double2 *buf, long long stride) {
    constexpr int EPW = 32 / W;
    const int m = B.S.cnt[C_M];
    const int g = lane / W;
    const int k = (int)(unit_in_inst * EPW) + g;
    const auto R = PolesOf<KIND_ARROW>::make(B.S, m);
    double2 *tb = buf ? buf + g * stride : nullptr;
    if constexpr (W == 32) {
        if (k <= m) eig_item<KIND_ARROW>(R, WarpTeam{lane}, B.S, k, o, tb);
    } else {
        const unsigned mask = ((1u << W) - 1u) << (lane & ~(W - 1));
        if (k <= m) eig_item<KIND_ARROW>(R, SubWarpTeam<W>{lane & (W - 1), mask}, B.S, k, o, tb);
    }
}

__global__ void __launch_bounds__(256, 3) k_batch_eig(const BatchInst *__restrict__ I, int count,
                                                   const long long *__restrict__ uoff,
                                                   BatchCtl *ctl, SolveOpts o, double2 *wbuf,
                                                   long long wstride, int slices) {
    const int lane = threadIdx.x & 31;
    const long long total = uoff[count];
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    double2 *buf = wbuf ? wbuf + gw * slices * wstride : nullptr;
    for (;;) {
        long long u = 0;
        if (lane == 0) u = atomicAdd(&ctl->tick_eig, 1);
        u = __shfl_sync(FULL, u, 0);
        if (u >= total) break;
        const int i = find_inst(uoff, count, u);
        const BatchInst &B = I[i];
        const long long ui = u - uoff[i];
        switch (B.team) {
            case 8: batch_unit<8>(B, ui, lane, o, buf, wstride); break;
            case 16: batch_unit<16>(B, ui, lane, o, buf, wstride); break;
            default: batch_unit<32>(B, ui, lane, o, buf, wstride); break;
        }
        __syncwarp();
    }
}

__global__ void k_batch_fix_decide(const BatchInst *__restrict__ I, int count,
                                   const long long *__restrict__ eoff, double knu_max) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= eoff[count]) return;
    const int i = find_inst(eoff, count, t);
    fix_decide_item(KIND_ARROW, I[i].S, (int)(t - eoff[i]), knu_max);
}

// One warp per remedied eigenpair that k_ffix left to the FP64 solver.
__global__ void __launch_bounds__(256) k_batch_fix_solve(const BatchInst *__restrict__ I,
                                                         const int2 *fixlist, BatchCtl *ctl,
                                                         SolveOpts o, double2 *wbuf,
                                                         long long wstride, int slices) {
    const int lane = threadIdx.x & 31;
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    double2 *buf = wbuf ? wbuf + gw * slices * wstride : nullptr;
    for (;;) {
        int w = 0;
        if (lane == 0) w = atomicAdd(&ctl->tick_fix, 1);
        w = __shfl_sync(FULL, w, 0);
        if (w >= ctl->nfix) break;
        const int2 ik = fixlist[w];
        const Scratch &S = I[ik.x].S;
        const auto R = PolesOf<KIND_ARROW>::make(S, S.cnt[C_M]);
        fix_solve_item<KIND_ARROW>(R, WarpTeam{lane}, S, ik.y, o, buf);
        __syncwarp();
    }
}

__global__ void k_batch_status(const BatchInst *__restrict__ I, int count, int *status) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const int *c = I[i].S.cnt;
    status[i] = (c[C_FLAGS] & CF_BAD) ? AE_ERR_INPUT : (c[C_CAPPED] ? AE_ERR_NOCONV : AE_OK);
}

// ---------------------------------------------------------------------------
// tuner: eigenpair team width per order bucket, cached as JSON
// ---------------------------------------------------------------------------
static std::mutex g_tune_mu;
static std::map<int, int> g_tune;          // bucket -> W
static bool g_tune_loaded = false;

static const char *build_tag() { return __DATE__ " " __TIME__; }

static int bucket_of(int n) {
    int b = 32;
    while (b < n && b < (1 << 24)) b <<= 1;
    return b;
}

static int default_team(int n) { return n <= 48 ? 8 : (n <= 160 ? 16 : 32); }

static std::string device_key() {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceProp p;
    if (cudaGetDeviceProperties(&p, dev) != cudaSuccess) return "unknown";
    return std::string(p.name) + "|" + build_tag();
}

static std::string cache_path() {
    const char *e = getenv("AE_TUNE_CACHE");
    if (e && *e) return e;
    const char *h = getenv("HOME");
    return std::string(h ? h : "/tmp") + "/.cache/arrowhead_tune.json";
}

// file format: {"key": "<device>|<build>", "team": {"32": 8, "64": 16, ...}}
static void load_cache_locked() {
    if (g_tune_loaded) return;
    g_tune_loaded = true;
    FILE *f = fopen(cache_path().c_str(), "r");
    if (!f) return;
    std::string s;
    char buf[4096];
    size_t k;
    while ((k = fread(buf, 1, sizeof buf, f)) > 0) s.append(buf, k);
    fclose(f);
    const std::string want = "\"key\": \"" + device_key() + "\"";
    if (s.find(want) == std::string::npos) return;   // another device or build
    size_t p = s.find("\"team\"");
    if (p == std::string::npos) return;
    p = s.find('{', p);
    while (p != std::string::npos) {
        const size_t q = s.find('"', p + 1);
        if (q == std::string::npos) break;
        const size_t r = s.find('"', q + 1);
        const size_t c = s.find(':', r);
        if (r == std::string::npos || c == std::string::npos) break;
        const int b = atoi(s.substr(q + 1, r - q - 1).c_str());
        const int w = atoi(s.c_str() + c + 1);
        if (b > 0 && (w == 8 || w == 16 || w == 32)) g_tune[b] = w;
        p = s.find(',', c);
    }
}

static void save_cache_locked() {
    const std::string path = cache_path();
    const size_t slash = path.rfind('/');
    if (slash != std::string::npos) {
        const std::string dir = path.substr(0, slash);
        for (size_t i = 1; i <= dir.size(); ++i)
            if (i == dir.size() || dir[i] == '/') mkdir(dir.substr(0, i).c_str(), 0755);
    }
    FILE *f = fopen(path.c_str(), "w");
    if (!f) return;
    fprintf(f, "{\"key\": \"%s\", \"team\": {", device_key().c_str());
    bool first = true;
    for (auto &kv : g_tune) {
        fprintf(f, "%s\"%d\": %d", first ? "" : ", ", kv.first, kv.second);
        first = false;
    }
    fprintf(f, "}}\n");
    fclose(f);
}

int team_for(int n) {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    load_cache_locked();
    auto it = g_tune.find(bucket_of(n));
    return it != g_tune.end() ? it->second : default_team(n);
}


// ---------------------------------------------------------------------------
// plans
// ---------------------------------------------------------------------------
static int sm_count_b() {
    int dev = 0, c = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
    return c > 0 ? c : 1;
}

static int batch_eig_grid() {
    static int per_sm = 0;
    if (!per_sm) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch_eig, 256, 0);
        if (per_sm <= 0) per_sm = 1;
    }
    return sm_count_b() * per_sm;
}

struct Plan {
    int count = 0;
    long long total_n = 0;
    // `slices` slices of stored pairs per warp of the FP64 kernels (`grid` CTAs)
    double2 *wbuf = nullptr;
    long long wstride = 0;
    int slices = 4, grid = 0;
    BatchInst *d_inst = nullptr;
    // prefix tables: eigenpairs, FP64 team units, units of 8 and of 32 eigenpairs
    // (count + 1 entries each, one after another)
    long long *d_eoff = nullptr, *d_uoff = nullptr, *d_off8 = nullptr, *d_off32 = nullptr;
    long long n8 = 0, n32 = 0;   // units in all
    int2 *d_fix = nullptr, *d_old = nullptr, *d_more = nullptr;
    bool fast = true, vectors = false;
    BatchCtl *d_ctl = nullptr;
    void *scratch = nullptr;
    int *status = nullptr;
    SolveOpts so{};
    RunOpts ro{};
    cudaGraphExec_t exec = nullptr;
    std::vector<BatchInst> host;
};

// bytes of one instance's scratch and fixed-point data
static size_t inst_bytes(int n) {
    return ((arrow_scratch_bytes(n) + 255) & ~(size_t)255) + ((fast_bytes(n) + 255) & ~(size_t)255);
}
static Scratch carve_inst(char *base, int n, bool fast) {
    Scratch S = carve_scratch(base, n);
    if (fast) S.f = carve_fast(base + ((arrow_scratch_bytes(n) + 255) & ~(size_t)255), n);
    return S;
}

// the prefix tables of `count` instances of orders ns[i] and team widths W[i]
static std::vector<long long> prefix_tables(int count, const int *ns, const int *W, Plan &P) {
    std::vector<long long> t(4 * (size_t)(count + 1), 0);
    long long *e = t.data(), *u = e + count + 1, *a = u + count + 1, *b = a + count + 1;
    for (int i = 0; i < count; ++i) {
        const long long n = ns[i], epw = 32 / W[i];
        e[i + 1] = e[i] + n;
        u[i + 1] = u[i] + (n + epw - 1) / epw;
        a[i + 1] = a[i] + (n + 7) / 8;
        b[i + 1] = b[i] + (n + 31) / 32 + 1;          // (unit 0: the outermost two)
    }
    P.total_n = e[count];
    P.n8 = a[count];
    P.n32 = b[count];
    return t;
}
static void set_tables(Plan &P, long long *d) {
    P.d_eoff = d;
    P.d_uoff = d + (P.count + 1);
    P.d_off8 = d + 2 * (size_t)(P.count + 1);
    P.d_off32 = d + 3 * (size_t)(P.count + 1);
}

static void enqueue(const Plan &P, cudaStream_t st) {
    const unsigned g = (unsigned)((P.total_n + 255) / 256), g1 = (unsigned)((P.total_n + 63) / 64);
    const unsigned gm = (unsigned)std::min<long long>(P.total_n, 4 * sm_count_b());
    const SrcMany src{P.d_inst, P.count, P.d_eoff, P.d_off8, P.d_off32, P.d_ctl, P.d_old, P.d_fix, P.d_more,
                      P.wbuf, P.slices * P.wstride};
    k_batch_prep<<<P.count, 1024, 0, st>>>(P.d_inst, P.d_ctl);
    if (P.fast) {
        if (P.wstride > kFarFrom) k_fgroup<KIND_ARROW><<<(unsigned)P.n32, 256, 0, st>>>(src);
        k_fopen<KIND_ARROW><<<(unsigned)P.n32, 256, 0, st>>>(src, P.so);
        k_feval<<<(unsigned)P.n8, 256, 0, st>>>(src);
        k_fstep<KIND_ARROW><<<g1, 64, 0, st>>>(src, P.so, 0);
        k_fmore<KIND_ARROW><<<gm, 256, 0, st>>>(src, P.so, 0, 0);
        k_fold<KIND_ARROW><<<P.grid, 256, 0, st>>>(src, P.so);
    } else {
        k_batch_eig<<<P.grid, 256, 0, st>>>(P.d_inst, P.count, P.d_uoff, P.d_ctl, P.so, P.wbuf,
                                            P.wstride, P.slices);
    }
    if (P.ro.fixup) {
        k_batch_fix_decide<<<g, 256, 0, st>>>(P.d_inst, P.count, P.d_eoff, P.ro.knu_max);
        k_ffix<KIND_ARROW><<<g1, 64, 0, st>>>(src);
        if (P.fast) k_fmore<KIND_ARROW><<<gm, 256, 0, st>>>(src, P.so, 1, 0);
        k_batch_fix_solve<<<P.grid, 256, 0, st>>>(P.d_inst, P.d_fix, P.d_ctl, P.so, P.wbuf,
                                                  P.wstride, P.slices);
    }
    k_fout<KIND_ARROW><<<g1, 64, 0, st>>>(src);
    if (P.vectors) {
        if (P.fast) k_fcols<KIND_ARROW><<<(unsigned)P.n32, 256, 0, st>>>(src);
        k_vectors<KIND_ARROW><<<gm, 256, 0, st>>>(src);
    }
    if (P.status) k_batch_status<<<(P.count + 255) / 256, 256, 0, st>>>(P.d_inst, P.count, P.status);
}

static void free_plan(Plan *P) {
    if (!P) return;
    if (P->exec) cudaGraphExecDestroy(P->exec);
    cudaFree(P->d_inst);
    cudaFree(P->d_eoff);         // (the other tables lie behind it)
    cudaFree(P->d_fix);
    cudaFree(P->d_old);
    cudaFree(P->d_more);
    cudaFree(P->d_ctl);
    cudaFree(P->scratch);
    cudaFree(P->wbuf);
    delete P;
}

// an instance's descriptor (alpha lives on the device)
static BatchInst make_inst(int n, const double *d, const double *z, const double *alpha,
                           double *lambda, double *V, const Scratch &S, int team) {
    BatchInst B;
    B.n = n;
    B.n1 = n - 1;
    B.d = d;
    B.z = z;
    B.alpha = alpha;
    B.S = S;
    Outputs out{};
    out.lambda = lambda;
    out.V = V;
    out.ldv = n;
    B.va = VecArgs{n, n - 1, d, z, z, nullptr, 0.0, 1.0, out};
    B.team = team;
    return B;
}

// Build the descriptor table and scratch; `force_team` > 0 overrides the tuner
// and takes the FP64 solver (the tuner times it).
static cudaError_t build_plan(Plan *P, int count, const long long *n_off, const long long *v_off,
                              const double *d_all, const double *z_all, const double *alpha_all,
                              double *lambda_all, double *V_all, int *status_all,
                              const RunOpts &ro, int force_team, cudaStream_t st) {
    P->count = count;
    P->status = status_all;
    P->ro = ro;
    P->so = SolveOpts{ro.max_iter, ro.precision, ro.finish, ro.bgate, ro.kb_max};
    P->fast = force_team <= 0 && ro.max_iter >= kMinIterCap;
    P->vectors = V_all != nullptr;
    std::vector<size_t> soff(count + 1, 0);
    std::vector<int> ns(count), W(count);
    for (int i = 0; i < count; ++i) {
        ns[i] = (int)(n_off[i + 1] - n_off[i]);
        W[i] = force_team > 0 ? force_team : team_for(ns[i]);
        soff[i + 1] = soff[i] + inst_bytes(ns[i]);
    }
    const std::vector<long long> tab = prefix_tables(count, ns.data(), W.data(), *P);
    const size_t items = (size_t)(P->total_n > 0 ? P->total_n : 1);
    long long *d_tab = nullptr;
    cudaError_t e;
    if ((e = cudaMalloc(&P->scratch, soff[count] + 256))) return e;
    if ((e = cudaMalloc(&P->d_inst, sizeof(BatchInst) * count))) return e;
    if ((e = cudaMalloc(&d_tab, sizeof(long long) * tab.size()))) return e;
    set_tables(*P, d_tab);
    if ((e = cudaMalloc(&P->d_fix, sizeof(int2) * items))) return e;
    if ((e = cudaMalloc(&P->d_old, sizeof(int2) * items))) return e;
    if ((e = cudaMalloc(&P->d_more, sizeof(int2) * items))) return e;
    if ((e = cudaMalloc(&P->d_ctl, sizeof(BatchCtl)))) return e;
    long long nmax = 1;
    for (int i = 0; i < count; ++i) nmax = std::max<long long>(nmax, ns[i]);
    P->wstride = (nmax + 1) & ~1LL;
    P->grid = batch_eig_grid();
    if ((e = cudaMalloc(&P->wbuf, sizeof(double2) * P->wstride * P->slices *
                                      (size_t)P->grid * 8)))
        return e;
    P->host.resize(count);
    long long vo = 0;
    for (int i = 0; i < count; ++i) {
        const int n = ns[i];
        const long long vi = v_off ? v_off[i] : vo;
        P->host[i] = make_inst(n, d_all + (n_off[i] - i), z_all + (n_off[i] - i), alpha_all + i,
                               lambda_all + n_off[i], V_all ? V_all + vi : nullptr,
                               carve_inst((char *)P->scratch + soff[i], n, P->fast), W[i]);
        vo += (long long)n * n;
    }
    if ((e = cudaMemcpyAsync(P->d_inst, P->host.data(), sizeof(BatchInst) * count,
                             cudaMemcpyHostToDevice, st)))
        return e;
    if ((e = cudaMemcpyAsync(d_tab, tab.data(), sizeof(long long) * tab.size(),
                             cudaMemcpyHostToDevice, st)))
        return e;
    return cudaStreamSynchronize(st);
}

// ---------------------------------------------------------------------------
// a batch of separate requests (the serving loop): instances with their own
// input and output buffers, solved by one pass of the batched stages
// ---------------------------------------------------------------------------
// Layout of the one device block a request batch needs: descriptors, prefix
// tables, remedy list, control block, corners, per-instance scratch and the
// stored-pair slices (one a warp, since a warp has one eigenpair, and no more
// warps than eigenpairs: two requests of n = 1000 take 32 MB); every part 256-byte
// aligned.
struct ReqBatchLayout {
    size_t inst, tab, fix, old, more, ctl, alpha, scratch, wbuf, total;
    long long wstride;
    int grid;
    std::vector<size_t> soff;
};

static ReqBatchLayout req_batch_layout(int count, const int *ns) {
    ReqBatchLayout L;
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    long long total_n = 0, nmax = 1;
    L.soff.assign(count + 1, 0);
    for (int i = 0; i < count; ++i) {
        total_n += ns[i];
        nmax = std::max<long long>(nmax, ns[i]);
        L.soff[i + 1] = L.soff[i] + inst_bytes(ns[i]);
    }
    L.wstride = (nmax + 1) & ~1LL;
    size_t p = 0;
    L.inst = p; p += up(sizeof(BatchInst) * count);
    L.tab = p;  p += up(sizeof(long long) * 4 * (count + 1));
    L.fix = p;  p += up(sizeof(int2) * (size_t)(total_n > 0 ? total_n : 1));
    L.old = p;  p += up(sizeof(int2) * (size_t)(total_n > 0 ? total_n : 1));
    L.more = p; p += up(sizeof(int2) * (size_t)(total_n > 0 ? total_n : 1));
    L.ctl = p;  p += up(sizeof(BatchCtl));
    L.alpha = p; p += up(sizeof(double) * count);
    L.scratch = p; p += L.soff[count];
    L.grid = (int)std::min<long long>(batch_eig_grid(), (total_n + 7) / 8);
    L.wbuf = p; p += sizeof(double2) * (size_t)L.wstride * (size_t)L.grid * 8;
    L.total = p + 256;
    return L;
}

size_t req_batch_bytes(int count, const int *ns) { return req_batch_layout(count, ns).total; }

// Solve `count` arrowhead requests (orders ns, inputs d[i], z[i] with corner
// alpha[i], outputs lam[i] and V[i] with ld = n) with the batched stages on
// `st`, using the device block `block` of req_batch_bytes() bytes.  Each
// result has the bits the single-instance solve gives (remedies the FP64
// solver takes, by a warp here and by a team as wide as one wave allows there,
// agree within the tolerance).  cnt[i]
// receives the device address of instance i's counters (C_COUNT ints).
cudaError_t launch_req_batch(int count, const int *ns, const double *const *d,
                             const double *const *z, const double *alpha, double *const *lam,
                             double *const *V, void *block, const RunOpts &ro, cudaStream_t st,
                             const int **cnt) {
    const ReqBatchLayout L = req_batch_layout(count, ns);
    char *b = (char *)(((uintptr_t)block + 255) & ~(uintptr_t)255);
    Plan P;
    P.count = count;
    P.ro = ro;
    P.so = SolveOpts{ro.max_iter, ro.precision, ro.finish, ro.bgate, ro.kb_max};
    P.fast = ro.max_iter >= kMinIterCap;
    P.d_inst = (BatchInst *)(b + L.inst);
    P.d_fix = (int2 *)(b + L.fix);
    P.d_old = (int2 *)(b + L.old);
    P.d_more = (int2 *)(b + L.more);
    P.d_ctl = (BatchCtl *)(b + L.ctl);
    P.wbuf = (double2 *)(b + L.wbuf);
    P.wstride = L.wstride;
    P.slices = 1;
    P.grid = L.grid;
    double *d_alpha = (double *)(b + L.alpha);
    std::vector<BatchInst> host(count);
    const std::vector<int> W(count, 32);
    const std::vector<long long> tab = prefix_tables(count, ns, W.data(), P);
    set_tables(P, (long long *)(b + L.tab));
    for (int i = 0; i < count; ++i) {
        double *Vi = V ? V[i] : nullptr;
        P.vectors |= Vi != nullptr;
        host[i] = make_inst(ns[i], d[i], z[i], d_alpha + i, lam[i], Vi,
                            carve_inst(b + L.scratch + L.soff[i], ns[i], P.fast), 32);
        cnt[i] = host[i].S.cnt;
    }
    // (pageable sources: each copy is staged before the call returns)
    cudaError_t e = cudaMemcpyAsync(P.d_inst, host.data(), sizeof(BatchInst) * count,
                                    cudaMemcpyHostToDevice, st);
    if (!e) e = cudaMemcpyAsync(P.d_eoff, tab.data(), sizeof(long long) * tab.size(),
                                cudaMemcpyHostToDevice, st);
    if (!e) e = cudaMemcpyAsync(d_alpha, alpha, sizeof(double) * count, cudaMemcpyHostToDevice,
                                st);
    if (e) return e;
    enqueue(P, st);
    return cudaGetLastError();
}

static cudaError_t capture_plan(Plan *P) {
    cudaStream_t cs;
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e) return e;
    cudaGraph_t g = nullptr;
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (!e) {
        enqueue(*P, cs);
        e = cudaStreamEndCapture(cs, &g);
    }
    if (!e) e = cudaGraphInstantiate(&P->exec, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    return e;
}

static cudaError_t plan_info(const Plan &P, ae_info *info, cudaStream_t st) {
    std::vector<int> cnt((size_t)P.count * C_COUNT);
    std::vector<unsigned long long> c64((size_t)P.count * C64_COUNT);
    for (int i = 0; i < P.count; ++i) {
        cudaError_t e = cudaMemcpyAsync(&cnt[(size_t)i * C_COUNT], P.host[i].S.cnt,
                                        sizeof(int) * C_COUNT, cudaMemcpyDeviceToHost, st);
        if (!e) e = cudaMemcpyAsync(&c64[(size_t)i * C64_COUNT], P.host[i].S.cnt64,
                                    sizeof(unsigned long long) * C64_COUNT,
                                    cudaMemcpyDeviceToHost, st);
        if (e) return e;
    }
    cudaError_t e = cudaStreamSynchronize(st);
    if (e) return e;
    memset(info, 0, sizeof(*info));
    for (int i = 0; i < P.count; ++i) {
        const int *c = &cnt[(size_t)i * C_COUNT];
        const unsigned long long *u = &c64[(size_t)i * C64_COUNT];
        info->n_reduced += c[C_M] + 1;
        info->n_deflated += c[C_ND];
        info->n_nearzero += c[C_NEARZERO];
        info->n_otherpole += c[C_OTHERPOLE];
        info->n_dpr1shift += c[C_DPR1];
        info->n_capped += c[C_CAPPED];
        info->n_fp32_fallback += c[C_FP32FB];
        info->n_ddb += c[C_DDB];
        info->n_mid64 += c[C_MID64];
        info->total_deriv += (long long)u[C64_DERIV];
        info->n_f32_passes += (long long)u[C64_F32];
        info->n_df_passes += (long long)u[C64_DF];
        if (c[C_MAXIT] > info->max_iter_used) info->max_iter_used = c[C_MAXIT];
        info->total_iter += (long long)u[C64_ITERS];
        info->fix_iter += (long long)u[C64_ITERS_FIX];
        double kb, kn;
        memcpy(&kb, &u[C64_MAXKB], sizeof kb);
        memcpy(&kn, &u[C64_MAXKNU], sizeof kn);
        if (kb > info->max_Kb) info->max_Kb = kb;
        if (kn > info->max_Knu) info->max_Knu = kn;
    }
    return cudaSuccess;
}

// synthetic instances for the tuner's timing runs (not part of any solve):
// d_r strictly decreasing in [-10, 10], z_r in (0, 1], alpha in [-1, 1]
__device__ __forceinline__ double hash01(unsigned long long x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    x ^= x >> 31;
    return (double)(x >> 11) * 0x1p-53;
}

__global__ void k_gen_uniform(int count, int n, double *d, double *z, double *alpha) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long rows = (long long)count * (n - 1);
    if (t < rows) {
        const int r = (int)(t % (n - 1));
        d[t] = 10.0 - 20.0 * (r + 0.25 + 0.5 * hash01(2 * t)) / (n - 1);
        z[t] = 1.0 - 0.95 * hash01(2 * t + 1);
    }
    if (t < count) alpha[t] = 2.0 * hash01(~t) - 1.0;
}

static cudaError_t time_team(int n, int W, float *ms, cudaStream_t st) {
    const int count = (int)std::max(2LL, std::min(4096LL, (1LL << 19) / n));
    std::vector<long long> n_off(count + 1);
    for (int i = 0; i <= count; ++i) n_off[i] = (long long)i * n;
    double *buf = nullptr;
    const size_t rows = (size_t)count * (n - 1);
    cudaError_t e = cudaMalloc(&buf, sizeof(double) * (2 * rows + count + (size_t)count * n));
    if (e) return e;
    double *d = buf, *z = buf + rows, *al = z + rows, *lam = al + count;
    k_gen_uniform<<<(unsigned)((rows + 255) / 256) + 1, 256, 0, st>>>(count, n, d, z, al);
    Plan *P = new Plan();
    RunOpts ro{};
    resolve_opts(nullptr, ro);
    ro.precision = AE_FP32_BRACKET;
    e = build_plan(P, count, n_off.data(), nullptr, d, z, al, lam, nullptr, nullptr, ro, W, st);
    cudaEvent_t a = nullptr, b = nullptr;
    if (!e) e = cudaEventCreate(&a);
    if (!e) e = cudaEventCreate(&b);
    if (!e) {
        enqueue(*P, st);   // warm-up
        cudaEventRecord(a, st);
        for (int r = 0; r < 2; ++r) enqueue(*P, st);
        cudaEventRecord(b, st);
        e = cudaEventSynchronize(b);
        if (!e) e = cudaEventElapsedTime(ms, a, b);
    }
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    free_plan(P);
    cudaFree(buf);
    return e;
}

}  // namespace ae

struct ae_batch {
    ae::Plan *p;
};

namespace {
int batch_args(int count, const long long *n_off, const double *d_all, const double *z_all,
               const double *alpha_all, const double *lambda_all) {
    if (count < 1) return -2;
    if (!n_off || n_off[0] != 0) return -3;
    for (int i = 0; i < count; ++i)
        if (n_off[i + 1] - n_off[i] < 1 || n_off[i + 1] - n_off[i] > (1 << 30)) return -3;
    if (n_off[count] > count && (!d_all || !z_all)) return -5;
    if (!alpha_all) return -7;
    if (!lambda_all) return -8;
    return 0;
}

int resolve(const ae_opts *o, ae::RunOpts &ro) { return ae::resolve_opts(o, ro); }

int fail(cudaError_t e) {
    ae::record_cuda_error(e);
    return AE_ERR_CUDA;
}
}  // namespace

extern "C" {

int ae_batch_create(ae_batch **plan, int count, const long long *n_off, const long long *v_off,
                    const double *d_all, const double *z_all, const double *alpha_all,
                    double *lambda_all, double *V_all, int *status_all, const ae_opts *opts,
                    void *stream) {
    if (!plan) return -1;
    *plan = nullptr;
    const int a = batch_args(count, n_off, d_all, z_all, alpha_all, lambda_all);
    if (a) return a;
    ae::RunOpts ro;
    if (resolve(opts, ro)) return -11;
    ae::Plan *P = new ae::Plan();
    cudaError_t e = ae::build_plan(P, count, n_off, v_off, d_all, z_all, alpha_all, lambda_all,
                                   V_all, status_all, ro, 0, (cudaStream_t)stream);
    if (!e) e = ae::capture_plan(P);
    if (e) {
        ae::free_plan(P);
        return fail(e);
    }
    *plan = new ae_batch{P};
    return AE_OK;
}

int ae_batch_run(ae_batch *plan, void *stream) {
    if (!plan || !plan->p) return -1;
    cudaError_t e = cudaGraphLaunch(plan->p->exec, (cudaStream_t)stream);
    return e ? fail(e) : AE_OK;
}

int ae_batch_info(ae_batch *plan, ae_info *info, void *stream) {
    if (!plan || !plan->p) return -1;
    if (!info) return -2;
    cudaError_t e = ae::plan_info(*plan->p, info, (cudaStream_t)stream);
    if (e) return fail(e);
    return AE_OK;
}

void ae_batch_destroy(ae_batch *plan) {
    if (!plan) return;
    cudaDeviceSynchronize();
    ae::free_plan(plan->p);
    delete plan;
}

int arrow_eig_batched(int count, const long long *n_off, const long long *v_off,
                      const double *d_all, const double *z_all, const double *alpha_all,
                      double *lambda_all, double *V_all, int *status_all, const ae_opts *opts,
                      ae_info *info, void *stream) {
    const int a = batch_args(count, n_off, d_all, z_all, alpha_all, lambda_all);
    if (a) return a;
    ae::RunOpts ro;
    if (resolve(opts, ro)) return -10;
    cudaStream_t st = (cudaStream_t)stream;
    ae::Plan *P = new ae::Plan();
    cudaError_t e = ae::build_plan(P, count, n_off, v_off, d_all, z_all, alpha_all, lambda_all,
                                   V_all, status_all, ro, 0, st);
    if (!e) {
        ae::enqueue(*P, st);
        e = cudaGetLastError();
    }
    int status = AE_OK;
    if (!e && info) {
        e = ae::plan_info(*P, info, st);
        if (!e && info->n_capped) status = AE_ERR_NOCONV;
    }
    if (!e) e = cudaStreamSynchronize(st);   // the plan's buffers are freed below
    ae::free_plan(P);
    return e ? fail(e) : status;
}

int ae_autotune(int n_max, void *stream) {
    if (n_max < 2) return -1;
    cudaStream_t st = (cudaStream_t)stream;
    std::map<int, int> found;
    for (int b = 32; b <= 256 && b <= std::max(32, n_max); b <<= 1) {
        int best = 32;
        float best_ms = 0.f;
        for (int W : {8, 16, 32}) {
            float ms = 0.f;
            cudaError_t e = ae::time_team(b, W, &ms, st);
            if (e) return fail(e);
            if (W == 8 || ms < best_ms) {
                best = W;
                best_ms = ms;
            }
        }
        found[b] = best;
    }
    for (int b = 512; b <= n_max && b <= (1 << 24); b <<= 1) found[b] = 32;
    std::lock_guard<std::mutex> lk(ae::g_tune_mu);
    ae::load_cache_locked();
    for (auto &kv : found) ae::g_tune[kv.first] = kv.second;
    ae::save_cache_locked();
    return AE_OK;
}

int ae_team_width(int n) { return n < 1 ? -1 : ae::team_for(n); }

}  // extern "C"
