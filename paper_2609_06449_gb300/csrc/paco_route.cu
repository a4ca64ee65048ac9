// paco_route.cu -- how paco_execute runs a plan: two to four passes of
// paco_fold.cuh.
//
// The route is the paper's composition Phase I -> redistribution -> Phase III
// with the factors chosen for the machine: a pass keeps its tile in one CTA,
// so a transform takes ceil(log2 N / 10) of them (complex64; 9 for complex128),
// the first with the redistribution in its stores, the others in place in the
// output (Phase III's length split further, Sect. 4.1).  The result does not
// depend on the factors (Theorem 3); the plan's own N1, N2 and W stay what
// paco_execute_stage1 / _stage2 / _phase1 use.  The weighted power runs the
// plan's own two stages (paco_power.cuh).
#include <cuda_runtime.h>

#include <array>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>

#include "paco_common.cuh"
#include "paco_fold.cuh"
#include "paco_power.cuh"
#include "paco_plan.h"
#include "paco_stage_args.cuh"
#include "paco_tcpass.cuh"
#include "paco_whole.cuh"

namespace paco {

constexpr int MAX_PASSES = 4;
constexpr int DIRECT_LG = 20;      // passes up to K L = 2^20 keep all their factors in a table (4 MiB, 8 in FP64)

struct Route {
    int n = 0;                     // passes of paco_execute (0: the stage kernels)
    WholeKernel whole;             // n = 1: whole transforms in a CTA
    WholeKernel whole_scaled;      //   of a scaled input
    FoldKernel k[MAX_PASSES];
    FoldKernel scaled;                 // k[0] for a scaled input (complex64)
    int twmode[MAX_PASSES] = {};       // FoldCfg::TW
    FoldArgs<float> f[MAX_PASSES];     // by the plan's precision
    FoldArgs<double> d[MAX_PASSES];
    TcPassArgs t[MAX_PASSES];
    PowerKernel pk[2];              // the stages of the weighted power (fn == nullptr: the stage kernels)
    PowerArgs pa[2];
    std::shared_ptr<void> tw[MAX_PASSES];   // the factors of every pass (shared_table)
};

// pi over `bits` bits with digits of t bits (host copy of digit_reverse).
static unsigned rev_host(unsigned u, int bits, int t)
{
    return bits == 0 ? u : (unsigned)paco_digit_reverse((int64_t)u, 1 << t, bits / t);
}

void route_destroy(Route *r)
{
    delete r;
}

// A table of factors, one for all plans that are alive on a device and need the
// same one: it depends on the lengths alone, and a program keeps a plan for every
// batch size and stream that it meets.  key: what tells the tables apart (the
// device and the kind among it).  make(&p) allocates and enqueues; every plan waits
// for the device before it is handed out, so a table found here is complete by
// then whichever plan made it.  Freed with the last plan that holds it.
using TableKey = std::array<int, 7>;
template <class Make>
static paco_status_t shared_table(const TableKey &key, std::shared_ptr<void> *out, const Make &make)
{
    static std::mutex &mutex = *new std::mutex;        // (not torn down before the last plan)
    static auto &tables = *new std::map<TableKey, std::weak_ptr<void>>;
    std::lock_guard<std::mutex> lock(mutex);
    std::weak_ptr<void> &known = tables[key];
    if ((*out = known.lock())) return PACO_OK;
    void *p = nullptr;
    const paco_status_t st = make(&p);
    if (st != PACO_OK) {
        cudaFree(p);
        return st;
    }
    *out = std::shared_ptr<void>(p, [](void *q) { cudaFree(q); });
    known = *out;
    return PACO_OK;
}
enum { TABLE_FOLD, TABLE_WHOLE, TABLE_ROOTS };

// Tables of a pass's factors, each rounded once, over K = 2^lgK columns (kappa).
enum TauKind {
    TAU_LEVELS,     // entry q A' + k_lo: w_{K A' n}^{-(kappa + K k_lo + K A' s)}, q = tau_index(n, s), A' = 2^lgA
    TAU_ROWS,       // entry r: w_{K A'}^{-kappa r}
    TAU_POWERS      // entry i: w_{K A'}^{-kappa 2^i}
};
struct Roots {
    const cx<double> *lo = nullptr, *hi = nullptr;   // (nullptr: by sincospi)
    int lg = 0, lo_bits = 0;                         // of w_{2^lg}
};
template <typename R>
__global__ void tau_gen_kernel(cx<R> *out, long long count, int kind, int lgA, int lgK, bool no_kappa, Roots roots)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const long long kap = no_kappa ? 0 : i & ((1ll << lgK) - 1);
    const int q = (int)(i >> lgK);
    long long e;
    int lgM = lgK + lgA;
    if (kind == TAU_LEVELS) {
        const int klo = q & ((1 << lgA) - 1), t = q >> lgA;
        const int lgq = t ? 31 - __clz(t) : 0, s = t ? t - (1 << lgq) : 0;
        e = kap + ((long long)klo << lgK) + ((long long)s << lgM);
        lgM += t ? lgq + 2 : 1;
    } else {
        e = kind == TAU_ROWS ? kap * q : kap << q;
    }
    if (roots.lo) {
        // the product of two FP64 roots, rounded once (a tenth of sincospi's work)
        const unsigned x = (unsigned)(e << (roots.lg - lgM));
        const cx<double> w = cmul(roots.lo[x & ((1u << roots.lo_bits) - 1u)], roots.hi[x >> roots.lo_bits]);
        out[i] = make_cx<R>((R)w.x, (R)w.y);
        return;
    }
    double sn, cs;
    sincospi(2.0 * (double)e / (double)(1ll << lgM), &sn, &cs);
    out[i] = make_cx<R>((R)cs, (R)(-sn));
}

// lo[r] = w^{-r}, r < 2^lo_bits, then hi[r] = w^{-(r << lo_bits)}, w = w_{2^lg}.
__global__ void roots_gen_kernel(cx<double> *out, int lg, int lo_bits)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, nlo = 1 << lo_bits;
    if (i >= nlo + (1 << (lg - lo_bits))) return;
    const long long e = i < nlo ? i : (long long)(i - nlo) << lo_bits;
    double sn, cs;
    sincospi(2.0 * (double)e / (double)(1ll << lg), &sn, &cs);
    out[i] = make_cx<double>(cs, -sn);
}

template <typename R>
static cx<R> *tau_gen(cx<R> *t, int entries, int kind, int lgA, int lgK, bool no_kappa = false, const Roots &roots = Roots())
{
    const long long count = (long long)entries << lgK;
    tau_gen_kernel<R><<<(unsigned)((count + 255) / 256), 256>>>(t, count, kind, lgA, lgK, no_kappa, roots);
    return t + count;
}

// Entries of FoldArgs::tau in mode FoldCfg::TW over 2^lgK columns.
static long long fold_entries(bool fp64, const FoldKernel &k, int mode, int lgK)
{
    const int A = 1 << k.lgA, B = 1 << k.lgB, nA = fp64 ? A : A / 2;
    if (mode == 0 && fold_plain(fp64, k.lgB)) return A * B;
    return mode == 1 ? (long long)(nA + A * B / 2) << lgK : A * B / 2 + (mode == 2 ? (long long)(nA + k.lgB) << lgK : 0);
}

template <typename R>
paco_status_t fold_table(void **dst, const FoldKernel &k, int mode, int lgK, bool no_kappa, size_t skip)
{
    const int A = 1 << k.lgA, B = 1 << k.lgB, lgL = k.lgA + k.lgB;
    const bool fp64 = sizeof(R) == 8;
    if (mode == 0 && fold_plain(fp64, k.lgB)) return gen_table((int)sizeof(cx<R>), dst, A * B, A * B, 1, 0);
    const int nA = fp64 ? A : A / 2;
    const long long count = fold_entries(fp64, k, mode, lgK);
    // FP32 tables of many entries: FP64 roots of w_{K L} behind the table
    Roots roots;
    size_t bytes = skip + (((size_t)count * sizeof(cx<R>) + 15) & ~(size_t)15);
    const bool by_roots = !fp64 && mode != 0 && !no_kappa;
    if (by_roots) {
        roots.lg = lgK + lgL;
        roots.lo_bits = (roots.lg + 1) / 2;
    }
    const int nroots = by_roots ? (1 << roots.lo_bits) + (1 << (roots.lg - roots.lo_bits)) : 0;
    PACO_CUDA_TRY(cudaMalloc(dst, bytes + (size_t)nroots * sizeof(cx<double>)));
    if (by_roots) {
        cx<double> *q = reinterpret_cast<cx<double> *>(static_cast<char *>(*dst) + bytes);
        roots_gen_kernel<<<(nroots + 255) / 256, 256>>>(q, roots.lg, roots.lo_bits);
        roots.lo = q;
        roots.hi = q + (1 << roots.lo_bits);
    }
    cx<R> *t = reinterpret_cast<cx<R> *>(static_cast<char *>(*dst) + skip);
    if (mode == 1) {
        t = fp64 ? tau_gen(t, A, TAU_ROWS, k.lgA, lgK, no_kappa) : tau_gen(t, nA, TAU_LEVELS, 0, lgK, no_kappa, roots);
        tau_gen(t, A * B / 2, TAU_LEVELS, k.lgA, lgK, no_kappa, roots);
    } else {
        t = tau_gen(t, A * B / 2, TAU_LEVELS, k.lgA, 0);
        if (mode == 2) {
            t = fp64 ? tau_gen(t, A, TAU_ROWS, k.lgA, lgK) : tau_gen(t, nA, TAU_LEVELS, 0, lgK, false, roots);
            tau_gen(t, k.lgB, TAU_POWERS, lgL, lgK, false, roots);
        }
    }
    PACO_CUDA_TRY(cudaGetLastError());
    return PACO_OK;
}

template paco_status_t fold_table<float>(void **, const FoldKernel &, int, int, bool, size_t);

void fold_levels(void *dst, const FoldKernel &k) { tau_gen(static_cast<cx<float> *>(dst), 1 << (k.lgA + k.lgB - 1), TAU_LEVELS, k.lgA, 0); }

paco_status_t whole_table(int lgN, void **dst)
{
    int k[4], n = 0, total = 0;                            // log2 of the frequencies known before every step
    k[0] = 0;
    for (; n < 3 && whole_radix(lgN, n); ++n) k[n + 1] = k[n] + ilog2_exact(whole_radix(lgN, n));
    for (int i = 1; i < n; ++i) total += 1 << (k[i + 1] - 1);
    PACO_CUDA_TRY(cudaMalloc(dst, (size_t)total * 8));
    cx<float> *t = static_cast<cx<float> *>(*dst);
    for (int i = 1; i < n; ++i) t = tau_gen(t, 1 << (k[i + 1] - 1), TAU_LEVELS, k[i], 0);
    PACO_CUDA_TRY(cudaGetLastError());
    return PACO_OK;
}

// A pass's columns are the frequencies of the passes before it (the first
// pass: all other rows of the view).
template <typename R>
void fold_pass_args(FoldArgs<R> *a, const FoldKernel &k, const int *f, int n, int i, int t)
{
    memset(a, 0, sizeof(*a));
    int lgN = 0, lgK = 0;
    for (int j = 0; j < n; ++j) {
        lgN += f[j];
        if (j < i) lgK += f[j];
    }
    const int lgL = f[i], lgC = i == 0 ? lgN - lgL : lgK;
    a->bstride = 1LL << lgN;
    a->ld_in = 1u << lgC;
    a->ld_out = i == 0 ? 1u << lgL : 1u << lgC;
    a->rev_bits = i == 0 ? 0 : lgL;
    a->rev_t = t;
    for (int j = 0; j < (1 << k.lgA); ++j) a->rowA[j] = rev_host((unsigned)j << k.lgB, a->rev_bits, t) << lgC;
    for (int j = 0; j < (1 << k.lgB); ++j) a->rowK[j] = (unsigned)j << (k.lgA + lgC);
    a->crev_bits = i == 0 ? lgC : 0;
    a->crev_t = t;
    a->lg_tiles = lgC - k.lgW;
    a->lg_all = lgN - lgL - k.lgW;
    a->blk_stride = i == 0 || i == n - 1 ? 0u : 1u << (lgK + lgL);
    a->lg_n = lgN;
    a->lg_k = lgK;
    a->mult = R(1);
}
template void fold_pass_args<float>(FoldArgs<float> *, const FoldKernel &, const int *, int, int, int);

// Pass i of the plan's route: launch constants and tables.
template <typename R>
static paco_status_t pass_setup(const paco_plan *pl, Route *r, FoldArgs<R> *a, const int *f, int n, int i, int t)
{
    const FoldKernel &k = r->k[i];
    fold_pass_args(a, k, f, n, i, t);
    PACO_CUDA_TRY(cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem));
    const int lgK = r->twmode[i] ? a->lg_k : 0;             // (mode 0: one column)
    const paco_status_t st = shared_table({pl->device, TABLE_FOLD, (int)sizeof(R), k.lgA, k.lgB, r->twmode[i], lgK}, &r->tw[i],
                                          [&](void **p) { return fold_table<R>(p, k, r->twmode[i], lgK); });
    a->tau = static_cast<const cx<R> *>(r->tw[i].get());
    return st;
}

// Stage i of the weighted power over the plan's factors.
static paco_status_t power_setup(const paco_plan *pl, PowerArgs *a, const PowerKernel &k, const int *lg, int i)
{
    memset(a, 0, sizeof(*a));
    const int lgL = lg[i], lgC = lg[1 - i];
    a->bstride = pl->N;
    a->ld_in = 1u << lgC;
    a->ld_out = i == 0 ? 1u << lgL : 1u << lgC;
    a->rev_bits = i == 0 ? 0 : lgL;
    a->rev_t = a->crev_t = pl->t;
    for (int j = 0; j < (1 << k.lgA); ++j) a->rowA[j] = rev_host((unsigned)j << k.lgB, a->rev_bits, pl->t) << lgC;
    for (int j = 0; j < (1 << k.lgB); ++j) a->rowK[j] = (unsigned)j << (k.lgA + lgC);
    a->crev_bits = i == 0 ? lgC : 0;
    a->lg_all = lgC - k.lgW;
    a->lo = static_cast<const cx<float> *>(pl->twN_lo);
    a->hi = static_cast<const cx<float> *>(pl->twN_hi);
    a->lo_bits = pl->twN_lo_bits;
    a->n_mask = (unsigned)(pl->N - 1);
    PACO_CUDA_TRY(cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem));
    a->twL = static_cast<const cx<float> *>(pl->twP[i]);
    return PACO_OK;
}

// Factors of the route, log2, first pass first; returns their number (0: none).
static int route_factors(const paco_plan *pl, int lg1, int lg2, int *f)
{
    if (pl->dims >= 2) {
        f[0] = lg1;
        f[1] = pl->dims == 3 ? pl->lgLa3 : lg2;
        f[2] = lg2 - f[1];
        return pl->dims;
    }
    // as even as possible, the larger ones first (the first pass has no twiddles)
    const int lg = lg1 + lg2, most = pl->esize == 8 ? 10 : 9;
    int n = (lg + most - 1) / most;
    if (n < 2) n = 2;
    for (int i = 0, left = lg; i < n; ++i) {
        f[i] = (left + n - i - 1) / (n - i);
        left -= f[i];
    }
    return n;
}

// The passes of a tensor-core form: 2^5..2^8 points each, at most four
// contractions in all (the stage kernels' number: the error is theirs).
static paco_status_t tc_setup(paco_plan *pl, Route *r, int lgN)
{
    int f[MAX_PASSES], n = (lgN + 7) / 8;
    for (int i = 0, left = lgN; i < n; ++i) {
        f[i] = (left + n - i - 1) / (n - i);
        left -= f[i];
    }
    int t = pl->t, extra = 4 - n;
    for (int i = 1; i < n; ++i)
        if (f[i] % t) t = 1;
    for (int i = 0, lgK = 0; i < n; lgK += f[i], ++i) {
        const bool tc2 = f[i] == 8 && extra-- > 0;
        r->k[i] = tcpass_kernel(pl->form, i == 0, tc2, f[i], i == 0 ? lgN - f[0] : lgK);
        if (!r->k[i].fn) return PACO_OK;
        TcPassArgs &a = r->t[i];
        fold_pass_args(&a.f, r->k[i], f, n, i, t);
        a.lo_bits = pl->twN_lo_bits;
        a.lo = static_cast<const cx<float> *>(pl->twN_lo);
        a.hi = static_cast<const cx<float> *>(pl->twN_hi);
        a.frag = static_cast<const uint4 *>(pl->tc);
        PACO_CUDA_TRY(cudaFuncSetAttribute(r->k[i].fn, cudaFuncAttributeMaxDynamicSharedMemorySize, r->k[i].smem));
        const paco_status_t st = shared_table({pl->device, TABLE_ROOTS, 8, f[i], 0, 0, 0}, &r->tw[i],
                                              [&](void **p) { return gen_table(8, p, 1LL << f[i], 1LL << f[i], 1, 0); });
        if (st != PACO_OK) return st;
        a.twL = static_cast<const cx<float> *>(r->tw[i].get());
    }
    r->n = n;
    return PACO_OK;
}

// Builds pl->route; its n stays 0 where the stage kernels run the plan.
paco_status_t route_setup(paco_plan *pl)
{
    // the plain forms with no stage option asked for
    if (pl->shard_G || pl->req_split || pl->req_ctas || pl->req_tile) return PACO_OK;
    Route *r = new (std::nothrow) Route();
    if (!r) return fail(PACO_ERR_NOMEM, "out of host memory");
    pl->route = r;                                     // freed with the plan
    const int lg[2] = {ilog2_exact(pl->N1), ilog2_exact(pl->N2)}, lgN = lg[0] + lg[1];
    if (pl->form) return pl->dims == 1 ? tc_setup(pl, r, lgN) : PACO_OK;
    int f[MAX_PASSES] = {0, 0, 0, 0};
    // short transforms: one CTA holds them whole.  2^13 and 2^14 points from a batch
    // of 32 on: fewer spread better over the SMs in two passes.  us in a graph, whole
    // and in passes: 2^13 x 1 4.8 and 3.9, x 32 5.3 and 5.0, x 48 5.3 and 5.8, x 128 5.5
    // and 9.1, x 512 14.6 and 16.1; 2^14 x 1 8.2 and 4.9, x 32 8.7 and 6.0, x 48 8.7
    // and 9.0, x 128 8.9 and 10.5, x 512 (in L2) 40 and 37.
    const bool whole = pl->dims == 1 && pl->esize == 8 && (lgN < 13 || pl->batch >= 32);
    if (whole && (r->whole = whole_kernel(lgN, false)).fn) {
        const paco_status_t st = shared_table({pl->device, TABLE_WHOLE, 8, lgN, 0, 0, 0}, &r->tw[0],
                                              [&](void **p) { return whole_table(lgN, p); });
        if (st != PACO_OK) return st;
        r->whole_scaled = whole_kernel(lgN, true);
        for (const WholeKernel *k : {&r->whole, &r->whole_scaled})
            PACO_CUDA_TRY(cudaFuncSetAttribute(k->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, k->smem));
        r->n = 1;
    }
    int n = pl->fused || r->n ? 0 : route_factors(pl, lg[0], lg[1], f);
    for (int i = 0, lgK = 0; i < n; lgK += f[i], ++i) {
        const int lgC = i == 0 ? lgN - f[0] : lgK;
        r->twmode[i] = i == 0 || pl->dims >= 2 ? 0 : lgK + f[i] <= DIRECT_LG ? 1 : 2;
        r->k[i] = pl->esize == 8 ? fold_kernel_f32(i == 0, r->twmode[i], f[i], lgC, pl->N * pl->batch <= (int64_t)1 << 24)
                                 : fold_kernel_f64(i == 0, r->twmode[i], f[i], lgC, n > 2);
        if (!r->k[i].fn) n = 0;
        if (i == 0 && pl->esize == 8)
            r->scaled = fold_kernel_f32(true, 0, f[i], lgC, pl->N * pl->batch <= (int64_t)1 << 24, true);
    }
    if (n && r->scaled.fn)
        PACO_CUDA_TRY(cudaFuncSetAttribute(r->scaled.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, r->scaled.smem));
    // pi of the redistribution: the plan's base where its digits fit the factors
    int t = pl->t;
    for (int i = 1; i < n; ++i)
        if (f[i] % t) t = 1;
    paco_status_t st = PACO_OK;
    for (int i = 0; i < n && st == PACO_OK; ++i)
        st = pl->esize == 8 ? pass_setup(pl, r, &r->f[i], f, n, i, t) : pass_setup(pl, r, &r->d[i], f, n, i, t);
    if (n) r->n = n;
    if (pl->dims == 3 || pl->esize != 8) return st;
    for (int i = 0; i < 2 && st == PACO_OK; ++i) {
        r->pk[i] = power_kernel(i == 0, lg[i], lg[1 - i]);
        if (r->pk[i].fn) st = power_setup(pl, &r->pa[i], r->pk[i], lg, i);
    }
    return st;
}

int route_passes(const paco_plan *pl) { return pl->route ? pl->route->n : 0; }

static paco_status_t launch(const paco_plan *pl, const void *fn, void *args, long long ctas, int threads, int smem,
                            bool pdl, cudaStream_t stream)
{
    if (ctas > INT32_MAX) return fail(PACO_ERR_UNSUPPORTED, "batch of %lld transforms is too large", (long long)pl->batch);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    // Programmatic serialisation from two CTAs an SM on (77 x 2^18: 111 -> 106
    // us): a smaller grid's CTAs would be placed beside the ones still running
    // instead of one to an SM (2^20: 12.3 -> 14.6 us).
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // the kernel waits (griddepcontrol)
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl && ctas > 2 * pl->num_sms ? 1 : 0;
    void *params[] = {args};
    PACO_CUDA_TRY(cudaLaunchKernelExC(&cfg, fn, params));
    return PACO_OK;
}

template <typename R>
static paco_status_t run_passes(const paco_plan *pl, const FoldArgs<R> *args, const void *in, void *out, int dir,
                                const StageTerms *terms, cudaStream_t stream)
{
    const Route &r = *pl->route;
    for (int i = 0; i < r.n; ++i) {
        FoldArgs<R> a = args[i];
        a.in = static_cast<const cx<R> *>(i == 0 ? in : out);
        a.out = static_cast<cx<R> *>(out);
        a.conj = dir == 1;
        a.reverse = i & 1;
        const bool scaled = terms && i == 0;
        if (scaled) {
            a.mult = (R)terms->ld_mult;
            a.scale = terms->ld_scale;
        }
        const FoldKernel &k = scaled ? r.scaled : r.k[i];
        const paco_status_t st = launch(pl, k.fn, &a, (long long)pl->batch << a.lg_all, k.threads, k.smem, true, stream);
        if (st != PACO_OK) return st;
    }
    return PACO_OK;
}

paco_status_t route_run(const paco_plan *pl, const void *in, void *out, int dir, const StageTerms *terms,
                        cudaStream_t stream)
{
    const Route &r = *pl->route;
    if (r.whole.fn) {
        WholeArgs a;
        a.in = static_cast<const float2 *>(in);
        a.out = static_cast<float2 *>(out);
        a.batch = pl->batch;
        a.tau = static_cast<const float2 *>(r.tw[0].get());
        a.conj = dir == 1;
        a.mult = terms ? terms->ld_mult : 1.f;
        a.scale = terms ? terms->ld_scale : nullptr;
        return launch(pl, terms ? r.whole_scaled.fn : r.whole.fn, &a, (pl->batch + r.whole.per_cta - 1) / r.whole.per_cta, r.whole.threads,
                      r.whole.smem, false, stream);
    }
    if (pl->form) {
        for (int i = 0; i < r.n; ++i) {
            TcPassArgs a = r.t[i];
            a.f.in = static_cast<const cx<float> *>(i == 0 ? in : out);
            a.f.out = static_cast<cx<float> *>(out);
            a.f.conj = dir == 1;
            a.f.reverse = i & 1;
            const paco_status_t st = launch(pl, r.k[i].fn, &a, (long long)pl->batch << a.f.lg_all, r.k[i].threads,
                                            r.k[i].smem, true, stream);
            if (st != PACO_OK) return st;
        }
        return PACO_OK;
    }
    return pl->esize == 8 ? run_passes(pl, pl->route->f, in, out, dir, terms, stream)
                          : run_passes(pl, pl->route->d, in, out, dir, terms, stream);
}

bool route_has_power(const paco_plan *pl, int stage) { return pl->route && pl->route->pk[stage].fn; }

paco_status_t route_power(const paco_plan *pl, int stage, const void *in, void *out, int dir, const StageTerms &terms,
                          cudaStream_t stream)
{
    const PowerKernel &k = pl->route->pk[stage];
    PowerArgs a = pl->route->pa[stage];
    a.in = static_cast<const cx<float> *>(in);
    a.out = static_cast<cx<float> *>(out);
    a.conj = dir == 1;
    a.w = terms.st_w;
    a.loss = terms.st_loss;
    a.store_weighted = terms.st_weighted;
    a.reverse = stage;
    return launch(pl, k.fn, &a, (long long)pl->batch << a.lg_all, k.threads, k.smem, true, stream);
}

} // namespace paco
