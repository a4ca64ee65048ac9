// paco_route.cu -- how paco_execute runs a complex64 transform: two or three
// passes of paco_pass.cuh.
//
// The route is the paper's composition Phase I -> redistribution -> Phase III
// with the two factors chosen for the machine: a pass of up to 2^10 points
// keeps its tile in one CTA and runs near the copy rate, so a transform of up
// to 2^20 points takes two of them and a longer one three (Phase III's length
// L2 L3 split once more, both halves in place in the output).  The result does
// not depend on the factors (Theorem 3); the plan's own N1, N2 and W stay what
// paco_execute_stage1 / _stage2 / _phase1 use.
#include <cuda_runtime.h>

#include <cstring>
#include <new>

#include "paco_common.cuh"
#include "paco_pass.cuh"
#include "paco_plan.h"
#include "paco_stage_args.cuh"

namespace paco {

struct Pass {
    PassKernel k;
    PassArgs a;
    void *tw = nullptr;            // w_L^{-r}
};

struct Route {
    int n = 0;                     // passes of paco_execute (0: the two stages)
    Pass p[3];
    Pass power[2];                 // the stages of the weighted power (fn == nullptr: the stage kernels)
};

// pi over `bits` bits with digits of t bits (host copy of digit_reverse).
static unsigned rev_host(unsigned u, int bits, int t)
{
    return bits == 0 ? u : (unsigned)paco_digit_reverse((int64_t)u, 1 << t, bits / t);
}

void route_destroy(Route *r)
{
    if (!r) return;
    for (Pass &p : r->p) cudaFree(p.tw);
    for (Pass &p : r->power) cudaFree(p.tw);
    delete r;
}

// Pass i of the n factors f: strides, row maps and tables.
static paco_status_t pass_setup(const paco_plan *pl, Pass *p, const int *f, int n, int i, int t)
{
    PassArgs &a = p->a;
    const PassKernel &k = p->k;
    memset(&a, 0, sizeof(a));
    int lgN = 0;
    for (int j = 0; j < n; ++j) lgN += f[j];
    const int lgL = f[i];
    const int lgC = (i == 0 || i == n - 1) ? lgN - lgL : f[0];      // columns of one row block, and the row stride
    a.bstride = pl->N;
    a.ld_in = 1u << lgC;
    a.ld_out = i == 0 ? 1u << lgL : 1u << lgC;
    a.rev_bits = i == 0 ? 0 : lgL;
    a.rev_t = t;
    for (int j = 0; j < (1 << k.lgA); ++j) a.rowA[j] = rev_host((unsigned)j << k.lgB, a.rev_bits, t) << lgC;
    for (int j = 0; j < (1 << k.lgB); ++j) a.rowK[j] = (unsigned)j << (k.lgA + lgC);
    a.crev_bits = i == 0 ? lgC : (i < n - 1) ? f[2] : 0;
    a.crev_t = t;
    a.lg_tiles = lgC - k.lgW;
    a.blk_stride = 1u << (f[0] + f[1]);
    a.lg_all = lgN - lgL - k.lgW;
    a.lo = static_cast<const cx<float> *>(pl->twN_lo);
    a.hi = static_cast<const cx<float> *>(pl->twN_hi);
    a.lo_bits = pl->twN_lo_bits;
    a.tw_mul = 1u << f[0];
    a.n_mask = (unsigned)(pl->N - 1);
    a.mult = 1.f;
    PACO_CUDA_TRY(cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem));
    const paco_status_t st = gen_table(8, &p->tw, 1LL << lgL, 1LL << lgL, 1, 0);
    a.twL = static_cast<const cx<float> *>(p->tw);
    return st;
}

// Factors of the route, log2, first pass first; returns their number (0: none).
static int route_factors(const paco_plan *pl, int lg1, int lg2, int *f)
{
    if (pl->dims == 3) {
        f[0] = lg1;
        f[1] = pl->lgLa3;
        f[2] = lg2 - pl->lgLa3;
        return 3;
    }
    if (pl->dims == 2) {
        f[0] = lg1;
        f[1] = lg2;
        return 2;
    }
    const int lg = lg1 + lg2;
    if (lg < 10 || lg > 30) return 0;
    if (lg <= 20) {
        f[0] = lg / 2;
        f[1] = lg - f[0];
        return 2;
    }
    f[0] = (lg + 2) / 3;
    f[1] = (lg - f[0] + 1) / 2;
    f[2] = lg - f[0] - f[1];
    return 3;
}

// Builds pl->route; leaves it nullptr where the stage kernels run the plan.
paco_status_t route_setup(paco_plan *pl)
{
    // the plain complex64 form with no stage option asked for
    if (pl->form || pl->shard_G || pl->esize != 8 || pl->req_split || pl->req_ctas || pl->req_tile) return PACO_OK;
    Route *r = new (std::nothrow) Route();
    if (!r) return fail(PACO_ERR_NOMEM, "out of host memory");
    pl->route = r;                                     // freed with the plan
    const int lg[2] = {ilog2_exact(pl->N1), ilog2_exact(pl->N2)}, lgN = lg[0] + lg[1];
    int f[3] = {0, 0, 0};
    int n = pl->fused ? 0 : route_factors(pl, lg[0], lg[1], f);
    for (int i = 0; i < n; ++i) {
        const int lgC = (i == 0 || i == n - 1) ? lgN - f[i] : f[0];
        r->p[i].k = i == 0 ? pass_kernel_first(f[i], lgC) : i == n - 1 ? pass_kernel_last(f[i], lgC)
                                                                       : pass_kernel_middle(f[i], lgC);
        if (!r->p[i].k.fn) n = 0;
    }
    // pi of the redistribution: the plan's base where its digits fit the factors
    int t = pl->t;
    for (int i = 1; i < n; ++i)
        if (f[i] % t) t = 1;
    paco_status_t st = PACO_OK;
    for (int i = 0; i < n && st == PACO_OK; ++i) st = pass_setup(pl, &r->p[i], f, n, i, t);
    r->n = n;
    if (pl->dims == 3) return st;
    for (int i = 0; i < 2 && st == PACO_OK; ++i) {
        r->power[i].k = i == 0 ? pass_kernel_first_stage(lg[0], lg[1]) : pass_kernel_last_loss(lg[1], lg[0]);
        if (r->power[i].k.fn) st = pass_setup(pl, &r->power[i], lg, 2, i, pl->t);
    }
    return st;
}

int route_passes(const paco_plan *pl) { return pl->route ? pl->route->n : 0; }

static paco_status_t launch_pass(const paco_plan *pl, const PassKernel &k, PassArgs &a, const void *in, void *out,
                                 int dir, cudaStream_t stream)
{
    a.in = static_cast<const cx<float> *>(in);
    a.out = static_cast<cx<float> *>(out);
    a.conj = dir == 1;
    const long long tiles = (long long)pl->batch << a.lg_all;
    if (tiles > INT32_MAX) return fail(PACO_ERR_UNSUPPORTED, "batch of %lld transforms is too large", (long long)pl->batch);
    void *params[] = {&a};
    PACO_CUDA_TRY(cudaLaunchKernel(k.fn, dim3((unsigned)tiles), dim3((unsigned)k.threads), params, (size_t)k.smem,
                                   stream));
    return PACO_OK;
}

paco_status_t route_run(const paco_plan *pl, const void *in, void *out, int dir, const StageTerms *terms,
                        cudaStream_t stream)
{
    const Route &r = *pl->route;
    for (int i = 0; i < r.n; ++i) {
        PassArgs a = r.p[i].a;
        if (terms && i == 0) {
            a.mult = terms->ld_mult;
            a.scale = terms->ld_scale;
        }
        const paco_status_t st = launch_pass(pl, r.p[i].k, a, i == 0 ? in : out, out, dir, stream);
        if (st != PACO_OK) return st;
    }
    return PACO_OK;
}

bool route_has_power(const paco_plan *pl, int stage) { return pl->route && pl->route->power[stage].k.fn; }

paco_status_t route_power(const paco_plan *pl, int stage, const void *in, void *out, int dir, const StageTerms &terms,
                          cudaStream_t stream)
{
    PassArgs a = pl->route->power[stage].a;
    a.w = terms.st_w;
    a.loss = terms.st_loss;
    a.store_weighted = terms.st_weighted;
    return launch_pass(pl, pl->route->power[stage].k, a, in, out, dir, stream);
}

} // namespace paco
