// paco_power.cu -- the kernels of paco_power.cuh by stage length.  The tiles
// and the factors A * B are the stage kernels', so that a thread's partial sums
// cover the same results.
#include "paco_plan.h"
#include "paco_power.cuh"

namespace paco {

template <int LGA, int LGB, int LGW, bool FIRST>
static PowerKernel kernel_of()
{
    using CFG = PowerCfg<LGA, LGB, LGW, FIRST>;
    PowerKernel k;
    k.fn = reinterpret_cast<const void *>(&paco_power_kernel<CFG>);
    k.lgA = LGA;
    k.lgB = LGB;
    k.lgW = LGW;
    k.threads = CFG::NT;
    k.smem = CFG::SMEM;
    return k;
}

template <bool FIRST>
static PowerKernel pick(int lgL, int lgC)
{
    switch (lgL) {
    case 5: return lgC >= 6 ? kernel_of<3, 2, 6, FIRST>() : PowerKernel();
    case 6: return lgC >= 5 ? kernel_of<3, 3, 5, FIRST>() : PowerKernel();
    case 7: return lgC >= 4 ? kernel_of<4, 3, 4, FIRST>() : PowerKernel();
    case 8: return lgC >= 4 ? kernel_of<4, 4, 4, FIRST>() : PowerKernel();
    case 9: return lgC >= 4 ? kernel_of<5, 4, 4, FIRST>() : PowerKernel();
    case 10: return lgC >= 3 ? kernel_of<5, 5, 3, FIRST>() : PowerKernel();
    default: return PowerKernel();
    }
}

// Entry r < count: w_M^{-r mult}, or (split) the product of entries r mod split and
// the rest of r, as the weighted power's stages take it.
struct TableSpec {
    void *out;
    long long M, mult;
    int count, split;
};
struct TableSpecs {
    TableSpec t[7];
};
template <typename R>
__global__ void plan_tables_kernel(const __grid_constant__ TableSpecs specs)
{
    const TableSpec &t = specs.t[blockIdx.y];
    auto root = [&](long long r) {
        double sn, cs;
        sincospi(2.0 * (double)((r * t.mult) % t.M) / (double)t.M, &sn, &cs);
        return make_cx<R>((R)cs, (R)(-sn));
    };
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < t.count; r += gridDim.x * blockDim.x) {
        cx<R> w = root(t.split ? r & (t.split - 1) : r);
        if constexpr (sizeof(R) == 4)
            if (t.split) {
                const cx<R> hi = root(r & ~(t.split - 1));
                w = t.count > 64 ? st::mul<1>(w, hi) : st::mul<0>(w, hi);
            }
        static_cast<cx<R> *>(t.out)[r] = w;
    }
}

paco_status_t plan_tables(paco_plan *pl, bool power)
{
    const int lgN = ilog2_exact(pl->N);
    pl->twN_lo_bits = (lgN + 1) / 2;
    const long long nlo = 1LL << pl->twN_lo_bits, nhi = pl->N / nlo, Mtw = pl->dims >= 2 ? 1 : pl->N;
    auto split = [](int64_t L) { return 1 << ((ilog2_exact(L) + 1) / 2); };
    struct { void **dst; TableSpec t; } want[7] = {
        {&pl->twL1, {nullptr, pl->N1, 1, (int)pl->N1, 0}},
        {&pl->twL2, {nullptr, pl->N2, 1, (int)pl->N2, 0}},
        {&pl->twN_lo, {nullptr, Mtw, 1, (int)nlo, 0}},
        {&pl->twN_hi, {nullptr, Mtw, nlo, (int)nhi, 0}},
        {&pl->tw_ones, {nullptr, 1, 1, pl->dims == 3 ? (int)pl->N2 : 0, 0}},
        {&pl->twP[0], {nullptr, pl->N1, 1, power ? (int)pl->N1 : 0, split(pl->N1)}},
        {&pl->twP[1], {nullptr, pl->N2, 1, power ? (int)pl->N2 : 0, split(pl->N2)}}};
    size_t bytes = 0;
    TableSpecs specs;
    int n = 0;
    for (auto &w : want) bytes += ((size_t)w.t.count * pl->esize + 255) & ~(size_t)255;
    PACO_CUDA_TRY(cudaMalloc(&pl->tables, bytes));
    bytes = 0;
    for (auto &w : want) {
        if (!w.t.count) continue;
        w.t.out = *w.dst = static_cast<char *>(pl->tables) + bytes;
        specs.t[n++] = w.t;
        bytes += ((size_t)w.t.count * pl->esize + 255) & ~(size_t)255;
    }
    if (pl->esize == 8) plan_tables_kernel<float><<<dim3(64, n), 256>>>(specs);
    else plan_tables_kernel<double><<<dim3(64, n), 256>>>(specs);
    PACO_CUDA_TRY(cudaGetLastError());
    return PACO_OK;
}

PowerKernel power_kernel(bool first, int lgL, int lgC) { return first ? pick<true>(lgL, lgC) : pick<false>(lgL, lgC); }

} // namespace paco
