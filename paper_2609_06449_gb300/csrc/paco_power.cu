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

__global__ void power_table_kernel(const cx<float> *w, cx<float> *out, int lgL)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x, s = 1 << ((lgL + 1) / 2);
    if (r >= 1 << lgL) return;
    const cx<float> lo = w[r & (s - 1)], hi = w[r & ~(s - 1)];
    out[r] = lgL > 6 ? st::mul<1>(lo, hi) : st::mul<0>(lo, hi);
}

paco_status_t power_table(const cx<float> *w, int lgL, void **dst)
{
    PACO_CUDA_TRY(cudaMalloc(dst, (size_t)8 << lgL));
    power_table_kernel<<<((1 << lgL) + 255) / 256, 256>>>(w, static_cast<cx<float> *>(*dst), lgL);
    PACO_CUDA_TRY(cudaGetLastError());
    return PACO_OK;
}

PowerKernel power_kernel(bool first, int lgL, int lgC) { return first ? pick<true>(lgL, lgC) : pick<false>(lgL, lgC); }

} // namespace paco
