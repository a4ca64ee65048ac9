// paco_power.cu -- the kernels of paco_power.cuh by stage length.  The tiles
// and the factors A * B are the stage kernels', so that a thread's partial sums
// cover the same results.
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

PowerKernel power_kernel(bool first, int lgL, int lgC) { return first ? pick<true>(lgL, lgC) : pick<false>(lgL, lgC); }

} // namespace paco
