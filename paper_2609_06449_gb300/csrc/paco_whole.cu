// paco_whole.cu -- the kernels of paco_whole.cuh by length.
#include "paco_whole.cuh"

namespace paco {

template <int LG, int EPT, int NT>
static WholeKernel kernel_of(bool scaled)
{
    using CFG = WholeCfg<LG, EPT, NT>;
    WholeKernel k;
    k.fn = scaled ? reinterpret_cast<const void *>(&paco_whole_kernel<LG, EPT, NT, true>)
                  : reinterpret_cast<const void *>(&paco_whole_kernel<LG, EPT, NT, false>);
    k.threads = NT;
    k.smem = CFG::SMEM;
    k.per_cta = CFG::G;
    return k;
}

WholeKernel whole_kernel(int lgN, bool scaled)
{
    switch (lgN) {
    case 4: return kernel_of<4, 16, 256>(scaled);
    case 5: return kernel_of<5, 16, 256>(scaled);
    case 6: return kernel_of<6, 16, 256>(scaled);
    case 7: return kernel_of<7, 16, 256>(scaled);
    case 8: return kernel_of<8, 16, 256>(scaled);
    case 9: return kernel_of<9, 16, 256>(scaled);
    case 10: return kernel_of<10, 16, 256>(scaled);
    case 11: return kernel_of<11, 16, 256>(scaled);
    case 12: return kernel_of<12, 16, 256>(scaled);
    case 13: return kernel_of<13, 32, 256>(scaled);
    case 14: return kernel_of<14, 32, 512>(scaled);
    default: return WholeKernel();
    }
}

} // namespace paco
