// paco_tcpass.cu -- the tensor-core passes by form and length.
#include "paco_tcpass.cuh"

namespace paco {

template <int FORM, int LGB, int LGW, bool FIRST, bool TC2>
static FoldKernel kernel_of(int lgC)
{
    using CFG = TcPassCfg<FORM, LGB, LGW, FIRST, TC2>;
    FoldKernel k;
    if (lgC < LGW) return k;
    k.fn = reinterpret_cast<const void *>(&paco_tcpass_kernel<CFG>);
    k.lgA = 4;
    k.lgB = LGB;
    k.lgW = LGW;
    k.threads = CFG::NT;
    k.smem = CFG::SMEM;
    return k;
}

template <int FORM>
static FoldKernel pick(bool first, bool tc2, int lgL, int lgC)
{
    switch (lgL) {
    case 5: return first ? FoldKernel() : kernel_of<FORM, 1, 5, false, false>(lgC);
    case 6: return first ? kernel_of<FORM, 2, 5, true, false>(lgC) : kernel_of<FORM, 2, 5, false, false>(lgC);
    case 7: return first ? kernel_of<FORM, 3, 4, true, false>(lgC) : kernel_of<FORM, 3, 5, false, false>(lgC);
    case 8:
        if (first) return kernel_of<FORM, 4, 4, true, true>(lgC);
        return tc2 ? kernel_of<FORM, 4, 4, false, true>(lgC) : kernel_of<FORM, 4, 4, false, false>(lgC);
    default: return FoldKernel();
    }
}

FoldKernel tcpass_kernel(int form, bool first, bool tc2, int lgL, int lgC)
{
    return form == TC_BF16X3 ? pick<TC_BF16X3>(first, tc2, lgL, lgC) : pick<TC_FP16>(first, tc2, lgL, lgC);
}

} // namespace paco
