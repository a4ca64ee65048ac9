// paco_fold_f64.cu -- the complex128 passes.
#include "paco_fold.cuh"

namespace paco {

template <bool FIRST, int TW>
static FoldKernel pick(int lgL, int lgC)
{
#define PACO_FOLD(LGA, LGB, LGW) (lgC >= LGW ? fold_kernel_of<FoldCfg<double, LGA, LGB, LGW, FIRST, TW>>() : FoldKernel())
    switch (lgL) {
    case 5: return PACO_FOLD(4, 1, 5);
    case 6: return PACO_FOLD(3, 3, 4);
    case 7: return PACO_FOLD(4, 3, 3);
    case 8: return PACO_FOLD(4, 4, 3);
    case 9: return PACO_FOLD(5, 4, 3);
    default: return FoldKernel();
    }
}

FoldKernel fold_kernel_f64(bool first, int tw, int lgL, int lgC)
{
    if (first) return pick<true, 0>(lgL, lgC);
    return tw == 0 ? pick<false, 0>(lgL, lgC) : tw == 1 ? pick<false, 1>(lgL, lgC) : pick<false, 2>(lgL, lgC);
}

} // namespace paco
