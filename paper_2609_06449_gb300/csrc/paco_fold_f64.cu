// paco_fold_f64.cu -- the complex128 passes.
#include "paco_fold.cuh"

namespace paco {

// Built: the lengths that a route has in each mode (2^5..2^9; from three passes on
// 2^6, and 2^7 with TW 2).
template <bool FIRST, int TW, bool CLOSER, int LGA, int LGB, int LGW>
static FoldKernel kernel_of(int lgC)
{
    if constexpr (LGA + LGB >= (TW == 2 ? 7 : CLOSER ? 6 : 5))
        if (lgC >= LGW) return fold_kernel_of<FoldCfg<double, LGA, LGB, LGW, FIRST, TW, 0, false, CLOSER>>();
    return FoldKernel();
}

template <bool FIRST, int TW, bool CLOSER = false>
static FoldKernel pick(int lgL, int lgC)
{
#define PACO_FOLD(LGA, LGB, LGW) kernel_of<FIRST, TW, CLOSER, LGA, LGB, LGW>(lgC)
    switch (lgL) {
    case 5: return PACO_FOLD(4, 1, 5);
    case 6: return PACO_FOLD(3, 3, 4);
    case 7: return PACO_FOLD(4, 3, 3);
    case 8: return PACO_FOLD(4, 4, 3);
    case 9: return PACO_FOLD(5, 4, 3);
    default: return FoldKernel();
    }
}

FoldKernel fold_kernel_f64(bool first, int tw, int lgL, int lgC, bool closer)
{
    if (first) return pick<true, 0>(lgL, lgC);
    if (tw == 0) return pick<false, 0>(lgL, lgC);
    if (tw == 2) return pick<false, 2>(lgL, lgC);
    return closer ? pick<false, 1, true>(lgL, lgC) : pick<false, 1>(lgL, lgC);
}

} // namespace paco
