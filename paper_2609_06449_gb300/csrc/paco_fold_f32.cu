// paco_fold_f32.cu -- the complex64 passes.
#include "paco_fold.cuh"

namespace paco {

// narrow: tiles of eight columns at 2^8 and 2^9 points, which put more CTAs on
// an SM, where the data stays in L2 and 64-byte rows cost nothing (one 2^16:
// 6.3 -> 5.1 us, one 2^24: 142 -> 135; out of L2 77 x 2^18 would lose 106 -> 112).
// The first pass of 2^8 points is the better for them at any size (2^28 points:
// 0.676 -> 0.618 ms).
template <bool FIRST, int TW, bool SCALED = false>
static FoldKernel pick(int lgL, int lgC, bool narrow)
{
#define PACO_FOLD(LGA, LGB, LGW) (lgC >= LGW ? fold_kernel_of<FoldCfg<float, LGA, LGB, LGW, FIRST, TW, 0, SCALED>>() : FoldKernel())
    switch (lgL) {
    case 5: return PACO_FOLD(4, 1, 6);
    case 6: return PACO_FOLD(4, 2, 5);
    case 7: return FIRST ? PACO_FOLD(4, 3, 4) : PACO_FOLD(4, 3, 5);
    case 8: return narrow || FIRST ? PACO_FOLD(4, 4, 3) : PACO_FOLD(4, 4, 4);
    case 9: return narrow ? PACO_FOLD(5, 4, 3) : PACO_FOLD(5, 4, 4);
    case 10: return !FIRST && lgC >= 17 ? PACO_FOLD(5, 5, 4) : PACO_FOLD(5, 5, 3);
    default: return FoldKernel();
    }
}

FoldKernel fold_kernel_f32(bool first, int tw, int lgL, int lgC, bool narrow, bool scaled)
{
    if (first) return scaled ? pick<true, 0, true>(lgL, lgC, narrow) : pick<true, 0>(lgL, lgC, narrow);
    return tw == 0 ? pick<false, 0>(lgL, lgC, narrow)
                   : tw == 1 ? pick<false, 1>(lgL, lgC, narrow) : pick<false, 2>(lgL, lgC, narrow);
}

} // namespace paco
