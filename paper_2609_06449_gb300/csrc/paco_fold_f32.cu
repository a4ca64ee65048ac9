// paco_fold_f32.cu -- the complex64 passes.
#include "paco_fold.cuh"

namespace paco {

// narrow: tiles of eight columns at 2^8 and 2^9 points, which put more CTAs on
// an SM, where the data stays in L2 and 64-byte rows cost nothing (one 2^16:
// 6.3 -> 5.1 us, one 2^24: 142 -> 135; out of L2 77 x 2^18 would lose 106 -> 112).
// The first pass of 2^8 points is the better for them at any size (2^28 points:
// 0.676 -> 0.618 ms).
// Built: the lengths that a route has in each mode (a first pass and the 2-D and 3-D
// forms 2^5..2^10; TW 1 2^6..2^10; TW 2, from three passes on, 2^7..2^9).
template <bool FIRST, int TW, bool SCALED, int LGA, int LGB, int LGW>
static FoldKernel kernel_of(int lgC)
{
    constexpr int LG = LGA + LGB;
    if constexpr (TW == 0 || (TW == 1 && LG >= 6) || (TW == 2 && LG >= 7 && LG <= 9))
        if (lgC >= LGW) return fold_kernel_of<FoldCfg<float, LGA, LGB, LGW, FIRST, TW, 0, SCALED>>();
    return FoldKernel();
}

template <bool FIRST, int TW, bool SCALED = false>
static FoldKernel pick(int lgL, int lgC, bool narrow)
{
#define PACO_FOLD(LGA, LGB, LGW) kernel_of<FIRST, TW, SCALED, LGA, LGB, LGW>(lgC)
    switch (lgL) {
    case 5: return PACO_FOLD(4, 1, 6);
    case 6: return PACO_FOLD(4, 2, 5);
    case 7: return FIRST ? PACO_FOLD(4, 3, 4) : PACO_FOLD(4, 3, 5);
    case 8: return narrow || FIRST ? PACO_FOLD(4, 4, 3) : PACO_FOLD(4, 4, 4);
    case 9: return narrow ? PACO_FOLD(5, 4, 3) : PACO_FOLD(5, 4, 4);
    case 10: return PACO_FOLD(5, 5, 3);
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
