// paco_pass_first.cu -- the "first" passes (Phase I with the redistribution).
#include "paco_pass.cuh"

namespace paco {

PassKernel pass_kernel_first(int lgL, int lgC)
{
    switch (lgL) {
    case 5: return lgC >= 6 ? pass_kernel_of<4, 1, 6, 1>() : PassKernel();
    case 6: return lgC >= 5 ? pass_kernel_of<4, 2, 5, 1>() : PassKernel();
    case 7: return lgC >= 4 ? pass_kernel_of<4, 3, 4, 1>() : PassKernel();
    case 8: return lgC >= 4 ? pass_kernel_of<4, 4, 4, 1>() : PassKernel();
    case 9: return lgC >= 4 ? pass_kernel_of<5, 4, 4, 1>() : PassKernel();
    case 10: return lgC >= 3 ? pass_kernel_of<5, 5, 3, 1>() : PassKernel();
    default: return PassKernel();
    }
}

} // namespace paco
