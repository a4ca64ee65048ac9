// paco_pass_last.cu -- the "last" passes (Phase III).
#include "paco_pass.cuh"

namespace paco {

PassKernel pass_kernel_last(int lgL, int lgC)
{
    switch (lgL) {
    case 5: return lgC >= 6 ? pass_kernel_of<4, 1, 6, 0>() : PassKernel();
    case 6: return lgC >= 5 ? pass_kernel_of<4, 2, 5, 0>() : PassKernel();
    case 7: return lgC >= 5 ? pass_kernel_of<4, 3, 5, 0>() : PassKernel();
    case 8: return lgC < 4 ? PassKernel() : lgC >= 17 ? pass_kernel_of<4, 4, 5, 0>() : pass_kernel_of<4, 4, 4, 0>();
    case 9: return lgC >= 4 ? pass_kernel_of<5, 4, 4, 0>() : PassKernel();
    case 10: return lgC < 3 ? PassKernel() : lgC >= 17 ? pass_kernel_of<5, 5, 4, 0>() : pass_kernel_of<5, 5, 3, 0>();
    default: return PassKernel();
    }
}

} // namespace paco
