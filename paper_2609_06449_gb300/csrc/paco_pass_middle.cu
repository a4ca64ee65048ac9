// paco_pass_middle.cu -- the "middle" passes (first half of a split Phase III).
#include "paco_pass.cuh"

namespace paco {

PassKernel pass_kernel_middle(int lgL, int lgC)
{
    switch (lgL) {
    case 5: return lgC >= 6 ? pass_kernel_of<4, 1, 6, 2>() : PassKernel();
    case 6: return lgC >= 5 ? pass_kernel_of<4, 2, 5, 2>() : PassKernel();
    case 7: return lgC >= 5 ? pass_kernel_of<4, 3, 5, 2>() : PassKernel();
    case 8: return lgC >= 4 ? pass_kernel_of<4, 4, 4, 2>() : PassKernel();
    case 9: return lgC >= 4 ? pass_kernel_of<5, 4, 4, 2>() : PassKernel();
    case 10: return lgC >= 4 ? pass_kernel_of<5, 5, 4, 2>() : PassKernel();
    default: return PassKernel();
    }
}

} // namespace paco
