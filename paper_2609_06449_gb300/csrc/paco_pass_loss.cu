// paco_pass_loss.cu -- the two passes of the weighted power of the spectrum.
#include "paco_pass.cuh"

namespace paco {

PassKernel pass_kernel_first_stage(int lgL, int lgC)
{
    switch (lgL) {
    case 5: return lgC >= 6 ? pass_kernel_of<3, 2, 6, 4>() : PassKernel();
    case 6: return lgC >= 5 ? pass_kernel_of<3, 3, 5, 4>() : PassKernel();
    case 7: return lgC >= 4 ? pass_kernel_of<4, 3, 4, 4>() : PassKernel();
    case 8: return lgC >= 4 ? pass_kernel_of<4, 4, 4, 4>() : PassKernel();
    case 9: return lgC >= 4 ? pass_kernel_of<5, 4, 4, 4>() : PassKernel();
    case 10: return lgC >= 3 ? pass_kernel_of<5, 5, 3, 4>() : PassKernel();
    default: return PassKernel();
    }
}

PassKernel pass_kernel_last_loss(int lgL, int lgC)
{
    switch (lgL) {
    case 5: return lgC >= 6 ? pass_kernel_of<3, 2, 6, 3>() : PassKernel();
    case 6: return lgC >= 5 ? pass_kernel_of<3, 3, 5, 3>() : PassKernel();
    case 7: return lgC >= 4 ? pass_kernel_of<4, 3, 4, 3>() : PassKernel();
    case 8: return lgC >= 4 ? pass_kernel_of<4, 4, 4, 3>() : PassKernel();
    case 9: return lgC >= 4 ? pass_kernel_of<5, 4, 4, 3>() : PassKernel();
    case 10: return lgC >= 3 ? pass_kernel_of<5, 5, 3, 3>() : PassKernel();
    default: return PassKernel();
    }
}

} // namespace paco
