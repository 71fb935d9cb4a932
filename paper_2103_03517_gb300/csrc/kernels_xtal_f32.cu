// kernels_xtal_f32.cu -- float instances of the crystal kernels (xtal_pass.cuh).
#include "xtal_pass.cuh"

namespace mcgb {
namespace {

using R = float;

#include "xtal_launch.cuh"

}  // namespace

const XtalKernels& xtal_f32() {
    static const XtalKernels k{pass, sample, field};
    return k;
}

}  // namespace mcgb
