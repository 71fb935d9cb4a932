// kernels_xtal_f64.cu -- double instances of the crystal kernels (xtal_pass.cuh).
// Built with -fmad=false, as kernels_f64.cu.
#include "xtal_pass.cuh"

namespace mcgb {
namespace {

using R = double;

#include "xtal_launch.cuh"

}  // namespace

const XtalKernels& xtal_f64() {
    static const XtalKernels k{pass, sample, field};
    return k;
}

}  // namespace mcgb
