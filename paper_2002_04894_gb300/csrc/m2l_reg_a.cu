// Instances of the register-resident M2L (m2l_reg.cuh).
#include "m2l_reg.cuh"

namespace fmm {
namespace reg {
FMM_M2L_REG(, 12)
}  // namespace reg
}  // namespace fmm
