// Instances of the register-resident M2L (m2l_reg.cuh).
#include "m2l_reg.cuh"

namespace fmm {
namespace reg {
FMM_M2L_REG(, 9)
FMM_M2L_REG(, 4)
}  // namespace reg
}  // namespace fmm
