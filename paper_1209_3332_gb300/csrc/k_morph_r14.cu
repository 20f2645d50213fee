// The passes of the opening for radius 14 (k_morph.cu).
#include "morph.cuh"

namespace nucseg {

MORPH_PASS(14)

}  // namespace nucseg
