// The passes of the opening for radius 12 (k_morph.cu).
#include "morph.cuh"

namespace nucseg {

MORPH_PASS(12)

}  // namespace nucseg
