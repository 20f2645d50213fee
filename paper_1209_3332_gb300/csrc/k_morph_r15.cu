// The passes of the opening for radius 15 (k_morph.cu).
#include "morph.cuh"

namespace nucseg {

MORPH_PASS(15)

}  // namespace nucseg
