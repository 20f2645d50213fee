// The passes of the opening for radii 10, 11 (k_morph.cu).
#include "morph.cuh"

namespace nucseg {

MORPH_PASS(10)
MORPH_PASS(11)

}  // namespace nucseg
