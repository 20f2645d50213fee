// The passes of the opening for radii 7, 8 (k_morph.cu).
#include "morph.cuh"

namespace nucseg {

MORPH_PASS(7)
MORPH_PASS(8)

}  // namespace nucseg
