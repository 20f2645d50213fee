// The passes of the opening for radii 1, 2, 3, 4, 5, 6 (k_morph.cu).
#include "morph.cuh"

namespace nucseg {

MORPH_PASS(1)
MORPH_PASS(2)
MORPH_PASS(3)
MORPH_PASS(4)
MORPH_PASS(5)
MORPH_PASS(6)

}  // namespace nucseg
