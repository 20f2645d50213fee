// The passes of the opening for radius 13 (k_morph.cu).
#include "morph.cuh"

namespace nucseg {

MORPH_PASS(13)

}  // namespace nucseg
