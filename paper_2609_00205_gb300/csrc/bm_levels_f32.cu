// Line passes of the global levels instantiated for float fields.
#include "bm_levels.cuh"

namespace bm {

BM_LEVELS(float)

}  // namespace bm
