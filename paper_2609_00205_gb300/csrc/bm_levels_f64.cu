// Line passes of the global levels instantiated for double fields.
#include "bm_levels.cuh"

namespace bm {

BM_LEVELS(double)

}  // namespace bm
