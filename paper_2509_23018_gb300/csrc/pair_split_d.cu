// Middle- and first-axis kernels of the tensor-core route, axis lengths 60, 64, 72.
#include "pair_split64_ct.cuh"

namespace gw {

GW_PAIR_SPLIT_DEF(60)
GW_PAIR_SPLIT_DEF(64)
GW_PAIR_SPLIT_DEF(72)
GW_PAIR_SPLIT64_DEF(60)
GW_PAIR_SPLIT64_DEF(64)
GW_PAIR_SPLIT64_DEF(72)

} // namespace gw
