// Middle- and first-axis kernels of the tensor-core route, axis lengths 32, 36, 40, 45.
#include "pair_split64_ct.cuh"

namespace gw {

GW_PAIR_SPLIT_DEF(32)
GW_PAIR_SPLIT_DEF(36)
GW_PAIR_SPLIT_DEF(40)
GW_PAIR_SPLIT_DEF(45)
GW_PAIR_SPLIT64_DEF(32)
GW_PAIR_SPLIT64_DEF(36)
GW_PAIR_SPLIT64_DEF(40)
GW_PAIR_SPLIT64_DEF(45)

} // namespace gw
