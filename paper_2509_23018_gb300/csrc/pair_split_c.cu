// Middle- and first-axis kernels of the tensor-core route, axis lengths 48, 50, 54.
#include "pair_split64_ct.cuh"

namespace gw {

GW_PAIR_SPLIT_DEF(48)
GW_PAIR_SPLIT_DEF(50)
GW_PAIR_SPLIT_DEF(54)
GW_PAIR_SPLIT64_DEF(48)
GW_PAIR_SPLIT64_DEF(50)
GW_PAIR_SPLIT64_DEF(54)

} // namespace gw
