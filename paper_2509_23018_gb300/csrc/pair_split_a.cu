// Middle- and first-axis kernels of the tensor-core route, axis lengths 20, 24, 25, 27, 30.
#include "pair_split64_ct.cuh"

namespace gw {

GW_PAIR_SPLIT_DEF(20)
GW_PAIR_SPLIT_DEF(24)
GW_PAIR_SPLIT_DEF(25)
GW_PAIR_SPLIT_DEF(27)
GW_PAIR_SPLIT_DEF(30)
GW_PAIR_SPLIT64_DEF(20)
GW_PAIR_SPLIT64_DEF(24)
GW_PAIR_SPLIT64_DEF(25)
GW_PAIR_SPLIT64_DEF(27)
GW_PAIR_SPLIT64_DEF(30)

} // namespace gw
