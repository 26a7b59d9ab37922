// The paired ping-pong step with population loads that leave L2 first (l2_policy in
// lbm_kernels.cu): for lattices of which one population copy fits L2, whose next step then finds
// most of its inputs there.
#define LBM_L2_FIRST
#include "lbm_pair.cu"
