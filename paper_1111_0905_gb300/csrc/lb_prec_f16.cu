// Launch table of the __half population storage (see lb_launch.cuh).
#include "lb_launch.cuh"

namespace tlbm {
const PrecOps kOpsF16 = {sizeof(__half), 1, &OpsImpl<__half>::prepare, &OpsImpl<__half>::fused,
                    &OpsImpl<__half>::init, &OpsImpl<__half>::pops,
                    &OpsImpl<__half>::tile_ok, &OpsImpl<__half>::info,
                    &OpsImpl<__half>::setpops, &OpsImpl<__half>::split,
                    &OpsImpl<__half>::march, &OpsImpl<__half>::step_info, OpsImpl<__half>::MTY, OpsImpl<__half>::MTY2, slots<__half>()};
}  // namespace tlbm
