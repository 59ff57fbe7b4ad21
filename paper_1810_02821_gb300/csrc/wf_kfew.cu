// Few fields up to 256x256: one thread-block cluster per field.
#define WF_LAUNCH_DEFINE_FEW
#include "wf_launch.h"

namespace wf {
WF_INSTANTIATE_FEW(64)
WF_INSTANTIATE_FEW(128)
WF_INSTANTIATE_FEW(256)
WF_INSTANTIATE_FEW2(128)
}  // namespace wf
