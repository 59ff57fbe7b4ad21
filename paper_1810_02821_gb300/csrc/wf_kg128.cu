// Cooperative multi-phase kernels for few 128x128 fields (fields in global memory).
#define WF_LAUNCH_DEFINE_GLOBAL
#include "wf_launch.h"

namespace wf {
WF_INSTANTIATE_GLOBAL_ONE(128)
WF_INSTANTIATE_GSPIN2(128)
}  // namespace wf
