// Few fields of 128x128 and 256x256, one thread-block cluster each.
#define WF_LAUNCH_DEFINE_GCLUSTER
#include "wf_launch.h"

namespace wf {
WF_INSTANTIATE_GCLUSTER(128)
WF_INSTANTIATE_GCLUSTER(256)
}  // namespace wf
