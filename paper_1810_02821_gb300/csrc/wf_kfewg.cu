// Few large fields: a block of rows and of columns per CTA, the half spectrum in global memory.
#define WF_LAUNCH_DEFINE_FEW
#include "wf_launch.h"

namespace wf {
WF_INSTANTIATE_FEW(512)
WF_INSTANTIATE_FEW(1024)
WF_INSTANTIATE_FEW2(256)
WF_INSTANTIATE_FEW2(512)
}  // namespace wf
