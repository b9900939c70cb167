// zoom_inst_9.cu -- instances of zoom_kernel, group 9 of zoom_list.h (a
// translation unit of its own so that the groups compile in parallel).
#include "zoom.h"

namespace cwtk {

CWT_ZOOM_GROUP_9(CWT_ZOOM_DEFINE)

}  // namespace cwtk
