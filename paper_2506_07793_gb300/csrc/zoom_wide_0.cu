// zoom_wide_0.cu -- instances of wide_rest_kernel, group 0 of zoom_wide_list.h.
#include "zoom.h"

namespace cwtk {

CWT_WIDE_REST_0(CWT_WIDE_DEFINE)

}  // namespace cwtk
