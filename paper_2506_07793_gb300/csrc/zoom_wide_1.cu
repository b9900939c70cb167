// zoom_wide_1.cu -- instances of wide_rest_kernel, group 1 of zoom_wide_list.h.
#include "zoom.h"

namespace cwtk {

CWT_WIDE_REST_1(CWT_WIDE_DEFINE)

}  // namespace cwtk
