// zoom_wide_2.cu -- instances of wide_rest_kernel, group 2 of zoom_wide_list.h.
#include "zoom.h"

namespace cwtk {

CWT_WIDE_REST_2(CWT_WIDE_DEFINE)

}  // namespace cwtk
