// zoom_wide_3.cu -- instances of wide_rest_kernel, group 3 of zoom_wide_list.h.
#include "zoom.h"

namespace cwtk {

CWT_WIDE_REST_3(CWT_WIDE_DEFINE)

}  // namespace cwtk
