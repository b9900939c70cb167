// zoom_wide_first.cu -- instances of wide_first_kernel (zoom_wide_list.h).
#include "zoom.h"

namespace cwtk {

const void *wide_first_entry(int i) {
    switch (i) {
#define CWT_WIDE_CASE(I, QA) \
    case I: return (const void *)&wide_first_kernel<QA>;
        CWT_WIDE_FIRST(CWT_WIDE_CASE)
#undef CWT_WIDE_CASE
        default: return nullptr;
    }
}

}  // namespace cwtk
