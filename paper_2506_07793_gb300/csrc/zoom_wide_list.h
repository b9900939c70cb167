// zoom_wide_list.h -- the instances of wide_first_kernel (index, QA) and of
// wide_rest_kernel (index, QB, QC, P, T, CTAs per SM; zoom_wide.cuh): first
// radices up to 32 over remaining lengths of 256 ... 1024 points, so that a
// padded length finds one for any band up to 20000 bins.  Translation units
// zoom_wide_first.cu and zoom_wide_<g>.cu.
#pragma once

#define CWT_WIDE_FIRST(X) \
    X(0, 2) X(1, 3) X(2, 4) X(3, 5) X(4, 6) X(5, 7) X(6, 8) X(7, 9) X(8, 10) X(9, 12) X(10, 14) X(11, 15) X(12, 16) X(13, 18) X(14, 20) X(15, 21) X(16, 24) X(17, 25) X(18, 27) X(19, 28) X(20, 30) X(21, 32)
#define CWT_WIDE_REST_0(X) \
    X(0, 16, 16, 16, 128, 5) \
    X(4, 16, 20, 16, 128, 4) \
    X(8, 15, 24, 16, 128, 4) \
    X(12, 14, 28, 16, 128, 3) \
    X(16, 15, 28, 16, 128, 3) \
    X(20, 16, 28, 16, 128, 3) \
    X(24, 18, 28, 16, 128, 2) \
    X(28, 20, 28, 16, 128, 2) \
    X(32, 25, 25, 16, 256, 2) \
    X(36, 25, 27, 16, 256, 2) \
    X(14, 32, 32, 8, 256, 2)
#define CWT_WIDE_REST_1(X) \
    X(1, 15, 18, 16, 128, 4) \
    X(5, 18, 18, 16, 128, 4) \
    X(9, 15, 25, 16, 128, 4) \
    X(13, 16, 25, 16, 128, 3) \
    X(17, 16, 27, 16, 128, 3) \
    X(21, 20, 24, 16, 128, 3) \
    X(25, 16, 32, 16, 128, 3) \
    X(29, 21, 27, 16, 256, 2) \
    X(33, 20, 32, 16, 256, 2) \
    X(37, 25, 28, 16, 256, 2)
#define CWT_WIDE_REST_2(X) \
    X(2, 12, 24, 16, 128, 4) \
    X(6, 14, 24, 16, 128, 4) \
    X(10, 14, 27, 16, 128, 4) \
    X(18, 21, 21, 16, 128, 3) \
    X(22, 18, 27, 16, 128, 3) \
    X(26, 21, 25, 16, 128, 2) \
    X(30, 24, 24, 16, 256, 2) \
    X(34, 24, 27, 16, 256, 2) \
    X(38, 27, 27, 8, 128, 4)
#define CWT_WIDE_REST_3(X) \
    X(3, 15, 20, 16, 128, 4) \
    X(7, 14, 25, 16, 128, 4) \
    X(11, 16, 24, 16, 128, 4) \
    X(15, 15, 27, 16, 128, 3) \
    X(19, 15, 30, 16, 128, 3) \
    X(23, 20, 25, 16, 128, 2) \
    X(27, 18, 30, 16, 128, 2) \
    X(31, 24, 25, 16, 256, 2) \
    X(35, 24, 28, 16, 256, 2) \
    X(39, 28, 28, 8, 128, 3)
#define CWT_WIDE_REST(X) CWT_WIDE_REST_0(X) CWT_WIDE_REST_1(X) CWT_WIDE_REST_2(X) CWT_WIDE_REST_3(X)

namespace cwtk {
constexpr int kWideFirst = 22, kWideRest = 40;
}
