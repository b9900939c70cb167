// zoom_list.h -- the instances of zoom_kernel (zoom.cuh): QA, QB, QC (1: two
// passes), columns P and threads T per CTA, CTAs per SM of the register
// budget, and the cost in ps per output point (mean of power-only and
// complex-and-power launches of 32 Mi points on a GB300, R = 64 residues).
// Chosen among 950 timed combinations: those that lower the mean cost of rows
// with padded lengths of 100 ... 131072 points (powers of two, smooth lengths
// and whole seconds, decimations 1 ... 8) and bands of 0.4 ... 30% of the row.
// Two-pass instances hold about 8192 points of tile on 128 threads, several
// CTAs per SM: 8 x 32 on 256 threads, three CTAs of 32 columns, takes 1.76 /
// 2.20 ps per point (power / complex and power) against 1.64 / 2.03.  Above
// Q = 1024 the tile leaves 4 columns, whose stores are 16-byte pieces; wider
// bands take the two kernels of zoom_wide.cuh.
// The groups are translation units (zoom_inst_<g>.cu).
#pragma once

#define CWT_ZOOM_GROUP_0(X) \
    X(0, 5, 5, 1, 32, 128, 6, 2.28f) \
    X(12, 6, 9, 1, 32, 128, 6, 1.95f) \
    X(24, 7, 21, 1, 32, 128, 4, 1.94f) \
    X(35, 15, 25, 1, 16, 128, 4, 2.29f) \
    X(47, 24, 28, 1, 16, 256, 2, 2.56f) \
    X(59, 8, 15, 16, 4, 256, 2, 4.29f) \
    X(71, 9, 21, 21, 4, 512, 1, 5.03f) \
    X(79, 10, 25, 25, 2, 512, 1, 7.8f)
#define CWT_ZOOM_GROUP_1(X) \
    X(1, 4, 7, 1, 32, 128, 6, 2.02f) \
    X(13, 5, 12, 1, 32, 128, 6, 1.78f) \
    X(25, 9, 18, 1, 32, 128, 4, 1.9f) \
    X(36, 14, 28, 1, 16, 128, 3, 2.19f) \
    X(48, 7, 7, 14, 8, 256, 3, 3.34f) \
    X(60, 10, 14, 14, 4, 256, 2, 4.68f) \
    X(72, 10, 20, 20, 4, 512, 1, 4.87f)
#define CWT_ZOOM_GROUP_2(X) \
    X(2, 5, 6, 1, 32, 128, 6, 1.98f) \
    X(14, 7, 9, 1, 32, 128, 6, 1.9f) \
    X(26, 7, 25, 1, 32, 128, 4, 2.08f) \
    X(37, 20, 20, 1, 16, 128, 3, 2.15f) \
    X(49, 27, 27, 1, 8, 128, 4, 2.84f) \
    X(61, 9, 15, 15, 4, 256, 2, 4.68f) \
    X(73, 15, 15, 18, 4, 512, 1, 5.31f)
#define CWT_ZOOM_GROUP_3(X) \
    X(3, 4, 8, 1, 32, 128, 6, 1.75f) \
    X(15, 4, 16, 1, 32, 128, 6, 1.67f) \
    X(27, 9, 21, 1, 32, 128, 4, 2.06f) \
    X(38, 21, 21, 1, 16, 128, 3, 2.5f) \
    X(50, 7, 7, 15, 8, 256, 3, 3.3f) \
    X(62, 8, 16, 16, 8, 512, 1, 3.72f) \
    X(74, 16, 16, 16, 4, 512, 1, 4.67f)
#define CWT_ZOOM_GROUP_4(X) \
    X(4, 5, 7, 1, 32, 128, 6, 2.12f) \
    X(16, 5, 15, 1, 32, 128, 6, 1.89f) \
    X(28, 10, 20, 1, 32, 128, 3, 1.92f) \
    X(39, 20, 24, 1, 16, 128, 3, 2.26f) \
    X(51, 25, 30, 1, 8, 128, 3, 3.02f) \
    X(63, 12, 12, 15, 4, 256, 2, 4.42f) \
    X(75, 10, 21, 21, 4, 512, 1, 4.97f)
#define CWT_ZOOM_GROUP_5(X) \
    X(5, 6, 6, 1, 32, 128, 6, 1.88f) \
    X(17, 9, 9, 1, 32, 128, 6, 1.95f) \
    X(29, 8, 30, 1, 32, 128, 3, 1.96f) \
    X(40, 7, 7, 10, 16, 256, 3, 2.74f) \
    X(52, 28, 28, 1, 8, 128, 3, 2.88f) \
    X(64, 10, 14, 16, 4, 256, 2, 4.61f) \
    X(76, 16, 16, 18, 4, 512, 1, 4.65f)
#define CWT_ZOOM_GROUP_6(X) \
    X(6, 4, 10, 1, 32, 128, 6, 1.79f) \
    X(18, 10, 10, 1, 32, 128, 6, 1.86f) \
    X(30, 10, 25, 1, 32, 128, 3, 2.21f) \
    X(41, 21, 24, 1, 16, 128, 3, 2.37f) \
    X(53, 28, 32, 1, 8, 128, 3, 2.83f) \
    X(65, 10, 12, 20, 4, 512, 1, 4.87f) \
    X(77, 14, 16, 21, 4, 512, 1, 4.94f)
#define CWT_ZOOM_GROUP_7(X) \
    X(7, 6, 7, 1, 32, 128, 6, 2.05f) \
    X(19, 7, 15, 1, 32, 128, 6, 1.84f) \
    X(42, 16, 32, 1, 16, 128, 3, 2.21f) \
    X(54, 32, 32, 1, 8, 256, 2, 2.79f) \
    X(66, 9, 18, 18, 4, 512, 1, 5.33f)
#define CWT_ZOOM_GROUP_8(X) \
    X(8, 5, 9, 1, 32, 128, 6, 2.04f) \
    X(20, 7, 16, 1, 32, 128, 6, 1.79f) \
    X(31, 8, 32, 1, 16, 128, 5, 1.83f) \
    X(43, 21, 25, 1, 16, 128, 2, 2.55f) \
    X(55, 9, 9, 15, 4, 256, 3, 4.48f) \
    X(67, 12, 16, 16, 4, 512, 1, 4.67f) \
    X(78, 16, 18, 18, 4, 512, 1, 4.82f)
#define CWT_ZOOM_GROUP_9(X) \
    X(9, 4, 12, 1, 32, 128, 6, 1.71f) \
    X(21, 5, 25, 1, 32, 128, 4, 2.22f) \
    X(32, 10, 28, 1, 32, 128, 2, 2.06f) \
    X(44, 18, 30, 1, 16, 128, 2, 2.35f) \
    X(56, 9, 12, 12, 4, 256, 3, 4.25f) \
    X(68, 15, 15, 15, 4, 512, 1, 4.99f)
#define CWT_ZOOM_GROUP_10(X) \
    X(10, 7, 7, 1, 32, 128, 6, 1.98f) \
    X(22, 8, 16, 1, 32, 128, 6, 1.73f) \
    X(33, 16, 18, 1, 16, 128, 4, 2.1f) \
    X(45, 25, 25, 1, 16, 256, 2, 2.83f) \
    X(57, 10, 10, 14, 4, 256, 3, 4.34f) \
    X(69, 9, 18, 21, 4, 512, 1, 5.01f)
#define CWT_ZOOM_GROUP_11(X) \
    X(11, 5, 10, 1, 32, 128, 6, 1.82f) \
    X(23, 9, 15, 1, 32, 128, 5, 1.98f) \
    X(34, 15, 21, 1, 16, 128, 4, 2.17f) \
    X(46, 20, 32, 1, 16, 256, 2, 2.62f) \
    X(58, 7, 15, 15, 4, 256, 3, 4.34f) \
    X(70, 12, 16, 20, 4, 512, 1, 4.8f)
#define CWT_ZOOM_ALL(X) \
    CWT_ZOOM_GROUP_0(X) CWT_ZOOM_GROUP_1(X) CWT_ZOOM_GROUP_2(X) CWT_ZOOM_GROUP_3(X) CWT_ZOOM_GROUP_4(X) CWT_ZOOM_GROUP_5(X) CWT_ZOOM_GROUP_6(X) CWT_ZOOM_GROUP_7(X) CWT_ZOOM_GROUP_8(X) CWT_ZOOM_GROUP_9(X) CWT_ZOOM_GROUP_10(X) CWT_ZOOM_GROUP_11(X)

namespace cwtk {
constexpr int kZoomInstances = 80;
}
