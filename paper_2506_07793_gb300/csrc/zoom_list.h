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
// Q = 1024 the tile leaves 4 columns, then 2, whose stores are 16- and 8-byte
// pieces.
// The groups are translation units (zoom_inst_<g>.cu).
#pragma once

#define CWT_ZOOM_GROUP_0(X) \
    X(0, 5, 5, 1, 32, 128, 6, 2.28f) \
    X(12, 6, 9, 1, 32, 128, 6, 1.95f) \
    X(24, 7, 21, 1, 32, 128, 4, 1.94f) \
    X(36, 15, 25, 1, 16, 128, 4, 2.29f) \
    X(48, 24, 28, 1, 16, 256, 2, 2.56f) \
    X(60, 8, 15, 16, 4, 256, 2, 4.29f) \
    X(72, 9, 21, 21, 4, 512, 1, 5.03f) \
    X(84, 10, 25, 25, 2, 512, 1, 7.8f)
#define CWT_ZOOM_GROUP_1(X) \
    X(1, 4, 7, 1, 32, 128, 6, 2.02f) \
    X(13, 5, 12, 1, 32, 128, 6, 1.78f) \
    X(25, 9, 18, 1, 32, 128, 4, 1.9f) \
    X(37, 14, 28, 1, 16, 128, 3, 2.19f) \
    X(49, 7, 7, 14, 8, 256, 3, 3.34f) \
    X(61, 10, 14, 14, 4, 256, 2, 4.68f) \
    X(73, 10, 20, 20, 4, 512, 1, 4.87f) \
    X(85, 14, 16, 28, 2, 512, 1, 7.36f)
#define CWT_ZOOM_GROUP_2(X) \
    X(2, 5, 6, 1, 32, 128, 6, 1.98f) \
    X(14, 7, 9, 1, 32, 128, 6, 1.9f) \
    X(26, 7, 25, 1, 32, 128, 4, 2.08f) \
    X(38, 20, 20, 1, 16, 128, 3, 2.15f) \
    X(50, 27, 27, 1, 8, 128, 4, 2.84f) \
    X(62, 9, 15, 15, 4, 256, 2, 4.68f) \
    X(74, 15, 15, 18, 4, 512, 1, 5.31f) \
    X(86, 15, 21, 21, 2, 512, 1, 7.53f)
#define CWT_ZOOM_GROUP_3(X) \
    X(3, 4, 8, 1, 32, 128, 6, 1.75f) \
    X(15, 4, 16, 1, 32, 128, 6, 1.67f) \
    X(27, 9, 21, 1, 32, 128, 4, 2.06f) \
    X(39, 21, 21, 1, 16, 128, 3, 2.5f) \
    X(51, 7, 7, 15, 8, 256, 3, 3.3f) \
    X(63, 8, 16, 16, 8, 512, 1, 3.72f) \
    X(75, 16, 16, 16, 4, 512, 1, 4.67f) \
    X(87, 16, 18, 24, 2, 512, 1, 7.49f)
#define CWT_ZOOM_GROUP_4(X) \
    X(4, 5, 7, 1, 32, 128, 6, 2.12f) \
    X(16, 5, 15, 1, 32, 128, 6, 1.89f) \
    X(28, 10, 20, 1, 32, 128, 3, 1.92f) \
    X(40, 20, 24, 1, 16, 128, 3, 2.26f) \
    X(52, 25, 30, 1, 8, 128, 3, 3.02f) \
    X(64, 12, 12, 15, 4, 256, 2, 4.42f) \
    X(76, 10, 21, 21, 4, 512, 1, 4.97f) \
    X(88, 18, 18, 24, 2, 512, 1, 7.47f)
#define CWT_ZOOM_GROUP_5(X) \
    X(5, 6, 6, 1, 32, 128, 6, 1.88f) \
    X(17, 9, 9, 1, 32, 128, 6, 1.95f) \
    X(29, 8, 30, 1, 32, 128, 3, 1.96f) \
    X(41, 7, 7, 10, 16, 256, 3, 2.74f) \
    X(53, 28, 28, 1, 8, 128, 3, 2.88f) \
    X(65, 10, 14, 16, 4, 256, 2, 4.61f) \
    X(77, 16, 16, 18, 4, 512, 1, 4.65f) \
    X(89, 16, 21, 24, 2, 512, 1, 7.28f)
#define CWT_ZOOM_GROUP_6(X) \
    X(6, 4, 10, 1, 32, 128, 6, 1.79f) \
    X(18, 10, 10, 1, 32, 128, 6, 1.86f) \
    X(30, 10, 25, 1, 32, 128, 3, 2.21f) \
    X(42, 21, 24, 1, 16, 128, 3, 2.37f) \
    X(54, 28, 32, 1, 8, 128, 3, 2.83f) \
    X(66, 10, 12, 20, 4, 512, 1, 4.87f) \
    X(78, 14, 16, 21, 4, 512, 1, 4.94f) \
    X(90, 16, 20, 28, 2, 512, 1, 7.26f)
#define CWT_ZOOM_GROUP_7(X) \
    X(7, 6, 7, 1, 32, 128, 6, 2.05f) \
    X(19, 7, 15, 1, 32, 128, 6, 1.84f) \
    X(31, 10, 25, 1, 32, 128, 3, 2.21f) \
    X(43, 16, 32, 1, 16, 128, 3, 2.21f) \
    X(55, 32, 32, 1, 8, 256, 2, 2.79f) \
    X(67, 9, 18, 18, 4, 512, 1, 5.33f) \
    X(79, 14, 14, 25, 2, 512, 1, 7.79f) \
    X(91, 21, 21, 21, 2, 512, 1, 7.62f)
#define CWT_ZOOM_GROUP_8(X) \
    X(8, 5, 9, 1, 32, 128, 6, 2.04f) \
    X(20, 7, 16, 1, 32, 128, 6, 1.79f) \
    X(32, 8, 32, 1, 16, 128, 5, 1.83f) \
    X(44, 21, 25, 1, 16, 128, 2, 2.55f) \
    X(56, 9, 9, 15, 4, 256, 3, 4.48f) \
    X(68, 12, 16, 16, 4, 512, 1, 4.67f) \
    X(80, 16, 18, 18, 4, 512, 1, 4.82f) \
    X(92, 15, 25, 25, 2, 512, 1, 7.67f)
#define CWT_ZOOM_GROUP_9(X) \
    X(9, 4, 12, 1, 32, 128, 6, 1.71f) \
    X(21, 5, 25, 1, 32, 128, 4, 2.22f) \
    X(33, 10, 28, 1, 32, 128, 2, 2.06f) \
    X(45, 18, 30, 1, 16, 128, 2, 2.35f) \
    X(57, 9, 12, 12, 4, 256, 3, 4.25f) \
    X(69, 15, 15, 15, 4, 512, 1, 4.99f) \
    X(81, 14, 15, 25, 2, 512, 1, 7.8f)
#define CWT_ZOOM_GROUP_10(X) \
    X(10, 7, 7, 1, 32, 128, 6, 1.98f) \
    X(22, 8, 16, 1, 32, 128, 6, 1.73f) \
    X(34, 16, 18, 1, 16, 128, 4, 2.1f) \
    X(46, 25, 25, 1, 16, 256, 2, 2.83f) \
    X(58, 10, 10, 14, 4, 256, 3, 4.34f) \
    X(70, 9, 18, 21, 4, 512, 1, 5.01f) \
    X(82, 15, 15, 25, 2, 512, 1, 7.54f)
#define CWT_ZOOM_GROUP_11(X) \
    X(11, 5, 10, 1, 32, 128, 6, 1.82f) \
    X(23, 9, 15, 1, 32, 128, 5, 1.98f) \
    X(35, 15, 21, 1, 16, 128, 4, 2.17f) \
    X(47, 20, 32, 1, 16, 256, 2, 2.62f) \
    X(59, 7, 15, 15, 4, 256, 3, 4.34f) \
    X(71, 12, 16, 20, 4, 512, 1, 4.8f) \
    X(83, 15, 18, 21, 2, 512, 1, 8.13f)
#define CWT_ZOOM_ALL(X) \
    CWT_ZOOM_GROUP_0(X) CWT_ZOOM_GROUP_1(X) CWT_ZOOM_GROUP_2(X) CWT_ZOOM_GROUP_3(X) CWT_ZOOM_GROUP_4(X) CWT_ZOOM_GROUP_5(X) CWT_ZOOM_GROUP_6(X) CWT_ZOOM_GROUP_7(X) CWT_ZOOM_GROUP_8(X) CWT_ZOOM_GROUP_9(X) CWT_ZOOM_GROUP_10(X) CWT_ZOOM_GROUP_11(X)

namespace cwtk {
constexpr int kZoomInstances = 93;
}
