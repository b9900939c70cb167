// zoom.h -- the host's view of the zoom_kernel instances (zoom.cuh,
// zoom_list.h): which scales run on which instance, and the launch of one
// class of scales (zoom.cu).  Used by plans (zoom.cu) and batches (batch.cu).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "zoom.cuh"
#include "zoom_list.h"
#include "zoom_wide.cuh"
#include "zoom_wide_list.h"

namespace cwtk {

// The kernel of instance I: zoom_kernel MODE 0 or 1, or (2) zoom_row_kernel
// (zoom_inst_<g>.cu), null where its rows of two residues are too long for that.
template <int I>
const void *zoom_entry(int mode);

// The longest rows that zoom_row_kernel holds on T threads.
constexpr int zoom_row_points(int T) { return T > 128 ? kZoomRowPoints : 5632; }
template <class Z>
const void *zoom_row_entry() {
    if constexpr (2 * Z::Q <= zoom_row_points(Z::T)) return (const void *)&zoom_row_kernel<Z>;
    else return nullptr;
}

#define CWT_ZOOM_DEFINE(I, QA, QB, QC, P, T, MINB, COST)                        \
    template <>                                                                 \
    const void *zoom_entry<I>(int mode) {                                       \
        using Z = ZoomCfg<QA, QB, QC, P, T, MINB>;                              \
        return mode == 0   ? (const void *)&zoom_kernel<Z, 0>                   \
               : mode == 1 ? (const void *)&zoom_kernel<Z, 1>                   \
                           : zoom_row_entry<Z>();                               \
    }

// The kernels of zoom_wide.cuh: first radix i, remaining length I in MODE 0 or 1.
const void *wide_first_entry(int i);
template <int I>
const void *wide_rest_entry(int mode);

#define CWT_WIDE_DEFINE(I, QB, QC, P, T, MINB)                                                          \
    template <>                                                                                         \
    const void *wide_rest_entry<I>(int mode) {                                                          \
        using Z = WideCfg<QB, QC, P, T, MINB>;                                                          \
        return mode == 0 ? (const void *)&wide_rest_kernel<Z, 0> : (const void *)&wide_rest_kernel<Z, 1>; \
    }

// Scales [first, first + ns) of a device list on one instance of zoom_kernel, of
// zoom_row_kernel (rows), or on first radix `wide` and remaining length `inst`
// of zoom_wide.cuh.
struct ZoomClass {
    int inst, first, ns;
    bool rows;
    int wide;  // -1: not wide
};

// What zoom_select decides from: a row on M points of which every sub-th is kept,
// output rows of n_out samples (0: of any length), the cost of a row (ps) on the
// kernels that take the rest and, if that is on kernels compiled for the plan, its
// cost there (else 0), and whether the phase, and whether more than one output
// array, is asked for.
struct ZoomShape {
    int M, sub, n_out;
    double rest_cost, compiled_cost;
    bool phase, both;
    bool rows_only, wide;  // only zoom_row_kernel; zoom_wide.cuh allowed
    double channels;  // nominal, for the cost of a launch against that of its rows
    // the part of the row that the outputs cover
    double kept() const { return n_out ? std::min(1.0, (double)n_out * sub / M) : 1.0; }
};

// Splits S scales with bands band[2 s] (start), band[2 s + 1] (length) into
// classes, their entries for the device in *list, and the rest.
void zoom_select(const ZoomShape &z, int S, const int *band, std::vector<ZoomClass> *classes,
                 std::vector<int4> *list, std::vector<int> *rest);
int zoom_class_L(const ZoomClass &c, int M);  // points of its first pass's table
// Launch class c for `chans` channels: a holds the pointers, N, M, tws, S,
// n_out, sub, n_keep, after and the batch's fields.
cudaError_t zoom_launch(const ZoomClass &c, ZoomArgs a, long long chans, const float2 *twl, const int4 *d_list,
                        cudaStream_t st);
// Launch wide class c with a workspace of two halves of z_rows rows of M
// points, used by turns (*turn counts on from class to class).
cudaError_t wide_launch(const ZoomClass &c, const ZoomArgs &a, long long chans, const float2 *twl, const int4 *d_list,
                        float2 *Z, int z_rows, int *turn, cudaStream_t st);

}  // namespace cwtk
