// zoom_wide.cuh -- bands too wide for one CTA's columns: the residue-class
// transform of zoom.cuh in two kernels with a workspace between them.
//
// A column of Q points (Q >= the band) leaves a CTA's tile room for few
// columns once Q passes 1024: their stores become pieces of 16 or 8 bytes and
// one CTA fills an SM.  The first pass of that transform, over the QA bins b +
// Q' g of one b (Q = QA Q'), turns the residues r mod M / Q into the residues
// t' = r + (M / Q) k1 mod R' = M / Q', whose remaining transforms have Q' points
// and are again independent:
//   wide_first_kernel  Z[b][t'] = sum_g Y[b + Q' g] w_M^(Q' g t'), every b < Q'
//                      and t' < R' of a row, as M / Q butterflies of QA points
//                      per b;
//   wide_rest_kernel   c[t' + R' h] = sum_b Z[b][t'] w_M^(b t') w_Q'^(b h) for P
//                      consecutive t' per CTA, two passes Q' = QB QC over a
//                      tile in shared memory, stores as zoom_kernel's.
// Z takes 8 bytes per output each way.  The host runs the rows in chunks whose
// Z stays in L2 (zoom.cu), in two halves of the workspace by turns: the first
// kernel of a chunk starts as the second of the chunk before it runs out of
// CTAs to launch (each waits, as programmatic dependents, only for what it
// needs).  Bound by instruction issue like zoom_kernel.
#pragma once

#include "zoom.cuh"

namespace cwtk {

struct WideArgs {
    ZoomArgs z;          // spec, bank, list, tables, outputs; z.R = M / Q, z.L = R'
    float2 *Z;           // [rows of the chunk][Q'][R']
    int row0, nrows;     // first row of the chunk and its rows
    int Qp, bb, groups;  // Q'; positions per CTA of the first kernel; its CTAs per row
    unsigned magG;       // zoom_magic(groups), of either kernel
};

constexpr int kWideThreads = 128;

template <int QA>
__global__ void __launch_bounds__(kWideThreads, QA <= 16 ? 5 : 4) wide_first_kernel(const WideArgs w) {
    constexpr int T = kWideThreads;
    // up to 16 points the modulation stays in registers, above it takes them
    // from the butterfly (QA = 32: 2.9 ps per point) and is read per use
    constexpr bool kKeep = QA <= 16;
    extern __shared__ float2 wsm[];
    const ZoomArgs &a = w.z;
    const int R = a.R, N = a.N, Qp = w.Qp, Q = QA * Qp, Rp = a.L, bb = w.bb;
    float2 *const Y = wsm, *const E = wsm + QA * bb;  // [QA][bb]; [QA + 1][R], or [2][QA][R] for b from and below rho
    const int tid = (int)threadIdx.x;
    int lrow, grp, th, r, c, si;
    zoom_divmod(blockIdx.x, (unsigned)w.groups, w.magG, lrow, grp);
    zoom_divmod((unsigned)tid, (unsigned)R, a.magR, th, r);
    const int TP = T / R;  // threads per residue; R <= T
    zoom_divmod((unsigned)(w.row0 + lrow), (unsigned)a.ns, a.magNs, c, si);
    const int4 sc = __ldg(&a.list[si]);
    const int g0 = sc.w / Qp, rho = sc.w - g0 * Qp, pst = g0 % QA;
    if (th < TP) {  // w_M^(Q' g r) = w_R'^(g r), as zoom_kernel's E
        unsigned i = zoom_mod((unsigned)(g0 + th) * (unsigned)r, (unsigned)Rp, a.magL);
        const unsigned stride = zoom_mod((unsigned)(TP * r), (unsigned)Rp, a.magL);
#pragma unroll 2
        for (int j = th; j <= QA; j += TP) {
            int p = pst + j;
            if (p >= QA) p -= QA;
            const float2 e = __ldg(&a.twl[i]);
            if constexpr (kKeep) {
                *CWT_SMEM(&E[(j == QA ? QA : p) * R + r]) = e;
            } else {
                if (j < QA) *CWT_SMEM(&E[p * R + r]) = e;
                if (j > 0) *CWT_SMEM(&E[(QA + (j == QA ? pst : p)) * R + r]) = e;
            }
            i += stride;
            if (i >= (unsigned)Rp) i -= (unsigned)Rp;
        }
    }
    // The spectra are complete when a.after.  This half of Z is free: the kernel
    // before has passed its wait for a kernel that outlived its last reader.
    if (!a.after) griddep_wait();
    griddep_launch();
    const int b0 = grp * bb, nb = min(bb, Qp - b0), wm = sc.w % Q;
    const float2 *X = a.spec + (size_t)c * N;
    const float *W = a.bank + (size_t)sc.x * N;
#pragma unroll 4
    for (int i = tid; i < QA * bb; i += T) {
        const int p = i / bb, j = i - p * bb;
        int k = b0 + j + Qp * p - wm;  // the bin of the window at this position
        k += k < 0 ? Q + sc.w : sc.w;
        float2 y = make_float2(0.f, 0.f);
        if (j < nb && (unsigned)(k - sc.y) < (unsigned)sc.z) {
            if (k >= N) k -= N;
            const float2 x = __ldcg(X + CWT_IDX(k, N));
            const float v = __ldg(W + k);
            y = make_float2(x.x * v, x.y * v);
        }
        *CWT_SMEM(&Y[i]) = y;
    }
    __syncthreads();
    // one CTA outlives the second kernel of the chunk before
    if (a.after && blockIdx.x == gridDim.x - 1) griddep_wait();
    if (th >= TP) return;
    float2 e[kKeep ? QA : 1], ex = make_float2(0.f, 0.f);
    if constexpr (kKeep) {
#pragma unroll
        for (int p = 0; p < QA; ++p) e[p] = *CWT_SMEM(&E[p * R + r]);
        ex = *CWT_SMEM(&E[QA * R + r]);
    }
    bool wrapped = false;
    float2 *out = w.Z + ((size_t)lrow * Qp + b0) * Rp + r;
#pragma unroll 1
    for (int j = th; j < nb; j += TP) {
        float2 v[QA];
        if constexpr (kKeep) {
            if ((b0 + j < rho) != wrapped) {
                wrapped = !wrapped;
                const float2 t = ex;
#pragma unroll
                for (int p = 0; p < QA; ++p)
                    if (p == pst) {
                        ex = e[p];
                        e[p] = t;
                    }
            }
#pragma unroll
            for (int p = 0; p < QA; ++p) v[p] = cmul(*CWT_SMEM(&Y[p * bb + j]), e[p]);
        } else {
            const float2 *ep = E + (b0 + j < rho ? QA * R : 0) + r;
#pragma unroll
            for (int p = 0; p < QA; ++p) v[p] = cmul(*CWT_SMEM(&Y[p * bb + j]), *CWT_SMEM(&ep[p * R]));
        }
        dft_r<QA, +1>(v);
        float2 *o = out + (size_t)j * Rp;
#pragma unroll
        for (int k = 0; k < QA; ++k) o[k * R] = v[k];
    }
}

template <int QB_, int QC_, int P_, int T_, int MINB_>
struct WideCfg {
    static constexpr int QB = QB_, QC = QC_, P = P_, T = T_, MINB = MINB_, Qp = QB * QC;
    static constexpr int QCP = P < 16 ? (QC | 1) : QC;  // a half-warp then meets different banks
    static constexpr int SMEM = QB * QCP * P * 8;
    static_assert((P & (P - 1)) == 0 && T % P == 0, "T / P threads per column");
};

template <class Z, int MODE>
__global__ void __launch_bounds__(Z::T, Z::MINB) wide_rest_kernel(const WideArgs w) {
    constexpr int QB = Z::QB, QC = Z::QC, P = Z::P, T = Z::T, TP = T / P, QCP = Z::QCP;
    extern __shared__ float2 wsm[];
    const ZoomArgs &a = w.z;
    const int Rp = a.L, tid = (int)threadIdx.x, col = tid % P, th = tid / P;
    int lrow, grp, c, si;
    zoom_divmod(blockIdx.x, (unsigned)w.groups, w.magG, lrow, grp);
    const bool in = grp * P + col < Rp;
    const int t1 = in ? grp * P + col : Rp - 1;  // residue t'; columns past the last repeat it
    zoom_divmod((unsigned)(w.row0 + lrow), (unsigned)a.ns, a.magNs, c, si);
    const int s = __ldg(&a.list[si].x);
    const float2 wb = __ldg(&a.tw[QC * t1 * a.tws]);
    const float2 wb8 = zoom_w8<QB>(a.tw, (unsigned)(QC * t1), (unsigned)a.M, a.magM, a.tws);
    float2 wn = __ldg(&a.tw[(t1 + Rp * th) * a.tws]);
    float2 w8n = zoom_w8<QC>(a.tw, (unsigned)(t1 + Rp * th), (unsigned)a.M, a.magM, a.tws);
    griddep_wait();  // Z
    griddep_launch();
    const float2 *src = w.Z + (size_t)lrow * Z::Qp * Rp + t1;
#pragma unroll 1
    for (int b1 = th; b1 < QC; b1 += TP) {
        float2 v[QB];
#pragma unroll
        for (int b = 0; b < QB; ++b) v[b] = __ldcg(src + (b1 + QC * b) * Rp);
        zoom_twiddle<QB>(v, wb, wb8);
        dft_r<QB, +1>(v);
        float2 *x = wsm + b1 * P + col;
#pragma unroll
        for (int k = 0; k < QB; ++k) *CWT_SMEM(&x[k * (QCP * P)]) = v[k];
    }
    const int step = Rp * QB, n_keep = in ? a.n_keep : 0;
    const size_t obase = (size_t)(c * a.S + s) * (size_t)a.n_out;
    __syncthreads();
#pragma unroll 1
    for (int k2 = th; k2 < QB; k2 += TP) {
        const int t0 = t1 + Rp * k2;
        const float2 wt = wn, w8 = w8n;
        if (k2 + TP < QB) {
            wn = __ldg(&a.tw[(t0 + Rp * TP) * a.tws]);
            w8n = zoom_w8<QC>(a.tw, (unsigned)(t0 + Rp * TP), (unsigned)a.M, a.magM, a.tws);
        }
        if (t0 >= n_keep) continue;
        const float2 *x = wsm + k2 * (QCP * P) + col;
        float2 v[QC];
#pragma unroll
        for (int b = 0; b < QC; ++b) v[b] = *CWT_SMEM(&x[b * P]);
        zoom_twiddle<QC>(v, wt, w8);
        dft_r<QC, +1>(v);
        zoom_emit<QC, MODE>(a, obase, t0, step, n_keep, v);
    }
}

}  // namespace cwtk
