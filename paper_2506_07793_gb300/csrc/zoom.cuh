// zoom.cuh -- the inverse FFT of a band-limited row, by output residue classes.
//
// A scale's wavelet occupies B of the M bins of its row (Eq. 3-5: a bump
// around the carrier; B / M is 0.005 ... 0.2 for EEG scales), so the row's
// inverse FFT (Eq. 2) is an interpolation.  With Q >= B a divisor of M and
// R = M / Q, the outputs t = r + R h of one residue class r are the Q-point
// inverse FFT of the band, modulated by w_M^(k r) and laid out by k mod Q:
//     c[r + R h] = sum_k Y[k] w_M^(k r) w_Q^(k h),   w_L = exp(2 pi i / L),
// each residue of k mod Q meeting the band at most once.  The classes are
// independent: no pass over the M-point row, no row in shared memory, no
// cluster for long rows, and log2 Q instead of log2 M stages per output.
//
// One CTA takes a column group: G <= P consecutive residues of a row (or all
// residues of several short rows), the columns of a [Q][P] tile in shared
// memory, and runs the Q-point FFT of every column in two or three Stockham
// passes Q = QA QB (QC).  Consecutive threads take consecutive columns, so
//  * twiddles of a pass that depend on the position alone are warp-uniform,
//    the tile is read and written without bank conflicts at immediate offsets,
//    and stores go to consecutive output samples;
//  * the first pass reads the band product Y (computed once per CTA into
//    shared memory) as a broadcast and multiplies it by the modulation
//    E[p][col] = w_M^(QP g_p r), QP = QB QC, a table of QA P entries per CTA;
//    the rest of the modulation commutes with the passes: a pass whose inputs
//    b (stride QC or 1) belong to the partial residue t0 takes the twiddles
//    w_M^(stride b t0), one table entry and a multiplication chain.
//  * passes after the first read and write the same slots, one barrier each.
#pragma once

#include "mixed_radix.cuh"
#include "phase.cuh"

namespace cwtk {

// An epoch of a batch: element offsets of channel 0's spectrum and outputs.
struct ZoomEpoch {
    long long spec, out, in;  // element offsets of channel 0: window of bins, output, input
    int n_out, n_keep, n, pad;
};

struct ZoomArgs {
    const float2 *spec;  // [C][N]
    const float *bank;   // [S][N]
    const float2 *tw;    // w_M^i = tw[i tws], i < M
    const float2 *twl;   // w_L^i, i < L = QA R
    const int4 *list;    // [ns] scales of this class: scale, band start, band length, window start
    float2 *oc;
    float *op, *oph;     // [C][S][n_out]
    int N, M, R, L, tws, ns, S, n_out;
    unsigned magM, magL, magR, magNs;  // zoom_magic of M, L, R, ns
    unsigned cols;       // C ns R columns
    int rows;            // most rows that one CTA's columns meet
    int sub, n_keep;     // outputs t = sub o, o < n_out; n_keep = sub (n_out - 1) + 1
    int after;           // 1: the spectra are complete when this kernel starts (see zoom.cu)
    // zoom_row_kernel: rows per CTA and of the launch, slots of a tile row, of
    // one position of it (QA R and padding) and of a row's last pass, zoom_magic
    // of nr R, the last pass's slots, QA R and sub
    int nr, nrows, rs, ps, js;
    unsigned magC, magJs, magL2, magSub;
    // batches: channel c is channel c mod C of epoch c / C (null: one epoch);
    // its spectrum holds the wn bins from w0 mod N (0 and N without epochs)
    const ZoomEpoch *epochs;
    int C, w0, wn;
    unsigned magCh;
};

// floor((2^32 - 1) / d): for x < 2^31, umulhi(x, mag) is x / d or one less.
__host__ __device__ constexpr unsigned zoom_magic(unsigned d) { return 0xffffffffu / d; }

__device__ __forceinline__ void zoom_divmod(unsigned x, unsigned d, unsigned mag, int &q, int &r) {
    unsigned qq = __umulhi(x, mag), rr = x - qq * d;
    if (rr >= d) {
        ++qq;
        rr -= d;
    }
    q = (int)qq;
    r = (int)rr;
}
__device__ __forceinline__ unsigned zoom_mod(unsigned x, unsigned d, unsigned mag) {
    const unsigned r = x - __umulhi(x, mag) * d;
    return r >= d ? r - d : r;
}

template <int QA_, int QB_, int QC_, int P_, int T_, int MINB_>
struct ZoomCfg {
    static constexpr int QA = QA_, QB = QB_, QC = QC_, P = P_, T = T_, MINB = MINB_;
    static constexpr int QP = QB * QC, Q = QA * QP;
    static constexpr int LAST = QC > 1 ? QC : QB;     // radix of the last pass
    static constexpr int K2 = QC > 1 ? QB : 1;        // outputs of the middle pass
    // positions b that a thread transforms at once in the first pass (Y is
    // then read two at a time); the window starts at a multiple of NB
    static constexpr int NB = QA <= 10 && QP % 2 == 0 ? 2 : 1;
    // pitch of the k1 index: odd when a half-warp spans several positions, so
    // that they fall into different banks
    static constexpr int QAP = P < 16 ? (QA | 1) : QA;
    static constexpr int TILE = QP * QAP * P;         // float2 slots
    static constexpr int ETAB = (QA + 1) * P;
    static constexpr int YP = (Q + 2) & ~1;           // pitch of a row's band product (even, not a multiple of 16)
    static_assert((P & (P - 1)) == 0 && T % P == 0, "T / P threads per column");
    static_assert(T / P <= Q, "first table entries of the last pass");
    __host__ __device__ static constexpr int smem(int rows) { return (TILE + ETAB + rows * YP) * 8; }
};

// The band product Y[k] = X[k] W[k] of a row by k mod Q, over the window
// [sc.w, sc.w + Q) of bins; X holds bins [w0, w0 + ...) mod N.  STEP threads
// take part, `lane` among them.
template <int Q, int STEP>
__device__ __forceinline__ void zoom_fill(float2 *Y, int lane, const int4 &sc, const float2 *X, int w0, int wn,
                                          const float *W, int N) {
    const int wm = sc.w % Q;
#pragma unroll 4
    for (int j = lane; j < Q; j += STEP) {
        int k = j - wm;
        k += k < 0 ? Q + sc.w : sc.w;  // in [sc.w, sc.w + Q)
        float2 y = make_float2(0.f, 0.f);
        if ((unsigned)(k - sc.y) < (unsigned)sc.z) {
            if (k >= N) k -= N;
            int kk = k - w0;
            if (kk < 0) kk += N;
            const float2 x = __ldcg(X + CWT_IDX(kk, wn));
            const float w = __ldg(W + k);
            y = make_float2(x.x * w, x.y * w);
        }
        *CWT_SMEM(&Y[j]) = y;
    }
}

// v[r] *= w1^r, r < R, as mr_twiddle, but with w8 = w1^8 from the table as
// well: the error of a power grows with its exponent over the entry it is
// formed from, here at most 7 + R / 8 instead of R - 1.
template <int R>
__device__ __forceinline__ void zoom_twiddle(float2 *v, float2 w1, float2 w8) {
    constexpr int LO = R < 8 ? R : 8;
    float2 wl[LO];
    wl[0] = make_float2(1.f, 0.f);
    wl[1] = w1;
#pragma unroll
    for (int r = 2; r < LO; ++r) wl[r] = (r & 1) ? cmul(wl[r - 1], w1) : cmul(wl[r >> 1], wl[r >> 1]);
#pragma unroll
    for (int r = 1; r < LO; ++r) v[r] = cmul(v[r], wl[r]);
    if constexpr (R > 8) {
        float2 wh = w8;
#pragma unroll
        for (int h = 1; 8 * h < R; ++h) {
            v[8 * h] = cmul(v[8 * h], wh);
#pragma unroll
            for (int l = 1; l < 8; ++l)
                if (8 * h + l < R) v[8 * h + l] = cmul(cmul(v[8 * h + l], wh), wl[l]);
            if (8 * (h + 1) < R) wh = cmul(wh, w8);
        }
    }
}
// w_M^(8 i) of that, i < M (not read for R <= 8).
template <int R>
__device__ __forceinline__ float2 zoom_w8(const float2 *tw, unsigned i, unsigned M, unsigned magM, int tws) {
    if constexpr (R > 8) return __ldg(&tw[zoom_mod(8u * i, M, magM) * (unsigned)tws]);
    else return make_float2(1.f, 0.f);
}

// fill(row, lane, int_c<threads of the row>) for each of n rows: all T threads
// one row after the other when there are few (each costs a load latency), a
// warp per row, or 8 threads.
template <int T, typename F>
__device__ __forceinline__ void zoom_rows(int n, int tid, const F &fill) {
    if (n < T / 32) {
#pragma unroll 1
        for (int i = 0; i < n; ++i) fill(i, tid, int_c<T>{});
    } else if (n <= T / 16) {
#pragma unroll 1
        for (int i = tid >> 5; i < n; i += T / 32) fill(i, tid & 31, int_c<32>{});
    } else {
#pragma unroll 1
        for (int i = tid >> 3; i < n; i += T / 8) fill(i, tid & 7, int_c<8>{});
    }
}

// Stores f(v[m]), m < min(L, left), at dst + m step.
template <int L, typename T, typename F>
__device__ __forceinline__ void zoom_store(T *dst, int step, int left, const float2 *v, const F &f) {
    if (left >= L) {
#pragma unroll
        for (int m = 0; m < L; ++m) __stcs(dst + (size_t)((unsigned)step) * m, f(v[m]));
    } else {
#pragma unroll
        for (int m = 0; m < L; ++m)
            if (m < left) __stcs(dst + (size_t)((unsigned)step) * m, f(v[m]));
    }
}

// The outputs t0 + step m < n_keep of one last-pass butterfly, MODE 0: complex
// and power at every sample; 1: also phase and sub > 1.
template <int L, int MODE>
__device__ __forceinline__ void zoom_emit(const ZoomArgs &a, size_t obase, int t0, int step, int n_keep,
                                          const float2 *v) {
    if constexpr (MODE == 0) {
        const int left = t0 + (L - 1) * step < n_keep ? L : (n_keep - t0 + step - 1) / step;
        if (a.oc) zoom_store<L>(a.oc + obase + t0, step, left, v, [](float2 x) { return x; });
        if (a.op)
            zoom_store<L>(a.op + obase + t0, step, left, v,
                          [](float2 x) { return fmaf(x.x, x.x, x.y * x.y); });
    } else {
#pragma unroll
        for (int m = 0; m < L; ++m) {
            const int t = t0 + m * step;
            if (t >= n_keep) continue;
            int o = t;
            if (a.sub != 1) {
                int rem;
                zoom_divmod((unsigned)t, (unsigned)a.sub, a.magSub, o, rem);
                if (rem != 0) continue;
            }
            if (a.oc) __stcs(a.oc + obase + o, v[m]);
            if (a.op) __stcs(a.op + obase + o, fmaf(v[m].x, v[m].x, v[m].y * v[m].y));
            if (a.oph) __stcs(a.oph + obase + o, phase_atan2(v[m].y, v[m].x));
        }
    }
}

// MODE as zoom_emit's.
template <class Z, int MODE>
__global__ void __launch_bounds__(Z::T, Z::MINB) zoom_kernel(const ZoomArgs a) {
    constexpr int QA = Z::QA, QB = Z::QB, QC = Z::QC, P = Z::P, T = Z::T, QP = Z::QP, Q = Z::Q, QAP = Z::QAP;
    constexpr int NB = Z::NB, LAST = Z::LAST, K2 = Z::K2;
    constexpr int TP = T / P;  // threads per column
    extern __shared__ float4 zsm4[];
    float2 *const Y = (float2 *)zsm4, *const tile = Y + a.rows * Z::YP, *const E = tile + Z::TILE;
    const int tid = (int)threadIdx.x, col = tid % P, th = tid / P;
    const int R = a.R, N = a.N;
    const unsigned gc0 = blockIdx.x * (unsigned)P;
    const int G = (int)min((unsigned)P, a.cols - gc0);  // columns of this CTA
    int row0, r0;
    zoom_divmod(gc0, (unsigned)R, a.magR, row0, r0);
    int nrow = 1, rl = 0, r = r0 + col;
    if (a.rows > 1) {  // columns past G repeat the last one
        int dummy;
        zoom_divmod((unsigned)(r0 + G - 1), (unsigned)R, a.magR, nrow, dummy);
        ++nrow;
        zoom_divmod((unsigned)(r0 + min(col, G - 1)), (unsigned)R, a.magR, rl, r);
    }
    int c, si;
    zoom_divmod((unsigned)(row0 + rl), (unsigned)a.ns, a.magNs, c, si);
    const int4 sc = __ldg(&a.list[si]);
    float2 wn = __ldg(&a.tw[(r + R * th) * a.tws]);  // the last pass's first table entries
    float2 w8n = zoom_w8<LAST>(a.tw, (unsigned)(r + R * th), (unsigned)a.M, a.magM, a.tws);
    // (before the wait: none of it depends on the forward FFTs)
    // modulation of the first pass: position p stands for the bins b + QP g,
    // g = p (mod QA) in [g0, g0 + QA), g0 = floor(window / QP), except that for
    // b < window mod QP the window reaches g0 + QA instead of g0 (row QA)
    const int g0 = sc.w / QP, rho = sc.w - g0 * QP, pst = g0 % QA;
    {
        const unsigned L = (unsigned)a.L;
        unsigned i = zoom_mod((unsigned)(g0 + th) * (unsigned)r, L, a.magL);
        const unsigned stride = zoom_mod((unsigned)(TP * r), L, a.magL);
#pragma unroll 2
        for (int j = th; j <= QA; j += TP) {
            int p = pst + j;
            if (p >= QA) p -= QA;
            *CWT_SMEM(&E[(j == QA ? QA : p) * P + col]) = __ldg(&a.twl[i]);
            i += stride;
            if (i >= L) i -= L;
        }
    }
    if (!a.after) griddep_wait();  // the forward FFTs
    griddep_launch();
    // band products of the CTA's rows by k mod Q (spectra through L2: a CTA may
    // share its SM with the kernel that wrote other spectra to the same address)
    zoom_rows<T>(nrow, tid, [&](int il, int lane, auto step) {
        int ic, is;
        zoom_divmod((unsigned)(row0 + il), (unsigned)a.ns, a.magNs, ic, is);
        const int4 z = __ldg(&a.list[is]);
        zoom_fill<Q, decltype(step)::value>(Y + il * Z::YP, lane, z, a.spec + (size_t)ic * N, 0, N,
                                            a.bank + (size_t)z.x * N, N);
    });
    __syncthreads();
    // first pass: DFT over p
    {
        const float2 *y = Y + rl * Z::YP;
        float2 e[QA];
#pragma unroll
        for (int p = 0; p < QA; ++p) e[p] = *CWT_SMEM(&E[p * P + col]);
        float2 ex = *CWT_SMEM(&E[QA * P + col]);
        bool wrapped = false;
#pragma unroll 1
        for (int b = NB * th; b < QP; b += NB * TP) {
            if ((b < rho) != wrapped) {
                wrapped = !wrapped;
                const float2 t = ex;
#pragma unroll
                for (int p = 0; p < QA; ++p)
                    if (p == pst) {
                        ex = e[p];
                        e[p] = t;
                    }
            }
            float2 *dst = tile + b * (QAP * P) + col;
            if constexpr (NB == 2) {
                float2 v[QA], u[QA];
#pragma unroll
                for (int p = 0; p < QA; ++p) {
                    const float4 y2 = *CWT_SMEM((const float4 *)(y + b + p * QP));
                    v[p] = cmul(make_float2(y2.x, y2.y), e[p]);
                    u[p] = cmul(make_float2(y2.z, y2.w), e[p]);
                }
                dft_r<QA, +1>(v);
                dft_r<QA, +1>(u);
#pragma unroll
                for (int k = 0; k < QA; ++k) {
                    *CWT_SMEM(&dst[k * P]) = v[k];
                    *CWT_SMEM(&dst[(QAP + k) * P]) = u[k];
                }
            } else {
                float2 v[QA];
#pragma unroll
                for (int p = 0; p < QA; ++p) v[p] = cmul(*CWT_SMEM(&y[b + p * QP]), e[p]);
                dft_r<QA, +1>(v);
#pragma unroll
                for (int k = 0; k < QA; ++k) *CWT_SMEM(&dst[k * P]) = v[k];
            }
        }
    }
    // middle pass: DFT over b2, b = b1 + QC b2, in place
    if constexpr (QC > 1) {
        __syncthreads();
#pragma unroll 1
        for (int q = th; q < QC * QA; q += TP) {
            const int b1 = q / QA, k1 = q - b1 * QA;
            float2 *x = tile + (b1 * QAP + k1) * P + col;
            const int i = QC * (r + R * k1);
            const float2 w = __ldg(&a.tw[i * a.tws]);
            const float2 w8 = zoom_w8<QB>(a.tw, (unsigned)i, (unsigned)a.M, a.magM, a.tws);
            float2 v[QB];
#pragma unroll
            for (int b = 0; b < QB; ++b) v[b] = *CWT_SMEM(&x[b * (QC * QAP * P)]);
            zoom_twiddle<QB>(v, w, w8);
            dft_r<QB, +1>(v);
#pragma unroll
            for (int k = 0; k < QB; ++k) *CWT_SMEM(&x[k * (QC * QAP * P)]) = v[k];
        }
    }
    // last pass: DFT over the remaining index, outputs t0 + step m
    const int step = R * QA * K2, n_keep = col < G ? a.n_keep : 0;
    const size_t obase = (size_t)(c * a.S + sc.x) * (size_t)a.n_out;
    __syncthreads();
#pragma unroll 1
    for (int q = th; q < QA * K2; q += TP) {
        const int k2 = q / QA, k1 = q - k2 * QA;
        const int t0 = r + R * q;  // q = k1 + QA k2
        const float2 w = wn, w8 = w8n;
        if (q + TP < QA * K2) {
            wn = __ldg(&a.tw[(t0 + R * TP) * a.tws]);
            w8n = zoom_w8<LAST>(a.tw, (unsigned)(t0 + R * TP), (unsigned)a.M, a.magM, a.tws);
        }
        if (t0 >= n_keep) continue;
        const float2 *x = tile + (QC * k2 * QAP + k1) * P + col;
        float2 v[LAST];
#pragma unroll
        for (int b = 0; b < LAST; ++b) v[b] = *CWT_SMEM(&x[b * (QAP * P)]);
        zoom_twiddle<LAST>(v, w, w8);
        dft_r<LAST, +1>(v);
        zoom_emit<LAST, MODE>(a, obase, t0, step, n_keep, v);
    }
    // complete in stream order: one CTA outlives the kernel before
    if (a.after && blockIdx.x == gridDim.x - 1) griddep_wait();
}

// Whole rows of M <= kZoomRowPoints points: a CTA holds all R residues of nr
// rows, so that its last pass can take its outputs in the order of t.  A store
// instruction then covers consecutive samples for any R, and starts on a
// 32-byte sector whatever the row's base (the slots of a row are shifted by
// base mod 8): a sector written in part costs L2 a read.
constexpr int kZoomRowPoints = 10240;

template <class Z>
__host__ __device__ constexpr int zoom_row_smem(int nr, int rs, int R) {
    return (nr * rs + (Z::QA + 1) * nr * R + nr * Z::YP) * 8 + nr * 24;
}

struct ZoomRow {
    long long base;  // element offset of the row's outputs
    int n_keep, shift, pad[2];
};
static_assert(sizeof(ZoomRow) == 24, "zoom_row_smem");

template <class Z>
__global__ void __launch_bounds__(Z::T, Z::MINB) zoom_row_kernel(const ZoomArgs a) {
    constexpr int QA = Z::QA, QB = Z::QB, QC = Z::QC, T = Z::T, QP = Z::QP, Q = Z::Q;
    constexpr int NB = Z::NB, LAST = Z::LAST, K2 = Z::K2;
    extern __shared__ float4 zsm4[];
    const int R = a.R, N = a.N, nr = a.nr, C = nr * R;
    float2 *const Y = (float2 *)zsm4, *const tile = Y + nr * Z::YP, *const E = tile + nr * a.rs;
    ZoomRow *const rows = (ZoomRow *)(E + (QA + 1) * C);
    const int tid = (int)threadIdx.x;
    const int row0 = (int)blockIdx.x * nr, last = a.nrows - 1;
    int th, col, rl, r;
    zoom_divmod((unsigned)tid, (unsigned)C, a.magC, th, col);
    zoom_divmod((unsigned)col, (unsigned)R, a.magR, rl, r);
    const int TP = T / C;  // threads per column; C <= T
    const bool on = th < TP;
    int c, si;
    zoom_divmod((unsigned)min(row0 + rl, last), (unsigned)a.ns, a.magNs, c, si);
    const int4 sc = __ldg(&a.list[si]);
    if (tid < nr) {
        int cc, ss;
        zoom_divmod((unsigned)min(row0 + tid, last), (unsigned)a.ns, a.magNs, cc, ss);
        const int s = __ldg(&a.list[ss].x);
        ZoomRow z;
        if (a.epochs) {
            int e, ch;
            zoom_divmod((unsigned)cc, (unsigned)a.C, a.magCh, e, ch);
            const ZoomEpoch ep = a.epochs[e];
            z.base = ep.out + ((long long)ch * a.S + s) * ep.n_out;
            z.n_keep = ep.n_keep;
        } else {
            z.base = ((long long)cc * a.S + s) * a.n_out;
            z.n_keep = a.n_keep;
        }
        if (row0 + tid > last) z.n_keep = 0;
        z.shift = (int)(z.base & 7);
        z.pad[0] = z.pad[1] = 0;
        rows[tid] = z;
    }
    // modulation of the first pass (see zoom_kernel)
    const int g0 = sc.w / QP, rho = sc.w - g0 * QP, pst = g0 % QA;
    if (on) {
        const unsigned L = (unsigned)a.L;
        unsigned i = zoom_mod((unsigned)(g0 + th) * (unsigned)r, L, a.magL);
        const unsigned stride = zoom_mod((unsigned)(TP * r), L, a.magL);
#pragma unroll 2
        for (int j = th; j <= QA; j += TP) {
            int p = pst + j;
            if (p >= QA) p -= QA;
            *CWT_SMEM(&E[(j == QA ? QA : p) * C + col]) = __ldg(&a.twl[i]);
            i += stride;
            if (i >= L) i -= L;
        }
    }
    if (!a.after) griddep_wait();  // the forward FFTs
    griddep_launch();
    // band products of the rows by k mod Q
    zoom_rows<T>(nr, tid, [&](int il, int lane, auto step) {
        int ic, is;
        zoom_divmod((unsigned)min(row0 + il, last), (unsigned)a.ns, a.magNs, ic, is);
        const int4 z = __ldg(&a.list[is]);
        const float2 *X = a.spec + (size_t)ic * N;
        if (a.epochs) {
            int e, ch;
            zoom_divmod((unsigned)ic, (unsigned)a.C, a.magCh, e, ch);
            X = a.spec + a.epochs[e].spec + (long long)ch * a.wn;
        }
        zoom_fill<Q, decltype(step)::value>(Y + il * Z::YP, lane, z, X, a.w0, a.wn, a.bank + (size_t)z.x * N, N);
    });
    __syncthreads();
    // first pass: DFT over p
    if (on) {
        const float2 *y = Y + rl * Z::YP;
        float2 e[QA];
#pragma unroll
        for (int p = 0; p < QA; ++p) e[p] = *CWT_SMEM(&E[p * C + col]);
        float2 ex = *CWT_SMEM(&E[QA * C + col]);
        bool wrapped = false;
#pragma unroll 1
        for (int b = NB * th; b < QP; b += NB * TP) {
            if ((b < rho) != wrapped) {
                wrapped = !wrapped;
                const float2 t = ex;
#pragma unroll
                for (int p = 0; p < QA; ++p)
                    if (p == pst) {
                        ex = e[p];
                        e[p] = t;
                    }
            }
            float2 *dst = tile + rl * a.rs + b * a.ps + r;
            if constexpr (NB == 2) {
                float2 v[QA], u[QA];
#pragma unroll
                for (int p = 0; p < QA; ++p) {
                    const float4 y2 = *CWT_SMEM((const float4 *)(y + b + p * QP));
                    v[p] = cmul(make_float2(y2.x, y2.y), e[p]);
                    u[p] = cmul(make_float2(y2.z, y2.w), e[p]);
                }
                dft_r<QA, +1>(v);
                dft_r<QA, +1>(u);
#pragma unroll
                for (int k = 0; k < QA; ++k) *CWT_SMEM(&dst[k * R]) = v[k];
                dst += a.ps;
#pragma unroll
                for (int k = 0; k < QA; ++k) *CWT_SMEM(&dst[k * R]) = u[k];
            } else {
                float2 v[QA];
#pragma unroll
                for (int p = 0; p < QA; ++p) v[p] = cmul(*CWT_SMEM(&y[b + p * QP]), e[p]);
                dft_r<QA, +1>(v);
#pragma unroll
                for (int k = 0; k < QA; ++k) *CWT_SMEM(&dst[k * R]) = v[k];
            }
        }
    }
    // middle pass: DFT over b2, b = b1 + QC b2, in place
    if constexpr (QC > 1) {
        __syncthreads();
        if (on) {
#pragma unroll 1
            for (int q = th; q < QC * QA; q += TP) {
                const int b1 = q / QA, k1 = q - b1 * QA;
                float2 *x = tile + rl * a.rs + b1 * a.ps + k1 * R + r;
                const int i = QC * (r + R * k1);
                const float2 w = __ldg(&a.tw[i * a.tws]);
                const float2 w8 = zoom_w8<QB>(a.tw, (unsigned)i, (unsigned)a.M, a.magM, a.tws);
                float2 v[QB];
#pragma unroll
                for (int b = 0; b < QB; ++b) v[b] = *CWT_SMEM(&x[b * (QC * a.ps)]);
                zoom_twiddle<QB>(v, w, w8);
                dft_r<QB, +1>(v);
#pragma unroll
                for (int k = 0; k < QB; ++k) *CWT_SMEM(&x[k * (QC * a.ps)]) = v[k];
            }
        }
    }
    __syncthreads();
    // last pass: DFT over the remaining index, outputs t0 + step m, t0 < step
    const int L1 = QA * R, step = L1 * K2;
#pragma unroll 1
    for (int i = tid; i < nr * a.js; i += T) {
        int il, j;
        zoom_divmod((unsigned)i, (unsigned)a.js, a.magJs, il, j);
        const ZoomRow z = rows[il];
        const int t0 = j - z.shift;
        if ((unsigned)t0 >= (unsigned)min(step, z.n_keep)) continue;
        const float2 w = __ldg(&a.tw[t0 * a.tws]);
        const float2 w8 = zoom_w8<LAST>(a.tw, (unsigned)t0, (unsigned)a.M, a.magM, a.tws);
        int at = t0;  // slot of (k2, k1, r): QC k2 ps + t0 mod L1
        if constexpr (K2 > 1) {
            int k2, tl;
            zoom_divmod((unsigned)t0, (unsigned)L1, a.magL2, k2, tl);
            at = QC * k2 * a.ps + tl;
        }
        const float2 *x = tile + il * a.rs + at;
        float2 v[LAST];
#pragma unroll
        for (int b = 0; b < LAST; ++b) v[b] = *CWT_SMEM(&x[b * a.ps]);
        zoom_twiddle<LAST>(v, w, w8);
        dft_r<LAST, +1>(v);
        if (a.sub != 1) {  // every sub-th sample: output o = t / sub
#pragma unroll
            for (int m = 0; m < LAST; ++m) {
                int o, rem;
                zoom_divmod((unsigned)(t0 + m * step), (unsigned)a.sub, a.magSub, o, rem);
                if (rem != 0 || t0 + m * step >= z.n_keep) continue;
                if (a.oc) __stcs(a.oc + z.base + o, v[m]);
                if (a.op) __stcs(a.op + z.base + o, fmaf(v[m].x, v[m].x, v[m].y * v[m].y));
            }
            continue;
        }
        const int left = t0 + (LAST - 1) * step < z.n_keep ? LAST : (z.n_keep - t0 + step - 1) / step;
        if (a.oc) zoom_store<LAST>(a.oc + z.base + t0, step, left, v, [](float2 x) { return x; });
        if (a.op)
            zoom_store<LAST>(a.op + z.base + t0, step, left, v,
                             [](float2 x) { return fmaf(x.x, x.x, x.y * x.y); });
    }
    // complete in stream order: one CTA outlives the kernel before
    if (a.after && blockIdx.x == gridDim.x - 1) griddep_wait();
}

}  // namespace cwtk
