// batch_forward.cu -- the forward FFTs of a batch's epochs where every scale
// runs by residue classes: only the window of bins that those read is kept.
//
// The signal is real: N samples are N / 2 complex ones, z[m] = x[2m] + i x[2m +
// 1], and with Z their FFT of M = N / 2 points
//   X[k] = E + w_N^k O,  E = (Z[k] + conj Z[-k]) / 2,  O = (Z[k] - conj Z[-k]) / 2i
// (indices mod M), formed for the bins of the window alone.  Bound by the
// latency of its passes through shared memory: a CTA holds one tile of 4096
// complex points (34 KB, three CTAs per SM), 16 per thread, whatever the length.
// 256 epochs of 64 channels x 256 ... 8192 samples: 187 us; in the persistent
// kernel, 8192 points on 104 KB beside its inverse rows, about 450.
#include <cuda_runtime.h>

#include "batch_kernel.cuh"
#include "fft_core.cuh"
#include "zoom.h"

namespace cwtk {
namespace {

constexpr int kFThreads = 256, kFR = 16, kFTile = kFThreads * kFR;
constexpr int kFSmem = (kFTile + (kFTile >> 4)) * 8;

template <int L>
__device__ __forceinline__ void forward_rows(const BatchForwardArgs &a, int group, float2 *sm) {
    constexpr int N = 1 << L, M = N / 2, T = M / kFR, P = kFThreads / T;
    using Shape = FftShape<M, kFR>;
    const int tid = (int)threadIdx.x, rl = tid / T, j = tid % T;
    const int row = group * P + rl;
    const float *x = a.in;
    int n = 0;
    if (row < a.rows[L]) {
        const int e = row / a.C, c = row - e * a.C;
        const ZoomEpoch ep = a.eps[L][e];
        x += ep.in + (long long)c * ep.n;
        n = ep.n;
    }
    auto load = [&](int m) -> float2 {
        return make_float2(2 * m < n ? __ldg(x + 2 * m) : 0.f, 2 * m + 1 < n ? __ldg(x + 2 * m + 1) : 0.f);
    };
    float2 *const Z = sm + rl * M;
    auto store = [&](int t, float2 v) { *CWT_SMEM(&Z[t]) = v; };  // one pass: nothing is staged
    float2 v[kFR];
    fft_pass0_dense<M, kFR, -1>(v, j, load);
    fft_finish<M, kFR, -1, decltype(store), true>(v, sm + rl * Shape::SMEM_F2, a.tw, j, store);
    if constexpr (Shape::NP > 1) {
        __syncthreads();  // every staging read is done before the spectra overwrite it
#pragma unroll
        for (int r = 0; r < kFR; ++r) *CWT_SMEM(&Z[j + r * T]) = v[r];
    }
    __syncthreads();
    const int wn = a.wn[L], w0 = a.w0[L];
    auto window = [&](int g, int lane, int step) {
        const int q = group * P + g;
        if (q >= a.rows[L]) return;
        const int e = q / a.C, c = q - e * a.C;
        float2 *out = a.ws + a.eps[L][e].spec + (long long)c * wn;
        const float2 *z = sm + g * M;
#pragma unroll 2
        for (int i = lane; i < wn; i += step) {
            const int k = (w0 + i) & (N - 1);
            const float2 p = *CWT_SMEM(&z[k & (M - 1)]), m = *CWT_SMEM(&z[-k & (M - 1)]);
            const float2 w = __ldg(&a.tw[k * (kTwN / N)]);  // conj w_N^k
            const float2 o = make_float2(0.5f * (p.y + m.y), 0.5f * (m.x - p.x));
            out[i] = make_float2(fmaf(0.5f, p.x + m.x, fmaf(w.x, o.x, w.y * o.y)),
                                 fmaf(0.5f, p.y - m.y, fmaf(w.x, o.y, -w.y * o.x)));
        }
    };
    if constexpr (P < 8) {
#pragma unroll 1
        for (int g = 0; g < P; ++g) window(g, tid, kFThreads);
    } else {
#pragma unroll 1
        for (int g = tid >> 5; g < P; g += kFThreads / 32) window(g, tid & 31, 32);
    }
}

__global__ void __launch_bounds__(kFThreads, 3) batch_forward_kernel(const BatchForwardArgs a) {
    extern __shared__ float2 fsm[];
    griddep_launch();
    int group = (int)blockIdx.x, L = kMaxBatchLog2;
    while (L > 5 && group >= a.groups[L]) group -= a.groups[L--];
    switch (L) {  // largest FFTs first
        case 5: forward_rows<5>(a, group, fsm); break;
        case 6: forward_rows<6>(a, group, fsm); break;
        case 7: forward_rows<7>(a, group, fsm); break;
        case 8: forward_rows<8>(a, group, fsm); break;
        case 9: forward_rows<9>(a, group, fsm); break;
        case 10: forward_rows<10>(a, group, fsm); break;
        case 11: forward_rows<11>(a, group, fsm); break;
        case 12: forward_rows<12>(a, group, fsm); break;
        default: forward_rows<13>(a, group, fsm); break;
    }
}

}  // namespace

cudaError_t launch_batch_forward(BatchForwardArgs a, cudaStream_t st) {
    long long blocks = 0;
    for (int L = 5; L <= kMaxBatchLog2; ++L) {
        const int P = 2 * kFTile >> L;  // rows per CTA
        a.groups[L] = (a.rows[L] + P - 1) / P;
        blocks += a.groups[L];
    }
    if (!blocks) return cudaSuccess;
    batch_forward_kernel<<<(unsigned)blocks, kFThreads, kFSmem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace cwtk
