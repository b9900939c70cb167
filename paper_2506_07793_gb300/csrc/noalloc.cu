// noalloc.cu -- cwt_execute_noalloc: the whole transform with no allocation.
//
// Some callers may not allocate GPU memory once they are running: real-time
// EEG / brain-machine-interface processing loops that must not block (a
// cudaMalloc or cudaFree can synchronise the device and stall the loop past
// its deadline), and plug-ins hosted by an application that owns the GPU
// memory budget.  This entry point serves them: the caller passes the signal
// and the outputs, and everything else the transform needs (twiddle table,
// wavelet bank, band table, spectra) lives in one file-scope device array of
// fixed size that every GPU loading this library holds until process exit.
//
// The arithmetic is the plan path's (FP64 bank evaluated in the same order,
// the same Stockham kernels), so the results match cwt_execute.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "fft_core.cuh"
#include "internal.h"
#include "phase.cuh"

namespace cwtk {
namespace {

constexpr size_t kScratchBytes = CWT_NOALLOC_SCRATCH_BYTES;
constexpr size_t kTwBytes = sizeof(float2) * (size_t)kTwN;  // twiddle table at offset 0
constexpr int kNaThreads = 256;

// The scratch.  Host code must not use this name as an address: it takes the
// device address from cudaGetSymbolAddress (per device) and passes pointers.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

__global__ void na_twiddle_kernel(float2 *tw) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < kTwN) {
        double s, c;
        sincospi(2.0 * (double)m / (double)kTwN, &s, &c);
        tw[m] = make_float2((float)c, (float)s);
    }
}

// F and sigma of up to kNaInline scales travel as kernel arguments; longer
// lists are copied into the scratch.
constexpr int kNaInline = 128;
struct NaScales {
    double F[kNaInline], sig[kNaInline];
};

// Eq. 3 (Morlet spectrum in Hz) in FP64 summed over aliases, in the plan
// generator's order.  Terms e^40 below the bin's largest (exponent `top`) are
// left out: together they are under 1e-15 of it.
__device__ __forceinline__ double na_alias_sum(double base, double r, double lo, double hi, double h, double kappa,
                                               double top) {
    const double q_lo = ceil(lo - base), q_hi = floor(hi - base);
    double v = 0.0;
    for (double q = q_lo; q <= q_hi; q += 1.0) {
        const double u = (base + q) * r;
        const double a = u - 1.0;
        const double e1 = -h * a * a, e2 = -h * u * u;
        double g = 0.0;
        if (e1 > top - 40.0) g = exp(e1);
        if (e2 - h > top - 40.0) g -= kappa * exp(e2);
        v += g;
    }
    return v;
}

// One CTA per scale: the spectrum of its bins in FP64, normalised to unit
// energy with the 1/N of the inverse FFT folded in, rounded to FP32, and its
// band.  Bound by FP64 exponentials (the pipe retires a warp instruction in 16
// cycles), so only bins whose exponent is within 27 of the scale's largest are
// evaluated, once, and no other takes an FP64 instruction: the others are at
// 2e-12 of the peak (a band's limit is 1e-10) and add under 1e-19 to the energy.
// Where the peak itself comes out far below its exponent (a carrier under the
// first bins, whose terms cancel) the bound says nothing and every bin is
// evaluated.  40 scales at N = 2048: 19 us, the forward FFTs beside it; two kernels
// that evaluated every bin three times took 112.
__global__ void __launch_bounds__(kNaThreads)
na_bank_kernel(int N, int S, double fs, const double *par, const __grid_constant__ NaScales inl,
               float *__restrict__ bank, int *__restrict__ band) {
    extern __shared__ double raw[];  // [N]
    __shared__ double sd[kNaThreads], sm[kNaThreads];
    __shared__ int smin[kNaThreads], smax[kNaThreads];
    griddep_launch();
    const int s = blockIdx.x, tid = threadIdx.x;
    const double F = par ? par[s] : inl.F[s], sg = par ? par[S + s] : inl.sig[s];
    const double hh = 0.5 * sg * sg, kappa = exp(-hh), r = fs / F, rN = 1.0 / (double)N;  // N is a power of two
    const double reach = 40.0 * F / sg, q_min = -reach / fs, q_max = (F + reach) / fs;
    const float h = (float)hh, du = (float)(r * rN), uN = (float)r;
    // The exponent of bin k's largest term: of its nearest aliases, u = nu / F in [0,
    // fs / F) with exponent -h (u - 1)^2 and v = u - fs / F with that of the
    // admissibility term, -h (v^2 + 1), kappa = exp(-h).  Squared after the difference:
    // u^2 + 1 - 2 u is off by 1e-7, which h makes more than the cut below from sigma =
    // 30000 up (bins beside the carrier were lost); this form by 2 h |u - 1| 1e-7, below
    // 1 wherever two bins of 16384 compare.
    auto exponent = [&](int k) {
        const float u = (float)k * du, d = u - 1.f, v = u - uN;
        return -h * fminf(d * d, v * v + 1.f);
    };
    __shared__ float sf[kNaThreads];
    float top = -INFINITY;
    for (int k = tid; k < N; k += kNaThreads) top = fmaxf(top, exponent(k));
    sf[tid] = top;
    __syncthreads();
    for (int w = kNaThreads / 2; w > 0; w >>= 1) {
        if (tid < w) sf[tid] = fmaxf(sf[tid], sf[tid + w]);
        __syncthreads();
    }
    const float peak = sf[0];
    float cut = peak - 27.f;
    double energy = 0.0, mx = 0.0;
    for (;;) {
        __syncthreads();
        double e = 0.0, m = 0.0;
        for (int k = tid; k < N; k += kNaThreads) {
            const float x = exponent(k);
            if (x > cut) {
                const double v = na_alias_sum((double)k * rN, r, q_min, q_max, hh, kappa,
                                              cut > -INFINITY ? (double)x : -1e300);
                raw[k] = v;
                e += v * v;
                m = fmax(m, fabs(v));
            }
        }
        sd[tid] = e;
        sm[tid] = m;
        __syncthreads();
        for (int w = kNaThreads / 2; w > 0; w >>= 1) {
            if (tid < w) {
                sd[tid] += sd[tid + w];
                sm[tid] = fmax(sm[tid], sm[tid + w]);
            }
            __syncthreads();
        }
        energy = sd[0];
        mx = sm[0];
        if (cut == -INFINITY || mx > exp((double)peak - 1.0)) break;
        cut = -INFINITY;
    }
    const double scale = energy > 0.0 ? 1.0 / sqrt((double)N * energy) : 0.0;
    const double thr = mx * kBandRelThreshold;
    float *b = bank + (size_t)s * N;
    int lo = N, hi = -N;
    for (int k = tid; k < N; k += kNaThreads) {
        float w = 0.f;
        if (exponent(k) > cut) {
            const double v = raw[k];
            w = (float)(v * scale);
            if (fabs(v) > thr) {
                const int ks = k < N / 2 ? k : k - N;
                lo = min(lo, ks);
                hi = max(hi, ks);
            }
        }
        b[k] = w;
    }
    smin[tid] = lo;
    smax[tid] = hi;
    __syncthreads();
    for (int w = kNaThreads / 2; w > 0; w >>= 1) {
        if (tid < w) {
            smin[tid] = min(smin[tid], smin[tid + w]);
            smax[tid] = max(smax[tid], smax[tid + w]);
        }
        __syncthreads();
    }
    if (tid == 0) {
        int start = 0, len = 0;
        if (smax[0] >= smin[0]) {
            start = smin[0] < 0 ? smin[0] + N : smin[0];
            len = smax[0] - smin[0] + 1;
        }
        band[2 * s] = start;
        band[2 * s + 1] = len;
    }
}

template <int N>
__global__ void __launch_bounds__(RowConfig<N>::THREADS)
na_forward_kernel(const float *__restrict__ x, int C, int n, float2 *__restrict__ spec,
                  const float2 *__restrict__ tw) {
    using RC = RowConfig<N>;
    extern __shared__ float2 na_smem[];
    griddep_launch();
    const int rl = threadIdx.x / RC::T, j = threadIdx.x % RC::T;
    const int row = blockIdx.x * RC::ROWS + rl;
    const bool act = row < C;
    float2 *sm = na_smem + rl * FftShape<N, RC::R>::SMEM_F2;
    const float *xr = x + (size_t)(act ? row : 0) * (size_t)n;
    float2 *out = spec + (size_t)(act ? row : 0) * (size_t)N;
    auto load = [&](int i) -> float2 { return make_float2((act && i < n) ? xr[i] : 0.f, 0.f); };
    auto store = [&](int t, float2 v) {
        if (act) out[t] = v;
    };
    fft_row<N, RC::R, -1>(sm, tw, j, load, store);
    griddep_wait();  // the bank, which this kernel overlaps: the stream's order holds
}

__device__ __noinline__ void na_store_phase(float *dst, float2 v) { *dst = phase_atan2(v.y, v.x); }

template <int N>
__global__ void __launch_bounds__(RowConfig<N>::THREADS)
na_scale_block_kernel(const float2 *__restrict__ spec, const float *__restrict__ bank,
                      const int *__restrict__ band, const float2 *__restrict__ tw, int S, int rows,
                      int n, float2 *oc, float *op, float *oph) {
    using RC = RowConfig<N>;
    extern __shared__ float2 na_smem[];
    const int rl = threadIdx.x / RC::T, j = threadIdx.x % RC::T;
    const int row = blockIdx.x * RC::ROWS + rl;
    const bool act = row < rows;
    const int c = act ? row / S : 0;
    const int s = act ? row - c * S : 0;
    griddep_wait();  // bank and spectra
    float2 *sm = na_smem + rl * FftShape<N, RC::R>::SMEM_F2;
    const float2 *X = spec + (size_t)c * N;
    const float *W = bank + (size_t)s * N;
    const int b0 = band[2 * s], B = act ? band[2 * s + 1] : 0;
    auto load = [&](int k) -> float2 {
        if (((k - b0) & (N - 1)) < B) {
            const float2 xv = X[k];
            const float w = W[k];
            return make_float2(xv.x * w, xv.y * w);
        }
        return make_float2(0.f, 0.f);
    };
    const size_t obase = (size_t)row * (size_t)n;
    auto store = [&](int t, float2 v) {
        if (!act || t >= n) return;
        if (oc) oc[obase + t] = v;
        if (op) op[obase + t] = fmaf(v.x, v.x, v.y * v.y);
        if (oph) na_store_phase(oph + obase + t, v);
    };
    fft_row<N, RC::R, +1>(sm, tw, j, load, store);
}

template <int N>
cudaError_t na_run(const float *x, int C, int n, int S, char *base, const double *par, const NaScales &inl,
                   size_t off_band, size_t off_bank, size_t off_spec, double fs, float2 *oc, float *op, float *oph,
                   cudaStream_t st) {
    using RC = RowConfig<N>;
    static std::atomic<unsigned> attr_b{0}, attr_f{0}, attr_s{0};
    cudaError_t e = ensure_smem_attr(na_bank_kernel, kMaxFft * (int)sizeof(double), &attr_b);
    if (e == cudaSuccess) e = ensure_smem_attr(na_forward_kernel<N>, RC::SMEM_BYTES, &attr_f);
    if (e == cudaSuccess) e = ensure_smem_attr(na_scale_block_kernel<N>, RC::SMEM_BYTES, &attr_s);
    if (e != cudaSuccess) return e;
    const float2 *tw = (const float2 *)base;
    int *band = (int *)(base + off_band);
    float *bank = (float *)(base + off_bank);
    float2 *spec = (float2 *)(base + off_spec);
    na_bank_kernel<<<S, kNaThreads, N * (int)sizeof(double), st>>>(N, S, fs, par, inl, bank, band);
    e = cudaGetLastError();
    // the forward FFTs run beside the bank, the rows wait for both
    if (e == cudaSuccess)
        e = launch_dependent(na_forward_kernel<N>, (C + RC::ROWS - 1) / RC::ROWS, RC::THREADS, RC::SMEM_BYTES, st, x, C,
                             n, spec, tw);
    const int rows = C * S;
    if (e == cudaSuccess)
        e = launch_dependent(na_scale_block_kernel<N>, (rows + RC::ROWS - 1) / RC::ROWS, RC::THREADS, RC::SMEM_BYTES, st,
                             (const float2 *)spec, (const float *)bank, (const int *)band, tw, S, rows, n, oc, op, oph);
    return e;
}

std::mutex g_na_mutex;
char *g_na_base[64] = {};

// Once per device, with that device current: resolve the scratch's device
// address and write the twiddle table into it.
cudaError_t na_setup(int dev, cudaStream_t st, char **base) {
    std::lock_guard<std::mutex> lk(g_na_mutex);
    if (!g_na_base[dev]) {
        void *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        na_twiddle_kernel<<<kTwN / 256, 256, 0, st>>>((float2 *)ptr);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return e;
        g_na_base[dev] = (char *)ptr;
    }
    *base = g_na_base[dev];
    return cudaSuccess;
}

bool na_dev_ptr(const void *p, int dev) {
    if (!p || (reinterpret_cast<uintptr_t>(p) & 15u)) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeManaged || (at.type == cudaMemoryTypeDevice && at.device == dev);
}

}  // namespace
}  // namespace cwtk

extern "C" cwt_status cwt_execute_noalloc(const float *d_signal, int channels, int samples,
                                          double fs, const double *freqs_hz,
                                          const double *n_cycles, int n_freqs, void *d_complex,
                                          float *d_power, float *d_phase, void *stream) {
    using namespace cwtk;
    // ---- host-side validation, before any CUDA call ----
    if (channels < 1 || samples < 1 || !(fs > 0.0) || !std::isfinite(fs) || !freqs_hz ||
        !n_cycles || n_freqs < 1 || (!d_complex && !d_power && !d_phase))
        return CWT_EINVAL;
    for (int i = 0; i < n_freqs; ++i) {
        if (!(freqs_hz[i] > 0.0) || !(freqs_hz[i] < 0.5 * fs) || !std::isfinite(freqs_hz[i]))
            return CWT_EINVAL;
        if (!(n_cycles[i] > 0.0) || !std::isfinite(n_cycles[i])) return CWT_EINVAL;
    }
    int N = 0;
    cwt_status stt = cwt_fft_length(samples, CWT_PAD_POW2, &N);
    if (stt != CWT_OK) return stt;
    if (!scales_on_grid(CWT_WAVELET_MORLET, freqs_hz, n_cycles, n_freqs, 3.0, fs, N)) return CWT_EINVAL;
    const int nblk = (N + kNaThreads - 1) / kNaThreads;
    const size_t off_par = align256(kTwBytes);
    // (a region that nothing uses any more: the documented limit counts it)
    const size_t off_part = off_par + align256(sizeof(double) * 2 * (size_t)n_freqs);
    const size_t off_band = off_part + align256(sizeof(double) * (size_t)n_freqs * nblk);
    const size_t off_bank = off_band + align256(sizeof(int) * 2 * (size_t)n_freqs);
    const size_t off_spec = off_bank + align256(sizeof(float) * (size_t)n_freqs * N);
    const size_t need = off_spec + sizeof(float2) * (size_t)channels * N;
    if (need > kScratchBytes || (long long)channels * n_freqs > (1ll << 30)) return CWT_EINVAL;

    // ---- device side ----
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return CWT_ECUDA;
    if (!na_dev_ptr(d_signal, dev) || (d_complex && !na_dev_ptr(d_complex, dev)) ||
        (d_power && !na_dev_ptr(d_power, dev)) || (d_phase && !na_dev_ptr(d_phase, dev)))
        return CWT_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    char *base = nullptr;
    // not inside a stream capture (see cwt.h), whether or not anything is copied;
    // asked before the set-up, whose launch and wait would invalidate the capture
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &cap);
    if (e == cudaSuccess && cap != cudaStreamCaptureStatusNone) return CWT_ECUDA;
    if (e == cudaSuccess) e = na_setup(dev, st, &base);
    NaScales inl;
    const double *par = nullptr;
    if (n_freqs <= kNaInline) {
        std::copy(freqs_hz, freqs_hz + n_freqs, inl.F);
        std::copy(n_cycles, n_cycles + n_freqs, inl.sig);
    } else {
        par = (const double *)(base + off_par);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(base + off_par, freqs_hz, sizeof(double) * n_freqs, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(base + off_par + sizeof(double) * n_freqs, n_cycles, sizeof(double) * n_freqs,
                                cudaMemcpyHostToDevice, st);
    }
    if (e == cudaSuccess) {
        float2 *oc = (float2 *)d_complex;
        const int S = n_freqs;
        switch (ilog2c(N)) {
#define CWT_NA_CASE(L)                                                                             \
    case L:                                                                                        \
        e = na_run<1 << L>(d_signal, channels, samples, S, base, par, inl, off_band, off_bank,    \
                           off_spec, fs, oc, d_power, d_phase, st);                                \
        break;
            CWT_NA_CASE(5) CWT_NA_CASE(6) CWT_NA_CASE(7) CWT_NA_CASE(8) CWT_NA_CASE(9)
            CWT_NA_CASE(10) CWT_NA_CASE(11) CWT_NA_CASE(12) CWT_NA_CASE(13) CWT_NA_CASE(14)
#undef CWT_NA_CASE
            default: return CWT_EUNSUPPORTED;
        }
    }
    if (e == cudaErrorMemoryAllocation) return CWT_ENOMEM;
#ifdef CWT_BOUNDS_CHECK
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && check_collect(nullptr)) return CWT_EDEVICE;
#endif
    return e == cudaSuccess ? CWT_OK : CWT_ECUDA;
}
