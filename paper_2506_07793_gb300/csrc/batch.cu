// batch.cu -- many epochs of uneven length in one call.
//
// The paper loops over recordings in Python (Sections "Comparison between
// devices and software" and "Wavelength and flexibility"); here a batch of
// epochs, each with its own length n_e and hence its own padded length
// N_e = next power of two >= max(n_e, 32) (Section "Fast Fourier transform"),
// is one launch per stage for all of them.
//
// The narrow-band scales (most or all: the band is 4 ... 36% of N_e / f on the
// batching workload) run by residue classes, zoom_row_kernel of zoom.cuh, one
// launch per padded length and class of scales over all its epochs.  They read
// a window of bins, an eighth of the spectrum; the workspace that carries it is
// kept below kWsBytes by taking the epochs in chunks.  Where every scale of a
// padded length does so, its forward FFTs are batch_forward.cu's.
//
// Otherwise a persistent kernel, replayed from a CUDA graph, takes work items
// of one epoch and G channels with G * N_e = one tile of kTile points (G capped
// by the channel count), from an atomic counter, largest FFTs first.  Per item
// the CTA
//   1. runs the forward FFT of the G channels (Eq. 2, one FFT per channel)
//      and keeps the spectra in shared memory -- they never reach HBM;
//   2. stores the window of bins that the narrow-band scales read;
//   3. for every (channel, scale) row of the other scales: band product with
//      the FP64-generated bank of length N_e (Eq. 3), spectral fold by the
//      power-of-two factor f of the decimation, inverse FFT of N_e / f points,
//      crop / decimate / reduce and coalesced stores (Section "Precision").
// Its rows take 16 points per thread (two CTAs per SM; 47 ms per batch of 2048
// epochs against 81 on 32 points), 32 only in batches with a row that 16 cannot
// stage, items largest first (59 and 131 ms in input order).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <new>
#include <numeric>
#include <vector>

#include "batch_kernel.cuh"
#include "zoom.h"

namespace cwtk {

const void *batch_kernel_ptr_16();
const void *batch_kernel_ptr_32();
const void *batch_kernel_ptr(int ri) { return ri == 16 ? batch_kernel_ptr_16() : batch_kernel_ptr_32(); }

// ---- host side -------------------------------------------------------------

constexpr size_t kWsBytes = (size_t)256 << 20;

// What a padded length needs: its bank, and which scales run how.
struct BatchLength {
    float *bank = nullptr;
    int *band = nullptr;
    int4 *d_list = nullptr;  // the classes' scales, then the rest's indices
    int *d_rest = nullptr;   // into d_list's allocation; null: every scale
    int nrest = 0, w0 = 0, wn = 0, M = 0;
    std::vector<ZoomClass> classes;
};

// Epochs of one workspace: their items, and per length the first and count of
// their ZoomEpochs.
struct BatchChunk {
    size_t item0 = 0, items = 0, ws = 0;
    size_t ep0[kMaxBatchLog2 + 1] = {}, eps[kMaxBatchLog2 + 1] = {};
};

struct BatchState {
    BatchLength len[kMaxBatchLog2 + 1];
    BatchItem *d_items = nullptr;
    size_t items_cap = 0;
    ZoomEpoch *d_eps = nullptr;
    size_t eps_cap = 0;
    float2 *d_ws = nullptr;
    size_t ws_cap = 0;  // elements
    int *d_counter = nullptr;
    // the shape that d_items and d_eps describe
    std::vector<cwt_epoch> shape;
    std::vector<BatchChunk> chunks;
    size_t n_items = 0;
    // CUDA graph: memset(counter) -> batch_kernel
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaGraphNode_t knode = nullptr;
    int graph_ri = 0;
    BatchArgs graph_args{};
    bool ready = false;
    int ri = 16;
    double tune_ms[4] = {0, 0, 0, 0};
    long long launches = 0;
    int grid = 0;
    size_t bytes = 0;
};

void free_batch_state(BatchState *b) {
    if (!b) return;
    for (BatchLength &l : b->len) {
        cudaFree(l.bank);
        cudaFree(l.band);
        cudaFree(l.d_list);
    }
    cudaFree(b->d_items);
    cudaFree(b->d_eps);
    cudaFree(b->d_ws);
    cudaFree(b->d_counter);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    delete b;
}

size_t batch_bytes(const BatchState *b) {
    if (!b) return 0;
    return b->bytes + b->items_cap * sizeof(BatchItem) + b->eps_cap * sizeof(ZoomEpoch) + b->ws_cap * sizeof(float2);
}

namespace {

template <int RI>
cudaError_t batch_attr() {
    static std::atomic<unsigned> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 32 && (done.load(std::memory_order_acquire) & (1u << dev))) return cudaSuccess;
    e = cudaFuncSetAttribute(batch_kernel_ptr(RI), cudaFuncAttributeMaxDynamicSharedMemorySize, batch_smem<RI>());
    if (e == cudaSuccess && dev < 32) done.fetch_or(1u << dev, std::memory_order_acq_rel);
    return e;
}

cudaError_t batch_grid(int ri, int *grid) {
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, batch_kernel_ptr(ri), kBThreads,
                                                          ri == 16 ? batch_smem<16>() : batch_smem<32>());
    if (e == cudaSuccess) *grid = sms * std::max(per, 1);
    return e;
}

// (Re)build the graph for radix `ri` with arguments `args`, or update its
// kernel node in place when only the arguments changed.
cudaError_t batch_graph(BatchState *b, int ri, const BatchArgs &args, int grid) {
    cudaKernelNodeParams kp{};
    void *kargs[] = {(void *)&args};
    kp.func = (void *)batch_kernel_ptr(ri);
    kp.gridDim = dim3(grid);
    kp.blockDim = dim3(kBThreads);
    kp.sharedMemBytes = ri == 16 ? batch_smem<16>() : batch_smem<32>();
    kp.kernelParams = kargs;
    if (b->exec && b->graph_ri == ri) {
        if (std::memcmp(&b->graph_args, &args, sizeof(args)) == 0) return cudaSuccess;
        cudaError_t e = cudaGraphExecKernelNodeSetParams(b->exec, b->knode, &kp);
        if (e == cudaSuccess) b->graph_args = args;
        return e;
    }
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
    cudaError_t e = cudaGraphCreate(&b->graph, 0);
    cudaGraphNode_t mnode;
    cudaMemsetParams mp{};
    mp.dst = b->d_counter;
    mp.elementSize = sizeof(int);
    mp.width = 1;
    mp.height = 1;
    mp.value = 0;
    if (e == cudaSuccess) e = cudaGraphAddMemsetNode(&mnode, b->graph, nullptr, 0, &mp);
    if (e == cudaSuccess) e = cudaGraphAddKernelNode(&b->knode, b->graph, &mnode, 1, &kp);
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
    if (e == cudaSuccess) {
        b->graph_ri = ri;
        b->graph_args = args;
    }
    return e;
}

}  // namespace

namespace {

// Bank, bands and the split of the scales for padded length 2^L.  Published
// only once complete, so a failure leaves nothing half-built for the next call.
cudaError_t make_length(cwt_plan_s *p, int L, cudaStream_t st, BatchLength *out) {
    const int S = p->S, N = 1 << L;
    BatchLength l;
    cudaError_t e = dmalloc(&l.bank, sizeof(float) * (size_t)S * N);
    if (e == cudaSuccess) e = dmalloc(&l.band, sizeof(int) * 2 * (size_t)S);
    if (e == cudaSuccess) e = launch_bank_n(p, N, l.bank, l.band, st, nullptr);
    std::vector<int> band(2 * (size_t)S), rest;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(band.data(), l.band, sizeof(int) * band.size(), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    std::vector<int4> list;
    if (e == cudaSuccess) {
        const int f = std::gcd(N, p->d);
        ZoomShape sh;
        sh.M = l.M = N / f;
        sh.sub = p->d / f;
        sh.n_out = 0;  // epochs of any length
        // ps: a row here takes 4.2 ps per point, and the first one brings the forward FFTs
        // of its length with it (7 of 64 scales of 8192-point rows: 6.3 ps per point in all,
        // 4.4 on 32 x 32 by residue classes)
        sh.rest_cost = 8.0 * batch_inverse_length(N, p->d);
        // rows subsampled past the fold (odd d) keep the kernel here: 0.92 against 0.99 ms
        // for 144 epochs of 8 channels at d = 5
        sh.phase = (p->outputs & CWT_OUT_PHASE) != 0 || sh.sub != 1;
        sh.rows_only = true;
        sh.wide = false;
        sh.channels = 4096;  // epochs x channels
        sh.both = false;
        sh.compiled_cost = 0;
        zoom_select(sh, S, band.data(), &l.classes, &list, &rest);
        l.nrest = (int)rest.size();
        if (!list.empty()) {
            int lo = N, hi = -N;
            for (const int4 &z : list) {  // the union of the bands, around bin 0
                const int b0 = z.y < N / 2 ? z.y : z.y - N;
                lo = std::min(lo, b0);
                hi = std::max(hi, b0 + z.z);
            }
            l.wn = std::min(N, std::max(hi - lo, 1));
            l.w0 = l.wn == N ? 0 : (lo + N) % N;
            e = dmalloc(&l.d_list, sizeof(int4) * list.size() + sizeof(int) * rest.size());
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(l.d_list, list.data(), sizeof(int4) * list.size(), cudaMemcpyHostToDevice, st);
            l.d_rest = (int *)(l.d_list + list.size());
            if (e == cudaSuccess && !rest.empty())
                e = cudaMemcpyAsync(l.d_rest, rest.data(), sizeof(int) * rest.size(), cudaMemcpyHostToDevice, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        }
    }
    if (e != cudaSuccess) {
        cudaFree(l.bank);
        cudaFree(l.band);
        cudaFree(l.d_list);
        return e;
    }
    *out = l;
    return cudaSuccess;
}

// Grow a device buffer to n elements; the old one is freed once the new exists.
template <class T>
cudaError_t grow(T **p, size_t *cap, size_t n) {
    if (n <= *cap) return cudaSuccess;
    T *d = nullptr;
    const cudaError_t e = dmalloc(&d, sizeof(T) * n);
    if (e != cudaSuccess) return e;
    cudaFree(*p);
    *p = d;
    *cap = n;
    return cudaSuccess;
}

int epoch_log2(const cwt_plan_s *p, const cwt_epoch &ep) {
    int N = kMinFft;
    while (N < ep.samples + p->pad_extra) N <<= 1;
    return ilog2c(N);
}

// Items, chunks of up to *ws_bytes (or one epoch) of workspace and epoch tables of a
// new shape, uploaded; *ws_bytes becomes the largest chunk's.
cudaError_t make_shape(cwt_plan_s *p, BatchState *b, const cwt_epoch *epochs, int n_epochs, size_t *ws_bytes,
                       cudaStream_t st) {
    const int C = p->C, S = p->S, d = p->d;
    std::vector<BatchItem> items;
    std::vector<ZoomEpoch> eps;
    std::vector<BatchChunk> chunks;
    size_t ws_max = 0, n_items = 0;
    int max_m = 0;
    b->ready = false;
    for (int first = 0; first < n_epochs;) {
        BatchChunk ch;
        ch.item0 = items.size();
        int last = first;
        for (; last < n_epochs; ++last) {
            const size_t w = (size_t)C * (size_t)b->len[epoch_log2(p, epochs[last])].wn;
            if (last > first && (ch.ws + w) * sizeof(float2) > *ws_bytes) break;
            ch.ws += w;
        }
        size_t ws = 0;
        for (int L = kMaxBatchLog2; L >= 0; --L) {  // largest FFTs first
            ch.ep0[L] = eps.size();
            for (int i = first; i < last; ++i) {
                const cwt_epoch &ep = epochs[i];
                if (epoch_log2(p, ep) != L) continue;
                const BatchLength &l = b->len[L];
                const int N = 1 << L, n_out = (ep.samples + d - 1) / d, sub = d / std::gcd(N, d);
                max_m = std::max(max_m, l.nrest ? batch_inverse_length(N, d) : 0);
                const int G = std::max(1, std::min(C, kTile / N));
                n_items += (size_t)((C + G - 1) / G);
                for (int c0 = 0; l.nrest && c0 < C; c0 += G) {  // the others: batch_forward.cu
                    BatchItem it{};
                    it.in_off = ep.in_offset + (long long)c0 * ep.samples;
                    it.out_off = ep.out_offset + (long long)c0 * S * n_out;
                    it.ws_off = (long long)ws + (long long)c0 * l.wn;
                    it.n = ep.samples;
                    it.log2n = L;
                    it.G = std::min(G, C - c0);
                    items.push_back(it);
                }
                eps.push_back({(long long)ws, ep.out_offset, ep.in_offset, n_out, sub * (n_out - 1) + 1, ep.samples, 0});
                ws += (size_t)C * (size_t)l.wn;
            }
            ch.eps[L] = eps.size() - ch.ep0[L];
        }
        ch.items = items.size() - ch.item0;
        ws_max = std::max(ws_max, ws);
        chunks.push_back(ch);
        first = last;
    }
    *ws_bytes = ws_max * sizeof(float2);
    cudaError_t e = grow(&b->d_items, &b->items_cap, std::max<size_t>(items.size(), 1));
    if (e == cudaSuccess) e = grow(&b->d_eps, &b->eps_cap, eps.size());
    if (e == cudaSuccess) e = grow(&b->d_ws, &b->ws_cap, ws_max);
    if (e == cudaSuccess && !items.empty())
        e = cudaMemcpyAsync(b->d_items, items.data(), items.size() * sizeof(BatchItem), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_eps, eps.data(), eps.size() * sizeof(ZoomEpoch), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // the host vectors go
    if (e != cudaSuccess) return e;
    // RI = 16 stages kBThreads * 16 points of inverse rows: only for batches
    // whose every inverse length fits (an 8192-point row at odd d needs RI = 32)
    const bool ri16 = max_m <= kBThreads * 16;
    b->ri = ri16 ? 16 : 32;
    for (int i = 0; i < 4; ++i) b->tune_ms[i] = !ri16 && i % 2 == 0 ? -1.0 : 0.0;
    b->shape.assign(epochs, epochs + n_epochs);
    b->chunks = chunks;
    b->n_items = n_items;
    b->ready = true;
    return cudaSuccess;
}

cudaError_t batch_prepare(cwt_plan_s *p, const cwt_epoch *epochs, int n_epochs, cudaStream_t st) {
    if (!p->batch) p->batch = new BatchState();
    BatchState *b = p->batch;
    cudaError_t e = cudaSuccess;
    if (!b->d_counter) e = dmalloc(&b->d_counter, sizeof(int));
    for (int i = 0; i < n_epochs && e == cudaSuccess; ++i) {
        const int L = epoch_log2(p, epochs[i]);
        if (b->len[L].bank) continue;
        e = make_length(p, L, st, &b->len[L]);
        if (e == cudaSuccess) b->bytes += (sizeof(float) * ((size_t)1 << L) + sizeof(int) * 2) * (size_t)p->S;
    }
    if (e == cudaSuccess) e = batch_attr<16>();
    if (e == cudaSuccess) e = batch_attr<32>();
    if (e != cudaSuccess) return e;
    const bool same = b->ready && b->shape.size() == (size_t)n_epochs &&
                      std::equal(b->shape.begin(), b->shape.end(), epochs, [](const cwt_epoch &x, const cwt_epoch &y) {
                          return x.in_offset == y.in_offset && x.out_offset == y.out_offset && x.samples == y.samples;
                      });
    if (same) return cudaSuccess;
    // more and smaller chunks where memory is short: slower, the same values
    size_t ws = kWsBytes, tried = (size_t)-1;
    while ((e = make_shape(p, b, epochs, n_epochs, &ws, st)) == cudaErrorMemoryAllocation && ws < tried) {
        cudaGetLastError();  // clear the non-sticky error
        tried = ws;
        ws /= 4;
    }
    return e;
}

cudaError_t batch_run(cwt_plan_s *p, const float *in, float2 *oc, float *op, float *oph, cudaStream_t st) {
    BatchState *b = p->batch;
    int grid = 0;
    cudaError_t e = batch_grid(b->ri, &grid);
    for (size_t k = 0; k < b->chunks.size() && e == cudaSuccess; ++k) {
        const BatchChunk &ch = b->chunks[k];
        BatchArgs a;
        std::memset(&a, 0, sizeof(a));  // padding too: the graph compares argument bytes
        a.in = in;
        a.oc = oc;
        a.op = op;
        a.oph = oph;
        a.items = b->d_items + ch.item0;
        a.n_items = (int)ch.items;
        a.counter = b->d_counter;
        a.ws = b->d_ws;
        for (int i = 0; i <= kMaxBatchLog2; ++i) {
            const BatchLength &l = b->len[i];
            a.bank[i] = l.bank;
            a.band[i] = l.band;
            a.rest[i] = l.classes.empty() ? nullptr : l.d_rest;
            a.nrest[i] = l.nrest;
            a.w0[i] = l.w0;
            a.wn[i] = l.wn;
        }
        a.tw = p->tw;
        a.S = p->S;
        a.d = p->d;
        if (ch.items) {
            e = batch_graph(b, b->ri, a, grid);
            if (e == cudaSuccess) e = cudaGraphLaunch(b->exec, st);
        }
        BatchForwardArgs f = {};
        f.in = in;
        f.ws = b->d_ws;
        f.tw = p->tw;
        f.C = p->C;
        for (int L = 0; L <= kMaxBatchLog2; ++L) {
            if (b->len[L].nrest || b->len[L].classes.empty()) continue;
            f.eps[L] = b->d_eps + ch.ep0[L];
            f.rows[L] = (int)ch.eps[L] * p->C;
            f.w0[L] = b->len[L].w0;
            f.wn[L] = b->len[L].wn;
        }
        if (e == cudaSuccess) e = launch_batch_forward(f, st);
        if (e != cudaSuccess) return e;
        b->grid = grid;
        ++b->launches;
        // the narrow-band scales, overlapping as in launch_scale_block_zoom
        bool after = false;
        for (int L = kMaxBatchLog2; L >= 0; --L) {
            const BatchLength &l = b->len[L];
            if (!ch.eps[L] || l.classes.empty()) continue;
            ZoomArgs z = {};
            z.spec = b->d_ws;
            z.bank = l.bank;
            z.tw = twiddles_pow2(p->tw, l.M);
            z.oc = oc;
            z.op = op;
            z.N = 1 << L;
            z.M = l.M;
            z.tws = 1;
            z.S = p->S;
            z.sub = p->d / std::gcd(z.N, p->d);
            z.epochs = b->d_eps + ch.ep0[L];
            z.C = p->C;
            z.magCh = zoom_magic((unsigned)p->C);
            z.w0 = l.w0;
            z.wn = l.wn;
            for (const ZoomClass &c : l.classes) {
                z.after = after;
                after = true;
                e = zoom_launch(c, z, (long long)ch.eps[L] * p->C, twiddles_pow2(p->tw, zoom_class_L(c, l.M)),
                                l.d_list, st);
                if (e != cudaSuccess) return e;
            }
        }
    }
    return e;
}

}  // namespace

cudaError_t batch_execute(cwt_plan_s *p, const cwt_epoch *epochs, int n_epochs, const float *in,
                          float2 *oc, float *op, float *oph, cudaStream_t st, bool prepare_only) {
    // A captured batch would replay into a workspace that a later shape replaces.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) return e;
    if (cap != cudaStreamCaptureStatusNone) return cudaErrorStreamCaptureUnsupported;
    if (!prepare_only) return batch_run(p, in, oc, op, oph, st);
    try {
        return batch_prepare(p, epochs, n_epochs, st);
    } catch (const std::bad_alloc &) {
        return cudaErrorMemoryAllocation;
    }
}

void batch_stats(const cwt_plan_s *p, cwt_batch_stats *s) {
    std::memset(s, 0, sizeof(*s));
    const BatchState *b = p->batch;
    if (!b) return;
    s->items = (int)b->n_items;
    s->grid = b->grid;
    s->inverse_radix = b->ri;
    s->order = 0;
    s->tuned = b->ready;
    for (int i = 0; i < 4; ++i) s->tune_ms[i] = b->tune_ms[i];
    s->graph_launches = b->launches;
    s->bank_bytes = b->bytes;
}

}  // namespace cwtk
