// zoom.cu -- which scales run by output residue classes (zoom.cuh), with which
// transform, and their launches.
//
// A row of N bins decimated by d is evaluated on the M = N / gcd(N, d) points
// that contain every kept sample (the spectral fold is implied: bins are
// taken mod M).  A scale whose band has B bins can run any instance with
// Q >= B and Q a divisor of M; the choice depends on the length and the bands
// alone, so that a shard of the channels gives the same bits as the whole.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <numeric>
#include <vector>

#include "internal.h"
#include "zoom.h"

namespace cwtk {

namespace {

struct ZoomInst {
    int QA, Q, NB, P, T, LAST;
    float cost;  // ps per point
};

// instance i of zoom_list.h (the groups list them out of order)
const ZoomInst &inst(int i) {
    static const std::vector<ZoomInst> table = [] {
        std::vector<ZoomInst> t(kZoomInstances);
#define CWT_ZOOM_ROW(I, QA, QB, QC, P, T, MINB, COST) \
    t[I] = ZoomInst{QA, QA * QB * QC, ZoomCfg<QA, QB, QC, P, T, MINB>::NB, P, T, ZoomCfg<QA, QB, QC, P, T, MINB>::LAST, COST};
        CWT_ZOOM_ALL(CWT_ZOOM_ROW)
#undef CWT_ZOOM_ROW
        return t;
    }();
    return table[(size_t)i];
}

}  // namespace

#define CWT_ZOOM_DECLARE(I, QA, QB, QC, P, T, MINB, COST) \
    template <>                                           \
    const void *zoom_entry<I>(int mode);
CWT_ZOOM_ALL(CWT_ZOOM_DECLARE)
#undef CWT_ZOOM_DECLARE
#define CWT_WIDE_DECLARE(I, QB, QC, P, T, MINB) \
    template <>                                 \
    const void *wide_rest_entry<I>(int mode);
CWT_WIDE_REST(CWT_WIDE_DECLARE)
#undef CWT_WIDE_DECLARE

namespace {

const void *kernel_of(int i, int mode) {
    switch (i) {
#define CWT_ZOOM_CASE(I, QA, QB, QC, P, T, MINB, COST) \
    case I: return zoom_entry<I>(mode);
        CWT_ZOOM_ALL(CWT_ZOOM_CASE)
#undef CWT_ZOOM_CASE
        default: return nullptr;
    }
}

int smem_of(int i, int rows) {
    switch (i) {
#define CWT_ZOOM_CASE(I, QA, QB, QC, P, T, MINB, COST) \
    case I: return ZoomCfg<QA, QB, QC, P, T, MINB>::smem(rows);
        CWT_ZOOM_ALL(CWT_ZOOM_CASE)
#undef CWT_ZOOM_CASE
        default: return 0;
    }
}

int row_smem_of(int i, int nr, int rs, int R) {
    switch (i) {
#define CWT_ZOOM_CASE(I, QA, QB, QC, P, T, MINB, COST) \
    case I: return zoom_row_smem<ZoomCfg<QA, QB, QC, P, T, MINB>>(nr, rs, R);
        CWT_ZOOM_ALL(CWT_ZOOM_CASE)
#undef CWT_ZOOM_CASE
        default: return 0;
    }
}

struct WideInst {
    int QB, QC, P, T, smem;
};

int wide_radix(int i) {
    static const int r[kWideFirst] = {
#define CWT_WIDE_ROW(I, QA) QA,
        CWT_WIDE_FIRST(CWT_WIDE_ROW)
#undef CWT_WIDE_ROW
    };
    return r[i];
}

const WideInst &wide_rest(int i) {
    static const std::vector<WideInst> table = [] {
        std::vector<WideInst> t(kWideRest);
#define CWT_WIDE_ROW(I, QB, QC, P, T, MINB) t[I] = WideInst{QB, QC, P, T, WideCfg<QB, QC, P, T, MINB>::SMEM};
        CWT_WIDE_REST(CWT_WIDE_ROW)
#undef CWT_WIDE_ROW
        return t;
    }();
    return table[(size_t)i];
}

const void *wide_kernel_of(int i, int mode) {
    switch (i) {
#define CWT_WIDE_CASE(I, QB, QC, P, T, MINB) \
    case I: return wide_rest_entry<I>(mode);
        CWT_WIDE_REST(CWT_WIDE_CASE)
#undef CWT_WIDE_CASE
        default: return nullptr;
    }
}

constexpr int kMaxSmem = 227 * 1024;
constexpr int kSms = 152;

// Rows that P consecutive columns, the first a multiple of P, can meet.
int rows_met(int P, int R) {
    if (R % P == 0) return 1;
    return P % R == 0 ? P / R : (P - 2) / R + 2;
}

// Slots of one position of a tile row (QA R and padding) and of a tile row.  A
// half-warp of the first pass that spans several rows, or the positions of
// several threads, then falls into different banks: rows start R and a
// thread's next NB positions nr R slots further, mod 16.
int position_stride(int i, int nr, int R) {
    const int C = nr * R, len = inst(i).QA * R;
    if (C >= 16) return len;
    const int nb = inst(i).NB, want = C / nb, mod = 16 / nb;
    return len + (((want - len) % mod) + mod) % mod;
}
int row_stride(int i, int nr, int R) {
    const int len = inst(i).Q / inst(i).QA * position_stride(i, nr, R);
    return R < 16 && nr > 1 ? len + ((R - len) & 15) : len;
}

// Rows per CTA of zoom_row_kernel for a launch of `rows`: the most threads at work
// on a tile of about 5000 points (several CTAs per SM), up to 8400; few enough
// that two CTAs per SM have rows.  A row's arithmetic does not depend on it.
int rows_per_cta(int i, int M, int R, long long rows) {
    const int T = inst(i).T;
    int best = 1;
    double score = -1;
    for (int nr = 1; nr * R <= T && (nr == 1 || (nr * M <= 8400 && (long long)nr * 2 * kSms <= rows)); ++nr) {
        const int C = nr * R;
        double v = (double)(T / C * C) / T;
        if (nr * M < 4000) v *= nr * M / 4000.0;
        if (nr * M > 5600) v *= 0.95;
        if (v > score) score = v, best = nr;
    }
    return best;
}

// Whether rows of M points, R residues, can run on instance i by whole rows (MODE
// 2, not for the phase), for any number of rows in a launch.
bool row_fits(int i, int M, int R) {
    if (R < 2 || R > inst(i).T || M > zoom_row_points(inst(i).T)) return false;
    for (int nr = rows_per_cta(i, M, R, 1ll << 40); nr >= 1; --nr)
        if (row_smem_of(i, nr, row_stride(i, nr, R), R) > kMaxSmem) return false;
    return true;
}

// Opt instance i (mode) into the largest shared memory, once per device.
cudaError_t ensure_smem(const void *kernel, std::atomic<unsigned> *done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 32 && (done->load(std::memory_order_acquire) & (1u << dev))) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e == cudaSuccess && dev < 32) done->fetch_or(1u << dev, std::memory_order_acq_rel);
    return e;
}
cudaError_t ensure_zoom_smem(int i, int mode) {
    static std::atomic<unsigned> done[kZoomInstances][3];
    return ensure_smem(kernel_of(i, mode), &done[i][mode]);
}
cudaError_t ensure_wide_smem(int i, int mode) {
    static std::atomic<unsigned> done[kWideRest][2];
    return ensure_smem(wide_kernel_of(i, mode), &done[i][mode]);
}

// Cost of one row (ps) on instance i by columns.  A run of R outputs starts at
// a multiple of R past the row's base: unless 8 divides both, its ends share
// 32-byte sectors with runs stored by other instructions.  With one output array
// that costs next to nothing (480 MB of power or of complex values: 0.95 of the
// instance's cost aligned, 1.0 not); with two, whose sectors compete for L2, it
// costs 1.25 at multiples of 4 and 1.3 ... 1.8 off them, against 1.15 (medians of
// 2200 launches of 40 Mi points at 39 lengths, by columns per CTA and residues).
double column_cost(int i, const ZoomShape &z) {
    const int R = z.M / inst(i).Q, P = inst(i).P;
    const bool eighth = R % 8 == 0 && z.n_out % 8 == 0, quarter = R % 4 == 0 && z.n_out % 4 == 0;
    const bool three = inst(i).Q / inst(i).QA != inst(i).LAST;  // passes
    double f;
    if (P <= 4) f = !z.both ? 0.92 : quarter ? 1.05 : 1.35;
    else if (!z.both) f = eighth ? 0.95 : R >= 32 ? 1.0 : 1.1;
    else if (quarter) f = eighth ? 1.15 : 1.25;
    else if (P <= 8) f = three ? 1.35 : R >= 8 ? 1.95 : 1.35;
    else f = P <= 16 ? 1.85 : R >= 128 ? 1.3 : R >= 64 ? 1.45 : R > P ? 1.75 : 1.55;  // R <= P: a CTA holds the row
    if (z.both && P > 4 && !quarter) f = 1.15 + (f - 1.15) * z.kept();
    if (R % P != 0 && P % R != 0) f *= 1.05;  // column groups that meet several rows form more band products
    // a division per output, and fewer of them stored
    if (z.sub != 1) f = three ? 1.25 : z.both ? 1.75 : 1.45;
    if ((P > 8 || (P > 4 && z.sub != 1)) && R < 8) f *= 1.4;
    return (double)z.M * inst(i).cost * f;
}

// Cost of one row (ps) on instance i by whole rows: 1.12 of the column cost,
// more where every row's band product serves few residues (8 x 16, power:
// 1.74 ps per point at R = 32, 1.84 at 16, 1.88 at 8, 2.06 at 4, 2.57 at 2)
// and where rows start off a sector, the more the fewer the slots of the last
// pass (1.93, 2.07, 2.21, 2.57, 3.36); 1.2 of that with two output arrays.
double whole_cost(int i, const ZoomShape &z) {
    const int R = z.M / inst(i).Q, J = z.M / inst(i).LAST;
    double f = 1.12 + 1.0 / R;
    if (z.n_out % 8 != 0 || z.n_out == 0) f += 0.08 + 6.0 / J;
    if (z.sub != 1) f *= 1.4;
    else if (z.both) f *= 1.2;
    return (double)z.M * inst(i).cost * f;
}

// Cost of one row (ps) with first radix i and remaining length j of
// zoom_wide.cuh, as above: 2500 launches of 40 ... 120 Mi points at 39 lengths
// within 7% rms for one output array, 10% for two.  The first kernel's stores are
// runs of R = M / Q points: 1.8 ps per point at R >= 16, 2.3 at 8, 3.1 at 4, 5.6
// at 2, 10.4 at 1 (QA = 16), where the whole-row kernels are the better ones.
double wide_cost(int i, int j, const ZoomShape &z) {
    const WideInst &w = wide_rest(j);
    const int Rp = z.M / (w.QB * w.QC), QA = wide_radix(i), R = Rp / QA;
    const bool eighth = Rp % 8 == 0 && z.n_out % 8 == 0, quarter = Rp % 4 == 0 && z.n_out % 4 == 0;
    double f = z.both ? (eighth ? 1.15 : quarter ? 1.25 : 1.15 + 0.6 * z.kept()) : eighth ? 0.95 : 1.0;
    if (z.sub != 1) f = 1.6;
    const double pad = (double)((Rp + w.P - 1) / w.P * w.P) / Rp;
    const double first = (QA <= 8 ? 1.4 : 1.4 + 0.025 * (QA - 8) + (QA > 16 ? 0.02 * (QA - 16) : 0.0)) +
                         0.58 * std::min(QA, 16) * std::pow((double)R, -1.15);
    const double rest = 1.95 + 0.0007 * (w.QB * w.QC) + ((w.QB % 5 == 0 || w.QB % 7 == 0 || w.QB % 3 == 0) ? 0.15 : 0.0) +
                  ((w.QC % 5 == 0 || w.QC % 7 == 0 || w.QC % 3 == 0) ? 0.15 : 0.0)  + (w.P < 16 ? 0.1 : 0.0);
    // and the wait of the second kernel for the first, shared by about ten scales
    return (double)z.M * (first + rest * f * pad) + 4e5 / z.channels;
}

constexpr int kWideCode = 1 << 20;  // candidate codes of zoom_select: + 1024 i + j

}  // namespace

int zoom_class_L(const ZoomClass &c, int M) {
    if (c.wide >= 0) return M / (wide_rest(c.inst).QB * wide_rest(c.inst).QC);
    return M / inst(c.inst).Q * inst(c.inst).QA;
}

void zoom_select(const ZoomShape &z, int S, const int *band, std::vector<ZoomClass> *classes,
                 std::vector<int4> *list, std::vector<int> *rest) {
    classes->clear();
    list->clear();
    rest->clear();
    // candidates: 2 i by columns, 2 i + 1 by whole rows, kWideCode + ... in two
    // kernels, kRest the whole-row FFT kernels; each with its cost of a row and
    // the widest band it takes wherever that starts
    constexpr int kRest = -1;
    struct Cand {
        int code;
        double cost;
        int cap;
    };
    std::vector<Cand> all{{kRest, z.rest_cost, 1 << 30}};
    for (int i = 0; i < kZoomInstances; ++i) {
        if (z.M % inst(i).Q != 0) continue;
        const int R = z.M / inst(i).Q, cap = inst(i).Q - (inst(i).NB - 1);  // the window starts at a multiple of NB
        // few residues leave a row's band product little use and its stores short
        if (!z.rows_only && (R >= 4 || inst(i).P <= 4) && smem_of(i, rows_met(inst(i).P, R)) <= kMaxSmem)
            all.push_back({2 * i, column_cost(i, z), cap});
        if (!z.phase && row_fits(i, z.M, R))
            all.push_back({2 * i + 1, whole_cost(i, z), cap});
    }
    if (z.wide)
        for (int j = 0; j < kWideRest; ++j) {
            const int Qp = wide_rest(j).QB * wide_rest(j).QC;
            if (z.M % Qp != 0) continue;
            for (int i = 0; i < kWideFirst; ++i)
                if ((z.M / Qp) % wide_radix(i) == 0 && z.M / Qp / wide_radix(i) <= kWideThreads)
                    all.push_back({kWideCode + 1024 * i + j, wide_cost(i, j, z), wide_radix(i) * Qp});
        }
    std::stable_sort(all.begin(), all.end(), [](const Cand &a, const Cand &b) { return a.cost < b.cost; });
    std::vector<Cand> open;  // those wider than every cheaper one, cheapest first
    for (const Cand &c : all)
        if (open.empty() || c.cap > open.back().cap) open.push_back(c);
    // every scale on its cheapest transform, then classes dissolved into the
    // remaining ones while the launches they save (3 us, 10 for two kernels) outweigh the dearer
    // transforms of their scales, at a nominal number of channels
    auto assign = [&](const std::vector<Cand> &o, std::vector<int> *to) -> double {
        double total = 0;
        std::vector<char> used(o.size(), 0);
        for (int s = 0; s < S; ++s) {
            size_t k = 0;
            while (k < o.size() && o[k].cap < band[2 * s + 1]) ++k;
            if (k == o.size()) return 1e300;
            total += z.channels * o[k].cost;
            used[k] = 1;
            if (to) (*to)[(size_t)s] = o[k].code;
        }
        for (size_t k = 0; k < o.size(); ++k)
            if (used[k]) total += o[k].code >= kWideCode ? 10e6 : 3e6;  // two kernels, the second after the first
        return total;
    };
    std::vector<int> to((size_t)S, kRest);
    double total = assign(open, &to);
    {
        std::vector<Cand> u;
        for (const Cand &c : open)
            if (std::find(to.begin(), to.end(), c.code) != to.end()) u.push_back(c);
        open = u;
    }
    while (open.size() > 1) {
        double best = total;
        size_t drop = open.size();
        for (size_t k = 0; k < open.size(); ++k) {
            std::vector<Cand> o = open;
            o.erase(o.begin() + (long)k);
            const double t = assign(o, nullptr);
            if (t < best) best = t, drop = k;
        }
        if (drop == open.size()) break;
        open.erase(open.begin() + (long)drop);
        total = assign(open, &to);
    }
    // rows compiled for the plan: scales whose class is dearer join them, if that
    // outweighs a launch of theirs alone
    if (z.compiled_cost > 0) {
        const bool rows = std::find(to.begin(), to.end(), kRest) != to.end();
        double gain = rows ? 3e6 : 0.0;
        std::vector<int> moved = to;
        for (const Cand &c : open)
            for (int s = 0; s < S; ++s)
                if (to[(size_t)s] == c.code && c.code != kRest && c.cost > z.compiled_cost) {
                    gain += z.channels * (c.cost - z.compiled_cost);
                    moved[(size_t)s] = kRest;
                }
        if (gain > 3e6) to = moved;
    }
    for (const Cand &cand : open) {
        const int k = cand.code;
        if (k == kRest) continue;
        const bool wide = k >= kWideCode;
        const int i = wide ? k & 1023 : k >> 1, first = (int)list->size(), nb = wide ? 1 : inst(i).NB;
        for (int s = 0; s < S; ++s)
            if (to[(size_t)s] == k)
                list->push_back(make_int4(s, band[2 * s], band[2 * s + 1], band[2 * s] / nb * nb));
        if ((int)list->size() > first)
            classes->push_back({i, first, (int)list->size() - first, !wide && (k & 1) != 0,
                                wide ? (k - kWideCode) >> 10 : -1});
    }
    for (int s = 0; s < S; ++s)
        if (to[(size_t)s] == kRest) rest->push_back(s);
    // wide classes, then the largest first: the last launch's tail is short
    std::stable_sort(classes->begin(), classes->end(), [](const ZoomClass &a, const ZoomClass &b) {
        return (a.wide >= 0) != (b.wide >= 0) ? a.wide >= 0 : a.ns > b.ns;
    });
}

cudaError_t zoom_launch(const ZoomClass &c, ZoomArgs a, long long chans, const float2 *twl, const int4 *d_list,
                        cudaStream_t st) {
    const ZoomInst &t = inst(c.inst);
    const int R = a.M / t.Q;
    const long long rows = chans * c.ns;
    a.R = R;
    a.L = R * t.QA;
    a.twl = twl;
    a.list = d_list + c.first;
    a.ns = c.ns;
    a.magM = zoom_magic((unsigned)a.M);
    a.magSub = zoom_magic((unsigned)a.sub);
    a.magL = zoom_magic((unsigned)a.L);
    a.magR = zoom_magic((unsigned)R);
    a.magNs = zoom_magic((unsigned)c.ns);
    // A column group that meets several rows forms their band products one after the
    // other, a load latency each, which a launch too small to fill the GPU does not
    // hide: such launches run by whole rows, the same arithmetic on the same tables
    // (16 x 32, 88 rows of 4096 points 6.4 us by columns, 3.9 by rows; 352 rows 9.0
    // and 6.3; 32 columns that meet two rows: 5.4 and 5.7 at 312).
    const int met = rows_met(t.P, R);
    const bool small = (double)rows * a.M <= (t.P <= 16 && met == 2 ? 1.5e6 : 5e5) && met >= (t.P >= 32 ? 3 : 2);
    const bool by_rows = c.rows || (small && !a.oph && row_fits(c.inst, a.M, R));
    // the kernels count rows, and columns those of all rows, in 31 bits
    if ((by_rows ? rows : rows * R) >= 2147483647ll) return cudaErrorInvalidValue;
    const int mode = by_rows ? 2 : a.oph || a.sub != 1 ? 1 : 0;
    cudaError_t e = ensure_zoom_smem(c.inst, mode);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3((unsigned)t.T);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (by_rows) {
        a.nr = rows_per_cta(c.inst, a.M, R, rows);
        a.nrows = (int)rows;
        a.ps = position_stride(c.inst, a.nr, R);
        a.rs = row_stride(c.inst, a.nr, R);
        const int J = a.M / t.LAST;  // last-pass slots of a row, and 7 for the shift
        a.js = !a.epochs && a.n_out % 8 == 0 ? J : (J + 14) & ~7;
        a.magC = zoom_magic((unsigned)(a.nr * R));
        a.magJs = zoom_magic((unsigned)a.js);
        a.magL2 = zoom_magic((unsigned)a.L);
        cfg.gridDim = dim3((unsigned)((rows + a.nr - 1) / a.nr));
        cfg.dynamicSmemBytes = (size_t)row_smem_of(c.inst, a.nr, a.rs, R);
    } else {
        a.cols = (unsigned)(rows * R);
        a.rows = rows_met(t.P, R);
        cfg.gridDim = dim3((a.cols + (unsigned)t.P - 1) / (unsigned)t.P);
        cfg.dynamicSmemBytes = (size_t)smem_of(c.inst, a.rows);
    }
    void *params[] = {&a};
    return cudaLaunchKernelExC(&cfg, kernel_of(c.inst, mode), params);
}

cudaError_t wide_launch(const ZoomClass &c, const ZoomArgs &args, long long chans, const float2 *twl,
                        const int4 *d_list, float2 *Z, int z_rows, int *turn, cudaStream_t st) {
    const WideInst &t = wide_rest(c.inst);
    const int QA = wide_radix(c.wide);
    WideArgs w;
    w.z = args;
    ZoomArgs &a = w.z;
    const long long rows = chans * c.ns;
    w.Qp = t.QB * t.QC;
    a.L = a.M / w.Qp;
    a.R = a.L / QA;
    a.twl = twl;
    a.list = d_list + c.first;
    a.ns = c.ns;
    a.magM = zoom_magic((unsigned)a.M);
    a.magSub = zoom_magic((unsigned)a.sub);
    a.magL = zoom_magic((unsigned)a.L);
    a.magR = zoom_magic((unsigned)a.R);
    a.magNs = zoom_magic((unsigned)c.ns);
    const int mode = a.oph || a.sub != 1 ? 1 : 0;
    cudaError_t e = ensure_wide_smem(c.inst, mode);
    if (e != cudaSuccess) return e;
    // positions per CTA of the first kernel: about 512 butterflies
    const int et = QA <= 16 ? QA + 1 : 2 * QA;  // its table's rows
    const int bb = std::max(4, std::min({w.Qp, 512 / a.R, (48 * 1024 / 8 - et * a.R) / QA}));
    const int smem1 = (QA * bb + et * a.R) * (int)sizeof(float2);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    for (long long r0 = 0; r0 < rows && e == cudaSuccess; r0 += z_rows) {
        w.row0 = (int)r0;
        w.Z = Z + (size_t)(*turn & 1) * (size_t)z_rows * (size_t)a.M;
        ++*turn;
        w.nrows = (int)std::min<long long>(z_rows, rows - r0);
        void *params[] = {&w};
        w.bb = bb;
        w.groups = (w.Qp + bb - 1) / bb;
        w.magG = zoom_magic((unsigned)w.groups);
        cfg.gridDim = dim3((unsigned)(w.nrows * w.groups));
        cfg.blockDim = dim3(kWideThreads);
        cfg.dynamicSmemBytes = (size_t)smem1;
        e = cudaLaunchKernelExC(&cfg, wide_first_entry(c.wide), params);
        if (e != cudaSuccess) return e;
        w.groups = (a.L + t.P - 1) / t.P;
        w.magG = zoom_magic((unsigned)w.groups);
        cfg.gridDim = dim3((unsigned)(w.nrows * w.groups));
        cfg.blockDim = dim3((unsigned)t.T);
        cfg.dynamicSmemBytes = (size_t)t.smem;
        e = cudaLaunchKernelExC(&cfg, wide_kernel_of(c.inst, mode), params);
        a.after = 1;
    }
    return e;
}

namespace {

// Half the workspace of zoom_wide.cuh: enough that more gains nothing (32 x 122880
// x 128 power: 1.80 ms with 28 MB, 1.69 with 40, then 1.61 ... 1.67 up to 400).
constexpr size_t kWideBytes = (size_t)56 << 20;

// Cost of one row (ps) on the whole-row kernels, for the bands that are left to
// them: wide ones, whose first pass is dense (medians of power alone and of
// complex and power, 40 Mi points; a narrow band takes 0.75 ... 0.9 of it); or on
// kernels compiled at the plan's creation, for lengths without compiled-in ones.
double row_cost(const cwt_plan_s *p, bool both, bool compiled) {
    if (p->precision != CWT_PREC_FP32)  // tensor-core stages: power of 1024 x 32768 340 us; two arrays at 131072
        return (double)p->N * (both ? 13.5 : 10.0);
    if (!p->mr) {
        const int L = p->M <= kMaxFft ? p->M : p->N;  // clusters transform all N points
        const double ps = L <= 256 ? 2.7 : L <= 4096 ? 3.1 : L <= 8192 ? 4.0 : L <= kMaxFft ? 5.0
                          : L <= 32768 ? 6.0 : L <= 65536 ? 7.1 : 9.5;
        // a folded row's first pass sums fold bins per point: 4096 / 4 3.4 ... 6.5, 16384 / 4 3.9 ... 6.5
        return (double)L * ((both ? 1.15 : 1.0) * ps + (L < p->N ? 1.5 : 0.0));
    }
    double ps;
    if (p->cl > 1)  // one kernel for two local rows per SM: 20000 5.7, 60000 8.4; 16464 12.7, 6.3 compiled for it
        ps = p->sch.fixed_cl >= 0 ? 6.2 : compiled ? 7.0 : 12.5;
    else  // 3000 4.3, 10000 4.0; 6400 5.2, 3200 6.3; 2304 8.1, 6300 9.4; compiled for the plan 2.9 ... 6.2
        ps = p->sch.fixed >= 0 ? 4.1 : compiled ? 4.7 : p->sch.fast >= 0 ? 5.7 : 8.6;
    return (double)p->N * (both ? 1.1 : 1.0) * ps;
}

}  // namespace

struct ZoomPlan {
    std::vector<ZoomClass> classes;
    std::vector<const float2 *> twl;  // per class: w_L^i, L = QA R
    int4 *d_list = nullptr;
    float2 *d_twl = nullptr;  // smooth lengths: those tables
    float2 *d_wide = nullptr;  // the wide classes' workspace, twice wide_rows rows of M points
    int wide_rows = 0;
    int M = 0, sub = 1, tws = 1;
    const float2 *tw = nullptr;
};

void free_zoom_plan(ZoomPlan *z) {
    if (!z) return;
    cudaFree(z->d_list);
    cudaFree(z->d_twl);
    cudaFree(z->d_wide);
    delete z;
}

void zoom_routes(const ZoomPlan *z, int *classes, int *two_kernels) {
    *classes = *two_kernels = 0;
    if (z)
        for (const ZoomClass &c : z->classes) (c.wide >= 0 ? *two_kernels : *classes) += c.ns;
}

static cudaError_t zoom_plan_build(cwt_plan_s *p, cudaStream_t st) {
    const int S = p->S;
    const int f = std::gcd(p->N, p->d), M = p->N / f;
    std::vector<int> band(2 * (size_t)S);
    cudaError_t e = cudaMemcpyAsync(band.data(), p->band, sizeof(int) * band.size(), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    std::vector<ZoomClass> classes;
    std::vector<int4> list;
    std::vector<int> rest;
    ZoomShape sh;
    sh.M = M;
    sh.sub = p->d / f;
    sh.n_out = p->n_out;
    sh.both = (p->outputs & (p->outputs - 1)) != 0;
    // a compiled plan starts from the split of one that is not, so that its results
    // are the same bits as far as the same scales stay on classes
    sh.rest_cost = row_cost(p, sh.both, false);
    sh.compiled_cost = p->compiled ? row_cost(p, sh.both, true) : 0.0;
    sh.phase = (p->outputs & CWT_OUT_PHASE) != 0;
    sh.rows_only = false;
    sh.wide = true;
    // between plans of a few channels, which would take launches that pay only
    // beyond them, and large ones, which want each scale on its cheapest form
    // (16384 x 100 at 64 channels: 272 us decided at 64, 258 at 32, 264 at 8; 2500 x
    // 100: 64, 64, 72; 2 x 30000: 48, 48, 37)
    sh.channels = 40;
    zoom_select(sh, S, band.data(), &classes, &list, &rest);
    // columns and grids stay within 31 bits
    for (const ZoomClass &c : classes)
        if ((double)p->C * c.ns * (c.wide >= 0 ? 1 : M / inst(c.inst).Q) >= 2147483647.0) list.clear();
    if (list.empty()) return cudaSuccess;
    ZoomPlan *z = new ZoomPlan;
    p->zoom = z;  // freed with the plan, also on failure
    z->classes = classes;
    z->M = M;
    z->sub = sh.sub;
    z->tw = p->mr ? p->twN : twiddles_pow2(p->tw, M);
    z->tws = p->mr ? p->N / M : 1;
    e = dmalloc(&z->d_list, sizeof(int4) * list.size());
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(z->d_list, list.data(), sizeof(int4) * list.size(), cudaMemcpyHostToDevice, st);
    // the first pass's tables w_L: powers of two from the device's, others here
    size_t total_l = 0, at = 0;
    for (const ZoomClass &c : classes) total_l += (size_t)zoom_class_L(c, M);
    if (e == cudaSuccess && p->mr) e = dmalloc(&z->d_twl, sizeof(float2) * total_l);
    for (const ZoomClass &c : classes) {
        const int L = zoom_class_L(c, M);
        if (e == cudaSuccess && p->mr) e = make_twiddles_n(L, z->d_twl + at, st);
        z->twl.push_back(p->mr ? z->d_twl + at : twiddles_pow2(p->tw, L));
        at += (size_t)L;
    }
    long long wide_rows = 0;
    for (const ZoomClass &c : classes)
        if (c.wide >= 0) wide_rows = std::max(wide_rows, (long long)p->C * c.ns);
    wide_rows = std::min(wide_rows, (long long)std::max<size_t>(1, kWideBytes / (sizeof(float2) * (size_t)M)));
    if (e == cudaSuccess && !rest.empty()) {
        e = dmalloc(&p->rest_list, sizeof(int) * rest.size());
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(p->rest_list, rest.data(), sizeof(int) * rest.size(), cudaMemcpyHostToDevice, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    // fewer rows at a time where memory is short: slower, the same values
    while (e == cudaSuccess && wide_rows) {
        e = dmalloc(&z->d_wide, 2 * sizeof(float2) * (size_t)M * (size_t)wide_rows);
        if (e != cudaErrorMemoryAllocation || wide_rows == 1) break;
        cudaGetLastError();  // clear the non-sticky error
        e = cudaSuccess;
        wide_rows = std::max(1ll, wide_rows / 4);
    }
    z->wide_rows = (int)wide_rows;
    p->rest_scales = (int)rest.size();
    p->bytes += sizeof(int4) * list.size() + sizeof(int) * rest.size() + (p->mr ? sizeof(float2) * total_l : 0) +
                2 * sizeof(float2) * (size_t)M * (size_t)wide_rows;
    return e;
}

cudaError_t zoom_plan_create(cwt_plan_s *p, cudaStream_t st) {
    p->rest_scales = p->S;
    // double outputs keep the whole-row kernels' bits
    if (p->io != CWT_DTYPE_F32 || p->whole_rows) return cudaSuccess;
    try {
        return zoom_plan_build(p, st);
    } catch (const std::bad_alloc &) {
        return cudaErrorMemoryAllocation;
    }
}

cudaError_t launch_scale_block_zoom(const cwt_plan_s *p, float2 *out_c, float *out_p, float *out_ph,
                                    cudaStream_t st) {
    const ZoomPlan *z = p->zoom;
    ZoomArgs a = {};
    a.spec = p->spec;
    a.bank = p->bank;
    a.tw = z->tw;
    a.oc = out_c;
    a.op = out_p;
    a.oph = out_ph;
    a.N = a.wn = p->N;
    a.M = z->M;
    a.tws = z->tws;
    a.S = p->S;
    a.n_out = p->n_out;
    a.sub = z->sub;
    a.n_keep = z->sub * (p->n_out - 1) + 1;
    // Launches overlap (programmatic dependent launch): the first after the
    // forward FFTs waits for them before it reads a spectrum; a later one may
    // start when every CTA of the one before has passed that point, reads the
    // spectra at once and waits at its end, so that the stream's order holds.
    int turn = 0;  // the workspace's halves
    bool after = p->rest_scales > 0;  // the whole-row kernel before saw the forward FFTs complete
    for (size_t k = 0; k < z->classes.size(); ++k) {
        a.after = after;
        after = true;
        const ZoomClass &c = z->classes[k];
        const cudaError_t e = c.wide >= 0 ? wide_launch(c, a, p->C, z->twl[k], z->d_list, z->d_wide, z->wide_rows,
                                                        &turn, st)
                                          : zoom_launch(c, a, p->C, z->twl[k], z->d_list, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace cwtk
