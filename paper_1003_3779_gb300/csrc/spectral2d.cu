// spectral2d.cu -- tables and launchers of the momentum-space torus kernels
// (k_spectral2d.cuh), FP32.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "qw_handle.h"
#include "k_spectral2d.cuh"

namespace qw {

// twiddles of every stage length, and the axis tables of both lengths.  The longer
// stages' twiddles also undo the norm lost by the 16-point transforms (DftGain):
// their own, and those of the stage of at most 128 (or, after 256, 16) points that
// follows, whose few twiddles round too alike (half of those of length 32 are 1).
// Rounded from many values, they do so on average to well below a rounding, which
// one float factor at the end could not.
__global__ void k_spec2_twiddles(S2 *tw) {
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id < 32 || id >= SPEC2_TW) return;
    const int n = 1 << (31 - __clz(id)), i = id - n, k = i / (n / 16), b = i % (n / 16);
    using Gain = DftGain<float>;
    double lost = 1.0;
    if (n >= 256) lost = Gain::of16 * (n <= 2048 ? Gain::of16 : 1.0) * (n == 2048 ? Gain::of8 : 1.0);
    // (the points with k = 0 are not multiplied, those with b = 0 by 1)
    const double up = 1.0 + (1.0 / lost - 1.0) / (15.0 / 16 * (1 - 16.0 / n));
    double s, c;
    sincospi(-2.0 * k * b / n, &s, &c);
    tw[id] = {(float)(c * up), (float)(s * up)};
}
// momentum / (2 pi) at place p; split: places of the even momenta of a cycle of
// 2^(L+1), then of the odd ones
__device__ __forceinline__ double spec2_momentum(int L, int p, int split) {
    const int n = 1 << L;
    return split ? (2.0 * spec2_freq(L, p % n) + p / n) / (2 * n) : (double)spec2_freq(L, p) / n;
}
__global__ void k_spec2_axis(Spec2Axis *ax, int L, int split) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= 1 << (L + split)) return;
    const double k = spec2_momentum(L, p, split);
    double s, c, h, g;
    sincospi(2.0 * k, &s, &c);
    sincospi(k, &h, &g);
    h *= h;
    g *= g;
    Spec2Axis a;
    a.s = (float)s;
    a.sh = (float)h; a.sl = (float)(h - a.sh);
    a.ch = (float)g; a.cl = (float)(g - a.ch);
    a.pad = 0.f;
    ax[p] = a;
}
// rows of (diag(e^{-ik}, e^{ik}) H)^K, or of its adjoint, by place
__global__ void k_spec2_tensor(SpecPair<float> *t, int L, int split, int K, int adj) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= 1 << (L + split)) return;
    using Z = Cx<double>;
    double s, c;
    sincospi(2.0 * spec2_momentum(L, p, split), &s, &c);
    const double r = 0.70710678118654752440;
    const Z u[4] = {{c * r, -s * r}, {c * r, -s * r}, {c * r, s * r}, {-c * r, -s * r}};
    Z m[4] = {u[0], u[1], u[2], u[3]};
    auto mul = [](const Z (&a)[4], const Z (&b)[4], Z (&o)[4]) {
        for (int i = 0; i < 2; ++i)
            for (int j = 0; j < 2; ++j) o[2 * i + j] = cfma(a[2 * i + 1], b[2 + j], cmul(a[2 * i], b[j]));
    };
    for (int bit = 30 - __clz(K); bit >= 0; --bit) {
        Z q[4];
        mul(m, m, q);
        if (K >> bit & 1) mul(q, u, m);
        else for (int i = 0; i < 4; ++i) m[i] = q[i];
    }
    if (adj) {
        const Z b = m[1];
        m[1] = {m[2].re, -m[2].im};
        m[2] = {b.re, -b.im};
        m[0].im = -m[0].im;
        m[3].im = -m[3].im;
    }
    for (int i = 0; i < 2; ++i)
        t[2 * p + i] = {{(float)m[2 * i].re, (float)m[2 * i].im}, {(float)m[2 * i + 1].re, (float)m[2 * i + 1].im}};
}

// tables: twiddles, the axes (places of 2^LX, then 2^LY), their 2 x 2 matrices
struct Spec2Tables {
    S2 *tw;
    Spec2Axis *ax, *ay;
    SpecPair<float> *tx, *ty;
};
static Spec2Tables tables(void *base) {
    Spec2Tables t;
    char *p = static_cast<char *>(base);
    t.tw = reinterpret_cast<S2 *>(p); p += sizeof(S2) * SPEC2_TW;
    t.tx = reinterpret_cast<SpecPair<float> *>(p); p += sizeof(SpecPair<float>) * 2 << SPEC2_MAX_LX;
    t.ty = reinterpret_cast<SpecPair<float> *>(p); p += sizeof(SpecPair<float>) * 2 << SPEC2_MAX_LX;
    t.ax = reinterpret_cast<Spec2Axis *>(p); p += sizeof(Spec2Axis) << SPEC2_MAX_LX;
    t.ay = reinterpret_cast<Spec2Axis *>(p);
    return t;
}
static constexpr size_t TABLE_BYTES = sizeof(S2) * SPEC2_TW + ((2 * sizeof(SpecPair<float>) * 2) << SPEC2_MAX_LX) +
                                      ((2 * sizeof(Spec2Axis)) << SPEC2_MAX_LX);

bool spectral2d_ok(int prec, int kind, int shift) {
    return prec == QW_F32 && (kind == CK_GROVER || (kind == CK_HH && shift == QW_SHIFT_DIAGONAL));
}

// How an axis of n sites is cut for K steps: the transform length, halo, outputs
// per block and blocks.
struct AxisCut {
    int L = 0, h = 0, split = 0;
    int64_t w = 0, blocks = 0;
    double points() const { return (double)blocks * (1 << L) * (L + 4); }   // (work: points times stages)
};
static AxisCut cut_axis(int64_t n, int K, int maxL, bool may_split = false) {
    for (int L = SPEC2_MIN_L; L <= maxL; ++L)
        if (n == (int64_t)1 << L) return {L, 0, 0, n, 1};   // a cycle of its own
    if (may_split && n == (int64_t)2 << maxL) return {maxL, 0, 1, n / 2, 2};   // ... in two halves
    AxisCut best;
    for (int L = SPEC2_MIN_L; L <= maxL; ++L) {
        const int64_t w = ((int64_t)1 << L) - 2 * K;
        if (w < 1) continue;
        AxisCut c{L, K, 0, std::min(w, n), (n + w - 1) / w};
        if (!best.L || c.points() < best.points()) best = c;
    }
    return best;
}

// both axes, and whether a batch of them fits the workspace (the halves of a split
// column are combined on the way back, so they are one batch: one block of rows)
static bool cut_axes(int64_t nx, int64_t ny, int K, size_t room, AxisCut &x, AxisCut &y) {
    x = cut_axis(nx, K, SPEC2_MAX_LX);
    y = cut_axis(ny, K, SPEC2_MAX_LY, x.blocks == 1);
    return x.L && y.L && ((size_t)32 << (x.L + y.L + y.split)) <= room;
}

// Workspace: the blocks of one batch, at least one of the largest that is planned.
size_t spectral2d_workspace(int64_t nx, int64_t ny) {
    const size_t want = (size_t)nx * ny * 32 * 4;
    return TABLE_BYTES + std::min<size_t>(size_t(1) << 31, std::max<size_t>(size_t(1) << 26, want));
}

// Steps per launch; fewer are only taken by a call of fewer (below, m launches
// would round more than stepping).
constexpr int SPEC2_LEAST_STEPS = 64, SPEC2_MOST_STEPS = 4000;
Spec2Plan spectral2d_plan(int64_t nx, int64_t ny, int64_t T, bool even) {
    // m launches of about T / m steps; a launch costs its points (about 7e8 point
    // stages per millisecond) and 20 us for its kernels.  Every m up to 100, then by
    // 2 %: with m <= 64 calls of more than 256000 steps were stepped, and shorter ones
    // off powers of two had only launches of deep halos (300 x 200, T = 100000:
    // 124 -> 27 ms).
    Spec2Plan best;
    const size_t room = spectral2d_workspace(nx, ny) - TABLE_BYTES;
    for (int64_t m = (T + SPEC2_MOST_STEPS - 1) / SPEC2_MOST_STEPS; m >= 1 && m <= T; m = std::max(m + 1, m * 102 / 100)) {
        int64_t K = (T + m - 1) / m;
        if (m > 1 && K < SPEC2_LEAST_STEPS) break;
        if (even) K += K & 1;
        if (K > SPEC2_MOST_STEPS) continue;
        AxisCut x, y;
        if (!cut_axes(nx, ny, (int)K, room, x, y)) continue;
        const double pts = (double)x.blocks * y.blocks * std::ldexp(1.0, x.L + y.L) * (x.L + y.L + 8);
        const double cost = (double)m * (pts / 7e8 + 0.02);
        if (best.K == 0 || cost < best.ms) { best.K = (int)K; best.ms = cost; }
    }
    return best;
}

cudaError_t launch_spectral2d_tables(void *work, cudaStream_t s) {
    k_spec2_twiddles<<<SPEC2_TW / 256, 256, 0, s>>>(tables(work).tw);
    return cudaGetLastError();
}

template <int L> static cudaError_t rows(const Spec2Args &a, bool inverse, cudaStream_t s) {
    constexpr int R = spec2_rows<L>(), TH = (1 << L) / 16 * R;
    constexpr size_t smem = spec2_row_smem<L>();
    auto kern = inverse ? k_spec2_rows_inverse<L> : k_spec2_rows_forward<L>;
    cudaError_t e = smem > 48 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) : cudaSuccess;
    if (e != cudaSuccess) return e;
    const int64_t n = (int64_t)a.nb * 4 * (inverse ? a.wy : (int64_t)1 << a.LY);
    kern<<<(unsigned)((n + R - 1) / R), TH, smem, s>>>(a);
    return cudaGetLastError();
}
static cudaError_t rows_any(const Spec2Args &a, bool inverse, cudaStream_t s) {
    switch (a.LX) {
        case 8: return rows<8>(a, inverse, s);
        case 9: return rows<9>(a, inverse, s);
        case 10: return rows<10>(a, inverse, s);
        case 11: return rows<11>(a, inverse, s);
        case 12: return rows<12>(a, inverse, s);
        case 13: return rows<13>(a, inverse, s);
    }
    return cudaErrorInvalidValue;
}
template <int L, int MODE> static cudaError_t columns(const Spec2Args &a, const Spec2Coin &c, cudaStream_t s) {
    constexpr size_t smem = spec2_col_smem<L>();
    auto kern = k_spec2_columns<L, MODE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((int64_t)a.nb * (1 << a.LX) / spec2_cols<L>()), spec2_cols<L>() * 4 * (1 << L) / 16, smem, s>>>(a, c);
    return cudaGetLastError();
}
template <int L> static cudaError_t columns_mode(int mode, const Spec2Args &a, const Spec2Coin &c, cudaStream_t s) {
    switch (mode) {
        case QW_SHIFT_MOVING: return columns<L, QW_SHIFT_MOVING>(a, c, s);
        case QW_SHIFT_FLIPFLOP: return columns<L, QW_SHIFT_FLIPFLOP>(a, c, s);
        case QW_SHIFT_DIAGONAL: return columns<L, QW_SHIFT_DIAGONAL>(a, c, s);
        case SPEC2_TENSOR: return columns<L, SPEC2_TENSOR>(a, c, s);
    }
    return cudaErrorInvalidValue;
}

// a.K steps (even for the Grover coin) from a.in to a.out, on the blocks of a
// launch of cut_K >= a.K; work: the workspace, with the twiddles in place.
cudaError_t launch_spectral2d(const Step2DArgs &a, int cut_K, int adjoint, void *work, cudaStream_t s) {
    const bool tensor = a.kind == CK_HH;
    const size_t room = spectral2d_workspace(a.nx, a.ny) - TABLE_BYTES;
    AxisCut x, y;
    if (a.K < 2 || a.K > cut_K || (!tensor && (a.K & 1)) || !cut_axes(a.nx, a.ny, cut_K, room, x, y)) return cudaErrorInvalidValue;
    const Spec2Tables t = tables(work);
    Spec2Args g{};
    g.in = a.in; g.out = a.out; g.nx = a.nx; g.ny = a.ny;
    g.wx = x.w; g.wy = y.w; g.hx = x.h; g.hy = y.h; g.nbx = (int)x.blocks; g.LX = x.L; g.LY = y.L; g.split = y.split;
    g.z = reinterpret_cast<S2 *>(static_cast<char *>(work) + TABLE_BYTES);
    g.tw = t.tw;
    g.scale = (float)(a.gain * std::ldexp(1.0, -(x.L + y.L + y.split)));
    Spec2Coin c{t.ax, t.ay, t.tx, t.ty, a.K, adjoint ? -1.f : 1.f};
    if (tensor) {
        k_spec2_tensor<<<(1 << x.L) / 32, 32, 0, s>>>(t.tx, x.L, 0, a.K, adjoint);
        k_spec2_tensor<<<(1 << (y.L + y.split)) / 32, 32, 0, s>>>(t.ty, y.L, y.split, a.K, adjoint);
    } else {
        k_spec2_axis<<<(1 << x.L) / 32, 32, 0, s>>>(t.ax, x.L, 0);
        k_spec2_axis<<<(1 << (y.L + y.split)) / 32, 32, 0, s>>>(t.ay, y.L, y.split);
    }
    cudaError_t e = cudaGetLastError();
    const int64_t blocks = x.blocks * y.blocks;
    const int64_t batch = std::min<int64_t>(blocks, (int64_t)(room / ((size_t)32 << (x.L + y.L))));
    for (int64_t b = 0; b < blocks && e == cudaSuccess; b += batch) {
        g.b0 = (int)b;
        g.nb = (int)std::min(batch, blocks - b);
        e = rows_any(g, false, s);
        const int mode = tensor ? SPEC2_TENSOR : a.shift;
        if (e == cudaSuccess) switch (y.L) {
            case 8: e = columns_mode<8>(mode, g, c, s); break;
            case 9: e = columns_mode<9>(mode, g, c, s); break;
            case 10: e = columns_mode<10>(mode, g, c, s); break;
            case 11: e = columns_mode<11>(mode, g, c, s); break;
            case 12: e = columns_mode<12>(mode, g, c, s); break;
            default: e = cudaErrorInvalidValue;
        }
        if (e == cudaSuccess) e = rows_any(g, true, s);
    }
    return e;
}

}  // namespace qw
