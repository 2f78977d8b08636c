// spectral1d.cu -- tables and launchers of the momentum-space kernel of the
// cycle walk (k_spectral1d.cuh).
#include <algorithm>
#include <cmath>

#include "qw_handle.h"
#include "k_spectral1d.cuh"

namespace qw {

// ------------------------------------------------------------------ double-double
// Unevaluated sums of two doubles (about 106 bits), for the matrices U^K of the
// double walks: repeated squaring doubles the relative error at each level, so
// in plain double U^1024 would be 1e-13 off, where stepping is 1e-14 off.
// TwoSum (Knuth), TwoProduct by FMA, sums and products as in Joldes, Muller &
// Popescu, ACM TOMS 44(2), 2017.
struct dd {
    double hi, lo;
};
__device__ __forceinline__ dd dd_fast(double a, double b) {
    const double s = __dadd_rn(a, b);
    return {s, __dsub_rn(b, __dsub_rn(s, a))};
}
__device__ __forceinline__ dd dd_sum(double a, double b) {
    const double s = __dadd_rn(a, b), t = __dsub_rn(s, a);
    return {s, __dadd_rn(__dsub_rn(a, __dsub_rn(s, t)), __dsub_rn(b, t))};
}
__device__ __forceinline__ dd operator+(dd x, dd y) {
    const dd s = dd_sum(x.hi, y.hi), t = dd_sum(x.lo, y.lo);
    const dd v = dd_fast(s.hi, __dadd_rn(s.lo, t.hi));
    return dd_fast(v.hi, __dadd_rn(t.lo, v.lo));
}
__device__ __forceinline__ dd operator-(dd x) { return {-x.hi, -x.lo}; }
__device__ __forceinline__ dd operator-(dd x, dd y) { return x + (-y); }
__device__ __forceinline__ dd operator*(dd x, dd y) {
    const double h = __dmul_rn(x.hi, y.hi), l = __fma_rn(x.hi, y.hi, -h);
    const double m = __fma_rn(x.lo, y.hi, __fma_rn(x.hi, y.lo, __dmul_rn(x.lo, y.lo)));
    return dd_fast(h, __dadd_rn(l, m));
}
template <class N> __device__ __forceinline__ N num(double a);
template <> __device__ __forceinline__ double num<double>(double a) { return a; }
template <> __device__ __forceinline__ dd num<dd>(double a) { return {a, 0.0}; }
__device__ __forceinline__ double to_double(double a) { return a; }
__device__ __forceinline__ double to_double(dd a) { return a.hi + a.lo; }

// cos and sin of pi p / B, B a power of two, 0 <= p < B
__device__ __forceinline__ void cos_sin_pi(int p, int B, double &c, double &s) { sincospi((double)p / B, &s, &c); }
// ... in double-double: the angle is folded into [0, pi/4], then Taylor's series
__device__ void cos_sin_pi(int p, int B, dd &c, dd &s) {
    const bool neg = 2 * p > B;                  // cos(pi - a) = -cos a, sin(pi - a) = sin a
    int q = neg ? B - p : p;                     // angle in [0, pi/2]
    const bool swap = 4 * q > B;
    if (swap) q = B / 2 - q;                     // angle in [0, pi/4]
    const dd pi{3.141592653589793116, 1.2246467991473532072e-16};
    const dd x = pi * num<dd>((double)q / B), x2 = -(x * x);
    dd cs = num<dd>(1.0), sn = x, ct = cs, st = x;
    for (int k = 1; k < 15; ++k) {               // (pi/4)^30 / 30! < 1e-35
        const double ic = 1.0 / ((2 * k - 1) * (2 * k)), is = 1.0 / ((2 * k) * (2 * k + 1));
        // the reciprocals to double-double: one Newton correction
        const dd rc{ic, __fma_rn(-ic, (double)((2 * k - 1) * (2 * k)), 1.0) * ic};
        const dd rs{is, __fma_rn(-is, (double)((2 * k) * (2 * k + 1)), 1.0) * is};
        ct = ct * x2 * rc;
        st = st * x2 * rs;
        cs = cs + ct;
        sn = sn + st;
    }
    c = swap ? sn : cs;
    s = swap ? cs : sn;
    if (neg) c = -c;
}

struct SpecCoin {
    double re[4], im[4];
};

// mat[(g, c, h, t)] = row h of scale * U(theta)^K (adj: of its adjoint) for the
// momentum that thread t of group g holds in register c: sublattice momentum
// p = G (a + 16 b + 256 c) + g, t = 16 a + b, theta = pi p / B per site.  For
// odd K the outputs sit one site further right, hence the factor e^{i theta}.
template <class R, class N>
__global__ void __launch_bounds__(32)
k_spec_matrices(SpecPair<R> *mat, SpecCoin coin, int G, int K, int flip, int adj, double scale) {
    const int id = blockIdx.x * 32 + threadIdx.x;           // (g, c, t)
    const int t = id % SPEC_GROUP, c = id / SPEC_GROUP % 16, g = id / (16 * SPEC_GROUP);
    if (g >= G) return;
    const int B = G * SPEC_POINTS, p = G * ((t >> 4) + 16 * (t & 15) + 256 * c) + g;
    using Z = Cx<N>;
    N cs, sn;
    cos_sin_pi(p, B, cs, sn);
    const Z e0{cs, sn}, e1{cs, -sn};
    auto mul = [](Z x, Z y) { return Z{x.re * y.re - x.im * y.im, x.re * y.im + x.im * y.re}; };
    auto add = [](Z x, Z y) { return Z{x.re + y.re, x.im + y.im}; };
    Z u[4];   // U(theta): coin 0 arrives from x + 1 (e^{i theta}), coin 1 from x - 1
    for (int k = 0; k < 2; ++k) {
        const Z r0 = mul(e0, Z{num<N>(coin.re[k]), num<N>(coin.im[k])});
        const Z r1 = mul(e1, Z{num<N>(coin.re[2 + k]), num<N>(coin.im[2 + k])});
        u[k] = flip ? r1 : r0;        // (flip-flop: they land in the other plane)
        u[2 + k] = flip ? r0 : r1;
    }
    Z m[4] = {u[0], u[1], u[2], u[3]};
    for (int bit = 30 - __clz(K); bit >= 0; --bit) {   // left to right: square, then times U
        const Z bc = mul(m[1], m[2]), tr = add(m[0], m[3]);
        const Z a = add(mul(m[0], m[0]), bc), d = add(mul(m[3], m[3]), bc);
        m[1] = mul(m[1], tr);
        m[2] = mul(m[2], tr);
        m[0] = a;
        m[3] = d;
        if (K >> bit & 1) {
            const Z w[4] = {m[0], m[1], m[2], m[3]};
            for (int r = 0; r < 2; ++r)
                for (int k = 0; k < 2; ++k) m[2 * r + k] = add(mul(w[2 * r], u[k]), mul(w[2 * r + 1], u[2 + k]));
        }
    }
    if (adj) {
        const Z b = m[1];
        m[1] = Z{m[2].re, -m[2].im};
        m[2] = Z{b.re, -b.im};
        m[0].im = -m[0].im;
        m[3].im = -m[3].im;
    }
    SpecPair<R> row[2];
    for (int h = 0; h < 2; ++h) {
        Z z[2];
        for (int k = 0; k < 2; ++k) z[k] = (K & 1) ? mul(m[2 * h + k], e0) : m[2 * h + k];
        row[h].a = {(R)(to_double(z[0].re) * scale), (R)(to_double(z[0].im) * scale)};
        row[h].b = {(R)(to_double(z[1].re) * scale), (R)(to_double(z[1].im) * scale)};
        mat[((g * 16 + c) * 2 + h) * SPEC_GROUP + t] = row[h];
    }
}

template <class R>
__global__ void k_spec_twiddles(SpecCx<R> *tw) {
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= SPEC_TW) return;
    int num, den;
    if (id < SPEC_TW2) { num = (id / 256) * (id % 256); den = 4096; }                                  // ta
    else if (id < SPEC_TWG) { num = ((id - SPEC_TW2) / 16) * ((id - SPEC_TW2) % 16); den = 256; }       // ub
    else { num = id - SPEC_TWG; den = 8192; }                                                          // j = t + 256 i
    double s, c;
    sincospi(-2.0 * num / den, &s, &c);
    tw[id] = {(R)c, (R)s};
}

template <int P, int G>
static cudaError_t go_spectral(const Spec1DArgs &a, cudaStream_t s) {
    using R = typename SpecReal<P>::type;
    constexpr size_t smem = spec_smem_bytes<R>(G);
    auto kern = k_spectral1d<P, G>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t W = 2 * ((int64_t)G * SPEC_POINTS - a.K), blocks = (a.n + W - 1) / W * 2;
    kern<<<(unsigned)blocks, G * SPEC_THREADS, smem, s>>>(a.in, a.out, a.n, a.K, W, a.table);
    return cudaGetLastError();
}

template <class R, class N>
static cudaError_t go_matrices(const Spec1DArgs &a, const double *coin, double scale, cudaStream_t s) {
    SpecCoin c;
    for (int i = 0; i < 4; ++i) { c.re[i] = coin[2 * i]; c.im[i] = coin[2 * i + 1]; }
    const int G = spectral1d_groups(a.tile);
    // (three 16-point transforms each way, whose norm the matrices put right: DftGain)
    if (sizeof(R) == sizeof(float)) scale /= std::pow(DftGain<R>::of16, 6);
    k_spec_matrices<R, N><<<G * SPEC_POINTS / 32, 32, 0, s>>>(static_cast<SpecPair<R> *>(a.table), c, G, a.K,
                                                              a.shift == QW_SHIFT_FLIPFLOP, a.adjoint,
                                                              scale / (G * SPEC_POINTS));
    return cudaGetLastError();
}

static bool spec_double(int prec) { return prec == QW_F64 || prec == QW_F32_COMP; }

// tile (sites per lane of a warp-sized view of the block, S / 32): 256 (S =
// 8192) and, for the float forms, 512 (S = 16384; two groups of double
// registers do not fit an SM)
int spectral1d_groups(int tile) { return tile == 512 ? 2 : 1; }

bool spectral1d_ok(int prec, int64_t n, int K, int tile) {
    if (!(tile == 256 || (tile == 512 && !spec_double(prec)))) return false;
    const int64_t W = 32LL * tile - 2LL * K;   // blocks of W sites, two CTAs each
    return K >= 1 && K < 16 * tile && (n + W - 1) / W < (int64_t(1) << 30);
}

size_t spectral1d_table_bytes(int prec, int tile) {
    const int G = spectral1d_groups(tile);
    return spec_double(prec) ? spec_table_bytes<double>(G) : spec_table_bytes<float>(G);
}

cudaError_t launch_spectral1d_twiddles(int prec, int tile, void *table, cudaStream_t s) {
    const int G = spectral1d_groups(tile);
    const unsigned blocks = (SPEC_TW + 127) / 128;
    char *t = static_cast<char *>(table);
    if (spec_double(prec)) k_spec_twiddles<double><<<blocks, 128, 0, s>>>(reinterpret_cast<SpecCx<double> *>(t + spec_matrix_bytes<double>(G)));
    else k_spec_twiddles<float><<<blocks, 128, 0, s>>>(reinterpret_cast<SpecCx<float> *>(t + spec_matrix_bytes<float>(G)));
    return cudaGetLastError();
}

cudaError_t launch_spectral1d_matrices(int prec, const Spec1DArgs &a, const double *coin, double scale, cudaStream_t s) {
    return spec_double(prec) ? go_matrices<double, dd>(a, coin, scale, s) : go_matrices<float, double>(a, coin, scale, s);
}

cudaError_t launch_spectral1d(int prec, const Spec1DArgs &a, cudaStream_t s) {
    if (!spectral1d_ok(prec, a.n, a.K, a.tile)) return cudaErrorInvalidValue;
    const bool two = spectral1d_groups(a.tile) == 2;
    switch (prec) {
        case QW_F64: return go_spectral<P_F64, 1>(a, s);
        case QW_F32_COMP: return go_spectral<P_COMP, 1>(a, s);
        case QW_F32: return two ? go_spectral<P_F32, 2>(a, s) : go_spectral<P_F32, 1>(a, s);
        case QW_F32_BF16STORE: return two ? go_spectral<P_BF16, 2>(a, s) : go_spectral<P_BF16, 1>(a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace qw
