// k_spectral1d.cuh -- K steps of the cycle walk with one coin for all sites, as
// a convolution done in momentum space block by block.
//
// With one coin C at every site the step U = S (I (x) C) of Sec. 2.1 commutes
// with translations: on a plane wave e^{i theta x} it is the 2 x 2 matrix
// U(theta) = diag(e^{i theta}, e^{-i theta}) C (moving shift; the flip-flop
// shift swaps the rows), so K steps are U(theta)^K, a convolution of the state
// with a kernel of 2K + 1 sites.  The walk is also bipartite: after K steps a
// site only depends on the sites x' with x' = x + K (mod 2), so even and odd
// sites (of the unrolled line) are two independent walks.  A CTA takes the B
// sites of one parity among S = 2B consecutive ones, transforms both coin
// planes (length B), multiplies each momentum by the 2 x 2 matrix U^K, and
// transforms back (overlap-save, Stockham Jr., "High-speed convolution and
// correlation", AFIPS 1966): the S - 2K sites in the middle of the block, whose
// light cone lies inside it, are the output.  Any n works: the block reads the
// cycle modulo n, as a stretch of the unrolled line.
//
// Why: stepping costs at least 4 additions per site and step (the sweep kernel
// is bound by their issue); this costs about 440 instructions per output site
// whatever K is, so at K = 4096 it needs 1/40 of them, and a state crosses HBM
// once per K <= S / 3 steps.  Rounding errors do not grow with K either: one
// transform pair adds 1.8e-7 (float) or 3.4e-16 (double) of the block's norm,
// where stepping is 3e-7 / 8e-16 off after 128 steps and 1.7e-6 / 6e-15 after
// 4096 / 1024 (Hadamard; against 64-bit and long double values).  The matrices
// U^K are formed in double (float walks) or double-double (double walks) by
// repeated squaring.
//
// Measured, stepping (autotuned) -> momentum space, per qw_step call:
//   n = 2^27 FP32, T = 4096: Hadamard class 73.7 -> 4.3 ms, complex coin 313 ->
//   4.3 ms; T = 1000: 18.1 -> 2.1 ms (G = 1), 76.4 -> 2.1 ms
//   n = 1000003 FP32 complex, T = 1000: 0.86 -> 0.031 ms
//   n = 2^20 FP64 real, T = 1000: 18.9 -> 0.57 ms; double-float: 6.2 -> 0.65 ms
// What bounds it (FP32, G = 2, 2^24 sites): latency.  One CTA fills an SM (139 KB
// of shared memory, all registers), so the loads of its block, the matrices and
// the barriers are only hidden by its own warps: issue 50 %, long scoreboard the
// first stall, DRAM 10 %.  Hence one plane per thread (1024 threads of 64
// registers; with both planes per thread, 512 of 128: issue 35 %, 5.0 ms), the
// next block's sites prefetched into L2 (4.8 ms without; two CTAs of G = 1 cover
// for each other, and gain nothing from it), and spec_reload.  FP64: its pipe.
//
// Layout of the transform.  512 threads hold 4096 points of both planes, 16 per
// thread, in registers: the lower half of a warp plane 0, the upper half plane 1
// at the same points, so that the 2 x 2 matrices take the other plane's value by
// a shuffle.  4096 = 16 x 16 x 16 (Cooley and Tukey, 1965): with j = t + 256 i, t = u + 16 v and p = a + 16 b + 256 c,
//   X[p] = sum_u w16^{uc} w256^{ub} sum_v w16^{vb} w4096^{ta} sum_i w16^{ia} x[j],
// so each sum is a 16-point transform inside a thread.  Between the first two
// the data change threads through shared memory (one block barrier); the second
// change is a 16 x 16 transpose inside a half warp (rows padded to 17), with no
// barrier.  Momenta stay in the order the threads hold them, the table of U^K
// is laid out in that order, and the inverse runs the same exchanges backward:
// two block barriers in all.  For G = 2 (B = 8192) two such groups share a CTA:
// group g transforms (x[j] +- x[j + 4096]) w8192^{gj} to the momenta 2r + g,
// and on the way back the groups swap half of their values.
#pragma once
#include "qw_internal.cuh"

namespace qw {

// compute precision of the transforms: float for FP32 and bf16 storage, double
// for FP64 and double-float (hi + lo fits a double)
template <int P> struct SpecReal { using type = float; };
template <> struct SpecReal<P_F64> { using type = double; };
template <> struct SpecReal<P_COMP> { using type = double; };

constexpr int SPEC_GROUP = 256;                       // threads per 4096 points of one plane
constexpr int SPEC_THREADS = 2 * SPEC_GROUP;          // ... of both planes
constexpr int SPEC_POINTS = 4096;                     // points per group and plane
constexpr int SPEC_ROW = 16 * 17;                     // one padded 16 x 16 tile
constexpr int SPEC_TW1 = 0;                           // twiddle tables, in elements: w4096^{ta} [a][t],
constexpr int SPEC_TW2 = 16 * 256;                    // w256^{ub} [b][u],
constexpr int SPEC_TWG = SPEC_TW2 + 16 * 16;          // w8192^{j} [i][t]
constexpr int SPEC_TW = SPEC_TWG + 16 * 256;

constexpr int SPEC_AHEAD = 152;                       // CTAs in flight (G = 2: one per SM)

template <class R> struct alignas(4 * sizeof(R)) SpecPair { Cx<R> a, b; };
template <class R> struct alignas(2 * sizeof(R)) SpecCx { R re, im; };

// bytes of the tables a handle keeps: U^K of every momentum, then the twiddles
template <class R> constexpr size_t spec_matrix_bytes(int G) { return (size_t)G * SPEC_POINTS * 4 * 2 * sizeof(R); }
template <class R> constexpr size_t spec_table_bytes(int G) { return spec_matrix_bytes<R>(G) + (size_t)SPEC_TW * 2 * sizeof(R); }
template <class R> constexpr size_t spec_smem_bytes(int G) { return (size_t)G * 2 * 16 * SPEC_ROW * 2 * sizeof(R); }

// site load / store in the compute precision of the transforms
template <int P> __device__ __forceinline__ Cx<typename SpecReal<P>::type> spec_ld(View v, int c, int64_t i) {
    const auto a = St<P>::ld(v, c, i);
    if constexpr (P == P_COMP)
        return {(double)a.re.hi + (double)a.re.lo, (double)a.im.hi + (double)a.im.lo};
    else
        return {a.re, a.im};
}
template <int P>
__device__ __forceinline__ void spec_st(View v, int c, int64_t i, Cx<typename SpecReal<P>::type> a) {
    if constexpr (P == P_COMP) {
        const float rh = (float)a.re, ih = (float)a.im;
        St<P>::st(v, c, i, Cx<ff>{{rh, (float)(a.re - (double)rh)}, {ih, (float)(a.im - (double)ih)}});
    } else {
        St<P>::st(v, c, i, a);
    }
}

// z * w, or z * conj(w) on the way back
template <int INV, class R> __device__ __forceinline__ Cx<R> spec_twiddle(Cx<R> z, Cx<R> w) {
    if (INV) return {z.re * w.re + z.im * w.im, z.im * w.re - z.re * w.im};
    return {z.re * w.re - z.im * w.im, z.im * w.re + z.re * w.im};
}
template <class R> __device__ __forceinline__ Cx<R> spec_tw(const SpecCx<R> *__restrict__ t, int i) {
    const SpecCx<R> w = t[i];
    return {w.re, w.im};
}

// The way back reads the twiddles (and in k_spec2_columns writes the addresses)
// of the way forth: without this the compiler keeps them in registers in
// between, and spills (190 bytes per thread here, 104 there, at 64 registers).
template <class T> __device__ __forceinline__ void spec_reload(T *&p) { asm volatile("" : "+l"(p)); }

// 4-point transform in place, w4 = -i (forward) or +i (inverse)
template <int INV, class R> __device__ __forceinline__ void dft4(Cx<R> &x0, Cx<R> &x1, Cx<R> &x2, Cx<R> &x3) {
    const Cx<R> s = cadd(x0, x2), d = csub(x0, x2), e = cadd(x1, x3), f = csub(x1, x3);
    x0 = cadd(s, e);
    x2 = csub(s, e);
    const Cx<R> p{d.re - f.im, d.im + f.re}, m{d.re + f.im, d.im - f.re};   // d + i f, d - i f
    x1 = INV ? p : m;
    x3 = INV ? m : p;
}

// cos and sin of pi / 8, cos of pi / 4
template <class R> struct Roots16 {
    static constexpr R C1 = (R)0.92387953251128675613, S1 = (R)0.38268343236508977173, H = (R)0.70710678118654752440;
};
// What the rounding of these constants does to the norm of a 16-point (and, of
// H alone, an 8-point) transform, as a factor on the amplitudes: all three floats
// lie below their values, so the float transforms shrink by 1.1e-8 each, always in
// the same sense.  The launchers undo it in tables that they round themselves (the
// cycle's matrices, the torus' twiddles).  Change of the norm by one launch, without
// and with that: cycle -1.6e-7, -2.5e-8; torus 256^2 -2.2e-7, 3.7e-8, 1024^2 -2.6e-7,
// -5.3e-8, 8192^2 -3.8e-7, -1.6e-8.  A quarter of the points meets w16, w16^3 or
// w16^9, a quarter H twice.
template <class R> struct DftGain {
    static constexpr double rot = (double)Roots16<R>::C1 * Roots16<R>::C1 + (double)Roots16<R>::S1 * Roots16<R>::S1;
    static constexpr double diag = 2.0 * (double)Roots16<R>::H * Roots16<R>::H;
    static constexpr double of16 = 1.0 + 0.5 * ((rot - 1.0) + (diag - 1.0)) / 4;
    static constexpr double of8 = 1.0 + 0.5 * (diag - 1.0) / 4;
};

// 16-point transform of x (index n) as 4 x 4; output k is left in x[out16(k)].
__host__ __device__ constexpr int out16(int k) { return 4 * (k & 3) + (k >> 2); }
template <int INV, class R> __device__ __forceinline__ void dft16(Cx<R> (&x)[16]) {
    constexpr R C1 = Roots16<R>::C1, S1 = Roots16<R>::S1, H = Roots16<R>::H;
#pragma unroll
    for (int b = 0; b < 4; ++b) dft4<INV>(x[b], x[4 + b], x[8 + b], x[12 + b]);
    const R g = INV ? (R)-1 : (R)1;   // w16 = C1 - i g S1
    auto mul = [](Cx<R> z, R wr, R wi) { return Cx<R>{z.re * wr - z.im * wi, z.im * wr + z.re * wi}; };
    // x[4c + b] *= w16^{bc}
    x[5] = mul(x[5], C1, -g * S1);
    x[6] = {H * (x[6].re + g * x[6].im), H * (x[6].im - g * x[6].re)};
    x[7] = mul(x[7], S1, -g * C1);
    x[9] = {H * (x[9].re + g * x[9].im), H * (x[9].im - g * x[9].re)};
    x[10] = {g * x[10].im, -g * x[10].re};
    x[11] = {H * (g * x[11].im - x[11].re), -H * (x[11].im + g * x[11].re)};
    x[13] = mul(x[13], S1, -g * C1);
    x[14] = {H * (g * x[14].im - x[14].re), -H * (x[14].im + g * x[14].re)};
    x[15] = mul(x[15], -C1, g * S1);
#pragma unroll
    for (int c = 0; c < 4; ++c) dft4<INV>(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
}
template <class R> __device__ __forceinline__ void order16(Cx<R> (&x)[16]) {   // x[k] = output k (a renaming)
    Cx<R> y[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) y[k] = x[out16(k)];
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = y[k];
}

__device__ __forceinline__ void spec_group_barrier(int G, int g) {
    if (G == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(SPEC_THREADS) : "memory");
}

// forward transform of one plane: x[i] = x(t + 256 i) -> x[c] = X(a + 16 b + 256 c)
// of thread t = 16 a + b.  `sm` is the plane's 16 padded tiles; the block
// barrier between first and second part is the caller's (shared by the planes).
template <class R>
__device__ __forceinline__ void spec_fwd1(Cx<R> (&x)[16], SpecCx<R> *sm, const SpecCx<R> *__restrict__ tw, int t) {
    dft16<0>(x);
#pragma unroll
    for (int a = 0; a < 16; ++a) {
        Cx<R> z = x[out16(a)];
        if (a) z = spec_twiddle<0>(z, spec_tw(tw + SPEC_TW1, a * 256 + t));
        sm[a * SPEC_ROW + t] = {z.re, z.im};
    }
}
template <class R>
__device__ __forceinline__ void spec_fwd2(Cx<R> (&x)[16], SpecCx<R> *sm, const SpecCx<R> *__restrict__ tw, int t) {
    SpecCx<R> *row = sm + (t >> 4) * SPEC_ROW;   // tile a: read and written by this half warp only
    const int u = t & 15;
#pragma unroll
    for (int v = 0; v < 16; ++v) { const SpecCx<R> z = row[u + 16 * v]; x[v] = {z.re, z.im}; }
    dft16<0>(x);
    __syncwarp();
#pragma unroll
    for (int b = 0; b < 16; ++b) {
        Cx<R> z = x[out16(b)];
        if (b) z = spec_twiddle<0>(z, spec_tw(tw + SPEC_TW2, b * 16 + u));
        row[b * 17 + u] = {z.re, z.im};
    }
    __syncwarp();
#pragma unroll
    for (int w = 0; w < 16; ++w) { const SpecCx<R> z = row[u * 17 + w]; x[w] = {z.re, z.im}; }
    dft16<0>(x);
    order16(x);
}
// the inverse, unnormalised (1 / B is folded into the matrices)
template <class R>
__device__ __forceinline__ void spec_inv1(Cx<R> (&x)[16], SpecCx<R> *sm, const SpecCx<R> *__restrict__ tw, int t) {
    SpecCx<R> *row = sm + (t >> 4) * SPEC_ROW;
    const int b = t & 15;
    dft16<1>(x);
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        Cx<R> z = x[out16(u)];
        if (u) z = spec_twiddle<1>(z, spec_tw(tw + SPEC_TW2, u * 16 + b));
        row[b * 17 + u] = {z.re, z.im};
    }
    __syncwarp();
#pragma unroll
    for (int w = 0; w < 16; ++w) { const SpecCx<R> z = row[w * 17 + b]; x[w] = {z.re, z.im}; }
    dft16<1>(x);
    __syncwarp();
#pragma unroll
    for (int v = 0; v < 16; ++v) { const Cx<R> z = x[out16(v)]; row[b + 16 * v] = {z.re, z.im}; }
}
template <class R>
__device__ __forceinline__ void spec_inv2(Cx<R> (&x)[16], const SpecCx<R> *sm, const SpecCx<R> *__restrict__ tw, int t) {
#pragma unroll
    for (int a = 0; a < 16; ++a) {
        const SpecCx<R> s = sm[a * SPEC_ROW + t];
        Cx<R> z{s.re, s.im};
        if (a) z = spec_twiddle<1>(z, spec_tw(tw + SPEC_TW1, a * 256 + t));
        x[a] = z;
    }
    dft16<1>(x);
    order16(x);
}

// Block blockIdx.x / 2 of W = 2 (G * 4096 - K) output sites, parity blockIdx.x & 1.
// table: U^K / B in the order the threads hold the momenta, then the twiddles.
template <int P, int G>
__global__ void __launch_bounds__(G *SPEC_THREADS, (G == 1 && sizeof(typename SpecReal<P>::type) == 4) ? 2 : 1)
k_spectral1d(View in, View out, int64_t n, int K, int64_t W, const void *__restrict__ table) {
    using R = typename SpecReal<P>::type;
    using C = Cx<R>;
    extern __shared__ __align__(16) unsigned char ssm[];
    const int g = G == 1 ? 0 : (int)threadIdx.x / SPEC_THREADS;   // uniform per warp
    const int h = (int)threadIdx.x >> 4 & 1;                      // the thread's plane
    const int t = ((int)threadIdx.x % SPEC_THREADS >> 5) * 16 + ((int)threadIdx.x & 15);
    SpecCx<R> *sm = reinterpret_cast<SpecCx<R> *>(ssm) + (size_t)(2 * g + h) * 16 * SPEC_ROW;
    const auto *mat = static_cast<const SpecPair<R> *>(table);
    const auto *tw = reinterpret_cast<const SpecCx<R> *>(static_cast<const char *>(table) + spec_matrix_bytes<R>(G));
    const int q = (int)(blockIdx.x & 1);
    const int64_t out0 = (int64_t)(blockIdx.x >> 1) * W;
    const int64_t wthis = min(W, n - out0);
    // first site of the block, inside the cycle: out0 - K modulo n
    int64_t x0 = (out0 - K + q) % n;
    if (x0 < 0) x0 += n;
    const bool once = n >= 2 * (int64_t)G * SPEC_POINTS;   // the block goes at most once past site n - 1
    auto site = [&](int j) {
        int64_t s = x0 + 2 * j;
        if (s >= n) s = once ? s - n : s % n;
        return s;
    };
    if constexpr (G == 2) {
        // the block that this SM takes next, into L2: 16 sites of plane q per thread
        const int64_t o1 = (int64_t)((blockIdx.x + SPEC_AHEAD) >> 1) * W, s1 = o1 - K + 16 * (int64_t)threadIdx.x;
        if (o1 < n && s1 >= 0 && s1 < n)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char *>(in.p) + (q * in.pitch + s1) * St<P>::SLOT_BYTES));
    }
    C f[16];
    if constexpr (G == 1) {
#pragma unroll
        for (int i = 0; i < 16; ++i) f[i] = spec_ld<P>(in, h, site(t + 256 * i));
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const C a = spec_ld<P>(in, h, site(t + 256 * i)), b = spec_ld<P>(in, h, site(t + 256 * i + SPEC_POINTS));
            f[i] = g == 0 ? cadd(a, b) : spec_twiddle<0>(csub(a, b), spec_tw(tw + SPEC_TWG, i * 256 + t));
        }
    }
    spec_fwd1(f, sm, tw, t);
    spec_group_barrier(G, g);
    spec_fwd2(f, sm, tw, t);
    // row h of the matrix: the other plane's value is 16 lanes away
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        const SpecPair<R> r = mat[((g * 16 + c) * 2 + h) * SPEC_GROUP + t];
        const C o{__shfl_xor_sync(0xffffffffu, f[c].re, 16), __shfl_xor_sync(0xffffffffu, f[c].im, 16)};
        const C z0 = h == 0 ? f[c] : o, z1 = h == 0 ? o : f[c];
        f[c] = cfma(r.b, z1, cmul(r.a, z0));
    }
    __syncwarp();   // the forward transposes' last reads of the tiles, before they are rewritten
    spec_reload(tw);
    spec_inv1(f, sm, tw, t);
    spec_group_barrier(G, g);
    spec_inv2(f, sm, tw, t);
    // point j is site out0 - K + o, o = 2j + q + (K mod 2); outputs have K <= o < K + wthis
    auto put = [&](int j, C v) {
        const int64_t o = 2 * (int64_t)j + q + (K & 1) - K;
        if (o >= 0 && o < wthis) spec_st<P>(out, h, out0 + o, v);
    };
    if constexpr (G == 1) {
#pragma unroll
        for (int i = 0; i < 16; ++i) put(t + 256 * i, f[i]);
    } else {
        // x[j] = z0 + z1 w8192^{-j}, x[j + 4096] = z0 - z1 w8192^{-j}: group 0 forms
        // them for i < 8, group 1 for i >= 8, after swapping the other half
        if (g == 1) {
#pragma unroll
            for (int i = 0; i < 16; ++i) f[i] = spec_twiddle<1>(f[i], spec_tw(tw + SPEC_TWG, i * 256 + t));
        }
        __syncthreads();   // every read of the tiles is done
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const C s = g == 0 ? f[8 + k] : f[k];
            sm[k * 256 + t] = {s.re, s.im};
        }
        __syncthreads();
        const SpecCx<R> *p = reinterpret_cast<const SpecCx<R> *>(ssm) + (size_t)(2 * (g ^ 1) + h) * 16 * SPEC_ROW;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const C m = g == 0 ? f[k] : f[8 + k], o{p[k * 256 + t].re, p[k * 256 + t].im};
            const C z0 = g == 0 ? m : o, z1 = g == 0 ? o : m;   // group 0's and group 1's value
            const int j = t + 256 * (g == 0 ? k : 8 + k);
            put(j, cadd(z0, z1));
            put(j + SPEC_POINTS, csub(z0, z1));
        }
    }
}

}  // namespace qw
