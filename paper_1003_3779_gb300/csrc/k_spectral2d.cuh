// k_spectral2d.cuh -- K steps of the torus walk with a Grover coin (any shift) or
// with H (x) H on the diagonal lattice, in momentum space.
//
// With one coin for all sites a step is a 4 x 4 matrix U(kx, ky) per momentum, so
// K steps are a transform of the four coin planes, U^K at each momentum, and the
// transform back, whatever K is (the 1D form: k_spectral1d.cuh).  An axis whose
// length is a power of two is transformed as the cycle it is; any other in blocks
// of B sites with K sites of halo per side (overlap-save), read modulo the torus.
// Three kernels per launch: rows forward into a workspace, columns forward, U^K
// and back, rows back into the state: the state crosses HBM three times per
// launch (a little more with halos), against once per 8 steps of streaming.
//
// U^K without a 4 x 4 power.  Write U = D M, D the shift's phases, M the coin
// (flip-flop: times the coin swap), real, symmetric, M^2 = 1.  For the Grover coin
// U has the eigenvalues 1, -1 and e^{+-i w}, cos w = -+ (cos kx + cos ky) / 2
// (moving / flip-flop; diagonal lattice: -cos kx cos ky).  X = (U - U^dagger) / 2
// vanishes on the first two eigenvectors and is +-i sin w on the others, so for
// even K
//     U^K = 1 + s_K X + 2 s_{K/2}^2 X^2,    s_n = sin(n w) / sin(w).
// s_n can be as large as n where w is near 0 or pi; X is small there, and is
// formed without cancellation as (E M - M E*) / 2 with E = D - 1 (or D + 1).
// cos(n w) and s_n come from repeated doubling in double-float, from
// sin^2(w/2) given to double-float accuracy.  The diagonal lattice with H (x) H is
// two independent 1D walks: U^K is a tensor product of two 2 x 2 matrices.
//
// Transforms: power-of-two lengths 256 .. 8192, 16 points per thread, radix-16
// stages in place in shared memory (the last one radix 2, 4 or 8 where 16 does
// not divide), in decimation-in-frequency order forward and the reverse order
// back, so momenta stay in digit-reversed places and nothing is reordered.
//
// Measured, streaming (8 steps per launch) -> momentum space, 1024 steps per call:
//   Grover 8192^2 106 -> 9.4 ms, 4096^2 29.2 -> 1.66 ms; H (x) H on the diagonal
//   lattice, 8192^2, 123 -> 8.6 ms; 300 x 200, 200 steps, with readout 1.12 -> 0.12 ms
// What bounds it (4096^2): the rows run at 61-66 % of the DRAM rate; the columns,
// three quarters of the time, are bound by the load queue and latency (issue 33 %):
// four planes of 4096 points take an SM, one column per CTA, whose 8-byte loads
// touch a 32-byte sector each.  A split axis of 8192 runs as even and odd momenta,
// and k and -k share their factors (15.3 -> 11.1 ms per call with copies).
#pragma once
#include "qw_internal.cuh"
#include "k_spectral1d.cuh"

namespace qw {

constexpr int SPEC2_MIN_L = 8, SPEC2_MAX_LX = 13, SPEC2_MAX_LY = 12;   // log2 of the transform lengths
// Twiddles of a stage of length n = 2^5 .. 2^13: w_n^{bk} at n + k n/16 + b.
constexpr int SPEC2_TW = 2 << SPEC2_MAX_LX;

// One momentum of an axis: sin, and sin^2 and cos^2 of half of it in double-float.
struct alignas(8) Spec2Axis {
    float s, sh, sl, ch, cl, pad;
};

__host__ __device__ inline int spec2_freq(int L, int p) {   // momentum at place p
    int n = 1 << L, f = 0, mult = 1;
    while (n > 1) {
        const int r = n >= 16 ? 16 : n, m = n / r;
        f += p / m * mult;
        p %= m;
        mult *= r;
        n = m;
    }
    return f;
}
__host__ __device__ inline int spec2_place(int L, int f) {   // place of momentum f
    int n = 1 << L, p = 0;
    while (n > 1) {
        const int r = n >= 16 ? 16 : n, m = n / r;
        p += f % r * m;
        f /= r;
        n = m;
    }
    return p;
}
__device__ __forceinline__ int spec2_at(int p) { return p + (p >> 4); }   // one pad slot per 16

template <int INV, class R> __device__ __forceinline__ void dft8(Cx<R> (&x)[8]) {
    constexpr R H = Roots16<R>::H;
    const R g = INV ? (R)-1 : (R)1;
    dft4<INV>(x[0], x[2], x[4], x[6]);
    dft4<INV>(x[1], x[3], x[5], x[7]);
    const Cx<R> o1 = x[3], o2 = x[5], o3 = x[7];
    const Cx<R> t1{H * (o1.re + g * o1.im), H * (o1.im - g * o1.re)}, t2{g * o2.im, -g * o2.re},
        t3{H * (g * o3.im - o3.re), -H * (o3.im + g * o3.re)};
    const Cx<R> e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6], o0 = x[1];
    x[0] = cadd(e0, o0); x[4] = csub(e0, o0);
    x[1] = cadd(e1, t1); x[5] = csub(e1, t1);
    x[2] = cadd(e2, t2); x[6] = csub(e2, t2);
    x[3] = cadd(e3, t3); x[7] = csub(e3, t3);
}

using S2 = SpecCx<float>;
using C2 = Cx<float>;

// the last stage, of length n = 2, 4 or 8, on 16 consecutive places per thread
template <int INV, int N> __device__ __forceinline__ void spec2_tail(S2 *sm, int t) {
    C2 x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) { const S2 z = sm[spec2_at(16 * t + i)]; x[i] = {z.re, z.im}; }
#pragma unroll
    for (int b = 0; b < 16; b += N) {
        if constexpr (N == 2) {
            const C2 u = x[b], v = x[b + 1];
            x[b] = cadd(u, v);
            x[b + 1] = csub(u, v);
        } else if constexpr (N == 4) {
            dft4<INV>(x[b], x[b + 1], x[b + 2], x[b + 3]);
        } else {
            C2 y[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) y[i] = x[b + i];
            dft8<INV>(y);
#pragma unroll
            for (int i = 0; i < 8; ++i) x[b + i] = y[i];
        }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) sm[spec2_at(16 * t + i)] = {x[i].re, x[i].im};
}

// a radix-16 stage of length n on the thread's places, forward: x holds them in
// order on entry; the results go to shared memory
template <int NN> __device__ __forceinline__ void spec2_put(C2 (&x)[16], S2 *sm, const S2 *__restrict__ tw, int base, int b) {
    dft16<0>(x);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        C2 z = x[out16(k)];
        if (NN > 16 && k) z = spec_twiddle<0>(z, spec_tw(tw, NN + k * (NN / 16) + b));
        sm[spec2_at(base + k * (NN / 16))] = {z.re, z.im};
    }
}
// backward: from shared memory, into x in order
template <int NN> __device__ __forceinline__ void spec2_get(C2 (&x)[16], const S2 *sm, const S2 *__restrict__ tw, int base, int b) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const S2 s = sm[spec2_at(base + k * (NN / 16))];
        C2 z{s.re, s.im};
        if (NN > 16 && k) z = spec_twiddle<1>(z, spec_tw(tw, NN + k * (NN / 16) + b));
        x[k] = z;
    }
    dft16<1>(x);
    order16(x);
}

// Forward transform of 2^L points: x[a] = point t + a 2^L / 16 on entry; the
// momenta are in sm (by place) on exit, before a barrier.
template <int L> __device__ __forceinline__ void spec2_forward(C2 (&x)[16], S2 *sm, const S2 *__restrict__ tw, int t) {
    constexpr int N = 1 << L, N2 = N / 16, N3 = N2 / 16;
    auto stage = [&](auto c) {
        constexpr int n = decltype(c)::value, m = n / 16;
        __syncthreads();
        const int base = t / m * n + t % m;
#pragma unroll
        for (int a = 0; a < 16; ++a) { const S2 z = sm[spec2_at(base + a * m)]; x[a] = {z.re, z.im}; }
        spec2_put<n>(x, sm, tw, base, t % m);
    };
    spec2_put<N>(x, sm, tw, t, t);
    if constexpr (N2 >= 16) stage(std::integral_constant<int, N2>{});
    if constexpr (N3 >= 16) stage(std::integral_constant<int, N3>{});
    if constexpr (L % 4 != 0) {
        __syncthreads();
        spec2_tail<0, 1 << (L % 4)>(sm, t);
    }
}
// The inverse (unnormalised): momenta in sm, after a barrier, to points in x.
template <int L> __device__ __forceinline__ void spec2_inverse(C2 (&x)[16], S2 *sm, const S2 *__restrict__ tw, int t) {
    constexpr int N = 1 << L, N2 = N / 16, N3 = N2 / 16;
    auto stage = [&](auto c) {
        constexpr int n = decltype(c)::value, m = n / 16;
        const int base = t / m * n + t % m;
        spec2_get<n>(x, sm, tw, base, t % m);
#pragma unroll
        for (int a = 0; a < 16; ++a) sm[spec2_at(base + a * m)] = {x[a].re, x[a].im};
        __syncthreads();
    };
    if constexpr (L % 4 != 0) {
        spec2_tail<1, 1 << (L % 4)>(sm, t);
        __syncthreads();
    }
    if constexpr (N3 >= 16) stage(std::integral_constant<int, N3>{});
    if constexpr (N2 >= 16) stage(std::integral_constant<int, N2>{});
    spec2_get<N>(x, sm, tw, t, t);
}

// One launch: blocks [b0, b0 + nb) of the lattice, block b = (b mod nbx, b / nbx)
// with wx x wy outputs from (b mod nbx) wx, (b / nbx) wy; hx, hy: halo (0 on a
// cyclic axis).  z: the workspace, [block][plane][row 2^LY][place 2^LX].
struct Spec2Args {
    View in, out;
    int64_t nx, ny, wx, wy;
    int hx, hy, nbx, b0, nb, LX, LY;
    int split;       // the y axis is a cycle of 2^(LY+1): block g transforms (row r +- row r + 2^LY) w^{gr}
    S2 *z;
    const S2 *tw;
    float scale;
};

// w_n^r, r < n/2, from the stage's twiddles: w_n^{bk} is at n + k n/16 + b, b < n/16
__device__ __forceinline__ C2 spec2_root(const S2 *tw, int n, int r) {
    const int m = n / 16, q = r / m;                    // r = q m + b: w^r = w^b w16^q
    const C2 w = spec_tw(tw, n + m + r % m);            // k = 1: w^b
    float s, c;
    sincospif(-0.125f * (float)q, &s, &c);
    return cmul(w, C2{c, s});
}

template <int L> constexpr int spec2_rows() { return L >= 12 ? 1 : 4096 >> L; }   // rows per CTA
template <int L> constexpr size_t spec2_row_smem() { return (size_t)spec2_rows<L>() * ((1 << L) * 17 / 16) * sizeof(S2); }

template <int L>
__global__ void __launch_bounds__((1 << L) / 16 * spec2_rows<L>())
k_spec2_rows_forward(Spec2Args a) {
    constexpr int N = 1 << L, TH = N / 16;
    extern __shared__ __align__(16) unsigned char ssm[];
    const int t = (int)threadIdx.x % TH, rr = (int)threadIdx.x / TH;
    S2 *sm = reinterpret_cast<S2 *>(ssm) + rr * (N * 17 / 16);
    const int NY = 1 << a.LY;
    const int64_t id = (int64_t)blockIdx.x * spec2_rows<L>() + rr;   // (block, plane, row), a whole number of CTAs
    const int r = (int)(id % NY), c = (int)(id / NY % 4), b = a.b0 + (int)(id / NY / 4);
    int64_t x0 = ((b % a.nbx) * a.wx - a.hx) % a.nx, y = a.split ? r : ((b / a.nbx) * a.wy - a.hy + r) % a.ny;
    if (x0 < 0) x0 += a.nx;
    if (y < 0) y += a.ny;
    const C2 w = a.split ? spec2_root(a.tw, 2 * NY, r) : C2{1.f, 0.f};
    C2 x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        int64_t s = x0 + t + i * TH;
        if (s >= a.nx) s = a.nx >= N ? s - a.nx : s % a.nx;
        x[i] = St<P_F32>::ld(a.in, c, y * a.nx + s);
        if (a.split) {
            const C2 q = St<P_F32>::ld(a.in, c, (y + NY) * a.nx + s);
            x[i] = b == 0 ? cadd(x[i], q) : spec_twiddle<0>(csub(x[i], q), w);
        }
    }
    spec2_forward<L>(x, sm, a.tw, t);
    __syncthreads();
    S2 *z = a.z + id * N;
#pragma unroll
    for (int i = 0; i < 16; ++i) z[t + i * TH] = sm[spec2_at(t + i * TH)];
}

template <int L>
__global__ void __launch_bounds__((1 << L) / 16 * spec2_rows<L>())
k_spec2_rows_inverse(Spec2Args a) {
    constexpr int N = 1 << L, TH = N / 16;
    extern __shared__ __align__(16) unsigned char ssm[];
    const int t = (int)threadIdx.x % TH, rr = (int)threadIdx.x / TH;
    S2 *sm = reinterpret_cast<S2 *>(ssm) + rr * (N * 17 / 16);
    const int64_t rows = (int64_t)a.nb * 4 * a.wy, id = min((int64_t)blockIdx.x * spec2_rows<L>() + rr, rows - 1);
    const int64_t r = id % a.wy;                                     // output row of the block
    const int c = (int)(id / a.wy % 4), bl = (int)(id / a.wy / 4), b = a.b0 + bl, NY = 1 << a.LY;
    const S2 *z = a.z + (((int64_t)(a.split ? 0 : bl) * 4 + c) * NY + a.hy + r) * N;
    if (!a.split) {
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[spec2_at(t + i * TH)] = z[t + i * TH];
    } else {   // rows r and r + 2^LY are even +- odd w^{-r}
        const C2 w = spec2_root(a.tw, 2 * NY, (int)r);
        const S2 *o = z + (int64_t)4 * NY * N;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const S2 e = z[t + i * TH], q = o[t + i * TH];
            const C2 u = spec_twiddle<1>(C2{q.re, q.im}, w);
            sm[spec2_at(t + i * TH)] = bl == 0 ? S2{e.re + u.re, e.im + u.im} : S2{e.re - u.re, e.im - u.im};
        }
    }
    __syncthreads();
    C2 x[16];
    spec2_inverse<L>(x, sm, a.tw, t);
    const int64_t x0 = (b % a.nbx) * a.wx, y = a.split ? r + (int64_t)bl * NY : (b / a.nbx) * a.wy + r;
    if (y >= a.ny || (int64_t)blockIdx.x * spec2_rows<L>() + rr >= rows) return;
    const int64_t w = min(a.wx, a.nx - x0);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int64_t j = (int64_t)(t + i * TH) - a.hx;
        if (j >= 0 && j < w) St<P_F32>::st(a.out, c, y * a.nx + x0 + j, rmul(a.scale, x[i]));
    }
}

// U^K at one momentum.  MODE: the shift of the Grover coin, or SPEC2_TENSOR.
constexpr int SPEC2_TENSOR = 3;
struct Spec2Coin {
    const Spec2Axis *ax, *ay;        // by place
    const SpecPair<float> *tx, *ty;  // SPEC2_TENSOR: the two rows of the axis' 2 x 2 matrix, by place
    int K;
    float sign;                      // +1, or -1 for the adjoint
};

template <int MODE> __device__ __forceinline__ void spec2_coin(C2 (&v)[4], const C2 (&e)[4], C2 (&x)[4]) {
    // x = (E M v - M E* v) / 2; M v = (sum v) / 2 - v (flip-flop: of the swapped plane)
    constexpr int SW = MODE == QW_SHIFT_FLIPFLOP ? 1 : 0;
    C2 w[4], p;
    C2 s = cadd(cadd(v[0], v[1]), cadd(v[2], v[3]));
#pragma unroll
    for (int c = 0; c < 4; ++c) w[c] = conjmul(e[c], v[c]);
    const C2 q = cadd(cadd(w[0], w[1]), cadd(w[2], w[3]));
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const C2 m{0.5f * s.re - v[c ^ SW].re, 0.5f * s.im - v[c ^ SW].im};
        const C2 n{0.5f * q.re - w[c ^ SW].re, 0.5f * q.im - w[c ^ SW].im};
        p = cmul(e[c], m);
        x[c] = {0.5f * (p.re - n.re), 0.5f * (p.im - n.im)};
    }
}

// The coefficients of one momentum: e = E, and s_K and 2 s_{K/2}^2 (the same for
// ky and -ky).
struct Spec2Factor {
    float sK, f2;
};
// sin^2(w'/2) and the sign of s_K (see above)
template <int MODE> __device__ __forceinline__ Spec2Factor spec2_factor(const Spec2Coin &k, const Spec2Axis &X, const Spec2Axis &Y) {
    const ff one = ff_from(1.f), two = ff_from(2.f);
    ff u;          // sin^2(w'/2), w' = w or pi - w, in [0, pi/2]
    float sgn;     // s_K(w) = sgn s_K(w')   (K even)
    if constexpr (MODE == QW_SHIFT_DIAGONAL) {
        const bool nx = X.sh > X.ch, ny = Y.sh > Y.ch;   // cos kx, cos ky < 0
        const ff hx = nx ? ff{X.ch, X.cl} : ff{X.sh, X.sl}, hy = ny ? ff{Y.ch, Y.cl} : ff{Y.sh, Y.sl};
        u = hx + hy - two * (hx * hy);
        sgn = nx == ny ? -1.f : 1.f;
    } else {
        const bool neg = X.sh + Y.sh > 1.f;              // cos kx + cos ky < 0
        const ff hx = neg ? ff{X.ch, X.cl} : ff{X.sh, X.sl}, hy = neg ? ff{Y.ch, Y.cl} : ff{Y.sh, Y.sl};
        u = hx + hy;
        u = {0.5f * u.hi, 0.5f * u.lo};
        sgn = (MODE == QW_SHIFT_FLIPFLOP) == neg ? -1.f : 1.f;
    }
    const ff c = one - two * u, s2 = two * two * u * (one - u);   // cos w', sin^2 w'
    ff C = c, S = one;                                            // of n = 1
    const int m = k.K / 2;
    for (int bit = 30 - __clz(m); bit >= 0; --bit) {
        const ff C1 = two * (C * C) - one;
        S = two * (S * C);
        C = C1;
        if (m >> bit & 1) {
            const ff C2n = C * c - S * s2;
            S = S * c + C;
            C = C2n;
        }
    }
    return {k.sign * sgn * 2.f * (S * C).hi, 2.f * (S * S).hi};
}
// U^K v at the momentum (X, Y), or with flip at (kx, -ky)
template <int MODE>
__device__ __forceinline__ void spec2_apply(const Spec2Axis &X, const Spec2Axis &Y, bool flip, Spec2Factor f, C2 (&v)[4]) {
    C2 e[4];
    const float ys = flip ? -Y.s : Y.s;
    if constexpr (MODE == QW_SHIFT_DIAGONAL) {
        const bool nx = X.sh > X.ch, ny = Y.sh > Y.ch;
        const float hx = nx ? X.ch : X.sh, hy = ny ? Y.ch : Y.sh, gx = nx ? -1.f : 1.f, gy = ny ? -1.f : 1.f;
        const C2 ex{-2.f * gx * hx, -X.s}, ey{-2.f * gy * hy, -ys};   // e^{-ik} - (its sign at w' = 0)
        const C2 p = cmul(ex, ey), q = conjmul(ey, ex);               // ex ey, ex conj(ey)
        e[0] = {gx * ey.re + gy * ex.re + p.re, gx * ey.im + gy * ex.im + p.im};
        e[1] = {gx * ey.re + gy * ex.re + q.re, -gx * ey.im + gy * ex.im + q.im};
        e[2] = {e[1].re, -e[1].im};
        e[3] = {e[0].re, -e[0].im};
    } else {
        const bool neg = X.sh + Y.sh > 1.f;
        const float g = neg ? -1.f : 1.f;
        const float dir = MODE == QW_SHIFT_FLIPFLOP ? 1.f : -1.f;     // moving: D_0 = e^{-ikx}; flip-flop: e^{ikx}
        e[0] = {-2.f * g * (neg ? X.ch : X.sh), dir * X.s};
        e[1] = {e[0].re, -e[0].im};
        e[2] = {-2.f * g * (neg ? Y.ch : Y.sh), dir * ys};
        e[3] = {e[2].re, -e[2].im};
    }
    C2 x1[4], x2[4];
    spec2_coin<MODE>(v, e, x1);
    spec2_coin<MODE>(x1, e, x2);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = rfma(f.f2, x2[q], rfma(f.sK, x1[q], v[q]));
}
// H (x) H on the diagonal lattice
__device__ __forceinline__ void spec2_tensor(const Spec2Coin &k, int px, int py, C2 (&v)[4]) {
    const SpecPair<float> a0 = k.tx[2 * px], a1 = k.tx[2 * px + 1], b0 = k.ty[2 * py], b1 = k.ty[2 * py + 1];
    C2 u[4];   // coin c = 2 j + k: j moves in x, k in y
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        u[q] = cfma(a0.b, v[2 + q], cmul(a0.a, v[q]));
        u[2 + q] = cfma(a1.b, v[2 + q], cmul(a1.a, v[q]));
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        v[2 * j] = cfma(b0.b, u[2 * j + 1], cmul(b0.a, u[2 * j]));
        v[2 * j + 1] = cfma(b1.b, u[2 * j + 1], cmul(b1.a, u[2 * j]));
    }
}

// columns per CTA: four where they fit, so that a warp's loads are whole sectors
template <int L> constexpr int spec2_cols() { return L >= 12 ? 1 : (L == 11 ? 2 : 4); }
template <int L> constexpr int spec2_col_stride() { return 4 * ((1 << L) * 17 / 16) + 4; }   // (4 mod 16: no bank conflicts)
template <int L> constexpr size_t spec2_col_smem() { return (size_t)spec2_cols<L>() * spec2_col_stride<L>() * sizeof(S2); }

template <int L, int MODE>
__global__ void __launch_bounds__(spec2_cols<L>() * 4 * (1 << L) / 16)
k_spec2_columns(Spec2Args a, Spec2Coin coin) {
    constexpr int N = 1 << L, TH = N / 16, C = spec2_cols<L>(), PL = N * 17 / 16;
    extern __shared__ __align__(16) unsigned char ssm[];
    S2 *all = reinterpret_cast<S2 *>(ssm);
    const int col = (int)threadIdx.x % C, t = (int)threadIdx.x / C % TH, c = (int)threadIdx.x / C / TH;
    S2 *sm = all + col * spec2_col_stride<L>() + c * PL;
    const int NX = 1 << a.LX, per = NX / C;
    const int bl = (int)(blockIdx.x / per), p0 = (int)(blockIdx.x % per) * C;
    S2 *z = a.z + ((int64_t)bl * 4 + c) * N * NX + p0 + col;
    C2 x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) { const S2 v = z[(int64_t)(t + i * TH) * NX]; x[i] = {v.re, v.im}; }
    spec2_forward<L>(x, sm, a.tw, t);
    __syncthreads();
    auto get = [&](int k, int p, C2 (&v)[4]) {
        const S2 *m = all + k * spec2_col_stride<L>() + spec2_at(p);
#pragma unroll
        for (int d = 0; d < 4; ++d) v[d] = {m[d * PL].re, m[d * PL].im};
    };
    auto put = [&](int k, int p, const C2 (&v)[4]) {
        S2 *m = all + k * spec2_col_stride<L>() + spec2_at(p);
#pragma unroll
        for (int d = 0; d < 4; ++d) m[d * PL] = {v[d].re, v[d].im};
    };
    const int odd = a.split ? a.b0 + bl : 0;             // the odd momenta of a split axis
    if constexpr (MODE == SPEC2_TENSOR) {
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
            const int id = (int)threadIdx.x + q * (4 * C * TH), k = id % C, p = id / C;
            C2 v[4];
            get(k, p, v);
            spec2_tensor(coin, p0 + k, odd * N + p, v);
            put(k, p, v);
        }
    } else {
        // the pairs ky, -ky share their factors: one of each pair has the last
        // digit of its place in the lower half; f = 0 and N / 2 are their own
        // partners (of the odd momenta, 2f + 1, none is)
        constexpr int R = L % 4 ? 1 << (L % 4) : 16, H = R / 2;
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
            const int id = (int)threadIdx.x + q * (4 * C * TH), k = id % C, h = id / C, p = h / H * R + h % H;
            const int f = spec2_freq(L, p), g = odd ? N - 1 - f : (N - f) % N;
            const int p2 = f == 0 && !odd ? spec2_place(L, N / 2) : spec2_place(L, g);
            const Spec2Axis X = coin.ax[p0 + k], Y = coin.ay[odd * N + p];
            const Spec2Factor fac = spec2_factor<MODE>(coin, X, Y);
            C2 v[4];
            get(k, p, v);
            spec2_apply<MODE>(X, Y, false, fac, v);
            put(k, p, v);
            get(k, p2, v);
            if (f == 0 && !odd) {
                const Spec2Axis Z = coin.ay[p2];
                spec2_apply<MODE>(X, Z, false, spec2_factor<MODE>(coin, X, Z), v);
            } else {
                spec2_apply<MODE>(X, Y, true, fac, v);
            }
            put(k, p2, v);
        }
    }
    __syncthreads();
    if constexpr (L >= 10) spec_reload(z);   // (shorter columns have the registers)
    spec2_inverse<L>(x, sm, a.tw, t);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int r = t + i * TH;
        if (r >= a.hy && r < a.hy + a.wy) z[(int64_t)r * NX] = {x[i].re, x[i].im};
    }
}

}  // namespace qw
