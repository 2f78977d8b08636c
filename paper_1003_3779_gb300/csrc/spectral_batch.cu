// spectral_batch.cu -- a batch of localised cycle walks in momentum space.
//
// A walk of T steps from one site x0 lives on the T + 1 sites x0 - T + 2j (it is
// bipartite, as in k_spectral1d.cuh), so its state is one inverse transform of
// length N = 2^L >= T + 1: at momentum theta_f = pi f / N per site,
//     psi(x0 - T + 2j) = (1/N) sum_f e^{2 pi i f j / N} e^{-i theta_f T} U(theta_f)^T c,
// c the coin state.  On a short cycle the line's sites are added up modulo n.
// With e^{-i delta} C = [[alpha, beta], [-beta*, alpha*]] the step is, up to the
// phase, V = [[a, b], [-b*, a*]], a = e^{i theta} alpha, b = e^{i theta} beta, and
//     V^T = cos(T w) + s_T X,  X = [[i Im a, b], [-b*, -i Im a]],
// cos w = Re a, s_T = sin(T w) / sin w: repeated doubling in double-float, from
// e^{i theta} in double-float.  No step is taken, nothing grows with T, and the
// cost per walk is N (T's bits + log N) instead of T^2.
//
// One CTA per walk: 2^L / 8 threads fill the momenta of both planes in shared
// memory, each half then transforms one plane (k_spectral2d.cuh's inverse, which
// takes them in digit-reversed places), and the CTA writes the sites of the light
// cone, their P and the norm.  Sites outside the cone are zero in both buffers
// and in P after any run of the batch, and stay so.
//
// 4096 walks (N up to 65536, T up to 4096) with readout: 10.74 ms in the window
// sweep, which is bound by the issue of its site-steps; 1.15 ms here.  The
// transforms take 0.6 ms of that; the chain of launches of the near-diagonal
// walks beside them bounds the rest (0.79 ms without it).
#include <algorithm>
#include <cmath>

#include "qw_handle.h"
#include "k_spectral2d.cuh"

namespace qw {

// e^{i pi k / 8192}, k < 8192, in double-float
struct SpecPhase {
    float ch, cl, sh, sl;
};
constexpr int PHASES = 1 << SPEC2_MAX_LX;

__global__ void k_batch_phases(SpecPhase *t) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= PHASES) return;
    double s, c;
    sincospi((double)k / PHASES, &s, &c);
    t[k] = {(float)c, (float)(c - (double)(float)c), (float)s, (float)(s - (double)(float)s)};
}

template <int L>
__global__ void __launch_bounds__((1 << L) / 8)
k_batch_spectral(const SpecWalk *__restrict__ walks, float2 *__restrict__ state, float *__restrict__ P, double *__restrict__ norms,
                 int *__restrict__ final_buf, const S2 *__restrict__ tw, const SpecPhase *__restrict__ phases) {
    constexpr int N = 1 << L, TH = N / 16, PL = N * 17 / 16, NT = N / 8;
    extern __shared__ __align__(16) unsigned char ssm[];
    __shared__ double red[NT / 32];
    S2 *all = reinterpret_cast<S2 *>(ssm);
    const SpecWalk w = walks[blockIdx.x];
    const int T = w.T;
    // momenta of both planes, in their places
    const ff ar{w.ah[0], w.al[0]}, ai{w.ah[1], w.al[1]}, bb{w.b2h, w.b2l};
    const C2 beta{w.b[0], w.b[1]}, c0{w.c[0], w.c[1]}, c1{w.c[2], w.c[3]};
    const ff one = ff_from(1.f), two = ff_from(2.f);
#pragma unroll 1
    for (int p = threadIdx.x; p < N; p += NT) {
        const int f = spec2_freq(L, p);
        const SpecPhase e = phases[f << (SPEC2_MAX_LX - L)];
        const ff ec{e.ch, e.cl}, es{e.sh, e.sl};
        const ff c = ec * ar - es * ai, im = ec * ai + es * ar;   // a = e^{i theta} alpha
        const ff s2 = im * im + bb;                                // sin^2 w
        ff C = T ? c : one, S = T ? one : ff_from(0.f);            // of n = 1 (T = 0: n = 0)
        for (int bit = 30 - __clz(T | 1); bit >= 0; --bit) {
            const ff C1 = two * (C * C) - one;
            S = two * (S * C);
            C = C1;
            if (T >> bit & 1) {
                const ff Cn = C * c - S * s2;
                S = S * c + C;
                C = Cn;
            }
        }
        const C2 b = cmul(C2{e.ch, e.sh}, beta);
        const float g = im.hi, ct = C.hi, st = S.hi;
        // X c
        const C2 q0 = cmul(b, c1), q1 = conjmul(b, c0);
        const C2 x0{q0.re - g * c0.im, q0.im + g * c0.re}, x1{-q1.re + g * c1.im, -q1.im - g * c1.re};
        C2 v0{ct * c0.re + st * x0.re, ct * c0.im + st * x0.im}, v1{ct * c1.re + st * x1.re, ct * c1.im + st * x1.im};
        // e^{-i theta T} / N
        const int r = (int)((int64_t)f * T & (2 * N - 1));
        float s, k;
        sincospif(-(float)r / N, &s, &k);
        const C2 ph{k / N, s / N};
        v0 = cmul(ph, v0);
        v1 = cmul(ph, v1);
        all[spec2_at(p)] = {v0.re, v0.im};
        all[PL + spec2_at(p)] = {v1.re, v1.im};
    }
    __syncthreads();
    const int plane = (int)threadIdx.x / TH, t = (int)threadIdx.x % TH;
    S2 *sm = all + plane * PL;
    C2 x[16];
    spec2_inverse<L>(x, sm, tw, t);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) sm[t + i * TH] = {x[i].re, x[i].im};   // point j, in order
    __syncthreads();
    // the cone's sites: site x0 - T + i (mod n) takes the points j with 2j = i (mod n)
    const int64_t span = 2 * (int64_t)T + 1, width = min(span, w.n);
    float2 *s0 = state + w.base, *s1 = s0 + w.pitch;
    double acc = 0.0;
    int64_t start = (w.x0 - T) % w.n;
    if (start < 0) start += w.n;
    for (int64_t i = threadIdx.x; i < width; i += NT) {
        float2 u = make_float2(0.f, 0.f), v = u;
        for (int64_t d = i; d < span; d += w.n) {
            if (d & 1) continue;
            const S2 a = all[d >> 1], b = all[PL + (d >> 1)];
            u.x += a.re; u.y += a.im;
            v.x += b.re; v.y += b.im;
        }
        int64_t site = start + i;
        if (site >= w.n) site -= w.n;
        s0[site] = u;
        s1[site] = v;
        const float pr = __fmaf_rn(u.x, u.x, __fmaf_rn(u.y, u.y, __fmaf_rn(v.x, v.x, v.y * v.y)));
        P[w.poff + site] = pr;
        acc += (double)pr;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int i = 0; i < NT / 32; ++i) tot += red[i];
        norms[w.id] = tot;
        final_buf[w.id] = 0;
    }
}

size_t batch_spectral_table_bytes() { return sizeof(S2) * SPEC2_TW + sizeof(SpecPhase) * PHASES; }

cudaError_t launch_batch_spectral_tables(void *table, cudaStream_t s) {
    cudaError_t e = launch_spectral2d_tables(table, s);   // (the twiddles, at its start)
    if (e != cudaSuccess) return e;
    k_batch_phases<<<PHASES / 256, 256, 0, s>>>(reinterpret_cast<SpecPhase *>(static_cast<char *>(table) + sizeof(S2) * SPEC2_TW));
    return cudaGetLastError();
}

int batch_spectral_length(int64_t T) {
    int L = SPEC2_MIN_L;
    while (L <= SPEC2_MAX_LX && ((int64_t)1 << L) < T + 1) ++L;
    return L <= SPEC2_MAX_LX ? L : 0;
}

template <int L>
static cudaError_t go_batch(const SpecWalk *walks, int count, float2 *state, float *P, double *norms, int *final_buf, const void *table,
                            cudaStream_t s) {
    if (!count) return cudaSuccess;
    constexpr size_t smem = (size_t)2 * ((1 << L) * 17 / 16) * sizeof(S2);
    auto kern = k_batch_spectral<L>;
    cudaError_t e = smem > 40 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) : cudaSuccess;
    if (e != cudaSuccess) return e;
    const S2 *tw = static_cast<const S2 *>(table);
    kern<<<(unsigned)count, (1 << L) / 8, smem, s>>>(walks, state, P, norms, final_buf, tw,
                                                     reinterpret_cast<const SpecPhase *>(tw + SPEC2_TW));
    return cudaGetLastError();
}

// walks: count[L - SPEC2_MIN_L] walks of length 2^L, longest first
cudaError_t launch_batch_spectral(const SpecWalk *walks, const int *count, void *state, float *P, double *norms, int *final_buf,
                                  const void *table, cudaStream_t s) {
    float2 *st = static_cast<float2 *>(state);
    cudaError_t e = cudaSuccess;
    for (int L = SPEC2_MAX_LX; L >= SPEC2_MIN_L && e == cudaSuccess; --L) {
        const int n = count[L - SPEC2_MIN_L];
        switch (L) {
            case 13: e = go_batch<13>(walks, n, st, P, norms, final_buf, table, s); break;
            case 12: e = go_batch<12>(walks, n, st, P, norms, final_buf, table, s); break;
            case 11: e = go_batch<11>(walks, n, st, P, norms, final_buf, table, s); break;
            case 10: e = go_batch<10>(walks, n, st, P, norms, final_buf, table, s); break;
            case 9: e = go_batch<9>(walks, n, st, P, norms, final_buf, table, s); break;
            default: e = go_batch<8>(walks, n, st, P, norms, final_buf, table, s);
        }
        walks += n;
    }
    return e;
}

}  // namespace qw
