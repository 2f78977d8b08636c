// k_window1d.cuh -- K generic forward steps of the 1D walk per launch: the segment
// and the line of Sec. 3, broken links, on the whole lattice or on the
// computation window of a localised walk (a walker started at MP steps only the
// sites [l_i, r_i] its light cone has reached).
//
// The 1D form of k_tile2d.cuh: a CTA keeps E sites in shared memory, in the
// walk's storage format, updates them in place for K steps (an amplitude stays
// in its slot while the lattice moves under it; a closed link swaps two slots)
// and writes the E - 2K sites whose light cone lies inside.  Every step applies
// the full coin row, the step's drift gain and the step's link draws, whatever
// the window, so clipped and full steps agree bit for bit.
//
// One step per launch of the whole lattice costs its round trip through HBM, and
// one CTA for a whole window is bound by one SM's issue (0.58 us per step for
// windows of up to 2049 sites); tiles of 256 sites spread a window over many SMs.
#pragma once
#include "k_generic.cuh"

namespace qw {

// drift gains of the launch's steps, in the compute real
template <class R>
struct WinGains {
    R v[WINDOW_MAX_STEPS];
};

// Slot of plane p at step t, as tile_slot of the 2D tiles: coin 0 moves to
// x - 1, coin 1 to x + 1.
template <int SH> __device__ __forceinline__ void win_slot(int p, int t, int &track, int &dx) {
    const int e = p == 0 ? -1 : 1;
    if (SH == QW_SHIFT_FLIPFLOP) {
        const int odd = t & 1;
        track = p ^ odd;
        dx = odd ? e : 0;
    } else {
        track = p;
        dx = -t * e;
    }
}

// Outputs: [o0, o0 + ow) modulo g.nx.
template <int P, int SH, int CK, int E, int TH>
__global__ void __launch_bounds__(TH)
k_step1d_window(View in, View out, GenGeom g, CoinP<typename St<P>::real> cp,
                const Cx<typename St<P>::real> *__restrict__ coins, int o0, int ow, int K,
                WinGains<typename St<P>::real> gains) {
    using S = St<P>;
    using real = typename S::real;
    using C = Cx<real>;
    constexpr int NS = E / TH, M = E - 1;
    static_assert(NS * TH == E && (E & M) == 0, "tile shape");
    extern __shared__ __align__(16) unsigned char wsm[];
    const View sv{wsm, E, 2};
    const int n = (int)g.nx, O = E - 2 * K;                     // n < 2^30 (launcher)
    const int b = (int)blockIdx.x * O - K;                      // tile site i is output b + i
    auto site = [&](int i) {
        int64_t x = (int64_t)o0 + b + i;                        // in [-K, 2n + E)
        if (n < E) { x %= n; return (int)(x < 0 ? x + n : x); }
        if (x < 0) x += n;
        if (x >= n) x -= n;
        return (int)(x >= n ? x - n : x);
    };
    C m[CK == CK_PERSITE ? NS : 1][4];
    unsigned char fixed[NS];
    PhiloxSite rnd[NS];
    int any = 0;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const int i = (int)threadIdx.x + k * TH, x = site(i);
#pragma unroll
        for (int c = 0; c < 2; ++c) S::st(sv, c, i, S::ld(in, c, x));
        if constexpr (CK == CK_PERSITE) {
#pragma unroll
            for (int e = 0; e < 4; ++e) m[k][e] = coins[4 * (int64_t)x + e];
        }
        fixed[k] = link_state(g, 0, x, 0, 0xffffffffu);
        any |= fixed[k];
        rnd[k] = philox_site((uint32_t)x, g.rk1);
    }
    // does any link of the tile ever close (or absorb)?
    const bool settle = __syncthreads_or(any) || g.rthr;
    for (int t = 0; t < K; ++t) {
        const real gain = gains.v[t];
        const bool one = is_one(gain);
        int st[NS];
        PhiloxStep ps;
        if (g.rthr) ps = philox_step(g.rstep + (uint32_t)t, g.rk0, g.rk1);
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const int i = (int)threadIdx.x + k * TH;
            int t0, d0, t1, d1;
            win_slot<SH>(0, t, t0, d0);
            win_slot<SH>(1, t, t1, d1);
            const int s0 = (i + d0) & M, s1 = (i + d1) & M;
            const C a0 = S::ld(sv, t0, s0), a1 = S::ld(sv, t1, s1);
            C v0, v1;
            if constexpr (CK == CK_REAL) {   // (the full row's products with its zero imaginary parts left out)
                v0 = rfma(cp.re[1], a1, rfma(cp.re[0], a0, czero<real>()));
                v1 = rfma(cp.re[3], a1, rfma(cp.re[2], a0, czero<real>()));
            } else {
                auto entry = [&](int e) { return CK == CK_PERSITE ? m[CK == CK_PERSITE ? k : 0][e] : C{cp.re[e], cp.im[e]}; };
                v0 = cfma(entry(1), a1, cfma(entry(0), a0, czero<real>()));
                v1 = cfma(entry(3), a1, cfma(entry(2), a0, czero<real>()));
            }
            if (!one) { v0 = rmul(gain, v0); v1 = rmul(gain, v1); }
            S::st(sv, t0, s0, v0);
            S::st(sv, t1, s1, v1);
            st[k] = fixed[k];
            if (g.rthr && philox_draw(rnd[k], ps, g.rk0, g.rk1).x < g.rthr) st[k] = 1;
        }
        __syncthreads();
        // each site settles the link to its right neighbour
        if (settle) {
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (!st[k]) continue;
                const int i = (int)threadIdx.x + k * TH;
                int t1, d1, t0, d0;
                win_slot<SH>(1, t, t1, d1);
                win_slot<SH>(0, t, t0, d0);
                const int q = (i + d1) & M, r = (i + 1 + d0) & M;
                const C u = st[k] == 1 ? S::ld(sv, t1, q) : czero<real>(), w = st[k] == 1 ? S::ld(sv, t0, r) : czero<real>();
                S::st(sv, t1, q, w);
                S::st(sv, t0, r, u);
            }
            __syncthreads();
        }
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const int i = (int)threadIdx.x + k * TH;
        if (i < K || i >= E - K || b + i >= ow) continue;
        const int x = site(i);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            int tr, d;
            win_slot<SH>(c, K, tr, d);
            S::st(out, c, x, S::ld(sv, tr, (i + d) & M));
        }
    }
}

}  // namespace qw
