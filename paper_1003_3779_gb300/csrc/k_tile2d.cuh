// k_tile2d.cuh -- K steps of the 2D walk per launch, a tile of the lattice in the
// shared memory of one CTA: for small lattices and light-cone windows, per-site
// phase coins, broken links and boundaries.
//
// The step is U = S (I (x) C) of Sec. 2.1 on the torus, the segment or the line
// (Sec. 3).  A CTA loads EX x EY sites, applies K steps and writes the
// (EX - 2K) x (EY - 2K) sites in the middle, whose light cone lies inside the
// tile.  The state is updated in place, with one barrier per step: an amplitude
// stays in its slot and the lattice moves under it.  With the moving shift,
// plane c of site x at step t lies in slot x - t e_c of track c; the coin at x
// reads its four slots and writes its four results back into them, and the
// shift is the change of t.  (Flip-flop: phi_c of x arrives at x + e_c in plane
// c xor 1, so at odd t plane p of x lies in track p xor 1, slot x + e_p, and at
// even t in track p, slot x.)  Slots are taken modulo the tile, so every slot
// belongs to one site at each step; what wraps round is garbage that never
// reaches the output.
//
// Links (Sec. 3, RBL): a closed link between x and x + e_c exchanges the
// destinations of phi_c(x) and phi_{c xor 1}(x + e_c), whatever the shift, so
// after the coins (and a second barrier) each site swaps the two slots of its
// own +x and +y links where they are closed, and zeroes them on an absorbing
// edge.  Nothing is drawn or decided twice.
//
// Why a tile: a launch per step costs 4 to 8 us whatever the lattice, and per
// step re-reads the state, the phases (and their sines) and re-draws halo
// links; here a site's phase factors stay in registers for K steps.  What
// bounds it: shared memory, 64 bytes per site and step (two sites per clock and
// SM), or the issue of the draws.
#pragma once
#include "qw_internal.cuh"
#include "k_generic.cuh"
#include "k_step2d.cuh"

namespace qw {

// Offset of the slot of plane p at step t from the site, and its track.
template <int SH> __device__ __forceinline__ void tile_slot(int p, int t, int &track, int &dx, int &dy) {
    if (SH == QW_SHIFT_FLIPFLOP) {
        const int odd = t & 1;
        track = p ^ odd;
        dx = odd ? dir_dx<SH>(p) : 0;
        dy = odd ? dir_dy<SH>(p) : 0;
    } else {
        track = p;
        dx = -t * dir_dx<SH>(p);
        dy = -t * dir_dy<SH>(p);
    }
}

// PH: per-site phase factors before the coin CK.
template <int P, int SH, int CK, bool PH, bool LINKS, int EX, int EY, int TH>
__global__ void __launch_bounds__(TH)
k_tile2d(View in, View out, GenGeom g, int64_t ox0, int64_t ow, int64_t oy0, int64_t oh, int K,
         CoinP<typename St<P>::real> cp, const float *__restrict__ phi, typename St<P>::real gain) {
    using S = St<P>;
    using real = typename S::real;
    using C = Cx<real>;
    struct alignas(2 * sizeof(real)) Slot { real re, im; };
    constexpr int NS = EX * EY / TH;            // sites per thread
    static_assert(NS * TH == EX * EY && (EX & (EX - 1)) == 0 && (EY & (EY - 1)) == 0 && TH % EX == 0, "tile shape");
    extern __shared__ __align__(16) unsigned char tsm[];
    Slot *sm = reinterpret_cast<Slot *>(tsm);   // [track][y][x]
    const int TX = EX - 2 * K, TY = EY - 2 * K;
    // the tile's first site (wrapped); its site (i, j) is lattice site (x0 + i, y0 + j)
    const int64_t bx = (int64_t)blockIdx.x * TX, by = (int64_t)blockIdx.y * TY;
    auto wrap = [](int64_t a, int64_t n, int e) {   // a is at most one period outside [0, n) where n >= e
        if (n < e) a %= n;
        return a < 0 ? a + n : (a >= n ? a - n : a);
    };
    const int64_t x0 = wrap(ox0 + bx - K, g.nx, EX), y0 = wrap(oy0 + by - K, g.ny, EY);
    const int i = (int)threadIdx.x % EX, j0 = (int)threadIdx.x / EX;   // site n of this thread: (i, j0 + n TH / EX)
    constexpr int DJ = TH / EX;
    int64_t gx = x0 + i;
    if (gx >= g.nx) gx = g.nx >= EX ? gx - g.nx : gx % g.nx;
    auto row = [&](int j) {
        int64_t y = y0 + j;
        if (y >= g.ny) y = g.ny >= EY ? y - g.ny : y % g.ny;
        return y;
    };
    SiteCoin<real> sc[PH ? NS : 1];
    unsigned char fixed[LINKS ? NS : 1];        // links closed or absorbing at every step
    PhiloxSite rnd[LINKS ? NS : 1];
    int any = 0;
#pragma unroll
    for (int n = 0; n < NS; ++n) {
        const int j = j0 + n * DJ;
        const int64_t gy = row(j), v = gy * g.nx + gx;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const C a = S::ld(in, c, v);
            sm[(c * EY + j) * EX + i] = {a.re, a.im};
        }
        if constexpr (PH) phase_of(phi, v, sc[n]);
        if constexpr (LINKS) {
            fixed[n] = (unsigned char)(link_state(g, 0, (int)gx, (int)gy, 0xffffffffu) |
                                       (link_state(g, 1, (int)gx, (int)gy, 0xffffffffu) << 2));
            any |= fixed[n];
            rnd[n] = philox_site((uint32_t)v, g.rk1);
        }
    }
    // does any link of the tile ever close (or absorb)?
    const bool settle = __syncthreads_or(any) || (LINKS && g.rthr);
    // slot of plane c of site (i, j) at step t
    auto slot = [&](int c, int t, int si, int sj) {
        int tr, dx, dy;
        tile_slot<SH>(c, t, tr, dx, dy);
        return (tr * EY + ((sj + dy) & (EY - 1))) * EX + ((si + dx) & (EX - 1));
    };
    auto coin = [&](int n, C (&a)[4], C (&p)[4]) {
        if constexpr (PH) {
#pragma unroll
            for (int c = 0; c < 4; ++c) a[c] = cmul(sc[n].e[c], a[c]);
        }
        coin4<CK, real>(cp, (const C *)nullptr, sc[0], a, p);
    };
    for (int t = 0; t < K; ++t) {
        unsigned st[LINKS ? NS : 1];
        PhiloxStep ps;
        if (LINKS && g.rthr) ps = philox_step(g.rstep + (uint32_t)t, g.rk0, g.rk1);
#pragma unroll
        for (int n = 0; n < NS; ++n) {
            const int j = j0 + n * DJ;
            C a[4], p[4];
            int at[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                at[c] = slot(c, t, i, j);
                const Slot s = sm[at[c]];
                a[c] = {s.re, s.im};
            }
            coin(n, a, p);
#pragma unroll
            for (int c = 0; c < 4; ++c) sm[at[c]] = {p[c].re, p[c].im};
            if constexpr (LINKS) {
                st[n] = fixed[n];
                if (g.rthr) {   // broken at random at this step: closed, whatever the boundary says
                    const uint2 w = philox_draw(rnd[n], ps, g.rk0, g.rk1);
                    if (w.x < g.rthr) st[n] = (st[n] & ~3u) | 1u;
                    if (w.y < g.rthr) st[n] = (st[n] & ~12u) | 4u;
                }
            }
        }
        if constexpr (LINKS) {
            // a site settles its +x and +y links: what each end sends across one
            // that is closed changes places, and is lost on an absorbing one
            if (settle) __syncthreads();
#pragma unroll
            for (int n = 0; n < NS; ++n) {
                const int j = j0 + n * DJ;
                if (!settle) break;
#pragma unroll
                for (int axis = 0; axis < 2; ++axis) {
                    const unsigned s = st[n] >> (2 * axis) & 3u;
                    if (!s) continue;
                    Slot *q = sm + slot(2 * axis, t, i, j);
                    Slot *r = sm + slot(2 * axis + 1, t, i + (axis == 0), j + axis);
                    const Slot u = s == 1 ? *q : Slot{0, 0}, v = s == 1 ? *r : Slot{0, 0};
                    *q = v;
                    *r = u;
                }
            }
        }
        __syncthreads();
    }
    if (i < K || i >= EX - K || bx + i - K >= ow) return;
#pragma unroll
    for (int n = 0; n < NS; ++n) {
        const int j = j0 + n * DJ;
        if (j < K || j >= EY - K || by + j - K >= oh) continue;
        const int64_t v = row(j) * g.nx + gx;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const Slot s = sm[slot(c, K, i, j)];
            C a{s.re, s.im};
            if (!is_one(gain)) a = rmul(gain, a);
            S::st(out, c, v, a);
        }
    }
}

}  // namespace qw
