// launch_step.cuh -- host-side launch of the step kernels for one precision.
// Included once per precision by step_<prec>.cu so the template instances of
// each precision compile in their own translation unit (in parallel).
#pragma once
#include "qw_internal.cuh"
#include "k_step1d.cuh"
#include "k_step2d.cuh"
#include "k_generic.cuh"
#include "k_window1d.cuh"

#include <algorithm>

namespace qw {

// Sites per lane compiled for the 1D kernel: two forward tiles, and the
// default tile used by the per-site coin and the adjoint.
template <int P> struct Tiles1D;
template <> struct Tiles1D<P_F32> { static constexpr int A = 8, B = 16, DEF = 16; };
template <> struct Tiles1D<P_BF16> { static constexpr int A = 8, B = 16, DEF = 16; };
template <> struct Tiles1D<P_F64> { static constexpr int A = 4, B = 8, DEF = 8; };
template <> struct Tiles1D<P_COMP> { static constexpr int A = 4, B = 8, DEF = 4; };

// Sites per lane of the 2D kernel (32 bytes of one plane per lane).
template <int P> struct Tile2D { static constexpr int R = 32 / St<P>::SLOT_BYTES < 1 ? 1 : 32 / St<P>::SLOT_BYTES; };
template <> struct Tile2D<P_COMP> { static constexpr int R = 4; };

// A third, short tile for narrow light-cone windows: an FP64 warp gets half a
// lane a clock from its scheduler, so a window runs faster on many short tiles
// (2001-site Hadamard cycle from one site, T = 1000: tiles of 8 sites per lane in
// blocks of four warps 2.3 ms, of 4 sites in blocks of one 0.82 ms, of 2 sites 0.59).
template <int P> struct WindowTile1D { static constexpr int R = 0; };
template <> struct WindowTile1D<P_F64> { static constexpr int R = 2; };

template <int P, int CK, int FF, int ADJ>
static void go1d_k1(const Step1DArgs &a, const CoinP<typename St<P>::real> &cp, cudaStream_t s) {
    using real = typename St<P>::real;
    const int64_t nwarps = (a.n + 32 * St<P>::VEC - 1) / (32 * St<P>::VEC);
    const int64_t blocks = (nwarps + 7) / 8;
    k_step1d_k1<P, CK, FF, ADJ><<<(unsigned)blocks, 256, 0, s>>>(
        a.in, a.out, a.n, nwarps, cp, static_cast<const Cx<real> *>(a.coins),
        real_from_double<real>(a.pre0), real_from_double<real>(a.pre1),
        real_from_double<real>(a.post0), real_from_double<real>(a.post1));
}

template <int P, int ADJ>
static bool go1d_k1_kind(const Step1DArgs &a, const CoinP<typename St<P>::real> &cp, cudaStream_t s) {
    const bool ff = a.shift == QW_SHIFT_FLIPFLOP;
    switch (a.kind) {
        case CK_REAL: ff ? go1d_k1<P, CK_REAL, 1, ADJ>(a, cp, s) : go1d_k1<P, CK_REAL, 0, ADJ>(a, cp, s); return true;
        case CK_COMPLEX: ff ? go1d_k1<P, CK_COMPLEX, 1, ADJ>(a, cp, s) : go1d_k1<P, CK_COMPLEX, 0, ADJ>(a, cp, s); return true;
        case CK_PERSITE: ff ? go1d_k1<P, CK_PERSITE, 1, ADJ>(a, cp, s) : go1d_k1<P, CK_PERSITE, 0, ADJ>(a, cp, s); return true;
        case CK_SIGN_P: if (ff) return false; go1d_k1<P, CK_SIGN_P, 0, ADJ>(a, cp, s); return true;
        case CK_SIGN_M: if (ff) return false; go1d_k1<P, CK_SIGN_M, 0, ADJ>(a, cp, s); return true;
        default: return false;
    }
}

// Outputs per warp of the temporal-blocking kernel: a multiple of VEC with
// 32R >= W + 2K + VEC - 1 (the tile origin is rounded down to VEC).
template <int P>
inline int64_t outputs_per_warp(int R, int K) {
    constexpr int V = St<P>::VEC;
    return (32LL * R - 2LL * K - (V - 1)) / V * V;
}

// The tiles that take factors between their steps (Step1DArgs::per): the widest of
// FP32 and bf16 storage and FP64's short one, for the coins that have factors.
template <int P> constexpr bool joins_1d(int R, int kind) {
    return (kind == CK_SIGN_P || kind == CK_SIGN_M) && (P == P_F64 ? R == WindowTile1D<P>::R : (P != P_COMP && R == Tiles1D<P>::B));
}

template <int P, int R, int CK, int FF, int ADJ>
static void go1d(const Step1DArgs &a, const CoinP<typename St<P>::real> &cp, cudaStream_t s) {
    const int64_t W = outputs_per_warp<P>(R, a.K);
    const bool win = a.oend > a.obeg;   // a light-cone window, else the whole cycle
    const int64_t ob = win ? a.obeg : 0, oe = win ? a.oend : a.n;
    const int64_t nwarps = (oe - ob + W - 1) / W;
    // a window of few tiles: one warp per block, so that each has a scheduler of
    // its own
    const int wpb = win && nwarps <= 4 * 152 ? 1 : 4;
    const int64_t blocks = (nwarps + wpb - 1) / wpb;
    auto kern = k_step1d<P, R, CK, FF, ADJ, false>;
    if constexpr (joins_1d<P>(R, CK)) {
        if (a.per) kern = k_step1d<P, R, CK, FF, ADJ, true>;
    }
    kern<<<(unsigned)blocks, 32 * wpb, 0, s>>>(
        a.in, a.out, a.n, a.K, W, ob, oe, nwarps, cp,
        static_cast<const Cx<typename St<P>::real> *>(a.coins),
        real_from_double<typename St<P>::real>(a.pre0), real_from_double<typename St<P>::real>(a.pre1),
        real_from_double<typename St<P>::real>(a.post0), real_from_double<typename St<P>::real>(a.post1),
        a.per, real_from_double<typename St<P>::real>(a.mid));
}

template <int P, int R, int ADJ>
static bool go1d_kind(const Step1DArgs &a, const CoinP<typename St<P>::real> &cp, cudaStream_t s) {
    const bool ff = a.shift == QW_SHIFT_FLIPFLOP;
    switch (a.kind) {
        case CK_REAL: ff ? go1d<P, R, CK_REAL, 1, ADJ>(a, cp, s) : go1d<P, R, CK_REAL, 0, ADJ>(a, cp, s); return true;
        case CK_COMPLEX: ff ? go1d<P, R, CK_COMPLEX, 1, ADJ>(a, cp, s) : go1d<P, R, CK_COMPLEX, 0, ADJ>(a, cp, s); return true;
        case CK_SIGN_P: if (ff) return false; go1d<P, R, CK_SIGN_P, 0, ADJ>(a, cp, s); return true;
        case CK_SIGN_M: if (ff) return false; go1d<P, R, CK_SIGN_M, 0, ADJ>(a, cp, s); return true;
        default: return false;
    }
}

// Sites per lane compiled for the sweep kernel (R * SLOT_BYTES / 16 = 2..16
// sixteen-byte units per lane and plane); the double-float form has none.
// The larger tile halves the per-level overhead (edge hand-over, shuffles)
// per site and allows deeper k; the smaller one takes cycles that are a
// multiple of half its chunk.
template <int P> struct SweepTiles { static constexpr int A = 16, B = 32; };
template <> struct SweepTiles<P_F64> { static constexpr int A = 8, B = 8; };
template <> struct SweepTiles<P_COMP> { static constexpr int A = 0, B = 0; };

// The sites per lane a sweep plan with this tile runs on a cycle of n sites:
// the requested tile if it is compiled, else the larger tile when the cycle
// holds at least two of its chunks, else the smaller one.
template <int P>
int sweep_tile(int64_t n, int tile) {
    using T = SweepTiles<P>;
    if constexpr (T::A == 0) {
        return 0;
    } else {
        if (tile == T::A || tile == T::B) return tile;
        return n >= 2 * 32LL * T::B ? T::B : T::A;
    }
}

template <int P, int R, int CK, int FF, int ADJ>
static cudaError_t go1d_sweep(const Step1DArgs &a, const CoinP<typename St<P>::real> &cp, cudaStream_t s) {
    using real = typename St<P>::real;
    using SW = Sweep<P, R>;
    constexpr int warps = 4;
    const size_t smem = warps * SW::warp_bytes(a.K);
    auto kfn = k_step1d_sweep<P, R, CK, FF, ADJ>;
    cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // Segments sized so that the whole launch is one wave of resident warps:
    // every warp sweeps about the same number of chunks, and the one warm-up
    // chunk per segment is a small fraction of it.
    int nch = a.chunks;
    if (nch <= 0) {
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, 32 * warps, smem);
        const int64_t resident = (int64_t)std::max(1, sms) * std::max(1, per_sm) * warps;
        const int64_t chunks = (a.n + SW::B - 1) / SW::B;
        nch = (int)std::max<int64_t>(1, (chunks + resident - 1) / resident);
    }
    const int64_t nseg = ((a.n + SW::B - 1) / SW::B + nch - 1) / nch;
    const int64_t blocks = (nseg + warps - 1) / warps;
    kfn<<<(unsigned)blocks, 32 * warps, smem, s>>>(a.in, a.out, a.n, a.K, nch, nseg, cp,
                                                  real_from_double<real>(a.pre0), real_from_double<real>(a.pre1),
                                                  real_from_double<real>(a.post0), real_from_double<real>(a.post1));
    return cudaGetLastError();
}

template <int P, int R, int ADJ>
static cudaError_t go1d_sweep_kind(const Step1DArgs &a, const CoinP<typename St<P>::real> &cp, cudaStream_t s) {
    const bool ff = a.shift == QW_SHIFT_FLIPFLOP;
    switch (a.kind) {
        case CK_REAL: return ff ? go1d_sweep<P, R, CK_REAL, 1, ADJ>(a, cp, s) : go1d_sweep<P, R, CK_REAL, 0, ADJ>(a, cp, s);
        case CK_COMPLEX: return ff ? go1d_sweep<P, R, CK_COMPLEX, 1, ADJ>(a, cp, s) : go1d_sweep<P, R, CK_COMPLEX, 0, ADJ>(a, cp, s);
        case CK_SIGN_P: return ff ? cudaErrorInvalidValue : go1d_sweep<P, R, CK_SIGN_P, 0, ADJ>(a, cp, s);
        case CK_SIGN_M: return ff ? cudaErrorInvalidValue : go1d_sweep<P, R, CK_SIGN_M, 0, ADJ>(a, cp, s);
        default: return cudaErrorInvalidValue;
    }
}

// Can the sweep kernel run this launch?  (n at least the chunk of the tile
// sweep_tile picks, 2 <= K < chunk / 2.)
template <int P>
bool sweep_ok(int64_t n, int K, int kind, int tile) {
    if (P == P_COMP || kind == CK_PERSITE || kind == CK_PHASE) return false;
    const int64_t B = 32LL * sweep_tile<P>(n, tile);
    return B > 0 && n >= B && K >= 2 && K <= B / 2 - 1;
}

// Largest K the 1D kernel accepts for tile R: at least half the tile is output
// (a quarter of the short window tile).
inline int max_k_1d(int R) { return R == 2 ? 24 : 8 * R; }

template <int P>
int tile1d_effective(int tile, int kind, int adj) {
    using T = Tiles1D<P>;
    if (adj || kind == CK_PERSITE) return T::DEF;
    return (tile == T::A || tile == T::B) ? tile : T::DEF;
}

template <int P>
cudaError_t step1d_t(const Step1DArgs &a0, const void *coinp, int adj, cudaStream_t s) {
    using T = Tiles1D<P>;
    const auto &cp = *static_cast<const CoinP<typename St<P>::real> *>(coinp);
    Step1DArgs a = a0;
    if (a.variant == 1) {   // time-skewed sweep
        if constexpr (P == P_COMP) {
            return cudaErrorInvalidValue;
        } else {
            using ST = SweepTiles<P>;
            if (!sweep_ok<P>(a.n, a.K, a.kind, a.tile)) return cudaErrorInvalidValue;
            if (sweep_tile<P>(a.n, a.tile) == ST::B)
                return adj ? go1d_sweep_kind<P, ST::B, 1>(a, cp, s) : go1d_sweep_kind<P, ST::B, 0>(a, cp, s);
            return adj ? go1d_sweep_kind<P, ST::A, 1>(a, cp, s) : go1d_sweep_kind<P, ST::A, 0>(a, cp, s);
        }
    }
    if constexpr (WindowTile1D<P>::R > 0) {
        constexpr int R = WindowTile1D<P>::R;
        if (a.tile == R && a.oend > a.obeg && a.kind != CK_PERSITE && a.K >= 1 && a.K <= max_k_1d(R)) {
            const bool ok = adj ? go1d_kind<P, R, 1>(a, cp, s) : go1d_kind<P, R, 0>(a, cp, s);
            return ok ? cudaGetLastError() : cudaErrorInvalidValue;
        }
    }
    a.tile = tile1d_effective<P>(a.tile, a.kind, adj);
    if (a.K < 1 || a.K > max_k_1d(a.tile) || (a.per && !joins_1d<P>(a.tile, a.kind))) return cudaErrorInvalidValue;
    const bool ff = a.shift == QW_SHIFT_FLIPFLOP;
    if (a.K == 1 && a.oend <= a.obeg) {   // one step per launch over the whole cycle: the streaming kernel
        const bool ok = adj ? go1d_k1_kind<P, 1>(a, cp, s) : go1d_k1_kind<P, 0>(a, cp, s);
        return ok ? cudaGetLastError() : cudaErrorInvalidValue;
    }
    if (!adj) {
        if (a.kind == CK_PERSITE) {
            ff ? go1d<P, T::DEF, CK_PERSITE, 1, 0>(a, cp, s) : go1d<P, T::DEF, CK_PERSITE, 0, 0>(a, cp, s);
        } else if (a.tile == T::A) {
            if (!go1d_kind<P, T::A, 0>(a, cp, s)) return cudaErrorInvalidValue;
        } else {
            if (!go1d_kind<P, T::B, 0>(a, cp, s)) return cudaErrorInvalidValue;
        }
    } else {
        if (a.kind == CK_PERSITE) {
            ff ? go1d<P, T::DEF, CK_PERSITE, 1, 1>(a, cp, s) : go1d<P, T::DEF, CK_PERSITE, 0, 1>(a, cp, s);
        } else if (!go1d_kind<P, T::DEF, 1>(a, cp, s)) {
            return cudaErrorInvalidValue;
        }
    }
    return cudaGetLastError();
}

template <int P, int CK, int FF, int ADJ>
static void go2d(const Step2DArgs &a, const CoinP<typename St<P>::real> &cp, cudaStream_t s) {
    // per-site phase coins in FP32: two sites per lane, for more warps in flight
    // (the step is latency-bound at 1024^2: 17.7 against 20.5 us per step with four)
    constexpr int R = (CK == CK_PHASE && P == P_F32) ? 2 : Tile2D<P>::R;
    const int64_t segs = (a.nx + 32 * R - 1) / (32 * R);
    // Rows and row segments to run.  A warp reads its row and writes planes to
    // the rows above and below; x-moving planes arrive from the neighbouring
    // columns.  So a state supported on the box [bx0, bx0 + bw) x [by0, by0 + bh)
    // needs the rows and columns of the box widened by one on each side (the
    // adjoint pulls from the same neighbours): every other output is zero and
    // already zero in the output buffer.
    int64_t r0 = 0, nr = a.ny, g0 = 0, ng = segs;
    if (a.bw > 0) {
        if (a.bh + 2 < a.ny) { r0 = (a.by0 - 1 + a.ny) % a.ny; nr = a.bh + 2; }
        if (a.bw + 2 < a.nx) {
            // columns [c0, c0 + cw) modulo nx; the last segment of a row may be short
            const int64_t c0 = (a.bx0 - 1 + a.nx) % a.nx, cw = a.bw + 2, S = 32 * R;
            g0 = c0 / S;
            ng = c0 + cw <= a.nx ? (c0 + cw - 1) / S - g0 + 1 : (segs - g0) + (c0 + cw - a.nx - 1) / S + 1;
            ng = std::min<int64_t>(segs, ng);
        }
    }
    const int64_t nwarps = ng * nr;
    const int64_t blocks = (nwarps + 3) / 4;
    k_step2d<P, R, CK, FF, ADJ><<<(unsigned)blocks, 128, 0, s>>>(
        a.in, a.out, a.nx, a.ny, segs, r0, nr, g0, ng, nwarps, cp, a.phi,
        static_cast<const Cx<typename St<P>::real> *>(a.coins),
        real_from_double<typename St<P>::real>(a.gain));
}

template <int P, int CK>
static void go2d_ff(const Step2DArgs &a, const CoinP<typename St<P>::real> &cp, int adj, cudaStream_t s) {
    switch (a.shift) {
        case QW_SHIFT_FLIPFLOP: adj ? go2d<P, CK, 1, 1>(a, cp, s) : go2d<P, CK, 1, 0>(a, cp, s); break;
        case QW_SHIFT_DIAGONAL: adj ? go2d<P, CK, 2, 1>(a, cp, s) : go2d<P, CK, 2, 0>(a, cp, s); break;
        default: adj ? go2d<P, CK, 0, 1>(a, cp, s) : go2d<P, CK, 0, 0>(a, cp, s); break;
    }
}

// Does the fast 2D kernel of precision P handle this coin kind?
template <int P>
constexpr bool fast2d_has_phase() { return P == P_F32 || P == P_F64; }

template <int P>
cudaError_t step2d_t(const Step2DArgs &a, const void *coinp, int adj, cudaStream_t s) {
    const auto &cp = *static_cast<const CoinP<typename St<P>::real> *>(coinp);
    switch (a.kind) {
        case CK_REAL: go2d_ff<P, CK_REAL>(a, cp, adj, s); break;
        case CK_COMPLEX: go2d_ff<P, CK_COMPLEX>(a, cp, adj, s); break;
        case CK_GROVER: go2d_ff<P, CK_GROVER>(a, cp, adj, s); break;
        case CK_HH: go2d_ff<P, CK_HH>(a, cp, adj, s); break;
        case CK_PHASE:
            if constexpr (fast2d_has_phase<P>()) { go2d_ff<P, CK_PHASE>(a, cp, adj, s); break; }
            return cudaErrorNotSupported;
        default: return cudaErrorNotSupported;
    }
    return cudaGetLastError();
}

// Tiles of T sites along an axis of n sites that hold the outputs of one step
// from a state supported on [c0, c0 + cw): that range widened by one site on
// each side (modulo n on the periodic lattice, cut at its ends otherwise).
// The last tile may be short.  cw = 0: every tile.
static inline void tile_range(int64_t c0, int64_t cw, int64_t n, int T, bool periodic, int &t0, int &nt) {
    const int64_t ntiles = (n + T - 1) / T;
    t0 = 0;
    nt = (int)ntiles;
    if (cw <= 0) return;
    int64_t a0, aw;
    if (periodic) {
        if (cw + 2 >= n) return;
        a0 = (c0 - 1 + n) % n;
        aw = cw + 2;
    } else {
        a0 = std::max<int64_t>(0, c0 - 1);
        aw = std::min<int64_t>(n, c0 + cw + 1) - a0;
    }
    t0 = (int)(a0 / T);
    const int64_t k = a0 + aw <= n ? (a0 + aw - 1) / T - t0 + 1 : (ntiles - t0) + (a0 + aw - n - 1) / T + 1;
    nt = (int)std::min<int64_t>(ntiles, k);
}

template <int P, int CK>
static void gogen(const StepGenericArgs &a, const CoinP<typename St<P>::real> &cp, cudaStream_t s) {
    GenGeom g{a.ndim, a.nx, a.ny, a.nx * a.ny, a.shift, a.bc, a.links, a.rthr, a.rk0, a.rk1, a.rstep, 0, 1, 0, 1};
    const int64_t blocks = (g.ns + 127) / 128;
    k_step_generic<P, CK><<<(unsigned)blocks, 128, 0, s>>>(
        a.in, a.out, g, a.adjoint, cp, static_cast<const Cx<typename St<P>::real> *>(a.coins), a.phi,
        real_from_double<typename St<P>::real>(a.gain));
}

// The tiled form serves the forward step on the 2D axis lattice (any coin,
// boundary and links); the grid's y extent limits ny to 65535 tiles.  (1D forward
// steps run k_step1d_window.)
template <int P>
static bool generic_tile_ok(const StepGenericArgs &a) {
    if (a.adjoint || !(a.shift == QW_SHIFT_MOVING || a.shift == QW_SHIFT_FLIPFLOP) || a.nx >= (int64_t(1) << 30))
        return false;
    return a.ndim == 2 && (a.ny + gt_y<P>() - 1) / gt_y<P>() <= 65535;
}

template <int P, int CK>
static void gotile(const StepGenericArgs &a, const CoinP<typename St<P>::real> &cp, cudaStream_t s) {
    using real = typename St<P>::real;
    const bool per = a.bc == QW_BC_PERIODIC;
    GenGeom g{a.ndim, a.nx, a.ny, a.nx * a.ny, a.shift, a.bc, a.links, a.rthr, a.rk0, a.rk1, a.rstep, 0, 1, 0, 1};
    const auto gain = real_from_double<real>(a.gain);
    const auto *coins = static_cast<const Cx<real> *>(a.coins);
    int gx = 0, gy = 0;
    tile_range(a.bx0, a.bw, a.nx, GT_X, per, g.tx0, gx);
    tile_range(a.by0, a.bw > 0 ? a.bh : 0, a.ny, gt_y<P>(), per, g.ty0, gy);
    g.ntx = (int)((a.nx + GT_X - 1) / GT_X);
    g.nty = (int)((a.ny + gt_y<P>() - 1) / gt_y<P>());
    const dim3 grid((unsigned)gx, (unsigned)gy);
    if (a.shift == QW_SHIFT_MOVING)
        k_step_generic_tile<P, QW_SHIFT_MOVING, CK><<<grid, GT_THREADS, 0, s>>>(a.in, a.out, g, cp, coins, a.phi, gain);
    else
        k_step_generic_tile<P, QW_SHIFT_FLIPFLOP, CK><<<grid, GT_THREADS, 0, s>>>(a.in, a.out, g, cp, coins, a.phi, gain);
}

template <int P>
cudaError_t generic_t(const StepGenericArgs &a, const void *coinp, cudaStream_t s) {
    const auto &cp = *static_cast<const CoinP<typename St<P>::real> *>(coinp);
    if (generic_tile_ok<P>(a)) {
        switch (a.kind) {
            case CK_PERSITE: gotile<P, CK_PERSITE>(a, cp, s); break;
            case CK_PHASE: gotile<P, CK_PHASE>(a, cp, s); break;
            case CK_GROVER: gotile<P, CK_GROVER>(a, cp, s); break;
            case CK_HH: gotile<P, CK_HH>(a, cp, s); break;
            case CK_REAL: gotile<P, CK_REAL>(a, cp, s); break;
            default: gotile<P, CK_COMPLEX>(a, cp, s); break;   // other global coins as a full matrix
        }
        return cudaGetLastError();
    }
    switch (a.kind) {
        case CK_PERSITE: gogen<P, CK_PERSITE>(a, cp, s); break;
        case CK_PHASE: gogen<P, CK_PHASE>(a, cp, s); break;
        default: gogen<P, CK_COMPLEX>(a, cp, s); break;  // every global coin as a full matrix
    }
    return cudaGetLastError();
}

// 1D generic forward steps: nsteps (at most WINDOW_MAX_STEPS) from the state in
// a.in on the output range [o0, o0 + ow) modulo nx; gains[i] is the drift gain of
// step i, a.rstep the random-link step of the first.  Ranges of up to
// WINDOW_SITES sites take tiles of 256, wider ones tiles of 2048, whose halos are
// a smaller share (a line of 2^20 sites from its middle, T = 1024, FP32: 593 us in
// one CTA, now under 150; the whole 2^27 line: 0.66 ms per step one by one).
template <int P, int CK, int SH, int E, int TH>
static cudaError_t gowin(const StepGenericArgs &a, const CoinP<typename St<P>::real> &cp, const double *gains, int nsteps,
                         int64_t o0, int64_t ow, cudaStream_t s) {
    using real = typename St<P>::real;
    GenGeom g{a.ndim, a.nx, a.ny, a.nx * a.ny, a.shift, a.bc, a.links, a.rthr, a.rk0, a.rk1, a.rstep, 0, 1, 0, 1};
    WinGains<real> gv{};
    for (int i = 0; i < nsteps; ++i) gv.v[i] = real_from_double<real>(gains[i]);
    auto kfn = k_step1d_window<P, SH, CK, E, TH>;
    constexpr size_t smem = (size_t)E * 2 * St<P>::SLOTS_PER_COIN * St<P>::SLOT_BYTES;
    // (set on every launch that needs it: the attribute is the current device's)
    cudaError_t e = smem > 48 * 1024 ? cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) : cudaSuccess;
    if (e != cudaSuccess) return e;
    const int64_t blocks = (ow + E - 2 * nsteps - 1) / (E - 2 * nsteps);
    kfn<<<(unsigned)blocks, TH, smem, s>>>(a.in, a.out, g, cp, static_cast<const Cx<real> *>(a.coins), (int)o0, (int)ow,
                                           nsteps, gv);
    return cudaGetLastError();
}

// the small tile: 256 sites; 64 in FP64, where a tile is bound by its SM's two
// lanes a clock (and takes at most 16 steps, see window1d_steps)
template <int P> struct WindowTile { static constexpr int E = 256; };
template <> struct WindowTile<P_F64> { static constexpr int E = 64; };

template <int P, int CK>
static cudaError_t gowin_shift(const StepGenericArgs &a, const CoinP<typename St<P>::real> &cp, const double *gains, int nsteps,
                               int64_t o0, int64_t ow, cudaStream_t s) {
    constexpr int E = WindowTile<P>::E;
    const bool narrow = ow <= WINDOW_SITES && 4 * nsteps <= E;
    if (a.shift == QW_SHIFT_MOVING)
        return narrow ? gowin<P, CK, QW_SHIFT_MOVING, E, E>(a, cp, gains, nsteps, o0, ow, s)
                      : gowin<P, CK, QW_SHIFT_MOVING, 2048, 512>(a, cp, gains, nsteps, o0, ow, s);
    if (a.shift == QW_SHIFT_FLIPFLOP)
        return narrow ? gowin<P, CK, QW_SHIFT_FLIPFLOP, E, E>(a, cp, gains, nsteps, o0, ow, s)
                      : gowin<P, CK, QW_SHIFT_FLIPFLOP, 2048, 512>(a, cp, gains, nsteps, o0, ow, s);
    return cudaErrorInvalidValue;
}

template <int P>
cudaError_t window1d_t(const StepGenericArgs &a, const void *coinp, const double *gains, int nsteps, int64_t o0, int64_t ow,
                       cudaStream_t s) {
    const auto &cp = *static_cast<const CoinP<typename St<P>::real> *>(coinp);
    if (a.ndim != 1 || a.adjoint || a.nx >= (int64_t(1) << 30) || nsteps < 1 || nsteps > WINDOW_MAX_STEPS || ow < 1)
        return cudaErrorInvalidValue;
    // (phase coins are expanded to per-site matrices in 1D)
    switch (a.kind) {
        case CK_PERSITE: return gowin_shift<P, CK_PERSITE>(a, cp, gains, nsteps, o0, ow, s);
        case CK_REAL: return gowin_shift<P, CK_REAL>(a, cp, gains, nsteps, o0, ow, s);
        default: return gowin_shift<P, CK_COMPLEX>(a, cp, gains, nsteps, o0, ow, s);
    }
}

}  // namespace qw

// One translation unit per precision defines these entry points.
#define QW_DEFINE_STEP_LAUNCHERS(PREC, SUFFIX)                                                          \
    namespace qw {                                                                                      \
    cudaError_t launch_step1d_##SUFFIX(const Step1DArgs &a, const void *cp, int adj, cudaStream_t s) {  \
        return step1d_t<PREC>(a, cp, adj, s);                                                           \
    }                                                                                                   \
    cudaError_t launch_step2d_##SUFFIX(const Step2DArgs &a, const void *cp, int adj, cudaStream_t s) {  \
        return step2d_t<PREC>(a, cp, adj, s);                                                           \
    }                                                                                                   \
    cudaError_t launch_generic_##SUFFIX(const StepGenericArgs &a, const void *cp, cudaStream_t s) {     \
        return generic_t<PREC>(a, cp, s);                                                               \
    }                                                                                                   \
    cudaError_t launch_window1d_##SUFFIX(const StepGenericArgs &a, const void *cp, const double *gains,  \
                                         int nsteps, int64_t o0, int64_t ow, cudaStream_t s) {          \
        return window1d_t<PREC>(a, cp, gains, nsteps, o0, ow, s);                                       \
    }                                                                                                   \
    int tile1d_##SUFFIX(int tile, int kind, int adj) { return tile1d_effective<PREC>(tile, kind, adj); } \
    bool sweep_ok_##SUFFIX(int64_t n, int K, int kind, int tile) { return sweep_ok<PREC>(n, K, kind, tile); } \
    int sweep_tile_##SUFFIX(int64_t n, int tile) { return sweep_tile<PREC>(n, tile); }                   \
    }
