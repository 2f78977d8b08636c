// tile2d.cu -- launcher of the 2D tile kernel (k_tile2d.cuh), FP32.
#include <algorithm>

#include "qw_handle.h"
#include "k_tile2d.cuh"

namespace qw {

template <int P, int SH, int CK, bool PH, bool LINKS, int EX, int EY, int TH>
struct TileShape {
    static constexpr size_t smem = (size_t)EX * EY * 4 * 2 * sizeof(typename St<P>::real);
    // CTAs of this shape the device holds at once (looked up once, by whichever
    // thread is first; every device here is the same part)
    static int64_t slots() {
        static const int64_t n = [] {
            auto kern = k_tile2d<P, SH, CK, PH, LINKS, EX, EY, TH>;
            int dev = 0, sms = 0, per_sm = 0;
            cudaGetDevice(&dev);
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TH, smem) != cudaSuccess || per_sm < 1) per_sm = 1;
            return (int64_t)sms * per_sm;
        }();
        return n;
    }
    static dim3 grid(const Tile2DArgs &a) {
        return dim3((unsigned)((a.ow + EX - 2 * a.K - 1) / (EX - 2 * a.K)), (unsigned)((a.oh + EY - 2 * a.K - 1) / (EY - 2 * a.K)));
    }
    static int64_t waves(const Tile2DArgs &a) {
        const dim3 g = grid(a);
        return ((int64_t)g.x * g.y + slots() - 1) / slots();
    }
    static cudaError_t launch(const Tile2DArgs &a, const void *coinp, cudaStream_t s) {
        auto kern = k_tile2d<P, SH, CK, PH, LINKS, EX, EY, TH>;
        // (set on every launch: the attribute belongs to the current device)
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid(a), TH, smem, s>>>(a.in, a.out, a.g, a.ox0, a.ow, a.oy0, a.oh, a.K,
                                       *static_cast<const CoinP<typename St<P>::real> *>(coinp), a.phi,
                                       real_from_double<typename St<P>::real>(a.gain));
        return cudaGetLastError();
    }
};

// 32 x 32 tiles (two sites per thread, several CTAs per SM), or 64 x 64 where
// the box has so many that their smaller share of halo sites counts: the shape
// whose waves process the fewer sites per SM.
template <int P, int SH, int CK, bool PH, bool LINKS>
static cudaError_t go_tile2d(const Tile2DArgs &a, const void *coinp, cudaStream_t s) {
    using Small = TileShape<P, SH, CK, PH, LINKS, 32, 32, 512>;
    using Large = TileShape<P, SH, CK, PH, LINKS, 64, 64, 1024>;
    const int64_t small = Small::waves(a) * Small::slots() * 32 * 32, large = Large::waves(a) * Large::slots() * 64 * 64;
    return large < small ? Large::launch(a, coinp, s) : Small::launch(a, coinp, s);
}

template <int P, int SH, bool LINKS>
static cudaError_t tile2d_kind(int kind, const Tile2DArgs &a, const void *coinp, cudaStream_t s) {
    if (a.phi) {   // phase coins: the base matrix in its Grover or its general form
        if (kind == CK_GROVER) return go_tile2d<P, SH, CK_GROVER, true, LINKS>(a, coinp, s);
        return go_tile2d<P, SH, CK_COMPLEX, true, LINKS>(a, coinp, s);
    }
    switch (kind) {
        case CK_REAL: return go_tile2d<P, SH, CK_REAL, false, LINKS>(a, coinp, s);
        case CK_COMPLEX: return go_tile2d<P, SH, CK_COMPLEX, false, LINKS>(a, coinp, s);
        case CK_GROVER: return go_tile2d<P, SH, CK_GROVER, false, LINKS>(a, coinp, s);
        case CK_HH: return go_tile2d<P, SH, CK_HH, false, LINKS>(a, coinp, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_tile2d(int shift, int kind, bool links, const Tile2DArgs &a, const void *coinp, cudaStream_t s) {
    if (a.K < 1 || a.K > TILE2D_MAX_STEPS || a.ow < 1 || a.oh < 1 || a.g.nx >= (int64_t(1) << 30) || a.g.ny >= (int64_t(1) << 30) ||
        a.g.nx * a.g.ny >= (int64_t(1) << 32) || (a.oh + 32 - 2 * a.K - 1) / (32 - 2 * a.K) > 65535)
        return cudaErrorInvalidValue;
    constexpr int P = P_F32;
    switch (shift) {
        case QW_SHIFT_MOVING:
            return links ? tile2d_kind<P, QW_SHIFT_MOVING, true>(kind, a, coinp, s) : tile2d_kind<P, QW_SHIFT_MOVING, false>(kind, a, coinp, s);
        case QW_SHIFT_FLIPFLOP:
            return links ? tile2d_kind<P, QW_SHIFT_FLIPFLOP, true>(kind, a, coinp, s) : tile2d_kind<P, QW_SHIFT_FLIPFLOP, false>(kind, a, coinp, s);
        case QW_SHIFT_DIAGONAL:
            return links ? cudaErrorInvalidValue : tile2d_kind<P, QW_SHIFT_DIAGONAL, false>(kind, a, coinp, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace qw
