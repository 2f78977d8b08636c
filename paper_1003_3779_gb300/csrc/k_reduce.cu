// k_reduce.cu -- coin marginals, norm, and state import/export kernels.
//
// P(v) = sum_c |psi(v,c)|^2 is the per-site term of the normalisation of the
// walker state (Sec. 2.2, and the two-qubit state of Sec. 3).  The norm
// sum_v P(v) is accumulated in double: each thread sums a fixed, strided set of
// sites, a block reduces its threads with warp shuffles, and a second one-block
// kernel adds the per-block partials in block order.  The grid size is fixed,
// so the summation order, and hence every bit of the result, does not depend
// on timing.  For float amplitudes with a float P the per-site sum of squares
// is formed in float (one rounding of 2^-24 per site) and only the running
// norm is double: double arithmetic runs at a small fraction of the float rate
// on this part.
#include <algorithm>
#include <type_traits>

#include "qw_internal.cuh"

namespace qw {

static constexpr int RED_THREADS = 256;
static constexpr int RED_BLOCKS = 152 * 4;   // a multiple of the SM count

int marginal_blocks() { return RED_BLOCKS; }

__device__ __forceinline__ double block_sum(double v, double *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
    return r;
}

// Is site i (linear) inside the box?  Both box axes are modulo the lattice.
__device__ __forceinline__ bool box_has(const SupportBox &b, int64_t i) {
    int64_t x = i, y = 0;
    if (b.ny > 1) {
        if (b.nx * b.ny < (int64_t(1) << 31)) { y = (uint32_t)i / (uint32_t)b.nx; x = (uint32_t)i - (uint32_t)y * (uint32_t)b.nx; }
        else { y = i / b.nx; x = i - y * b.nx; }
    }
    const int64_t dx = x - b.x0, dy = y - b.y0;
    return (dx >= 0 ? dx : dx + b.nx) < b.w && (dy >= 0 ? dy : dy + b.ny) < b.h;
}
template <int VEC> __device__ __forceinline__ bool box_meets(const SupportBox &b, int64_t i0) {
    bool in = false;
#pragma unroll
    for (int k = 0; k < VEC; ++k) in = in || box_has(b, i0 + k);
    return in;
}

// Each thread handles VEC consecutive sites per iteration with vector loads.
// box: the state is zero outside it (a clipped walk), so groups of sites that
// lie outside are not read; their P is zero and the norm's sum, in the same
// fixed order, keeps its bits.
template <int P, int PF32>
__global__ void __launch_bounds__(RED_THREADS)
k_marginals(View v, int64_t ns, void *P_out, double *partials, SupportBox box) {
    using S = St<P>;
    using real = typename S::real;
    __shared__ double sh[RED_THREADS / 32];
    const int d = v.d;
    double acc = 0.0;
    const int64_t ngroups = (ns + S::VEC - 1) / S::VEC;
    for (int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; gidx < ngroups;
         gidx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i0 = gidx * S::VEC;
        double p[S::VEC];
#pragma unroll
        for (int k = 0; k < S::VEC; ++k) p[k] = 0.0;
        if (box.w && !box_meets<S::VEC>(box, i0)) {
#pragma unroll
            for (int k = 0; k < S::VEC; ++k)
                if (P_out && i0 + k < ns) {
                    if (PF32) reinterpret_cast<float *>(P_out)[i0 + k] = 0.f;
                    else reinterpret_cast<double *>(P_out)[i0 + k] = 0.0;
                }
            continue;
        }
        if constexpr (PF32 && std::is_same<real, float>::value) {
          if (i0 + S::VEC <= ns) {
            // float amplitudes and a float P: |psi|^2 per site in float (FP64 is
            // slow on this part), the VEC sites summed in float, one double add
            float pf[S::VEC], grp = 0.f;
#pragma unroll
            for (int k = 0; k < S::VEC; ++k) pf[k] = 0.f;
            for (int c = 0; c < d; ++c) {
                Cx<real> a[S::VEC];
                S::ldv(v, c, i0, a);
#pragma unroll
                for (int k = 0; k < S::VEC; ++k) pf[k] = __fmaf_rn((float)a[k].re, (float)a[k].re, __fmaf_rn((float)a[k].im, (float)a[k].im, pf[k]));
            }
#pragma unroll
            for (int k = 0; k < S::VEC; ++k) {
                grp += pf[k];
                if (P_out) reinterpret_cast<float *>(P_out)[i0 + k] = pf[k];
            }
            acc += (double)grp;
            continue;
          }
        }
        if (i0 + S::VEC <= ns) {
            for (int c = 0; c < d; ++c) {
                Cx<real> a[S::VEC];
                S::ldv(v, c, i0, a);
#pragma unroll
                for (int k = 0; k < S::VEC; ++k) p[k] += norm2d(a[k]);
            }
        } else {
            for (int c = 0; c < d; ++c)
                for (int k = 0; k < S::VEC; ++k)
                    if (i0 + k < ns) p[k] += norm2d(S::ld(v, c, i0 + k));
        }
#pragma unroll
        for (int k = 0; k < S::VEC; ++k) {
            if (i0 + k < ns) {
                acc += p[k];
                if (P_out) {
                    if (PF32) reinterpret_cast<float *>(P_out)[i0 + k] = (float)p[k];
                    else reinterpret_cast<double *>(P_out)[i0 + k] = p[k];
                }
            }
        }
    }
    double b = block_sum(acc, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

__global__ void k_sum_partials(const double *partials, int n, double *out) {
    // one warp, lanes own fixed strided subsets, then a fixed shuffle tree
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += 32) v += partials[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) *out = v;
}

template <int P>
static cudaError_t marginals_t(View v, int64_t ns, void *P_out, int pf32, double *partials, int nblocks,
                               double *norm_dev, const SupportBox &box, cudaStream_t s) {
    if (pf32) k_marginals<P, 1><<<nblocks, RED_THREADS, 0, s>>>(v, ns, P_out, partials, box);
    else k_marginals<P, 0><<<nblocks, RED_THREADS, 0, s>>>(v, ns, P_out, partials, box);
    if (norm_dev) k_sum_partials<<<1, 32, 0, s>>>(partials, nblocks, norm_dev);
    return cudaGetLastError();
}

cudaError_t launch_marginals(int prec, View v, int64_t ns, void *P, int p_f32, double *partials,
                             int nblocks, double *norm_dev, const SupportBox &box, cudaStream_t s) {
    switch (prec) {
        case P_F64: return marginals_t<P_F64>(v, ns, P, p_f32, partials, nblocks, norm_dev, box, s);
        case P_F32: return marginals_t<P_F32>(v, ns, P, p_f32, partials, nblocks, norm_dev, box, s);
        case P_BF16: return marginals_t<P_BF16>(v, ns, P, p_f32, partials, nblocks, norm_dev, box, s);
        case P_COMP: return marginals_t<P_COMP>(v, ns, P, p_f32, partials, nblocks, norm_dev, box, s);
    }
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------- support box
// Bounding box of the nonzero amplitudes of a state (any coin, any plane):
// box[0..1] the smallest and largest column, box[2..3] the smallest and
// largest row, as unsigned 64-bit values for the atomics; box[0] > box[1]
// means the state is zero.  It is the starting window of the light-cone
// clipping of a localised walk (the "line" computation window of Sec. 3,
// which starts at the walker's site and widens by one site per step).
//
// The search runs with the copy of the caller's state into the walk's buffer
// (SRC: one read and one write of the state, at the copy rate) or over the
// buffer alone.  Each thread takes 16 bytes of every plane slot per round; a
// block keeps the range it has seen in registers and adds it to the box once,
// with four atomics.  (Four atomics per warp and tile on the same four words,
// and cudaMemcpy2DAsync for the copy, took 99 us to search a dense state of
// 10^6 sites and 1300 us to copy one of 2 GiB; now under 10 us and 650 us.)
// Over the buffer alone, a first block looks at the first and the last 256
// sites: a dense state fills the box there, and the search returns.
static constexpr int SUP_THREADS = 256;

// which of the vector's sites hold a nonzero amplitude (-0 is zero; a NaN is not)
template <int SB> __device__ __forceinline__ unsigned nonzero_sites(uint4 u) {
    if constexpr (SB == 16) return ((u.y << 1) | u.x | (u.w << 1) | u.z) != 0u;
    else if constexpr (SB == 8) return (((u.x << 1) | (u.y << 1)) != 0u) | ((((u.z << 1) | (u.w << 1)) != 0u) << 1);
    else return ((u.x & 0x7fff7fffu) != 0u) | (((u.y & 0x7fff7fffu) != 0u) << 1) |
                (((u.z & 0x7fff7fffu) != 0u) << 2) | (((u.w & 0x7fff7fffu) != 0u) << 3);
}

// the smallest / largest linear index and column of the sites a thread has seen
struct Seen {
    unsigned long long i0 = ~0ull, i1 = 0ull, x0 = ~0ull, x1 = 0ull;
    __device__ void site(int64_t i, int64_t nx, int64_t ns) {
        int64_t x = i;
        if (nx < ns) x = ns < (int64_t(1) << 31) ? (int64_t)((uint32_t)i % (uint32_t)nx) : i % nx;
        i0 = min(i0, (unsigned long long)i); i1 = max(i1, (unsigned long long)i);
        x0 = min(x0, (unsigned long long)x); x1 = max(x1, (unsigned long long)x);
    }
};
// add what the block has seen to the box
__device__ __forceinline__ void merge_seen(Seen v, int64_t nx, unsigned long long *box) {
    __shared__ unsigned long long sh[SUP_THREADS / 32][4];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.i0 = min(v.i0, __shfl_xor_sync(0xffffffffu, v.i0, o));
        v.i1 = max(v.i1, __shfl_xor_sync(0xffffffffu, v.i1, o));
        v.x0 = min(v.x0, __shfl_xor_sync(0xffffffffu, v.x0, o));
        v.x1 = max(v.x1, __shfl_xor_sync(0xffffffffu, v.x1, o));
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { sh[w][0] = v.i0; sh[w][1] = v.i1; sh[w][2] = v.x0; sh[w][3] = v.x1; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < SUP_THREADS / 32; ++k) {
            v.i0 = min(v.i0, sh[k][0]); v.i1 = max(v.i1, sh[k][1]);
            v.x0 = min(v.x0, sh[k][2]); v.x1 = max(v.x1, sh[k][3]);
        }
        if (v.i0 != ~0ull) {
            atomicMin(&box[0], v.x0);
            atomicMax(&box[1], v.x1);
            atomicMin(&box[2], v.i0 / (unsigned long long)nx);
            atomicMax(&box[3], v.i1 / (unsigned long long)nx);
        }
    }
}

// empties the box; with a state, looks at its first and last SUP_THREADS sites
template <int SB>
__global__ void __launch_bounds__(SUP_THREADS)
k_support_init(const char *state, int64_t slot_bytes, int nslots, int64_t nx, int64_t ns, unsigned long long *box) {
    if (threadIdx.x == 0) { box[0] = ~0ull; box[1] = 0ull; box[2] = ~0ull; box[3] = 0ull; }
    if (!state) return;
    __syncthreads();
    Seen v;
    for (int end = 0; end < 2; ++end) {
        const int64_t i = end ? ns - 1 - threadIdx.x : threadIdx.x;
        if (i < 0 || i >= ns) continue;
        for (int c = 0; c < nslots; ++c) {
            uint4 u = make_uint4(0, 0, 0, 0);
            const char *p = state + c * slot_bytes + i * SB;
            if constexpr (SB == 16) u = *reinterpret_cast<const uint4 *>(p);
            else if constexpr (SB == 8) { const uint2 a = *reinterpret_cast<const uint2 *>(p); u.x = a.x; u.y = a.y; }
            else u.x = *reinterpret_cast<const unsigned *>(p);
            if (nonzero_sites<SB>(u)) v.site(i, nx, ns);
        }
    }
    merge_seen(v, nx, box);
}

__device__ __forceinline__ uint4 widen(uint4 u) { return u; }
__device__ __forceinline__ uint4 widen(uint2 u) { return make_uint4(u.x, u.y, 0u, 0u); }

// SRC: src holds nslots dense planes of ns sites, which are copied to dst; else
// dst is searched alone.  V: the vector that every plane of src is aligned to,
// 16 bytes, or 8 for complex64 planes of an odd number of sites.
template <int SB, bool SRC, class V>
__global__ void __launch_bounds__(SUP_THREADS)
k_support(const char *__restrict__ src, char *__restrict__ dst, int64_t slot_bytes, int nslots, int64_t nx, int64_t ns,
          unsigned long long *box) {
    constexpr int SPV = (int)sizeof(V) / SB;   // sites per vector
    if (!SRC) {   // the box already spans the lattice: nothing left to find
        // (one thread looks for the block: other blocks are adding to the box, and
        // threads that saw different boxes would part before the shuffles below)
        __shared__ int full;
        if (threadIdx.x == 0) {
            const volatile unsigned long long *vb = box;
            full = vb[0] == 0ull && vb[1] == (unsigned long long)(nx - 1) && vb[2] == 0ull &&
                   vb[3] == (unsigned long long)(ns / nx - 1);
        }
        __syncthreads();
        if (full) return;
    }
    const int64_t nvec = (ns + SPV - 1) / SPV;
    Seen v;
    for (int64_t k = (int64_t)blockIdx.x * SUP_THREADS + threadIdx.x; k < nvec; k += (int64_t)gridDim.x * SUP_THREADS) {
        unsigned nz = 0;
        for (int c0 = 0; c0 < nslots; c0 += 2) {   // two slots in flight (nslots is even)
            V u[2];
#pragma unroll
            for (int c = 0; c < 2; ++c)
                u[c] = SRC ? __ldcs(reinterpret_cast<const V *>(src + (c0 + c) * ns * SB) + k)
                           : reinterpret_cast<const V *>(dst + (c0 + c) * slot_bytes)[k];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (SRC) reinterpret_cast<V *>(dst + (c0 + c) * slot_bytes)[k] = u[c];
                nz |= nonzero_sites<SB>(widen(u[c]));
            }
        }
        if (nz) {
#pragma unroll
            for (int i = 0; i < SPV; ++i)
                if ((nz >> i & 1u) && k * SPV + i < ns) v.site(k * SPV + i, nx, ns);   // (not the slot's padding)
        }
    }
    merge_seen(v, nx, box);
}

template <int SB, class V>
static cudaError_t support_t(const void *src, View v, int nslots, int64_t nx, int64_t ny, unsigned long long *box, cudaStream_t s) {
    constexpr int SPV = (int)sizeof(V) / SB;
    const int64_t ns = nx * ny, slot = v.pitch * SB;
    const int64_t tiles = ((ns + SPV - 1) / SPV + SUP_THREADS - 1) / SUP_THREADS;
    const unsigned grid = (unsigned)std::min<int64_t>(tiles, 152 * 8);
    char *dst = static_cast<char *>(v.p);
    // (the first look saves reading a dense state, but costs 2 us: not for small ones)
    const bool look = !src && nslots * ns * SB > (int64_t(32) << 20);
    k_support_init<SB><<<1, SUP_THREADS, 0, s>>>(look ? dst : nullptr, slot, nslots, nx, ns, box);
    if (src) k_support<SB, true, V><<<grid, SUP_THREADS, 0, s>>>(static_cast<const char *>(src), dst, slot, nslots, nx, ns, box);
    else k_support<SB, false, V><<<grid, SUP_THREADS, 0, s>>>(nullptr, dst, slot, nslots, nx, ns, box);
    return cudaGetLastError();
}

int dense_vector(const void *dense, int64_t ns, int slot_bytes) {
    for (int vb : {16, 8})
        if (vb >= slot_bytes && slot_bytes >= 8 && reinterpret_cast<uintptr_t>(dense) % vb == 0 && ns * slot_bytes % vb == 0)
            return vb;
    return 0;
}

cudaError_t launch_support(const void *src, View v, int nslots, int slot_bytes, int64_t nx, int64_t ny, unsigned long long *box,
                           cudaStream_t s) {
    const int vb = src ? dense_vector(src, nx * ny, slot_bytes) : 16;
    if (slot_bytes == 16 && vb == 16) return support_t<16, uint4>(src, v, nslots, nx, ny, box, s);
    if (slot_bytes == 8 && vb == 16) return support_t<8, uint4>(src, v, nslots, nx, ny, box, s);
    if (slot_bytes == 8 && vb == 8) return support_t<8, uint2>(src, v, nslots, nx, ny, box, s);
    if (slot_bytes == 4 && !src) return support_t<4, uint4>(nullptr, v, nslots, nx, ny, box, s);
    return cudaErrorInvalidValue;
}

// The state out into nslots dense planes (V as dense_vector): sites outside the
// box, where the state is zero, are written without a read.
template <int SB, class V>
__global__ void __launch_bounds__(SUP_THREADS)
k_store_state(const char *__restrict__ state, int64_t slot_bytes, int nslots, int64_t ns, char *__restrict__ out, SupportBox box) {
    constexpr int SPV = (int)sizeof(V) / SB;
    const int64_t nvec = ns / SPV;
    for (int64_t k = (int64_t)blockIdx.x * SUP_THREADS + threadIdx.x; k < nvec; k += (int64_t)gridDim.x * SUP_THREADS) {
        const bool in = box.w == 0 || box_meets<SPV>(box, k * SPV);
        for (int c0 = 0; c0 < nslots; c0 += 2) {
            V u[2] = {};
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (in) u[c] = reinterpret_cast<const V *>(state + (c0 + c) * slot_bytes)[k];
#pragma unroll
            for (int c = 0; c < 2; ++c) __stcs(reinterpret_cast<V *>(out + (c0 + c) * ns * SB) + k, u[c]);
        }
    }
}

cudaError_t launch_store_state(View v, int nslots, int slot_bytes, int64_t ns, void *out, const SupportBox &box, cudaStream_t s) {
    const int vb = dense_vector(out, ns, slot_bytes);
    if (!vb) return cudaErrorInvalidValue;
    const int64_t tiles = (ns / (vb / slot_bytes) + SUP_THREADS - 1) / SUP_THREADS;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(tiles, 152 * 8));
    const char *p = static_cast<const char *>(v.p);
    char *o = static_cast<char *>(out);
    if (slot_bytes == 16) k_store_state<16, uint4><<<grid, SUP_THREADS, 0, s>>>(p, v.pitch * 16, nslots, ns, o, box);
    else if (vb == 16) k_store_state<8, uint4><<<grid, SUP_THREADS, 0, s>>>(p, v.pitch * 8, nslots, ns, o, box);
    else k_store_state<8, uint2><<<grid, SUP_THREADS, 0, s>>>(p, v.pitch * 8, nslots, ns, o, box);
    return cudaGetLastError();
}

// Zero the box of every slot (columns and rows modulo the lattice).
template <class V>
__global__ void __launch_bounds__(SUP_THREADS)
k_clear_box(V *state, int64_t pitch, int nslots, SupportBox b) {
    const int64_t n = b.w * b.h;
    for (int64_t k = (int64_t)blockIdx.x * SUP_THREADS + threadIdx.x; k < n; k += (int64_t)gridDim.x * SUP_THREADS) {
        const int64_t r = k / b.w;
        int64_t x = b.x0 + (k - r * b.w), y = b.y0 + r;
        if (x >= b.nx) x -= b.nx;
        if (y >= b.ny) y -= b.ny;
        for (int c = 0; c < nslots; ++c) state[c * pitch + y * b.nx + x] = V{};
    }
}

cudaError_t launch_clear_box(View v, int nslots, int slot_bytes, const SupportBox &b, cudaStream_t s) {
    const int64_t tiles = (b.w * b.h + SUP_THREADS - 1) / SUP_THREADS;
    if (tiles <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)std::min<int64_t>(tiles, 152 * 8);
    switch (slot_bytes) {
        case 16: k_clear_box<uint4><<<grid, SUP_THREADS, 0, s>>>(static_cast<uint4 *>(v.p), v.pitch, nslots, b); break;
        case 8: k_clear_box<uint2><<<grid, SUP_THREADS, 0, s>>>(static_cast<uint2 *>(v.p), v.pitch, nslots, b); break;
        case 4: k_clear_box<unsigned><<<grid, SUP_THREADS, 0, s>>>(static_cast<unsigned *>(v.p), v.pitch, nslots, b); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- import / export
// Caller layout: d dense planes of nsites complex numbers (complex128 or
// complex64).  One launch converts `count` sites of plane `plane`, starting at
// site `first`; `src`/`dst` point at the first of those sites.
template <int P>
__global__ void k_import(View dst, const void *src, int c64, int64_t first, int64_t count, int plane) {
    using real = typename St<P>::real;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    double re, im;
    if (c64) {
        float2 a = reinterpret_cast<const float2 *>(src)[i];
        re = a.x; im = a.y;
    } else {
        double2 a = reinterpret_cast<const double2 *>(src)[i];
        re = a.x; im = a.y;
    }
    Cx<real> z;
    if constexpr (P == P_COMP) {
        float rh = (float)re, ih = (float)im;
        z = {{rh, (float)(re - (double)rh)}, {ih, (float)(im - (double)ih)}};
    } else {
        z = {(real)re, (real)im};
    }
    St<P>::st(dst, plane, first + i, z);
}

template <int P>
__global__ void k_export(View srcv, void *dst, int c64, int64_t first, int64_t count, int plane) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    auto z = St<P>::ld(srcv, plane, first + i);
    double re, im;
    if constexpr (P == P_COMP) {
        re = (double)z.re.hi + (double)z.re.lo;
        im = (double)z.im.hi + (double)z.im.lo;
    } else {
        re = (double)z.re; im = (double)z.im;
    }
    if (c64) reinterpret_cast<float2 *>(dst)[i] = make_float2((float)re, (float)im);
    else reinterpret_cast<double2 *>(dst)[i] = make_double2(re, im);
}

cudaError_t launch_import(int prec, View dst, int64_t nsites, const void *src, int src_c64,
                          int64_t first, int64_t count, int plane, cudaStream_t s) {
    (void)nsites;
    if (count <= 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((count + 255) / 256);
    switch (prec) {
        case P_F64: k_import<P_F64><<<blocks, 256, 0, s>>>(dst, src, src_c64, first, count, plane); break;
        case P_F32: k_import<P_F32><<<blocks, 256, 0, s>>>(dst, src, src_c64, first, count, plane); break;
        case P_BF16: k_import<P_BF16><<<blocks, 256, 0, s>>>(dst, src, src_c64, first, count, plane); break;
        case P_COMP: k_import<P_COMP><<<blocks, 256, 0, s>>>(dst, src, src_c64, first, count, plane); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_export(int prec, View src, int64_t nsites, void *dst, int dst_c64,
                          int64_t first, int64_t count, int plane, cudaStream_t s) {
    (void)nsites;
    if (count <= 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((count + 255) / 256);
    switch (prec) {
        case P_F64: k_export<P_F64><<<blocks, 256, 0, s>>>(src, dst, dst_c64, first, count, plane); break;
        case P_F32: k_export<P_F32><<<blocks, 256, 0, s>>>(src, dst, dst_c64, first, count, plane); break;
        case P_BF16: k_export<P_BF16><<<blocks, 256, 0, s>>>(src, dst, dst_c64, first, count, plane); break;
        case P_COMP: k_export<P_COMP><<<blocks, 256, 0, s>>>(src, dst, dst_c64, first, count, plane); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace qw
