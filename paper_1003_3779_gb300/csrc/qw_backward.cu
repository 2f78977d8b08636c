// qw_backward.cu -- gradient of a region's probability mass with respect to the
// per-site coin phases, by the adjoint of the walk.
//
// Walk: psi_{t+1} = S C psi_t on the torus (Sec. 2.2 / Sec. 3, U = S (C (x) I)),
// with the per-site coin C_v = B diag(e^{i phi_{v,k}}) (phase first).
// Loss: L = sum_{v in R, c} |psi_T(v, c)|^2.  With lambda_T = 1_R psi_T and
// lambda_t = U^dagger lambda_{t+1}, differentiating D_v = diag(e^{i phi_v})
// (dD_v / dphi_{v,k} = i E_kk D_v) gives
//     dL/dphi_{v,k} = sum_t 2 Re( conj(a_t(v)_k) i b_t(v)_k ) = sum_t -2 Im(conj(a_k) b_k),
//     a_t = B^dagger S^dagger lambda_{t+1},   b_t = D_v psi_t = B^dagger S^dagger psi_{t+1}.
// So one backward step pulls both lambda_{t+1} and psi_{t+1} through S^dagger,
// applies B^dagger to both, adds the gradient term to a per-segment
// accumulator in the compute precision (flushed into the double gradient at the
// end of every segment of K steps), and emits
// lambda_t = D^dagger a and psi_t = D^dagger b.  psi_t is rebuilt from psi_{t+1}
// (the walk is unitary) instead of stored; it is re-seeded from a forward
// checkpoint every K steps, which bounds the drift of the reconstruction to K
// steps.
//
// Light cones (the computation windows of Sec. 3, of the walk and of its
// adjoint): lambda_t is zero outside the region widened by T - t sites, and
// psi_t outside the start's support widened by t.  The product a b, and with it
// the gradient, is zero outside their intersection; lambda is only needed
// where psi will still be nonzero, which is that intersection too, and psi on
// the sites from which the rest of its segment is rebuilt.  A step runs on
// those sites only.  On a 1024^2 torus (T = 512, K = 64, a walker on one site,
// a 64 x 64 region) the sweep's sites fall to a tenth.
#include <algorithm>
#include <cmath>
#include <string>

#include "qw_handle.h"
#include "k_step2d.cuh"

namespace qw {

template <class R> __device__ __forceinline__ void expi(float a, Cx<R> &e);
template <> __device__ __forceinline__ void expi<float>(float a, Cx<float> &e) { float s, c; sincosf(a, &s, &c); e = {c, s}; }
template <> __device__ __forceinline__ void expi<double>(float a, Cx<double> &e) { double s, c; sincos((double)a, &s, &c); e = {c, s}; }

// An arc of a cycle of n sites: [a, a + w) modulo n.
struct Arc {
    int64_t a, w;
};
static bool arc_has(const Arc &r, int64_t x, int64_t n) {
    const int64_t d = x - r.a;
    return (d >= 0 ? d : d + n) < r.w;
}
// r widened by k sites on each side
static Arc arc_widen(Arc r, int64_t k, int64_t n) {
    if (r.w + 2 * k >= n) return {0, n};
    return {((r.a - k) % n + n) % n, r.w + 2 * k};
}
// one arc that covers the intersection of p and q (w = 0: they do not meet)
static Arc arc_cover(const Arc &p, const Arc &q, int64_t n) {
    if (p.w >= n) return q;
    if (q.w >= n) return p;
    const bool qp = arc_has(p, q.a, n), pq = arc_has(q, p.a, n);
    if (qp && pq && p.a != q.a) return p.w < q.w ? p : q;   // they may meet at both ends
    if (qp) { const int64_t d = (q.a - p.a + n) % n; return {q.a, std::min(q.w, p.w - d)}; }
    if (pq) { const int64_t d = (p.a - q.a + n) % n; return {p.a, std::min(p.w, q.w - d)}; }
    return {0, 0};
}
// how far x lies outside the arc: x is in the arc widened by k if and only if
// this is at most k
__device__ __forceinline__ int64_t arc_distance(const Arc &r, int64_t x, int64_t n) {
    int64_t d = x - r.a;
    if (d < 0) d += n;
    return d < r.w ? 0 : min(d - r.w + 1, n - d);
}

// One launch of K backward steps, t0 + K -> t0.
struct BackArgs {
    View lam_in, psi_in, lam_out, psi_out;
    int64_t nx, ny;
    int64_t cx, cw, cy, ch;          // the box of output sites (a cover of those that matter)
    Arc psi_x, psi_y, reg_x, reg_y;  // the start's support and the region
    int64_t t0, T, reach;            // psi_t0 is wanted up to `reach` sites from the region
    int K;
    const float *phi;
    void *gseg;
};

// Slot of plane c in the in-place update (k_tile2d.cuh), backward: the step from
// s to s + 1 steps before the launch's start reads plane c (flip-flop: c xor 1)
// at v + e_c, and plane c of v is written to the slot that was read.
template <int FF> __device__ __forceinline__ void back_slot(int c, int s, int &track, int &dx, int &dy) {
    const int k = FF ? (s & 1 ? 0 : 1) : s + 1;
    track = FF && !(s & 1) ? c ^ 1 : c;
    dx = k * dir_dx<0>(c);
    dy = k * dir_dy<0>(c);
}

// K backward steps in a tile of both fields in shared memory: one launch, one
// read of the phases (and their sines) and one update of the accumulator per K
// steps.  On the workload above the sweep took 512 launches of 4.0 us (6.2 us
// with the gaps between them), now 83 of 16 us.  64 registers a thread (a few
// spilled) for two CTAs per SM: 26 -> 16 us per launch.  What bounds it: latency
// for narrow windows, 128 bytes of shared memory per site and step for wide ones.
// Largest box that takes 8 steps per launch rather than 4; the whole gradient of
// the workload above at 0 / 40000 / 70000 / 120000 / no limit: 4.28 / 4.19 / 4.17
// / 4.12 / 4.24 ms.
constexpr int64_t BACK_DEEP_SITES = 120000;
constexpr int BACK_E = 32, BACK_TH = 512, BACK_NS = BACK_E * BACK_E / BACK_TH;   // tile, threads, sites per thread
template <int P, int FF, int GROVER>
__global__ void __launch_bounds__(BACK_TH, P == P_F32 ? 2 : 1)
k_backward2d(BackArgs a, CoinP<typename St<P>::real> cp) {
    using real = typename St<P>::real;
    using S = St<P>;
    using C = Cx<real>;
    struct alignas(2 * sizeof(real)) Slot { real re, im; };
    constexpr int E = BACK_E, M = E - 1;
    extern __shared__ __align__(16) unsigned char bsm[];
    Slot *lam = reinterpret_cast<Slot *>(bsm), *psi = lam + 4 * E * E;   // [track][y][x]
    const int O = E - 2 * a.K;
    auto wrap = [](int64_t q, int64_t n) {   // q is at most about a period outside [0, n): no division
        while (q < 0) q += n;
        while (q >= n) q -= n;
        return q;
    };
    const int64_t bx = (int64_t)blockIdx.x * O - a.K, by = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * O - a.K;
    if (by + a.K >= a.ch) return;   // (the last layer of a tall torus' rows of tiles: the whole block)
    const int i = (int)threadIdx.x % E, j0 = (int)threadIdx.x / E;
    const int64_t x = wrap(a.cx + bx + i, a.nx);
    const int64_t far_x = arc_distance(a.psi_x, x, a.nx), near_x = arc_distance(a.reg_x, x, a.nx);
    C e[BACK_NS][4];
    real g[BACK_NS][4];
    int64_t v[BACK_NS];
    int far[BACK_NS], near[BACK_NS];
#pragma unroll
    for (int n = 0; n < BACK_NS; ++n) {
        const int j = j0 + n * (BACK_TH / E);
        const int64_t y = wrap(a.cy + by + j, a.ny);
        v[n] = y * a.nx + x;
        // distances (cut at 2^30) from the start's support and from the region
        far[n] = (int)min((int64_t)1 << 30, max(far_x, arc_distance(a.psi_y, y, a.ny)));
        near[n] = (int)min((int64_t)1 << 30, max(near_x, arc_distance(a.reg_y, y, a.ny)));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const C l = S::ld(a.lam_in, c, v[n]), p = S::ld(a.psi_in, c, v[n]);
            lam[(c * E + j) * E + i] = {l.re, l.im};
            psi[(c * E + j) * E + i] = {p.re, p.im};
            g[n][c] = (real)0;
        }
        const float4 ph = reinterpret_cast<const float4 *>(a.phi)[v[n]];
        const float pk[4] = {ph.x, ph.y, ph.z, ph.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) expi<real>(pk[c], e[n][c]);
    }
    __syncthreads();
    for (int s = 0; s < a.K; ++s) {
        const int64_t t = a.t0 + a.K - 1 - s;   // this step forms time t
#pragma unroll
        for (int n = 0; n < BACK_NS; ++n) {
            const int j = j0 + n * (BACK_TH / E);
            C mu[4], nu[4];
            int at[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                int tr, dx, dy;
                back_slot<FF>(c, s, tr, dx, dy);
                at[c] = (tr * E + ((j + dy) & M)) * E + ((i + dx) & M);
                mu[c] = {lam[at[c]].re, lam[at[c]].im};
                nu[c] = {psi[at[c]].re, psi[at[c]].im};
            }
            // p = B^dagger mu, q = B^dagger nu
            C p[4], q[4];
            if (GROVER) {   // real symmetric: B^dagger = B = (1/2) J - I
                C sm = cadd(cadd(mu[0], mu[1]), cadd(mu[2], mu[3]));
                C sn = cadd(cadd(nu[0], nu[1]), cadd(nu[2], nu[3]));
                sm = rmul(cp.re[1], sm);
                sn = rmul(cp.re[1], sn);
#pragma unroll
                for (int k = 0; k < 4; ++k) { p[k] = csub(sm, mu[k]); q[k] = csub(sn, nu[k]); }
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    C aa = conjmul(C{cp.re[k], cp.im[k]}, mu[0]);
                    C bb = conjmul(C{cp.re[k], cp.im[k]}, nu[0]);
#pragma unroll
                    for (int r = 1; r < 4; ++r) {
                        const C br{cp.re[4 * r + k], cp.im[4 * r + k]};
                        aa = cadd(aa, conjmul(br, mu[r]));
                        bb = cadd(bb, conjmul(br, nu[r]));
                    }
                    p[k] = aa;
                    q[k] = bb;
                }
            }
            // the gradient term, where psi_t and lambda_t may both be nonzero
            // (elsewhere a field is zero, or was not rebuilt).  -2 Im(conj(p) q)
            // in the compute precision, as is the segment's running sum, which is
            // added into the double gradient once per segment of K steps (double
            // arithmetic is slow on this part)
            const bool lit = far[n] <= t && near[n] <= a.T - t;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (lit) g[n][k] += (p[k].im * q[k].re - p[k].re * q[k].im) * (real)2;
                const C l = conjmul(e[n][k], p[k]), w = conjmul(e[n][k], q[k]);
                lam[at[k]] = {l.re, l.im};
                psi[at[k]] = {w.re, w.im};
            }
        }
        __syncthreads();
    }
    if (i < a.K || i >= E - a.K || bx + i >= a.cw) return;
#pragma unroll
    for (int n = 0; n < BACK_NS; ++n) {
        const int j = j0 + n * (BACK_TH / E);
        if (j < a.K || j >= E - a.K || by + j >= a.ch) continue;
        const bool lit = near[n] <= a.T - a.t0;
        if (lit && far[n] < a.t0 + a.K) {
            real *gs = static_cast<real *>(a.gseg) + 4 * v[n];
#pragma unroll
            for (int k = 0; k < 4; ++k) gs[k] += g[n][k];
        }
        if (far[n] > a.t0 || near[n] > a.reach) continue;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            int tr, dx, dy;
            back_slot<FF>(c, a.K - 1, tr, dx, dy);
            const int at = (tr * E + ((j + dy) & M)) * E + ((i + dx) & M);
            if (lit) S::st(a.lam_out, c, v[n], C{lam[at].re, lam[at].im});
            S::st(a.psi_out, c, v[n], C{psi[at].re, psi[at].im});
        }
    }
}

// grad += gseg (double), gseg = 0: the end of one segment of the adjoint sweep.
template <class R>
__global__ void k_flush_segment(R *__restrict__ gseg, double *__restrict__ grad, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    grad[i] += (double)gseg[i];
    gseg[i] = (R)0;
}

// lambda_T = psi_T on the region (lam is zero elsewhere already), and per-block
// partial sums of |psi_T|^2 over it.
template <int P>
__global__ void __launch_bounds__(256)
k_seed_region(View psi, View lam, int64_t nx, int64_t rx, int64_t ry, int64_t rw, int64_t rh, double *partials) {
    using S = St<P>;
    __shared__ double sh[8];
    double acc = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rw * rh; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / rw, v = (ry + r) * nx + rx + (i - r * rw);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const auto z = S::ld(psi, c, v);
            acc += norm2d(z);
            S::st(lam, c, v, z);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = 0.0;
        for (int i = 0; i < 8; ++i) b += sh[i];
        partials[blockIdx.x] = b;
    }
}

__global__ void k_sum_blocks(const double *partials, int n, double *out) {
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += 32) v += partials[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) *out = v;
}

template <int P> constexpr size_t back_smem() { return (size_t)2 * 4 * BACK_E * BACK_E * 2 * sizeof(typename St<P>::real); }

template <int P, int FF, int GROVER>
static cudaError_t go_backward(const qw_walk *w, const BackArgs &a) {
    auto kern = k_backward2d<P, FF, GROVER>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)back_smem<P>());
    if (e != cudaSuccess) return e;
    const int O = BACK_E - 2 * a.K;
    // rows of tiles in layers of equal height, as the grid's second dimension ends at
    // 65535 (a one-dimensional grid's division cost 0.8 % of the gradient at 1024^2)
    const int64_t rows = (a.ch + O - 1) / O, layers = (rows + 65534) / 65535;
    const dim3 grid((unsigned)((a.cw + O - 1) / O), (unsigned)((rows + layers - 1) / layers), (unsigned)layers);
    kern<<<grid, BACK_TH, back_smem<P>(), w->stream>>>(a, *reinterpret_cast<const CoinP<typename St<P>::real> *>(w->coinp));
    return cudaGetLastError();
}

template <int P>
static cudaError_t backward_steps(const qw_walk *w, const BackArgs &a) {
    bool grover = true;
    for (int r = 0; r < 4; ++r)
        for (int c = 0; c < 4; ++c)
            grover = grover && w->coin_host[2 * (4 * r + c)] == (r == c ? -0.5 : 0.5) &&
                     w->coin_host[2 * (4 * r + c) + 1] == 0.0;
    if (w->shift == QW_SHIFT_FLIPFLOP) return grover ? go_backward<P, 1, 1>(w, a) : go_backward<P, 1, 0>(w, a);
    return grover ? go_backward<P, 0, 1>(w, a) : go_backward<P, 0, 0>(w, a);
}

}  // namespace qw

using namespace qw;

extern "C" qw_status qw_backward(qw_walk *w, const int64_t rect[4], int64_t T, int64_t K, double *loss_out,
                                 double *grad_phi, int on_device) {
    if (!w) return QW_EINVAL;
    NvtxRange nvtx("qw_backward");
    if (!rect || !grad_phi || T < 0 || K < 1) return set_error(w, QW_EINVAL, "bad rect, grad buffer, T or K");
    if (w->ndim != 2) return set_error(w, QW_EUNSUPPORTED, "qw_backward is defined on the torus");
    if (w->kind != CK_PHASE) return set_error(w, QW_ESTATE, "qw_backward needs a phase coin (qw_set_coin_phases)");
    if (w->prec != QW_F32 && w->prec != QW_F64) return set_error(w, QW_EUNSUPPORTED, "qw_backward runs in FP32 or FP64");
    if (w->bc != QW_BC_PERIODIC || links_on(w)) return set_error(w, QW_EUNSUPPORTED, "qw_backward needs the periodic torus");
    if (rect[0] < 0 || rect[1] < 0 || rect[2] < 0 || rect[3] < 0 || rect[0] + rect[2] > w->nx || rect[1] + rect[3] > w->ny)
        return set_error(w, QW_EINVAL, "rect outside the lattice");

    const int64_t nseg = (T + K - 1) / K;
    const size_t sb = w->state_bytes;
    const size_t gbytes = sizeof(double) * 4 * (size_t)w->ns;
    const size_t segbytes = (w->prec == QW_F32 ? 4 : 8) * 4 * (size_t)w->ns;   // per-segment accumulator
    const size_t need = (size_t)(nseg + 1) * sb + 2 * sb + (on_device ? 0 : gbytes) + segbytes + 256;
    cudaError_t e;
    if (w->grad_scratch_bytes < need) {
        cudaStreamSynchronize(w->stream);
        cudaFree(w->grad_scratch);
        w->grad_scratch = nullptr;
        w->grad_scratch_bytes = 0;
        if ((e = dev_alloc(&w->grad_scratch, need)) != cudaSuccess) return cuda_error(w, e, "gradient scratch");
        w->grad_scratch_bytes = need;
    }
    char *base = static_cast<char *>(w->grad_scratch);
    auto ckpt = [&](int64_t s) { return View{base + s * sb, w->pitch, w->d}; };
    View lam[2] = {View{base + (nseg + 1) * sb, w->pitch, w->d}, View{base + (nseg + 2) * sb, w->pitch, w->d}};
    double *grad = on_device ? grad_phi : reinterpret_cast<double *>(base + (nseg + 3) * sb);
    void *gseg = base + (nseg + 3) * sb + (on_device ? 0 : gbytes);

    // the start's support (the whole torus if nothing is known), searched here
    // when the steps are not clipped: the sweep's sites do not depend on that
    SupportBox start;
    qw_status rs = start_support(w, start);
    if (rs != QW_OK) return rs;
    const Arc psi_x = start.w ? Arc{start.x0, start.w} : Arc{0, w->nx}, psi_y = start.w ? Arc{start.y0, start.h} : Arc{0, w->ny};
    const Arc reg_x{rect[0], rect[2]}, reg_y{rect[1], rect[3]};

    // forward with a checkpoint every K steps
    e = cudaMemcpyAsync(ckpt(0).p, w->buf[w->cur], sb, cudaMemcpyDeviceToDevice, w->stream);
    if (e != cudaSuccess) return cuda_error(w, e, "checkpoint");
    for (int64_t s = 0; s < nseg; ++s) {
        qw_status st = run_steps(w, std::min(K, T - s * K), 0);
        if (st != QW_OK) return st;
        if ((e = cudaMemcpyAsync(ckpt(s + 1).p, w->buf[w->cur], sb, cudaMemcpyDeviceToDevice, w->stream)) != cudaSuccess)
            return cuda_error(w, e, "checkpoint");
    }

    // lambda_T and the loss; lambda is only ever written inside its light cone,
    // so both of its buffers start as zero
    const int nb = marginal_blocks();
    if ((e = cudaMemsetAsync(lam[0].p, 0, 2 * sb, w->stream)) != cudaSuccess) return cuda_error(w, e, "adjoint clear");
    if (w->prec == QW_F32)
        k_seed_region<P_F32><<<nb, 256, 0, w->stream>>>(ckpt(nseg), lam[0], w->nx, rect[0], rect[1], rect[2], rect[3], w->partials);
    else
        k_seed_region<P_F64><<<nb, 256, 0, w->stream>>>(ckpt(nseg), lam[0], w->nx, rect[0], rect[1], rect[2], rect[3], w->partials);
    k_sum_blocks<<<1, 32, 0, w->stream>>>(w->partials, nb, w->norm_dev);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_error(w, e, "region seed");
    if ((e = cudaMemsetAsync(grad, 0, gbytes, w->stream)) != cudaSuccess) return cuda_error(w, e, "gradient clear");
    if ((e = cudaMemsetAsync(gseg, 0, segbytes, w->stream)) != cudaSuccess) return cuda_error(w, e, "gradient clear");

    // backward, segment by segment, psi re-seeded from the checkpoint at each boundary
    int li = 0;
    for (int64_t s = nseg - 1; s >= 0; --s) {
        const int64_t t_hi = std::min((s + 1) * K, T), t_lo = s * K;
        View psi_in = ckpt(s + 1);
        int pi = 0;
        for (int64_t t = t_hi; t > t_lo;) {
            BackArgs a{};
            // 8 steps per launch where their tiles (16 x 16 outputs of 32 x 32) are
            // about one per SM, else 4 (24 x 24): the fewer sites for the halo
            for (int k : {8, 4}) {
                a.K = (int)std::min<int64_t>(k, t - t_lo);
                a.t0 = t - a.K;
                a.reach = (T - t_lo) + (a.t0 - t_lo);
                const Arc cx = arc_cover(arc_widen(psi_x, t - 1, w->nx), arc_widen(reg_x, a.reach, w->nx), w->nx);
                const Arc cy = arc_cover(arc_widen(psi_y, t - 1, w->ny), arc_widen(reg_y, a.reach, w->ny), w->ny);
                a.cx = cx.a; a.cw = cx.w; a.cy = cy.a; a.ch = cy.w;
                if (a.cw * a.ch <= BACK_DEEP_SITES) break;
            }
            a.lam_in = lam[li]; a.lam_out = lam[li ^ 1];
            a.psi_in = psi_in; a.psi_out = view_of(w, pi);
            a.nx = w->nx; a.ny = w->ny;
            a.psi_x = psi_x; a.psi_y = psi_y; a.reg_x = reg_x; a.reg_y = reg_y;
            a.T = T; a.phi = w->phi_dev; a.gseg = gseg;
            if (a.cw > 0 && a.ch > 0) {   // (else the cones do not meet: the gradient is zero)
                e = w->prec == QW_F32 ? backward_steps<P_F32>(w, a) : backward_steps<P_F64>(w, a);
                if (e != cudaSuccess) return cuda_error(w, e, "backward step");
            }
            li ^= 1;
            psi_in = a.psi_out;
            pi ^= 1;
            t = a.t0;
        }
        const int64_t n4 = 4 * w->ns;
        const unsigned fb = (unsigned)((n4 + 255) / 256);
        if (w->prec == QW_F32) k_flush_segment<float><<<fb, 256, 0, w->stream>>>(static_cast<float *>(gseg), grad, n4);
        else k_flush_segment<double><<<fb, 256, 0, w->stream>>>(static_cast<double *>(gseg), grad, n4);
        if ((e = cudaGetLastError()) != cudaSuccess) return cuda_error(w, e, "segment flush");
    }

    // leave the walk at psi_T; hand out the gradient and the loss (the sweep
    // used the walk's other buffer as scratch: it is no longer zero outside
    // the support box)
    w->next_clear = w->dirty_known = false;
    e = cudaMemcpyAsync(w->buf[w->cur], ckpt(nseg).p, sb, cudaMemcpyDeviceToDevice, w->stream);
    if (e == cudaSuccess && !on_device) e = cudaMemcpyAsync(grad_phi, grad, gbytes, cudaMemcpyDeviceToHost, w->stream);
    if (e == cudaSuccess && loss_out)
        e = cudaMemcpyAsync(w->host_scalar, w->norm_dev, sizeof(double), cudaMemcpyDeviceToHost, w->stream);
    if (e == cudaSuccess && (loss_out || !on_device)) e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess) return cuda_error(w, e, "gradient readout");
    if (loss_out) *loss_out = *w->host_scalar;
    return QW_OK;
}
