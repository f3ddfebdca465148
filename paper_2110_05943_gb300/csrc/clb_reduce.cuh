// clb_reduce.cuh -- FP64 reductions: mean Nusselt number of a wall (Sec. 3.2)
// and the steady-state residual.  Two-level and fixed-order (block tree of
// warp shuffles -> per-block partials -> one block), so results are
// bit-reproducible run to run.
#pragma once
#include "clb_kernels.cuh"

namespace clb {

constexpr int kRedThreads = 256;
constexpr int kMaxResidualBlocks = 2432;   // 152 SMs x 16 resident 256-thread blocks

// Number of partial slots a handle needs (per reduced quantity).
inline int reduce_partials(int nx, int ny) {
    const long long n = (long long)nx * ny;
    long long nb = (n + kRedThreads - 1) / kRedThreads;
    if (nb > kMaxResidualBlocks) nb = kMaxResidualBlocks;
    const int m = (nx > ny ? nx : ny);
    const long long nw = (m + kRedThreads - 1) / kRedThreads;
    return (int)(nb > nw ? nb : nw);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sum over a block of kRedThreads threads; the result is valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    v = warp_sum(v);
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    v = threadIdx.x < (kRedThreads / 32) ? sh[threadIdx.x] : 0.0;
    if (wid == 0) v = warp_sum(v);
    __syncthreads();
    return v;
}

// Temperature (Eq. 36) of node (x, y) at the current time level; wall nodes
// give their wall value or the second-order adiabatic extrapolation.
template <class P>
__device__ __forceinline__ double temperature_at(const BufT<const typename P::S>& B, const AuxT<typename P::R>& A,
                                                 const KParamsT<typename P::R>& K, int x, int y) {
    using R = typename P::R;
    WallInfo w;
    R v[5];
    // a rest-centred form carries T - T0
    const double toff = P::kCentred ? (double)K.T0 : 0.0;
    if (!wall_info(K.g, K.b, x, y, w)) {
        P::pull5(B, A, K, x, y, v);
        return toff + (double)(sum5(v) * K.p.inv_sigma);
    }
    if (w.st >= 0) return (double)K.b.Tw[w.st];
    P::pull5(B, A, K, x + w.dx, y + w.dy, v);
    const R Ts = sum5(v) * K.p.inv_sigma;
    P::pull5(B, A, K, x + 2 * w.dx, y + 2 * w.dy, v);
    const R Tss = sum5(v) * K.p.inv_sigma;
    return toff + (double)((R(4) * Ts - Tss) * R(1.0 / 3.0));
}

// Trapezoid-weighted local Nusselt number Nu = -L dT/dn / dT of node i of a
// wall of len nodes (FP64); `scale` = -L / (dT (len - 1)).
template <class P>
__device__ __forceinline__ double local_nusselt(const BufT<const typename P::S>& B, const AuxT<typename P::R>& A,
                                                const KParamsT<typename P::R>& K, int side, int i, int len,
                                                double scale) {
    const int e = (side == 1 ? K.g.nx : K.g.ny) - 1;
    double T[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        T[k] = side == 0   ? temperature_at<P>(B, A, K, k, i)
               : side == 1 ? temperature_at<P>(B, A, K, e - k, i)
               : side == 2 ? temperature_at<P>(B, A, K, i, k)
                           : temperature_at<P>(B, A, K, i, e - k);
    const double d = (side & 1) ? (3.0 * T[0] - 4.0 * T[1] + T[2]) * 0.5 : (-3.0 * T[0] + 4.0 * T[1] - T[2]) * 0.5;
    const double wgt = (i == 0 || i == len - 1) ? 0.5 : 1.0;
    return scale * d * wgt;
}

// Per-block partial sums of the local Nusselt numbers of one wall.
template <class P>
__global__ void __launch_bounds__(kRedThreads) k_nusselt_partial(const BufT<typename P::S> in,
                                                                 const AuxT<typename P::R> A,
                                                                 const KParamsT<typename P::R> K, int side,
                                                                 double scale, double* __restrict__ partial) {
    __shared__ double sh[kRedThreads / 32];
    const int len = side < 2 ? K.g.ny : K.g.nx;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double v = i < len ? local_nusselt<P>(as_const(in), A, K, side, i, len, scale) : 0.0;
    v = block_sum(v, sh);
    if (threadIdx.x == 0) partial[blockIdx.x] = v;
}

// Nusselt numbers of one wall of the cases of a batch, a block per case (each
// with two nodes along the wall and three across it at least):
// one launch and one copy for the whole batch (512 cases: 27 ms with two
// launches, a copy and a wait each, 0.1 ms now).  cur[c]: the case's current
// buffer; geom[c] = (L, dT).  The sums of 256 nodes and the sum over them run
// in the order of k_nusselt_partial and k_sum_partials: the same bits.
template <class P>
__global__ void __launch_bounds__(kRedThreads)
    k_nusselt_batch(const CaseT<typename P::R, typename P::S>* __restrict__ cases, const int* __restrict__ cur,
                    const double2* __restrict__ geom, int side, double* __restrict__ nu) {
    __shared__ double sh[kRedThreads / 32];
    __shared__ double part;
    const auto& C = cases[blockIdx.x];
    const BufT<const typename P::S> B = as_const(C.b[cur[blockIdx.x]]);
    const int len = side < 2 ? C.K.g.ny : C.K.g.nx;
    const double scale = -geom[blockIdx.x].x / geom[blockIdx.x].y / (double)(len - 1);
    double acc = 0.0;
    for (int b = 0; b * kRedThreads < len; ++b) {
        const int i = b * kRedThreads + threadIdx.x;
        const double v = block_sum(i < len ? local_nusselt<P>(B, C.A, C.K, side, i, len, scale) : 0.0, sh);
        if (threadIdx.x == 0) part = v;
        __syncthreads();
        if ((b & (kRedThreads - 1)) == (int)threadIdx.x) acc += part;
        __syncthreads();
    }
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) nu[blockIdx.x] = acc;
}

// Residual sums over all nodes: |u - u_ref|^2, |u|^2, (T - T_ref)^2, T^2;
// the reference is replaced by the current fields.  cur/ref hold
// (ux, uy, T) as three consecutive dense fields of n values.
__global__ void __launch_bounds__(kRedThreads) k_residual_partial(const double* __restrict__ cur,
                                                                  double* __restrict__ ref, long long n,
                                                                  double* __restrict__ partial, int nb) {
    __shared__ double sh[kRedThreads / 32];
    double du = 0.0, uu = 0.0, dt = 0.0, tt = 0.0;
    for (long long i = (long long)blockIdx.x * kRedThreads + threadIdx.x; i < n;
         i += (long long)gridDim.x * kRedThreads) {
        const double a = cur[i], b = cur[n + i], t = cur[2 * n + i];
        const double ea = a - ref[i], eb = b - ref[n + i], et = t - ref[2 * n + i];
        du = fma(ea, ea, fma(eb, eb, du));
        uu = fma(a, a, fma(b, b, uu));
        dt = fma(et, et, dt);
        tt = fma(t, t, tt);
        ref[i] = a;
        ref[n + i] = b;
        ref[2 * n + i] = t;
    }
    du = block_sum(du, sh);
    uu = block_sum(uu, sh);
    dt = block_sum(dt, sh);
    tt = block_sum(tt, sh);
    if (threadIdx.x == 0) {
        partial[0 * nb + blockIdx.x] = du;
        partial[1 * nb + blockIdx.x] = uu;
        partial[2 * nb + blockIdx.x] = dt;
        partial[3 * nb + blockIdx.x] = tt;
    }
}

// result[k] = sum_b partial[k * nb + b], k < nk, in a fixed order.
__global__ void __launch_bounds__(kRedThreads) k_sum_partials(const double* __restrict__ partial, int nb, int nk,
                                                              double* __restrict__ result) {
    __shared__ double sh[kRedThreads / 32];
    for (int k = 0; k < nk; ++k) {
        double v = 0.0;
        for (int b = threadIdx.x; b < nb; b += kRedThreads) v += partial[k * nb + b];
        v = block_sum(v, sh);
        if (threadIdx.x == 0) result[k] = v;
    }
}

}  // namespace clb
