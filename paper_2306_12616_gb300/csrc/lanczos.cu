// Lanczos spectral bounds: the tighter alternative to the Gershgorin discs.
//
// The expansion maps H onto [-1, 1] with its lowest and highest eigenvalues (Sec.
// "Chebyshev expansions with O(sqrt L) number of matrix multiplications"); Gershgorin discs
// enclose the spectrum but are several times wider than it for the tight-binding model, which
// costs resolution per term. K steps of the Lanczos process (float64, no reorthogonalisation:
// only the extreme Ritz values are used) give the extreme eigenvalues of the tridiagonal T_K;
// each is widened by its residual beta_{K+1} |y_K| (an eigenvalue of H lies that close) and by
// 1% of the width, and the result is intersected with the Gershgorin interval.
//
// Start vector: v_i = u_i - 1/2, u_i the i-th output of splitmix64 (Steele, Lea and Flood
// 2014) from a fixed seed, scaled to [0, 1): a counter-based draw, identical on any device.
#include <cooperative_groups.h>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace fo {
namespace {

constexpr uint64_t kLzSeed = 0x4C414E43ull;
constexpr double kLzMargin = 0.01;
constexpr int kLzLoads = 16;    // columns per lane in flight (matrix-vector product)
constexpr int kLzCluster = 8;   // one-warp blocks per instance of the update
constexpr int kLzKeep = 8;      // rows per thread of the update kept in registers

__device__ __forceinline__ double warp_sum_d(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ double block_sum_d(double v, double* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    v = warp_sum_d(v);
    __syncthreads();
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double t = lane < nw ? sh[lane] : 0.0;
        t = warp_sum_d(t);
        if (lane == 0) sh[32] = t;
    }
    __syncthreads();
    return sh[32];
}

// i-th splitmix64 output of the stream started at seed, in [0, 1).
__device__ __forceinline__ double splitmix_uniform(uint64_t seed, uint64_t i) {
    uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = z ^ (z >> 31);
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
}

// Per-instance state at in.lz: q_prev[np], q[np], w[np], alpha[kLzMax], beta[kLzMax + 1],
// steps done, stopped flag.
struct Lz {
    double *qp, *q, *w, *alpha, *beta, *meta;
};
__device__ __forceinline__ Lz lz_of(const Inst& in) {
    Lz z;
    z.qp = in.lz;
    z.q = z.qp + in.np;
    z.w = z.q + in.np;
    z.alpha = z.w + in.np;
    z.beta = z.alpha + kLzMax;
    z.meta = z.beta + kLzMax + 1;
    return z;
}

__global__ void k_lz_init(const Inst* __restrict__ insts, int batch) {
    pdl_sync();
    __shared__ double sh[33];
    const Inst& in = insts[blockIdx.x];
    const Lz z = lz_of(in);
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < in.np; i += blockDim.x) {
        const double v = i < in.n ? splitmix_uniform(kLzSeed, (uint64_t)i) - 0.5 : 0.0;
        z.q[i] = v;
        z.qp[i] = 0.0;
        s = fma(v, v, s);
    }
    s = block_sum_d(s, sh);
    const double inv = 1.0 / sqrt(s);
    for (int64_t i = threadIdx.x; i < in.np; i += blockDim.x) z.q[i] *= inv;
    if (threadIdx.x == 0) {
        z.beta[0] = 0.0;
        z.meta[0] = 0.0;   // steps done
        z.meta[1] = 0.0;   // stopped
    }
}

// w = H q - beta_j q_prev for the rows of this block (a warp per row); partial w . q. Bytes of H
// bound it (18 MB at N = 1501, from L2 after the first step): 16 columns per lane are loaded before
// they are used, in the order the sums take them (one load at a time kept 2 KB per warp in flight:
// 15.7 us per step at N = 1501, 12.3 now).
__global__ void __launch_bounds__(32 * kGershRows) k_lz_matvec(const Inst* __restrict__ insts,
                                                               const InstIO* io, Work wg, int j,
                                                               double* part) {
    pdl_sync();
    __shared__ double sp[kGershRows];
    const int b = blockIdx.x;
    const int i = inst_of(wg, b);
    const Inst& in = insts[i];
    const Lz z = lz_of(in);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = in.n, ld = io[i].ldh;
    const int64_t row = (int64_t)(b - wg.pre[i]) * kGershRows + warp;
    double d = 0.0;
    if (z.meta[1] == 0.0 && row < n) {
        const double* hr = io[i].H + row * ld;
        double s = 0.0;
        int64_t c = lane;
        for (; c + 32 * (kLzLoads - 1) < n; c += 32 * kLzLoads) {
            double hv[kLzLoads], qv[kLzLoads];
#pragma unroll
            for (int u = 0; u < kLzLoads; ++u) hv[u] = hr[c + 32 * u];
#pragma unroll
            for (int u = 0; u < kLzLoads; ++u) qv[u] = z.q[c + 32 * u];
#pragma unroll
            for (int u = 0; u < kLzLoads; ++u) s = fma(hv[u], qv[u], s);
        }
#pragma unroll 4
        for (; c < n; c += 32) s = fma(hr[c], z.q[c], s);
        s = warp_sum_d(s);
        const double wv = s - z.beta[j] * z.qp[row];
        if (lane == 0) z.w[row] = wv;
        d = wv * z.q[row];
    }
    if (lane == 0) sp[warp] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kGershRows; ++w) t += sp[w];
        part[b] = t;
    }
}

// alpha_j, w -= alpha_j q, beta_{j+1} = ||w||, q_prev = q, q = w / beta_{j+1}. Stops (for good) on
// an invariant subspace. One cluster of kLzCluster one-warp blocks per instance: row r belongs to
// thread r mod 256 of the cluster, the warps' sums are exchanged through distributed shared memory
// and added in warp order, as one block of 256 threads would (the same bits), but the float64
// divisions and shuffles, which one SM's float64 pipe (two lanes per clock) took 7 us for at
// N = 1501, run on eight. The partials of w . q are added in block order from shared memory (a
// thread adding them from global memory took 10 us).
__global__ void __cluster_dims__(kLzCluster, 1, 1) __launch_bounds__(32)
    k_lz_update(const Inst* __restrict__ insts, Work wg, int j, const double* part) {
    pdl_sync();
    constexpr int kChunk = 512;
    __shared__ double sp[kChunk];
    __shared__ double sh[kLzCluster];
    cg::cluster_group cl = cg::this_cluster();
    const int i = (int)blockIdx.x / kLzCluster, w = (int)cl.block_rank(), lane = threadIdx.x;
    const Inst& in = insts[i];
    const Lz z = lz_of(in);
    if (z.meta[1] != 0.0) return;   // written at the end of an earlier step: uniform over the cluster
    cl.sync();   // every block of the cluster runs before its shared memory is written
    const int64_t n = in.n;
    const double bj = z.beta[j];
    const int p0 = wg.pre[i], p1 = wg.pre[i + 1];
    // up to kLzKeep of this thread's rows stay in registers, requested before the sum of the partials
    double wk[kLzKeep], qk[kLzKeep];
#pragma unroll
    for (int u = 0; u < kLzKeep; ++u) {
        const int64_t r = w * 32 + lane + (int64_t)u * 32 * kLzCluster;
        wk[u] = r < n ? z.w[r] : 0.0;
        qk[u] = r < n ? z.q[r] : 0.0;
    }
    double a = 0.0;
    for (int c0 = p0; c0 < p1; c0 += kChunk) {
        const int m = p1 - c0 < kChunk ? p1 - c0 : kChunk;
        for (int q = lane; q < m; q += 32) sp[q] = part[c0 + q];
        __syncwarp();
#pragma unroll 8
        for (int q = 0; q < m; ++q) a += sp[q];   // every lane the same sum
        __syncwarp();
    }
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < kLzKeep; ++u) {
        if (w * 32 + lane + (int64_t)u * 32 * kLzCluster >= n) break;
        wk[u] = wk[u] - a * qk[u];
        s = fma(wk[u], wk[u], s);
    }
    const int64_t rest = w * 32 + lane + (int64_t)kLzKeep * 32 * kLzCluster;
    for (int64_t r = rest; r < n; r += 32 * kLzCluster) {
        const double wv = z.w[r] - a * z.q[r];
        z.w[r] = wv;
        s = fma(wv, wv, s);
    }
    s = warp_sum_d(s);
    if (lane < kLzCluster) *cl.map_shared_rank(&sh[w], lane) = s;
    cl.sync();
    const double bnext = sqrt(warp_sum_d(lane < kLzCluster ? sh[lane] : 0.0));
    // an invariant subspace, or n steps (the whole space)
    const bool stop = !(bnext > 1e-12 * (fabs(a) + bj)) || j + 1 >= n;
    if (!stop) {
#pragma unroll
        for (int u = 0; u < kLzKeep; ++u) {
            const int64_t r = w * 32 + lane + (int64_t)u * 32 * kLzCluster;
            if (r >= n) break;
            z.qp[r] = qk[u];
            z.q[r] = wk[u] / bnext;
        }
        for (int64_t r = rest; r < n; r += 32 * kLzCluster) {
            z.qp[r] = z.q[r];
            z.q[r] = z.w[r] / bnext;
        }
    }
    cl.sync();   // every block has read the record before it changes, and left the shared sums
    if (w == 0 && lane == 0) {
        z.alpha[j] = a;
        z.beta[j + 1] = bnext;
        z.meta[0] = (double)(j + 1);
        if (stop) z.meta[1] = 1.0;
    }
}

// Number of eigenvalues of the K x K tridiagonal below x (Sturm); beta2[j] = beta_j^2.
__device__ int sturm_count(const double* alpha, const double* beta2, int K, double x) {
    int c = 0;
    double d = alpha[0] - x;
    if (d < 0.0) ++c;
    for (int j = 1; j < K; ++j) {
        if (d == 0.0) d = 1e-300;
        d = (alpha[j] - x) - beta2[j] / d;
        if (d < 0.0) ++c;
    }
    return c;
}

// |last component| of the unit eigenvector for the eigenvalue theta (forward recurrence,
// the stable direction for an extreme eigenvalue), rescaled against overflow.
__device__ double last_component(const double* alpha, const double* beta, int K, double theta) {
    double ym = 0.0, y = 1.0, nrm = 1.0;
    for (int j = 0; j + 1 < K; ++j) {
        const double yn = ((theta - alpha[j]) * y - (j > 0 ? beta[j] * ym : 0.0)) / beta[j + 1];
        ym = y;
        y = yn;
        nrm += y * y;
        if (nrm > 1e200) {
            const double s = 1e-100;
            y *= s;
            ym *= s;
            nrm *= s * s;
        }
    }
    return fabs(y) / sqrt(nrm);
}

// One block of two warps per instance, a warp per end of the spectrum. The bisection's steps depend
// on one another, so a warp looks five of them ahead: lane i evaluates the Sturm count of node i
// of the tree of the next midpoints (31 nodes, each midpoint formed by the same halvings), and the
// path is then followed with the bisection's own test at every level: the same sequence, hence
// the same bits, in a fifth of the dependent rounds (40 steps: 2.13 ms with one thread, 0.24 now).
__global__ void __launch_bounds__(64) k_lz_bounds(const Inst* __restrict__ insts) {
    pdl_sync();
    __shared__ double alpha[kLzMax], beta[kLzMax + 1], beta2[kLzMax + 1], s_th[2], s_rs[2];
    const Inst& in = insts[blockIdx.x];
    const Lz z = lz_of(in);
    DevResult* res = in.res;
    const int K = (int)z.meta[0];
    if (K < 1) return;
    const int lane = threadIdx.x & 31, e = threadIdx.x >> 5;
    for (int j = threadIdx.x; j <= K; j += 64) {
        if (j < K) alpha[j] = z.alpha[j];
        const double b = z.beta[j];
        beta[j] = b;
        beta2[j] = b * b;
    }
    __syncthreads();
    // an enclosure of T's eigenvalues for the bisection
    double lo = INFINITY, hi = -INFINITY;
    for (int j = lane; j < K; j += 32) {
        const double r = (j > 0 ? fabs(beta[j]) : 0.0) + (j + 1 < K ? fabs(beta[j + 1]) : 0.0);
        lo = fmin(lo, alpha[j] - r);
        hi = fmax(hi, alpha[j] + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const int target = e == 0 ? 1 : K;   // smallest x with count(x) >= target
    double a = lo, b = hi;
    int it = 0;
    for (bool stop = false; !stop;) {
        // this lane's node: the bits of its index below the leading one are the turns from the
        // root (0: b = mid, 1: a = mid)
        double na = a, nb = b;
        const int depth = 31 - __clz(lane | 1);
        for (int d = depth - 1; d >= 0; --d) {
            const double mid = 0.5 * (na + nb);
            if ((lane >> d) & 1) na = mid;
            else nb = mid;
        }
        const bool left = lane > 0 && sturm_count(alpha, beta2, K, 0.5 * (na + nb)) >= target;
        const unsigned turns = __ballot_sync(0xffffffffu, left);
        int node = 1;
        for (int d = 0; d < 5; ++d) {
            if (!(it < 200 && b - a > 1e-15 * fmax(1.0, fmax(fabs(a), fabs(b))))) {
                stop = true;
                break;
            }
            const double mid = 0.5 * (a + b);
            const bool l = (turns >> node) & 1u;
            if (l) b = mid;
            else a = mid;
            node = 2 * node + (l ? 0 : 1);
            ++it;
        }
    }
    if (lane == 0) {
        const double th = 0.5 * (a + b);
        s_th[e] = th;
        s_rs[e] = K > 1 ? beta[K] * last_component(alpha, beta, K, th) : beta[K];
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double width = s_th[1] - s_th[0];
    double el = s_th[0] - s_rs[0] - kLzMargin * width;
    double eh = s_th[1] + s_rs[1] + kLzMargin * width;
    el = fmax(el, res->bounds[0]);
    eh = fmin(eh, res->bounds[1]);
    if (!(eh - el > 1e-12 * fmax(1.0, fmax(fabs(el), fabs(eh))))) {
        const double c = 0.5 * (el + eh);
        el = c - 1.0;
        eh = c + 1.0;
    }
    if (res->nonfinite) return;   // keep the Gershgorin record of a non-finite H
    res->bounds[0] = el;
    res->bounds[1] = eh;
}

}  // namespace

cudaError_t launch_lanczos(const Inst* in, const InstIO* io, int batch, Work wg, double* part, int steps,
                           cudaStream_t s, int* launches) {
    if (steps < 1) return cudaSuccess;
    if (steps > kLzMax) steps = kLzMax;
    launch_pdl(batch, k_lz_init, batch, 256, 0, s, in, batch);
    for (int j = 0; j < steps; ++j) {
        launch_pdl(batch, k_lz_matvec, wg.total, 32 * kGershRows, 0, s, in, io, wg, j, part);
        launch_pdl(batch, k_lz_update, batch * kLzCluster, 32, 0, s, in, wg, j, part);
    }
    launch_pdl(batch, k_lz_bounds, batch, 64, 0, s, in);
    if (launches) *launches += 2 + 2 * steps;
    return cudaGetLastError();
}

}  // namespace fo
