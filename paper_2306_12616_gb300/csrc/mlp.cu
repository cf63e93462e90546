// Learned chemical potential: features, the network (forward, backward, Adam), the
// proposal of mu and the trace judge with its corrections.
//
// The paper fixes mu by hand. Here a small fully connected network (68 -> 256 -> 256 -> 2,
// SiLU, float32) maps the moments tau_1..tau_64 / N that the baby steps already give (plus
// N_e / N, kT on the scaled axis and the bounds) to mu on the scaled axis and to the order
// of the expansion; it is trained on (H, mu) pairs the exact method generates. A proposed
// mu is only kept when the float64 trace of the resulting P meets the tolerance; otherwise
// mu is corrected from tr P and ||P||_F^2 (Newton, then secant) and P re-evaluated, and
// instances that still miss fall back to exact moments and bisection.
//
// Every reduction runs in a fixed order (one thread per output, sequential sums), so
// training and inference are deterministic.
#include <cooperative_groups.h>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace fo {
namespace {

__device__ __forceinline__ float silu_f(float z) { return z / (1.0f + expf(-z)); }
__device__ __forceinline__ float silu_grad_f(float z) {
    const float s = 1.0f / (1.0f + expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

// ------------------------------------------------------------------ rows of a batch
// Everything of a training step that is local to a row of the batch: gather and standardise, the
// three layers, the loss gradient and the gradients of the pre-activations. A cluster of kCl CTAs
// takes kRows rows; each CTA holds 256 / kCl hidden units of either layer: its rows of W1 and W2
// and its columns of W2 (the backward pass) are copied to shared memory at the start, while the
// first layer runs, and activations are exchanged through distributed shared memory (three
// times). The weights' bytes bound it: 145 KB per CTA from L2, about 2300 clocks, as long as the
// sums of a layer; one CTA per two rows would read all 580 KB. Every sum runs in the order of its
// definition, one term after another in one thread.
// One training step of 256 rows, with k_mlp_grad: 2 launches and 31 us, where 11 launches took about
// 205 us (20000 rows, two epochs: 33.5 -> 4.9 ms; 5.3 while the row indices, targets, biases and Adam's
// state were requested where they are used and the output sums read eight rows of one bank).
constexpr int kCl = 4;                          // CTAs per cluster
constexpr int kRows = 8;                        // rows per cluster
constexpr int kUnits = kMlpHidden / kCl;        // hidden units per CTA
constexpr int kRowThreads = kUnits * (kRows / 2);   // a thread: one unit, two rows
constexpr int kLd1 = kMlpIn;                    // shared strides: an odd number of 16-byte words, so that
constexpr int kLd2 = kMlpHidden + 4;            // the rows of a warp's lanes start in different banks
static_assert(kLd1 % 8 == 4 && kLd2 % 8 == 4, "strides");

struct RowSmem {
    float w1[kUnits * kLd1];          // rows of W1
    float w2r[kUnits * kLd2];         // rows of W2 (forward)
    float w2c[kMlpHidden * kUnits];   // columns of W2 (backward)
    float w3[kMlpOut * kMlpHidden];
    float x[kRows * kMlpIn];
    float a1[kRows * kMlpHidden];
    float a2[kRows * kMlpHidden];
    float dz2[kRows * kMlpHidden];
    float dy[kRows * kMlpOut];
};

struct RowArgs {
    const float *params, *src, *tsrc;   // parameters; features and targets [. x 68], [. x 2]
    const int* idx;                     // rows of src / tsrc (null: row b)
    const float* norm;                  // standardisation (null: src and tsrc are standardised)
    int B;
    float *x, *t;                       // standardised rows [B x 68], [B x 2] (training)
    float *a1, *a2, *dz1, *dz2;         // [B x 256]
    float *y, *dy;                      // [B x 2]
};

template <bool TRAIN>
__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(kRowThreads) k_mlp_rows(const RowArgs g) {
    extern __shared__ __align__(16) unsigned char raw[];
    RowSmem& sm = *reinterpret_cast<RowSmem*>(raw);
    cg::cluster_group cl = cg::this_cluster();
    const int c = (int)cl.block_rank(), u0 = c * kUnits;
    const int b0 = ((int)blockIdx.x / kCl) * kRows, tid = threadIdx.x;
    const float* W1 = g.params;
    const float* B1 = W1 + kMlpHidden * kMlpIn;
    const float* W2 = B1 + kMlpHidden;
    const float* B2 = W2 + kMlpHidden * kMlpHidden;
    const float* W3 = B2 + kMlpHidden;
    const float* B3 = W3 + kMlpOut * kMlpHidden;
    // this thread: hidden unit u0 + o of rows 2 rg, 2 rg + 1
    const int o = tid % kUnits, rg = tid / kUnits, r0 = 2 * rg;
    // what is read once and used late is requested first, ahead of the weights' copies: the rows (through
    // their indices), the biases and, in the threads of the outputs, their target
    constexpr int NX = (kRows * kMlpIn + kRowThreads - 1) / kRowThreads;
    float xv[NX], xm[NX], xs[NX];
#pragma unroll
    for (int u = 0; u < NX; ++u) {
        const int q = tid + u * kRowThreads, rr = q / kMlpIn, i = q - rr * kMlpIn, b = b0 + rr;
        xv[u] = xm[u] = 0.0f;
        xs[u] = 1.0f;
        if (q < kRows * kMlpIn && b < g.B) {
            xv[u] = g.src[(int64_t)(g.idx ? g.idx[b] : b) * kMlpIn + i];
            if (g.norm) {
                xm[u] = g.norm[i];
                xs[u] = g.norm[kMlpIn + i];
            }
        }
    }
    const float bias1 = B1[u0 + o], bias2 = B2[u0 + o];
    float bias3 = 0.0f, t = 0.0f;
    if (tid < kRows * kMlpOut) {
        const int rr = tid / kMlpOut, j = tid - rr * kMlpOut, b = b0 + rr;
        bias3 = B3[j];
        if (TRAIN && b < g.B) {
            t = g.tsrc[(int64_t)(g.idx ? g.idx[b] : b) * kMlpOut + j];
            if (g.norm) t = (t - g.norm[2 * kMlpIn + j]) / g.norm[2 * kMlpIn + kMlpOut + j];
        }
    }
    // group 0: W1; group 1: W2's rows and W3; group 2: W2's columns
    for (int q = tid; q < kUnits * (kMlpIn / 4); q += kRowThreads) {
        const int o = q / (kMlpIn / 4), i = 4 * (q - o * (kMlpIn / 4));
        cp_async16(&sm.w1[o * kLd1 + i], W1 + (u0 + o) * kMlpIn + i);
    }
    cp_async_commit();
    for (int q = tid; q < kUnits * (kMlpHidden / 4); q += kRowThreads) {
        const int o = q / (kMlpHidden / 4), i = 4 * (q - o * (kMlpHidden / 4));
        cp_async16(&sm.w2r[o * kLd2 + i], W2 + (u0 + o) * kMlpHidden + i);
    }
    for (int q = tid; q < kMlpOut * kMlpHidden; q += kRowThreads) sm.w3[q] = W3[q];
    cp_async_commit();
    if (TRAIN) {
        for (int q = tid; q < kMlpHidden * (kUnits / 4); q += kRowThreads) {
            const int o = q / (kUnits / 4), i = 4 * (q - o * (kUnits / 4));
            cp_async16(&sm.w2c[o * kUnits + i], W2 + o * kMlpHidden + u0 + i);
        }
    }
    cp_async_commit();
#pragma unroll
    for (int u = 0; u < NX; ++u) {
        const int q = tid + u * kRowThreads, rr = q / kMlpIn, i = q - rr * kMlpIn, b = b0 + rr;
        if (q >= kRows * kMlpIn) break;
        float v = xv[u];
        if (g.norm) v = (v - xm[u]) / xs[u];   // (0 past the batch)
        if (TRAIN && c == 0 && b < g.B) g.x[(int64_t)b * kMlpIn + i] = v;
        sm.x[q] = v;
    }
    cp_async_wait<2>();
    __syncthreads();
    cl.sync();   // every CTA of the cluster runs before its shared memory is written
    auto share = [&](float* dst, float v0, float v1) {   // into every CTA's copy
#pragma unroll
        for (int q = 0; q < kCl; ++q) {
            float* d = cl.map_shared_rank(dst, q);
            d[r0 * kMlpHidden + u0 + o] = v0;
            d[(r0 + 1) * kMlpHidden + u0 + o] = v1;
        }
    };
    auto keep = [&](float* dst, float v0, float v1) {     // [B x 256] in global memory
        if (b0 + r0 < g.B) dst[(int64_t)(b0 + r0) * kMlpHidden + u0 + o] = v0;
        if (b0 + r0 + 1 < g.B) dst[(int64_t)(b0 + r0 + 1) * kMlpHidden + u0 + o] = v1;
    };
    auto layer = [&](const float* w, const float* in, int n, float bias, float& s0, float& s1) {
        s0 = s1 = bias;
        const float *x0 = in + r0 * n, *x1 = x0 + n;
#pragma unroll 4
        for (int i = 0; i < n; i += 4) {
            const float4 wv = *reinterpret_cast<const float4*>(w + i);
            const float4 p = *reinterpret_cast<const float4*>(x0 + i), q = *reinterpret_cast<const float4*>(x1 + i);
            s0 = fmaf(p.x, wv.x, s0);
            s1 = fmaf(q.x, wv.x, s1);
            s0 = fmaf(p.y, wv.y, s0);
            s1 = fmaf(q.y, wv.y, s1);
            s0 = fmaf(p.z, wv.z, s0);
            s1 = fmaf(q.z, wv.z, s1);
            s0 = fmaf(p.w, wv.w, s0);
            s1 = fmaf(q.w, wv.w, s1);
        }
    };
    float z10, z11, z20, z21;
    layer(sm.w1 + o * kLd1, sm.x, kMlpIn, bias1, z10, z11);
    {
        const float v0 = silu_f(z10), v1 = silu_f(z11);
        share(sm.a1, v0, v1);
        if (TRAIN) keep(g.a1, v0, v1);
    }
    cp_async_wait<1>();
    cl.sync();
    layer(sm.w2r + o * kLd2, sm.a1, kMlpHidden, bias2, z20, z21);
    {
        const float v0 = silu_f(z20), v1 = silu_f(z21);
        share(sm.a2, v0, v1);
        if (TRAIN) keep(g.a2, v0, v1);
    }
    cp_async_wait<0>();
    cl.sync();
    if (tid < kRows * kMlpOut) {
        // the outputs, in every CTA (the backward pass of each needs them)
        const int rr = tid / kMlpOut, j = tid - rr * kMlpOut, b = b0 + rr;
        float s = bias3;
        const float *w = sm.w3 + j * kMlpHidden, *a = sm.a2 + rr * kMlpHidden;
        // (the eight rows lie in the same banks: one 16-byte read serves four terms)
#pragma unroll 4
        for (int i = 0; i < kMlpHidden; i += 4) {
            const float4 p = *reinterpret_cast<const float4*>(a + i), wv = *reinterpret_cast<const float4*>(w + i);
            s = fmaf(p.x, wv.x, s);
            s = fmaf(p.y, wv.y, s);
            s = fmaf(p.z, wv.z, s);
            s = fmaf(p.w, wv.w, s);
        }
        if (b < g.B) {
            if (c == 0) g.y[(int64_t)b * kMlpOut + j] = s;
            if (TRAIN) {
                const float wl = j ? kMlpLossW1 : kMlpLossW0;
                const float d = s - t;
                const float dv = 2.0f * wl * d / (float)g.B;
                sm.dy[tid] = dv;
                if (c == 0) {
                    g.t[(int64_t)b * kMlpOut + j] = t;
                    g.dy[(int64_t)b * kMlpOut + j] = dv;
                }
            }
        } else if (TRAIN) {
            sm.dy[tid] = 0.0f;
        }
    }
    if (!TRAIN) return;   // (no CTA touches another's shared memory past the last cl.sync)
    __syncthreads();
    {
        // dz2 = (sum_j dy_j W3[j, .]) silu'(z2)
        float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
        for (int j = 0; j < kMlpOut; ++j) {
            const float w = sm.w3[j * kMlpHidden + u0 + o];
            s0 = fmaf(sm.dy[r0 * kMlpOut + j], w, s0);
            s1 = fmaf(sm.dy[(r0 + 1) * kMlpOut + j], w, s1);
        }
        const float v0 = s0 * silu_grad_f(z20), v1 = s1 * silu_grad_f(z21);
        share(sm.dz2, v0, v1);
        keep(g.dz2, v0, v1);
    }
    cl.sync();
    {
        // dz1 = (sum_o dz2_o W2[o, .]) silu'(z1)
        float s0 = 0.0f, s1 = 0.0f;
        const float *p = sm.dz2 + r0 * kMlpHidden, *q = p + kMlpHidden;
#pragma unroll 4
        for (int k = 0; k < kMlpHidden; k += 4) {
            const float4 d0 = *reinterpret_cast<const float4*>(p + k), d1 = *reinterpret_cast<const float4*>(q + k);
            const float* w = sm.w2c + k * kUnits + o;
            s0 = fmaf(d0.x, w[0], s0);
            s1 = fmaf(d1.x, w[0], s1);
            s0 = fmaf(d0.y, w[kUnits], s0);
            s1 = fmaf(d1.y, w[kUnits], s1);
            s0 = fmaf(d0.z, w[2 * kUnits], s0);
            s1 = fmaf(d1.z, w[2 * kUnits], s1);
            s0 = fmaf(d0.w, w[3 * kUnits], s0);
            s1 = fmaf(d1.w, w[3 * kUnits], s1);
        }
        keep(g.dz1, s0 * silu_grad_f(z10), s1 * silu_grad_f(z11));
    }
}

// ------------------------------------------------------------------ weight gradients, Adam, loss
// dW[o, i] = sum_b dZ[b, o] A[b, i] (one thread per parameter group, b in order), db[o] = sum_b
// dZ[b, o] as the column i = I with A = 1, of all three layers in one launch, then either the
// gradient itself or one Adam step of the parameter (Kingma and Ba, bias-corrected, step from 1);
// one more block adds the loss. A block: kGo outputs x kGi inputs, 128 threads of 1 x 4 parameters;
// 16 x 32 tiles give 202 blocks for the 152 SMs. Latency bounds it, so dZ and A are requested whole
// (up to kGb rows) by asynchronous copies before any sum starts (four staged passes took a quarter longer).
constexpr int kGo = 16, kGi = 32, kGb = 256;
constexpr int kGradSmem = kGb * (kGo + kGi) * 4;
constexpr int kTilesI1 = (kMlpIn + 1 + kGi - 1) / kGi, kTilesI2 = (kMlpHidden + 1 + kGi - 1) / kGi;
constexpr int kTilesO = kMlpHidden / kGo;
constexpr int kGradBlocks = kTilesO * kTilesI1 + kTilesO * kTilesI2 + kTilesI2 + 1;

struct GradArgs {
    const float *x, *a1, *a2, *dz1, *dz2, *dy, *y, *t;
    int B;
    float* grad;          // gradient out (null: Adam)
    float *p, *m, *v;     // Adam: parameters and moments
    float lr;
    int step;
    float* loss;
};

__global__ void __launch_bounds__(128) k_mlp_grad(const GradArgs g) {
    extern __shared__ __align__(16) float gsm[];
    float (*sz)[kGo] = reinterpret_cast<float (*)[kGo]>(gsm);
    float (*sa)[kGi] = reinterpret_cast<float (*)[kGi]>(gsm + kGb * kGo);
    __shared__ float s_corr[2];
    const int tid = threadIdx.x;
    int blk = blockIdx.x;
    if (blk == kGradBlocks - 1) {
        // L = (1/B) sum_b sum_j w_j (y - t)^2: 256 strided float64 sums (two per thread here), a
        // shuffle tree per 32 of them, their eight results in order
        __shared__ double sh[8];
        for (int half = 0; half < 2; ++half) {
            double s = 0.0;
            for (int q = tid + 128 * half; q < 2 * g.B; q += 256) {
                const float w = (q & 1) ? kMlpLossW1 : kMlpLossW0;
                const float d = g.y[q] - g.t[q];
                s += (double)w * d * d;
            }
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if ((tid & 31) == 0) sh[4 * half + (tid >> 5)] = s;
        }
        __syncthreads();
        if (tid == 0) {
            double tot = 0.0;
            for (int w = 0; w < 8; ++w) tot += sh[w];
            *g.loss = (float)(tot / g.B);
        }
        return;
    }
    // layer, output tile, input tile; parameters W (O x I) at off, then the O biases
    const float *dz, *A;
    int O, I, off, ot, it;
    if (blk < kTilesO * kTilesI2) {
        dz = g.dz2;
        A = g.a1;
        O = kMlpHidden;
        I = kMlpHidden;
        off = kMlpHidden * kMlpIn + kMlpHidden;
        ot = blk / kTilesI2;
        it = blk - ot * kTilesI2;
    } else if ((blk -= kTilesO * kTilesI2) < kTilesO * kTilesI1) {
        dz = g.dz1;
        A = g.x;
        O = kMlpHidden;
        I = kMlpIn;
        off = 0;
        ot = blk / kTilesI1;
        it = blk - ot * kTilesI1;
    } else {
        blk -= kTilesO * kTilesI1;
        dz = g.dy;
        A = g.a2;
        O = kMlpOut;
        I = kMlpHidden;
        off = kMlpHidden * kMlpIn + kMlpHidden + kMlpHidden * kMlpHidden + kMlpHidden;
        ot = 0;
        it = blk;
    }
    const int o0 = ot * kGo, i0 = it * kGi;
    if (!g.grad && tid == 0) {
        s_corr[0] = 1.0f - powf(0.9f, (float)g.step);
        s_corr[1] = 1.0f - powf(0.999f, (float)g.step);
    }
    const int o = tid >> 3, i4 = (tid & 7) * 4;
    // Adam's state of this thread's parameters, requested before the sums
    float pm[4], pv[4], pp[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = i0 + i4 + u;
        const int q = i < I ? off + (o0 + o) * I + i : off + O * I + o0 + o;
        const bool mine = !g.grad && o0 + o < O && i <= I;
        pm[u] = mine ? g.m[q] : 0.0f;
        pv[u] = mine ? g.v[q] : 0.0f;
        pp[u] = mine ? g.p[q] : 0.0f;
    }
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int b0 = 0; b0 < g.B; b0 += kGb) {
        const int nb = g.B - b0 < kGb ? g.B - b0 : kGb;
        __syncthreads();
        if (O % 4 == 0) {
            for (int q = tid; q < nb * (kGo / 4); q += 128) {
                const int b = q / (kGo / 4), oo = 4 * (q % (kGo / 4));
                cp_async16(&sz[b][oo], dz + (int64_t)(b0 + b) * O + o0 + oo);
            }
        } else {
            for (int q = tid; q < nb * kGo; q += 128) {
                const int b = q / kGo, oo = q % kGo;
                sz[b][oo] = o0 + oo < O ? dz[(int64_t)(b0 + b) * O + o0 + oo] : 0.0f;
            }
        }
        for (int q = tid; q < nb * (kGi / 4); q += 128) {
            const int b = q / (kGi / 4), ii = 4 * (q % (kGi / 4));
            // (I is a multiple of 4: a group of four columns is inside the inputs, or starts at the
            // bias column, or lies past it)
            if (i0 + ii < I) cp_async16(&sa[b][ii], A + (int64_t)(b0 + b) * I + i0 + ii);
            else *reinterpret_cast<float4*>(&sa[b][ii]) = make_float4(i0 + ii == I ? 1.0f : 0.0f, 0.0f, 0.0f, 0.0f);
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
#pragma unroll 8
        for (int b = 0; b < nb; ++b) {
            const float z = sz[b][o];
            const float4 a = *reinterpret_cast<const float4*>(&sa[b][i4]);
            s[0] = fmaf(z, a.x, s[0]);
            s[1] = fmaf(z, a.y, s[1]);
            s[2] = fmaf(z, a.z, s[2]);
            s[3] = fmaf(z, a.w, s[3]);
        }
    }
    if (o0 + o >= O) return;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = i0 + i4 + u;
        if (i > I) break;
        const int q = i < I ? off + (o0 + o) * I + i : off + O * I + o0 + o;
        if (g.grad) {
            g.grad[q] = s[u];
        } else {
            const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
            // the products that are rounded by themselves, written out: left to the compiler, constant
            // b1 and b2 moved the contraction to the other product
            const float mq = fmaf(b1, pm[u], (1.0f - b1) * s[u]);
            const float vq = fmaf(b2, pv[u], (1.0f - b2) * s[u] * s[u]);
            g.m[q] = mq;
            g.v[q] = vq;
            const float mh = mq / s_corr[0];
            const float vh = vq / s_corr[1];
            g.p[q] = pp[u] - g.lr * mh / (sqrtf(vh) + eps);
        }
    }
}

// Column mean and standard deviation (float64 sums in row order); std floored at 1e-6 of
// max(1, |mean|) so that constant columns map to zero. One block per column.
__global__ void k_col_stats(const float* __restrict__ X, int n, int C, float* __restrict__ mean,
                            float* __restrict__ stdv) {
    __shared__ double sh[2][32];
    const int c = blockIdx.x;
    double s = 0.0, q = 0.0;
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        const double v = X[(int64_t)r * C + c];
        s += v;
        q += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = s; sh[1][threadIdx.x >> 5] = q; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ts = 0.0, tq = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { ts += sh[0][w]; tq += sh[1][w]; }
        const double mu = ts / n;
        const double var = fmax(tq / n - mu * mu, 0.0);
        mean[c] = (float)mu;
        stdv[c] = (float)fmax(sqrt(var), 1e-6 * fmax(1.0, fabs(mu)));
    }
}

// Features of every instance (row = caller index when rows_by_user, else plan order):
// tau_1..tau_64 / n (tau_j, j > 2k, zero), N_e / n, 2 kT / (e_b - e_a), e_a / 100, e_b / 100.
__global__ void k_features(const Inst* __restrict__ insts, const InstIO* io, int batch, int k,
                           int rows_by_user, float* __restrict__ feat) {
    const int i = blockIdx.x, c = threadIdx.x;
    if (i >= batch || c >= kMlpIn) return;
    const Inst& in = insts[i];
    const DevResult* r = in.res;
    const double n = (double)in.n;
    const double ea = r->bounds[0], eb = r->bounds[1];
    double v = 0.0;
    if (c < kMlpMoments) v = (c + 1 <= 2 * k) ? in.tau[c + 1] / n : 0.0;
    else if (c == kMlpMoments) v = io[i].n_e / n;
    else if (c == kMlpMoments + 1) v = 2.0 * io[i].kT / (eb - ea);
    else if (c == kMlpMoments + 2) v = ea / 100.0;
    else v = eb / 100.0;
    const int row = rows_by_user ? in.user : i;
    feat[(int64_t)row * kMlpIn + c] = (float)v;
}

// Targets (mu_x, log2(L*) / log2(n_terms)) of every instance, from its mu, bounds and
// coefficients c_j(mu) (L*: the smallest L with sum_{j >= L} |c_j| <= kOrderEps). Row =
// caller index.
__global__ void k_targets(const Inst* __restrict__ insts, int batch, int n_terms, float* __restrict__ tgt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= batch) return;
    const Inst& in = insts[i];
    const DevResult* r = in.res;
    const double ea = r->bounds[0], eb = r->bounds[1];
    // the order target: the smallest L with sum_{j >= L} |c_j| <= kOrderEps, so that the
    // expansion cut at L terms is within kOrderEps of the full one in the 2-norm
    double tail = 0.0;
    int L = n_terms;
    for (int j = n_terms - 1; j >= 1; --j) {
        tail += fabs(in.c[j]);
        if (tail > kOrderEps) break;
        L = j;
    }
    const double lg = n_terms > 1 ? log2((double)n_terms) : 1.0;
    tgt[(int64_t)in.user * 2] = (float)((2.0 * r->mu - (ea + eb)) / (eb - ea));
    tgt[(int64_t)in.user * 2 + 1] = (float)(log2((double)(L > 1 ? L : 1)) / lg);
}

// Low moments tau_0..tau_{2k} from the baby-step traces diag[0..k) (T_1..T_k) and
// gram[i-1] = <T_k, T_i>, i = 1..k: tau_{k+i} = 2 <T_k, T_i> - tau_{k-i} (Eq. identity).
__global__ void k_assemble_low(const Inst* __restrict__ insts, int batch, int k) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= batch) return;
    const Inst& in = insts[i];
    if (!in.res->active) return;
    double* tau = in.tau;
    tau[0] = (double)in.n;
    for (int j = 1; j <= k; ++j) tau[j] = in.diag[j - 1];
    for (int j = 1; j <= k; ++j) tau[k + j] = 2.0 * in.gram[j - 1] - tau[k - j];
}

// mu0 = mid + half (m_x + s_x y0) clamped into the bounds, order = n_terms^(m_o + s_o y1).
// The network's proposals: mu, and the expansion order L* (the number of terms whose
// coefficient tail sum_{j >= L*} |c_j| is at most kOrderEps). With use_order the instance's expansion is cut at
// n_eff = k m_eff coefficients, m_eff = ceil(margin L* / k) giant steps, clamped to [2, m]:
// every coefficient from n_eff on is zero, and the products whose outputs that leaves zero
// or unused are skipped (step_needed).
__global__ void k_learned_mu(const Inst* __restrict__ insts, int batch, const float* __restrict__ y,
                             const float* __restrict__ norm, int n_terms, int k, int m, int use_order,
                             double margin) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= batch) return;
    DevResult* r = insts[i].res;
    const double ea = r->bounds[0], eb = r->bounds[1];
    const float* tmean = norm + 2 * kMlpIn;
    const float* tstd = tmean + kMlpOut;
    const double mx = (double)tmean[0] + (double)tstd[0] * (double)y[2 * i];
    const double lo = (double)tmean[1] + (double)tstd[1] * (double)y[2 * i + 1];
    double mu = 0.5 * (ea + eb) + 0.5 * (eb - ea) * mx;
    mu = fmin(fmax(mu, ea), eb);
    r->mu = r->mu0 = mu;
    r->order = exp2(lo * log2((double)(n_terms > 1 ? n_terms : 2)));
    if (use_order && m >= 2 && isfinite(r->order)) {
        int me = (int)ceil(margin * fmax(r->order, 1.0) / (double)k);
        me = me < 2 ? 2 : (me > m ? m : me);
        r->m_eff = me;
        r->n_eff = k * me < n_terms ? k * me : n_terms;
    }
}

// The judge after evaluation `round` (0 = at the learned mu): accept when |tr P - N_e| <=
// tol (tol <= 0: 1e-8 max(1, N_e) for float64, 1e-7 n for the split forms); otherwise, if
// rounds remain, move mu by a Newton step on d tr P / d mu ~ tr(P (I - P)) / kT_p =
// (tr P - ||P||_F^2) / kT_p (first round; kT_p the effective temperature of the truncated
// expansion, k_poly_width, which is kT for an exact Fermi function) or a secant step
// through the previous evaluation, limited to 10 kT_p; else leave the instance active for
// the bisection fallback.
__global__ void k_learned_check(const Inst* __restrict__ insts, const InstIO* io, int batch,
                                int round, int max_rounds, double tol, int is64, int* __restrict__ active_count) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= batch) return;
    DevResult* r = insts[i].res;
    if (!r->active) return;
    const double n_e = io[i].n_e, kT = io[i].kT;
    // default: float64 meets the strict trace bar; the split forms are judged within the band
    // of their float32 rounding of tr P (the trace correction then removes that part)
    const double t = tol > 0.0 ? tol : (is64 ? 1e-8 * fmax(1.0, n_e) : 1e-7 * (double)insts[i].n);
    const double err = r->trace - n_e;
    r->evals = round + 1;
    if (fabs(err) <= t && isfinite(err)) {
        r->active = 0;
        r->learned_ok = 1;
        return;
    }
    if (round >= max_rounds) {
        r->learned_ok = 0;   // stays active: exact moments and bisection follow
        atomicAdd(active_count, 1);
        return;
    }
    const double kte = (r->kt_eff > 0.0 && isfinite(r->kt_eff)) ? fmax(r->kt_eff, kT) : kT;
    double slope = (r->trace - r->frob2) / kte;
    if (round > 0 && r->mu != r->mu_prev) {
        const double sec = (r->trace - r->tr_prev) / (r->mu - r->mu_prev);
        if (sec > 0.0 && isfinite(sec)) slope = sec;
    }
    double step = (slope > 0.0 && isfinite(slope)) ? -err / slope : 0.0;
    step = fmin(fmax(step, -10.0 * kte), 10.0 * kte);
    r->mu_prev = r->mu;
    r->tr_prev = r->trace;
    r->mu = r->mu + step;
    atomicAdd(active_count, 1);
}

}  // namespace

// ------------------------------------------------------------------ launchers
namespace {
template <bool TRAIN>
cudaError_t launch_rows(const RowArgs& a, cudaStream_t s) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_mlp_rows<TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RowSmem));
    if (e != cudaSuccess) return e;
    k_mlp_rows<TRAIN><<<(unsigned)((a.B + kRows - 1) / kRows * kCl), kRowThreads, sizeof(RowSmem), s>>>(a);
    return cudaGetLastError();
}
}  // namespace

cudaError_t mlp_forward(const float* params, const float* x, const float* norm, int B, float* y, cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    RowArgs a{};
    a.params = params;
    a.src = x;
    a.norm = norm;
    a.B = B;
    a.y = y;
    return launch_rows<false>(a, s);
}

cudaError_t mlp_step(const MlpStep& st, cudaStream_t s) {
    if (st.B <= 0) return cudaSuccess;
    const size_t B = (size_t)st.B;
    RowArgs a{};
    a.params = st.params;
    a.src = st.feat;
    a.tsrc = st.target;
    a.idx = st.idx;
    a.norm = st.norm;
    a.B = st.B;
    float* w = st.scratch;
    auto take = [&](size_t n) { float* r = w; w += (n + 3) & ~size_t(3); return r; };   // 16-byte aligned
    a.x = take(B * kMlpIn);
    a.t = take(B * kMlpOut);
    a.a1 = take(B * kMlpHidden);
    a.a2 = take(B * kMlpHidden);
    a.dz1 = take(B * kMlpHidden);
    a.dz2 = take(B * kMlpHidden);
    a.y = take(B * kMlpOut);
    a.dy = take(B * kMlpOut);
    const cudaError_t e = launch_rows<true>(a, s);
    if (e != cudaSuccess) return e;
    GradArgs g{};
    g.x = a.x;
    g.a1 = a.a1;
    g.a2 = a.a2;
    g.dz1 = a.dz1;
    g.dz2 = a.dz2;
    g.dy = a.dy;
    g.y = a.y;
    g.t = a.t;
    g.B = st.B;
    g.grad = st.grad;
    g.p = st.params;
    g.m = st.m;
    g.v = st.v;
    g.lr = st.lr;
    g.step = st.step;
    g.loss = st.loss;
    const cudaError_t eg = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, kGradSmem);
    if (eg != cudaSuccess) return eg;
    k_mlp_grad<<<kGradBlocks, 128, kGradSmem, s>>>(g);
    return cudaGetLastError();
}
size_t mlp_step_floats(int B) { return (size_t)B * (kMlpIn + 3 * kMlpOut + 4 * kMlpHidden) + 3 * 4; }

cudaError_t mlp_col_stats(const float* X, int n, int C, float* mean, float* stdv, cudaStream_t s) {
    k_col_stats<<<C, 256, 0, s>>>(X, n, C, mean, stdv);
    return cudaGetLastError();
}

cudaError_t launch_features(const Inst* in, const InstIO* io, int batch, int k, int rows_by_user, float* feat,
                            cudaStream_t s) {
    k_features<<<batch, 96, 0, s>>>(in, io, batch, k, rows_by_user, feat);
    return cudaGetLastError();
}

cudaError_t launch_targets(const Inst* in, int batch, int n_terms, float* tgt, cudaStream_t s) {
    k_targets<<<(batch + 127) / 128, 128, 0, s>>>(in, batch, n_terms, tgt);
    return cudaGetLastError();
}

cudaError_t launch_assemble_low(const Inst* in, int batch, int k, cudaStream_t s) {
    k_assemble_low<<<(batch + 127) / 128, 128, 0, s>>>(in, batch, k);
    return cudaGetLastError();
}

cudaError_t launch_learned_mu(const Inst* in, int batch, const float* y, const float* norm, int n_terms,
                              int k, int m, int use_order, double margin, cudaStream_t s) {
    k_learned_mu<<<(batch + 127) / 128, 128, 0, s>>>(in, batch, y, norm, n_terms, k, m, use_order, margin);
    return cudaGetLastError();
}

cudaError_t launch_learned_check(const Inst* in, const InstIO* io, int batch, int round, int max_rounds,
                                 double tol, int is64, int* active_count, cudaStream_t s) {
    k_learned_check<<<(batch + 127) / 128, 128, 0, s>>>(in, io, batch, round, max_rounds, tol, is64, active_count);
    return cudaGetLastError();
}

}  // namespace fo
