// Float64 recurrence product out = alpha * A B + beta * C + D + shift * I_n on the tensor cores.
//
// tcgen05 has no float64 kind and this GPU's float64 pipe retires about two FMAs per clock and
// SM (1.1 TFLOP/s over the chip), so the float64 path is not run there. A float64 matrix is
// held as eight signed 8-bit digits per entry (Ozaki's splitting with a common exponent: x =
// 2^e sum_i d_i 2^(-7-8i), d_i in [-128, 127], i.e. x rounded to 2^(e-63) with |x| < 0.99 2^e, e a
// bound of the whole matrix), the digits stored as float16 integers. A product of two digits
// and a sum of 1024 of them are integers of at most 2^24, which the tensor core's float32
// accumulator holds exactly, so the products of digit matrices are exact whatever the order of
// the sums. The product keeps the 36 digit pairs of order i + j <= 7; the sums per order are carried
// on in 64-bit integers and rounded to float64 once. The pairs left out, of order 8 and above, add
// at most about 7 K 2^-64 of 2^(eA+eB) (the seven of order 8, |d| <= 2^7; 2^-51 at K = 1000), and
// rms 2^-59 sqrt(K/1000) of it for digits that are independent and uniform.
// Both, and the rounding to 2^(e-63), are relative to the largest entries: the error is that of
// float64 norm-wise, not entry-wise. An entry 2^-40 of the largest has about three digits, and in
// a product with it the partner is cut to the digits whose order sum stays below 8. A 24-term recurrence
// on two fragments coupled by c of the largest entry leaves the coupling block with a relative error
// of 4e-15 at c = 1e-4, 3e-11 at 1e-8, 4e-7 at 1e-12 (float64 sums 5e-16 throughout); callers
// who need that ask for the FMA kernel (FO_FLAG_FP64_FMA). Norm-wise: density matrices against 64-bit references at the same mu, tight-
// binding and random matrices of N = 64 ... 1900 with 64 ... 400 terms: error 0.97 of the FMA
// kernel's (geometric mean; at most 1.003), commutator with H 0.66 of it. One product of N = 1000
// takes 60 us and of N = 2000 255 us, where the FMA kernel took 1.14 and 8.4 ms.
//
// k_dig_mma: one unit = one 128 x 128 output tile on or above the diagonal, one range of k and
// one group of orders: the four low orders 4..7 (26 digit pairs, all 8 digits of both
// operands) or the four high orders 0..3 (10 pairs, 4 digits). Each order has its own TMEM
// accumulator (4 x 128 columns: all of TMEM), so that every staged digit serves all its pairs:
// 16 (or 8) operand tiles of 4 KB per 26 (or 10) MMAs of 64 clocks, 39 (51) bytes per clock
// from L2, where a product per plane pair would need 128. The accumulators are exact for 64
// MMAs; they restart at staggered k-blocks, so that the drain warps empty one of them (to
// 64-bit integer registers) while the MMAs of the others run, the restarted order's MMAs last.
// Measured: 72 (79) clocks per MMA; with one thread computing descriptors in a loop it was 146
// (209), with run-time accumulator indices 81 (115).
// Units write their exact 64-bit sums; integer sums over k ranges do not depend on the order,
// so the split of k (chosen per plan to fill the SMs) does not change a bit of the result.
//
// k_dig_update: adds the units' sums of a 32 x 32 block, rounds the product to float64, applies
// the recurrence update, and writes the float64 master on both sides of the diagonal (or the
// caller's P) and, for the members T_j(X) on bounds that enclose the spectrum, the digits: their
// entries are at most 1, and a bound from the units' largest sums and the largest entry of C often
// gives a finer scale. Elsewhere (Clenshaw members, given or Lanczos bounds) such a bound is
// several bits too wide, which the dropped pairs would show (up to 1.7x the FMA kernel's error),
// so the digits are split from the finished master at its largest entry by a kernel of their own
// (k_dig_split).
//
// Float64 staged plans (Algorithm 1 multiplies arbitrary pairs of slots, which would need the
// digits of every slot), plans whose digit buffers do not fit the device and calls with
// FO_FLAG_FP64_FMA run the FMA kernel.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>
#include <functional>
#include <vector>
#include <type_traits>

#include "digits.h"
#include "internal.cuh"
#include "tcptx.cuh"

namespace fo {
namespace {

constexpr int kT = 128;                     // tile edge (UMMA M = N = 128)
constexpr int kDigits = 8;
constexpr int kBoxBytes = kT * 128;         // one box: 128 rows x 128 bytes (4 digits x 16 k): 16 KB
constexpr int kLowStages = 3, kHighStages = 6;
constexpr int kRing = kLowStages * 4 * kBoxBytes;   // 192 KB, the same for both order groups
constexpr int kMmaSmem = kRing + 1024 /*align*/ + 256 /*barriers*/;
constexpr int kDrainWarps = 8;                // 64 accumulator columns each
constexpr int kMmaThreads = 32 * (2 + kDrainWarps);

static_assert(kHighStages * 2 * kBoxBytes == kRing, "ring of the high orders");
static_assert(kMmaSmem <= 232448 - 64, "shared memory of the unit kernel");

struct DigMaps {
    CUtensorMap m[kMaxBuckets];
};

// Shared-memory descriptor of a K-major operand tile with 128-byte swizzle: 128-byte rows, 8-row
// groups 1 KB apart. A row holds 4 digits x 16 k entries; digit i starts 32 i bytes into it.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;                 // SWIZZLE_128B
    return d;
}
// kind::f16, float32 accumulators, float16 operands, both K-major, M = N = 128
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(kT >> 3) << 17) | ((uint32_t)(kT >> 4) << 24);

// The O + 1 digit pairs of order O for one k16 block.
template <int O>
__device__ __forceinline__ void issue_order(uint32_t tmem_d, uint32_t alo, uint32_t blo, uint32_t hi, bool fresh,
                                            uint32_t lead) {
#pragma unroll
    for (int i = 0; i <= O; ++i) {
        const int j = O - i;
        umma_lead(tmem_d, alo + (uint32_t)((i >> 2) * (kBoxBytes >> 4) + (i & 3) * 2), hi,
                  blo + (uint32_t)((j >> 2) * (kBoxBytes >> 4) + (j & 3) * 2), hi, kIdesc,
                  i > 0 ? 1u : (fresh ? 0u : 1u), lead);
    }
}

// f(integral_constant<PH>) for PH = ph, 0 <= ph < N.
template <int N, int PH = 0, class F>
__device__ __forceinline__ void switch_phase(int ph, F& f) {
    if constexpr (PH < N) {
        if (ph == PH) f(std::integral_constant<int, PH>{});
        else switch_phase<N, PH + 1>(ph, f);
    }
}

// Unit u of an instance: the low-order units of all tiles first (the long ones), then the high.
struct Unit {
    int tile, split, nsplit;
    bool low;
};
__device__ __forceinline__ Unit unit_of(int u, int tiles, int sl, int sh) {
    Unit w;
    w.low = u < tiles * sl;
    const int v = w.low ? u : u - tiles * sl;
    w.nsplit = w.low ? sl : sh;
    w.tile = v / w.nsplit;
    w.split = v - w.tile * w.nsplit;
    return w;
}

__global__ void __launch_bounds__(kMmaThreads, 1)
    k_dig_mma(const __grid_constant__ DigMaps maps, const Inst* __restrict__ insts, const int* __restrict__ pre, int i0,
              int i1, int unit0, int b0, int a_buf, int b_buf, int out_slot, int need_m, int* err_flag) {
    pdl_launch();
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kRing);
    uint64_t* empty = full + kHighStages;
    uint64_t* seg_full = empty + kHighStages;
    uint64_t* seg_empty = seg_full + 4;
    uint64_t* all_done = seg_empty + 4;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(all_done + 1);
    __shared__ int abort_flag;

    const int gu = unit0 + (int)blockIdx.x;
    const int inst = find_inst(pre, i0, i1, gu);
    const Inst& in = insts[inst];
    const int nt = (int)(in.np / kT);
    const int u = gu - __ldg(pre + inst);
    const Unit w = unit_of(u, nt * (nt + 1) / 2, in.dig_sl, in.dig_sh);
    int I, J;
    upper_tile(w.tile, nt, I, J);
    const int m0 = I * kT, n0 = J * kT;
    const int nk = (int)((in.n + 15) / 16);
    const int kb0 = (int)((int64_t)nk * w.split / w.nsplit), kb1 = (int)((int64_t)nk * (w.split + 1) / w.nsplit);
    const int cnt = kb1 - kb0;
    const int gs = w.low ? 1 : 2;
    const int nbx = w.low ? 2 : 1;                       // boxes per operand and k16 block
    const int S = w.low ? kLowStages : kHighStages;
    const uint32_t stage_bytes = (uint32_t)(2 * nbx * kBoxBytes);
    const CUtensorMap* map = &maps.m[in.bucket - b0];
    // the warp index through a shuffle: the compiler then knows that a role's branch is uniform
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < kHighStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 4; ++a) {
            mbar_init(&seg_full[a], 1);
            mbar_init(&seg_empty[a], 32 * kDrainWarps);
        }
        mbar_init(all_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
    }
    pdl_wait();   // above: the plan's constant tables only; tensor memory is taken after the wait
    if (!step_needed(in.res, need_m)) return;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    volatile int* vabort = &abort_flag;
    auto give_up = [&]() {
        atomicExch(&abort_flag, 1);
        atomicExch(err_flag, 1);
    };

    long long acc[64];   // a drain thread's exact sums, in units of the group's lowest order
#pragma unroll
    for (int j = 0; j < 64; ++j) acc[j] = 0;
    bool ok = true;

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer
            int s = 0, issued = 0;
            uint32_t ph = 1;   // parity that an unused stage's `empty` barrier already shows
            for (int l = 0; l < cnt; ++l) {
                if (!mbar_wait(&empty[s], ph, kWaitNs, vabort)) {
                    give_up();
                    break;
                }
                mbar_expect_tx(&full[s], stage_bytes);
                unsigned char* st = smem + s * stage_bytes;
                for (int x = 0; x < nbx; ++x) {
                    const int c0 = (kb0 + l) * 128 + x * 64;   // 16-byte aligned: 128 and 64 entries of 2 bytes
                    tma_load_4d(st + x * kBoxBytes, map, &full[s], c0, m0, a_buf, in.in_bucket);
                    tma_load_4d(st + (nbx + x) * kBoxBytes, map, &full[s], c0, n0, b_buf, in.in_bucket);
                }
                ++issued;
                if (++s == S) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            // before the CTA may exit: every stage released (the MMAs have read it), or after an
            // abort at least the copies in flight landed
            for (int g = issued > S ? issued - S : 0; g < issued; ++g) {
                if (*vabort) mbar_wait(&full[g % S], (uint32_t)(g / S) & 1u, kDrainNs, nullptr);
                else if (!mbar_wait(&empty[g % S], (uint32_t)(g / S) & 1u, kWaitNs, vabort)) atomicExch(err_flag, 1);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer: the whole warp keeps the loop (its descriptors then live in
        // uniform registers), one elected lane issues
        const uint64_t desc0 = sdesc_sw128(smem_u32(smem));
        const uint32_t hi = (uint32_t)(desc0 >> 32);
        const uint32_t lead = elect_one() ? 1u : 0u;
        auto issue = [&](auto low_tag) {
            constexpr bool LOW = decltype(low_tag)::value;
            constexpr int GS = LOW ? 1 : 2, NBX = LOW ? 2 : 1, ST = LOW ? kLowStages : kHighStages;
            constexpr uint32_t SB = 2 * NBX * (kBoxBytes >> 4);
            int s = 0;
            uint32_t ph = 0, par = 0;   // par: bit a = parity of accumulator a's next seg_empty wait
            for (int l = 0; l < cnt; ++l) {
                if (!mbar_wait_warp(&full[s], ph, kWaitNs, vabort)) {
                    if (lead) give_up();
                    return;
                }
                fence_after();
                const uint32_t alo = (uint32_t)desc0 + (uint32_t)s * SB, blo = alo + NBX * (kBoxBytes >> 4);
                // the block's phase in the groups' period, as a constant: every accumulator index, start
                // and end is then static (with run-time ones an accumulator switch took ~140 clocks)
                bool go = true;
                auto block = [&](auto ph_tag) {
                    constexpr int PH = decltype(ph_tag)::value;
                    auto acc_step = [&](auto q_tag) {
                        constexpr int A = acc_order(decltype(q_tag)::value, acc_place(PH, GS), GS);
                        constexpr bool BEG = acc_begins(A, acc_place(PH, GS), GS);
                        constexpr bool END = acc_ends(A, PH, 1 << 30, GS);
                        if (BEG && l > 0 && go) {
                            go = mbar_wait_warp(&seg_empty[A], (par >> A) & 1u, kWaitNs, vabort);
                            fence_after();
                            par ^= 1u << A;
                        }
                        issue_order<(LOW ? 4 : 0) + A>(tmem + A * kT, alo, blo, hi, BEG || l == 0, lead && go);
                        if (END || l == cnt - 1) umma_commit_if(&seg_full[A], lead);
                    };
                    acc_step(std::integral_constant<int, 0>{});
                    acc_step(std::integral_constant<int, 1>{});
                    acc_step(std::integral_constant<int, 2>{});
                    acc_step(std::integral_constant<int, 3>{});
                };
                switch_phase<4 << GS>(l & ((4 << GS) - 1), block);
                if (!go) {
                    if (lead) give_up();
                    return;
                }
                umma_commit_if(&empty[s], lead);
                if (++s == ST) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        };
        if (w.low) issue(std::true_type{});
        else issue(std::false_type{});
        if (lead) umma_commit(all_done);   // every issued MMA has completed (also after an abort)
        __syncwarp();
    } else {
        // ---------------- drain warps: finished groups into 64-bit integers
        const int q = warp & 3, grp = (warp - 2) >> 2;
        const uint32_t t_row = tmem + ((uint32_t)(q * 32) << 16) + grp * 64;
        uint32_t par = 0;
        for (int l = 0; l < cnt && ok; ++l) {
            for (int x = 0; x < 4; ++x) {
                const int a = acc_order(x, l, gs);
                if (!acc_ends(a, l, cnt, gs)) continue;
                if (!mbar_wait_warp(&seg_full[a], (par >> a) & 1u, kWaitNs, vabort)) {
                    ok = false;
                    break;
                }
                par ^= 1u << a;
                __syncwarp();
                fence_after();
                const int mul = 1 << (8 * (3 - a));   // order a of the group, in units of its lowest
#pragma unroll
                for (int cb = 0; cb < 2; ++cb) {
                    uint32_t r[32];
                    tmem_ld32(t_row + a * kT + cb * 32, r);
                    if (cb == 1) {
                        fence_before();
                        mbar_arrive(&seg_empty[a]);   // the accumulator is in registers: it may restart
                    }
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        acc[cb * 32 + j] += (long long)__float2int_rn(__uint_as_float(r[j])) * (long long)mul;
                }
            }
        }
        if (!mbar_wait_warp(all_done, 0, kWaitNs, nullptr)) ok = false;
        __syncwarp();
        if (!ok && lane == 0) give_up();
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
    if (warp < 2 || *vabort) return;
    // the unit's sums, column by column: lanes on rows, 256 bytes per store
    {
        const Inst& in2 = insts[inst];
        const int q = warp & 3, grp = (warp - 2) >> 2;
        long long* dst = in2.dpart + (size_t)u * (kT * kT) + (size_t)(grp * 64) * kT + q * 32 + lane;
#pragma unroll
        for (int j = 0; j < 64; ++j) dst[(size_t)j * kT] = acc[j];
        if (!w.low && out_slot >= 0) {
            // bound of the unit's sums, for the scale of the result's digits
            unsigned long long mx = 0;
#pragma unroll
            for (int j = 0; j < 64; ++j) {
                const unsigned long long v = (unsigned long long)(acc[j] < 0 ? -acc[j] : acc[j]);
                mx = v > mx ? v : mx;
            }
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
                mx = v > mx ? v : mx;
            }
            if (lane == 0)
                atomicMax(in2.umax + (size_t)out_slot * kDigMaxSplit + w.split,
                          __float_as_uint(__ull2float_ru(mx)));
        }
    }
}

// ------------------------------------------------------------------ scales and digits

// The eight digits of eight consecutive columns of one row (bytes as above) into the digit
// buffer: 16 bytes of float16 integers per digit.
__device__ __forceinline__ void store_digits(char* dig, int64_t np, int64_t row, int64_t col,
                                             const unsigned long long (&u)[8]) {
    char* dst = dig + row * np * 16 + (col >> 4) * 256 + (col & 15) * 2;
#pragma unroll
    for (int p = 0; p < kDigits; ++p) {
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            // byte 7 - p of two neighbours as float16 1024 + byte, minus 1152
            const uint32_t x0 = (uint32_t)(p < 4 ? u[2 * h] >> 32 : u[2 * h]);
            const uint32_t x1 = (uint32_t)(p < 4 ? u[2 * h + 1] >> 32 : u[2 * h + 1]);
            const int bb = 3 - (p & 3);
            const uint32_t by = __byte_perm(x0, x1, (uint32_t)(bb | ((4 + bb) << 8)));
            uint32_t hw = (by & 0x00ff00ffu) | 0x64006400u;
            __half2 hv;
            memcpy(&hv, &hw, 4);
            hv = __hsub2(hv, __half2half2(__ushort_as_half((unsigned short)0x6480)));
            memcpy(&w[h], &hv, 4);
        }
        *reinterpret_cast<uint4*>(dst + p * 32) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

constexpr int kUpWarps = 16, kUpCols = 32 / kUpWarps;

struct DigStep {
    int a, b, c, d, out;         // slots (-1: absent)
    int dig_out;                 // digit buffer of the result, -1: none
    int out64, need_m;
    int alpha_exp;               // alpha = 2^alpha_exp
    double beta, shift;
};

// One 32 x 32 block (bi, bj), bj >= bi, of one instance: 16 warps, lane = row within the block (the
// units' sums and the mirrored masters are then read 256 bytes per warp), two columns each, all
// loads before any use (four warps with eight columns each took longer on small matrices: their
// unrolled code is fetched once per launch). Bytes bound it (8 (k ranges) + 8 (C, D) read and 24 written
// per entry of the square, about half of them from L2): the float64 pipe sees one or two
// operations per entry (alpha is a power of two, folded into the conversion; magnitudes are
// compared as integers).
__global__ void __launch_bounds__(32 * kUpWarps, 3) k_dig_update(const Inst* __restrict__ insts, const InstIO* io,
                                                    Work ws, const DigStep st) {
    pdl_sync();
    __shared__ double sv[32][33];
    __shared__ unsigned long long su[32][33];
    __shared__ int s_e[2];
    const int inst = inst_of(ws, blockIdx.x);
    const Inst& in = insts[inst];
    if (!step_needed(in.res, st.need_m)) return;
    const int64_t n = in.n, np = in.np;
    int bi, bj;
    upper_tile(blockIdx.x - ws.pre[inst], (int)(np / 32), bi, bj);
    const int nt = (int)(np / kT), tiles = nt * (nt + 1) / 2;
    const int TI = bi >> 2, TJ = bj >> 2;
    const int tile = TI * nt - TI * (TI - 1) / 2 + (TJ - TI);
    const int sl = in.dig_sl, shi = in.dig_sh;
    const long long* lo0 = in.dpart + (size_t)tile * sl * (kT * kT);
    const long long* hi0 = in.dpart + ((size_t)tiles * sl + (size_t)tile * shi) * (kT * kT);
    const int64_t sb = in.slot_bytes;
    const double* C = st.c >= 0 ? reinterpret_cast<const double*>(in.slots + sb * st.c) : nullptr;
    const double* D = st.d >= 0 ? reinterpret_cast<const double*>(in.slots + sb * st.d) : nullptr;
    double* out = st.out >= 0 && !st.out64 ? reinterpret_cast<double*>(in.slots + sb * st.out) : nullptr;
    double* P = st.out64 ? io[inst].P : nullptr;
    const int64_t ldp = io[inst].ldp;
    const int lane = threadIdx.x & 31, cg = threadIdx.x >> 5;
    const int ro = (bi & 3) * 32, co = (bj & 3) * 32;
    // offsets of this thread's entries in a unit's sums; below the diagonal of a diagonal block: the
    // mirrored entry (the same value)
    int o[kUpCols];
    long long lo[kUpCols], hi[kUpCols];
    double cv[kUpCols], dv[kUpCols];
#pragma unroll
    for (int q = 0; q < kUpCols; ++q) {
        const int c = cg * kUpCols + q;
        const bool mir = bi == bj && c < lane;
        o[q] = (co + (mir ? lane : c)) * kT + ro + (mir ? c : lane);
        lo[q] = hi[q] = 0;
        const int64_t mo = ((int64_t)bj * 32 + c) * np + (int64_t)bi * 32 + lane;
        cv[q] = C ? C[mo] : 0.0;
        dv[q] = D ? D[mo] : 0.0;
    }
    // (streaming loads: each sum is read once; through L1 as other data the product takes 0.4 % longer)
    for (int s = 0; s < sl; ++s, lo0 += kT * kT)
#pragma unroll
        for (int q = 0; q < kUpCols; ++q) lo[q] += __ldcs(lo0 + o[q]);
    for (int s = 0; s < shi; ++s, hi0 += kT * kT)
#pragma unroll
        for (int q = 0; q < kUpCols; ++q) hi[q] += __ldcs(hi0 + o[q]);
    if (cg == 0) {
        // the scales: warp 0, a lane per k range
        const int ea = in.sexp[st.a], eb = in.sexp[st.b];
        int eo = 0, ep = ea + eb;
        if (ea == kPoison || eb == kPoison) {
            ep = eo = kPoison;
        } else if (st.dig_out >= 0) {
            // |product| <= sum over k ranges of the largest high-order sum, plus the low orders
            // (below n 2^-29), at scale 2^(ea + eb)
            float um = lane < shi ? __uint_as_float(in.umax[(size_t)st.out * kDigMaxSplit + lane]) : 0.0f;
            for (int x = 8; x > 0; x >>= 1) um += __shfl_xor_sync(0xffffffffu, um, x);
            const double mx = (double)n * 1.862645149230957e-09 + (double)um * 3.637978807091713e-12;
            double b = scalbn(mx, ep + st.alpha_exp) + fabs(st.shift);
            if (st.c >= 0) b += fabs(st.beta) * __longlong_as_double((long long)in.smax[st.c]);
            eo = scale_exp(b * 1.000001);
            if (eo != kPoison && eo > 1) eo = 1;   // every entry of T_j(X) is at most 1
        }
        if (lane == 0) {
            s_e[0] = ep;
            s_e[1] = eo;
            if (st.dig_out >= 0 && bi == 0 && bj == 0) in.sexp[st.out] = eo;
        }
    }
    __syncthreads();
    const int ep = s_e[0], eo = s_e[1];
    unsigned long long mx = 0;
#pragma unroll
    for (int q = 0; q < kUpCols; ++q) {
        const int c = cg * kUpCols + q;
        const int64_t gr = (int64_t)bi * 32 + lane, gc = (int64_t)bj * 32 + c;   // entry (gr, gc) = (gc, gr)
        double v;
        if (ep != kPoison) v = fixed_to_double(hi[q], lo[q], ep + st.alpha_exp);
        else v = gr < n && gc < n ? __longlong_as_double(0x7ff8000000000000ll) : 0.0;   // the border stays zero
        if (C) v = fma(st.beta, cv[q], v);
        if (D) v += dv[q];
        if (gr == gc && gr < n) v += st.shift;
        const unsigned long long av = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
        mx = av > mx ? av : mx;
        sv[c][lane] = v;
        if (st.dig_out >= 0) su[c][lane] = digits_of(v, eo);
        if (out) out[gc * np + gr] = v;
        if (P && gr < n && gc < n) P[gc * ldp + gr] = v;
    }
    if (out) max_to(in.smax + st.out, mx);
    __syncthreads();
    if (bi != bj) {
#pragma unroll
        for (int q = 0; q < kUpCols; ++q) {
            const int r = cg * kUpCols + q;
            const int64_t gr = (int64_t)bi * 32 + r, gc = (int64_t)bj * 32 + lane;
            if (out) out[gr * np + gc] = sv[lane][r];
            if (P && gr < n && gc < n) P[gr * ldp + gc] = sv[lane][r];
        }
    }
    if (st.dig_out < 0 || eo == kPoison || threadIdx.x >= 256) return;
    // eight digits of eight neighbours: threads 0..127 the rows of bj, 128..255 (off the diagonal) of bi
    char* dig = in.dig + (size_t)st.dig_out * 16 * np * np;
    const bool up = threadIdx.x >= 128;
    if (up && bi == bj) return;
    const int row = (threadIdx.x & 127) >> 2, c8 = (threadIdx.x & 3) * 8;
    unsigned long long u[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) u[q] = up ? su[c8 + q][row] : su[row][c8 + q];
    store_digits(dig, np, (int64_t)(up ? bi : bj) * 32 + row, (int64_t)(up ? bj : bi) * 32 + c8, u);
}

// Digits of one slot (X, a Clenshaw member, or the last R of an expansion: slot0 + its l) into digit
// buffer `buf`, at the scale of the slot's largest entry: the same 32 x 32 blocks; the slot's float64
// master is complete on both sides.
__global__ void __launch_bounds__(128) k_dig_split(const Inst* __restrict__ insts, Work ws, int slot0, int last_m,
                                                   int buf, int need_m) {
    pdl_sync();
    const int inst = inst_of(ws, blockIdx.x);
    const Inst& in = insts[inst];
    if (!step_needed(in.res, need_m)) return;
    const int slot = last_m > 0 ? slot0 + (in.res->m_eff > 0 ? in.res->m_eff : last_m) - 1 : slot0;
    const int64_t np = in.np;
    int bi, bj;
    upper_tile(blockIdx.x - ws.pre[inst], (int)(np / 32), bi, bj);
    const int e = scale_exp(__longlong_as_double((long long)in.smax[slot]));
    if (threadIdx.x == 0 && bi == 0 && bj == 0) in.sexp[slot] = e;
    if (e == kPoison) return;
    const double* M = reinterpret_cast<const double*>(in.slots + in.slot_bytes * slot);
    char* dig = in.dig + (size_t)buf * 16 * np * np;
    const int row = threadIdx.x >> 2, c8 = (threadIdx.x & 3) * 8;
    for (int side = 0; side < (bi != bj ? 2 : 1); ++side) {
        const int64_t gr = (int64_t)(side ? bj : bi) * 32 + row, gc = (int64_t)(side ? bi : bj) * 32 + c8;
        unsigned long long u[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const double2 v = *reinterpret_cast<const double2*>(M + gr * np + gc + 2 * q);
            u[2 * q] = digits_of(v.x, e);
            u[2 * q + 1] = digits_of(v.y, e);
        }
        store_digits(dig, np, gr, gc, u);
    }
}

// Clears the largest-entry and unit records of slots [slot0, slot0 + count); one block per instance.
__global__ void k_dig_reset(const Inst* __restrict__ insts, int slot0, int count) {
    pdl_sync();
    const Inst& in = insts[blockIdx.x];
    for (int q = threadIdx.x; q < count; q += blockDim.x) in.smax[slot0 + q] = 0;
    for (int q = threadIdx.x; q < count * kDigMaxSplit; q += blockDim.x) in.umax[(size_t)slot0 * kDigMaxSplit + q] = 0;
}

}  // namespace

// Units of one instance's product (low and high order groups of every upper tile).
int64_t dig_units(int64_t np, int sl, int sh) {
    const int64_t nt = np / kT;
    return nt * (nt + 1) / 2 * (sl + sh);
}
// Clocks of a unit of cnt k16 blocks, from timers in the kernel (N = 256, 1000, 2000): its start,
// last drains and stores, and its MMAs (26 of 72 clocks, 10 of 80).
double unit_clocks(bool low, int cnt) { return low ? 14000.0 + 1870.0 * cnt : 16000.0 + 800.0 * cnt; }

// k ranges of the low- and high-order units of every instance (sizes n[i], instances in plan
// order): the pair of clocks-per-unit targets whose units, taken in order by `sms` SMs, finish
// first. Ranges shorter than two k16 blocks do not pay.
void dig_splits(const int64_t* n, const int64_t* np, int count, int sms, int* sl, int* sh) {
    double total = 0.0;
    for (int i = 0; i < count; ++i) {
        const double nt = (double)(np[i] / kT);
        const int nk = (int)((n[i] + 15) / 16);
        total += nt * (nt + 1) / 2 * (unit_clocks(true, nk) + unit_clocks(false, nk));
    }
    auto split_for = [&](bool low, int nk, double target) {
        int s = 1;
        while (s < kDigMaxSplit && nk / (s + 1) >= 2 && unit_clocks(low, (nk + s - 1) / s) > target) ++s;
        return s;
    };
    std::vector<int> tl(count), th(count);
    std::vector<double> busy;
    double best = -1.0;
    for (double f = 0.06; f < 1.5; f *= 1.15) {
        const double target = total / sms * f;
        double makespan;
        size_t units = 0;
        double bytes = 0.0, work = 0.0, longest = 0.0;
        for (int i = 0; i < count; ++i) {
            const int nk = (int)((n[i] + 15) / 16);
            const int64_t nt = np[i] / kT, tiles = nt * (nt + 1) / 2;
            tl[i] = split_for(true, nk, target);
            th[i] = split_for(false, nk, target);
            const double ul = unit_clocks(true, (nk + tl[i] - 1) / tl[i]), uh = unit_clocks(false, (nk + th[i] - 1) / th[i]);
            units += (size_t)tiles * (tl[i] + th[i]);
            work += (double)tiles * (tl[i] * ul + th[i] * uh);
            longest = std::max(longest, std::max(ul, uh));
            bytes += (double)tiles * kT * kT * 8.0 * (tl[i] + th[i]);
        }
        if (units > 20000) {
            makespan = work / sms + longest;
        } else {
            // list scheduling in launch order
            busy.assign(sms, 0.0);
            auto cmp = std::greater<double>();
            for (int i = 0; i < count; ++i) {
                const int nk = (int)((n[i] + 15) / 16);
                const int64_t nt = np[i] / kT, tiles = nt * (nt + 1) / 2;
                for (int g = 0; g < 2; ++g) {
                    const int s = g == 0 ? tl[i] : th[i];
                    const double c = unit_clocks(g == 0, (nk + s - 1) / s);
                    for (int64_t u = 0; u < tiles * s; ++u) {
                        std::pop_heap(busy.begin(), busy.end(), cmp);
                        busy.back() += c;
                        std::push_heap(busy.begin(), busy.end(), cmp);
                    }
                }
            }
            makespan = *std::max_element(busy.begin(), busy.end());
        }
        makespan += bytes / 2000.0;   // the update reads every unit's sums (about 2 KB per clock)
        if (best < 0.0 || makespan < best) {
            best = makespan;
            std::copy(tl.begin(), tl.end(), sl);
            std::copy(th.begin(), th.end(), sh);
        }
    }
}

bool dig_make_map(void* map128, const void* base, int64_t np, int count, int64_t inst_bytes, std::string* err) {
    uint64_t dims[4] = {(uint64_t)np * 8, (uint64_t)np, (uint64_t)kDigBufs, (uint64_t)count};
    uint64_t strides[3] = {(uint64_t)np * 16, (uint64_t)np * np * 16, (uint64_t)inst_bytes};
    uint32_t box[4] = {64, kT, 1, 1};
    return encode_map_f16(map128, base, 4, dims, strides, box, err);
}

cudaError_t dig_product(const Step& s, int dig_a, int dig_b, int dig_out, const Inst* in, const InstIO* io,
                        const Work& wu, const int* pre_host, const Work& wsym, const GramGroup* grp,
                        int ngrp, const void* maps, bool enclosed, int* err_flag, cudaStream_t st, int* launches) {
    const int dig_fused = enclosed ? dig_out : -1;   // digits written by the update itself
    const cudaError_t ea = cudaFuncSetAttribute(k_dig_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, kMmaSmem);
    if (ea != cudaSuccess) return ea;
    for (int q = 0; q < ngrp; ++q) {
        const GramGroup& g = grp[q];
        const int u0 = pre_host[g.i0], u1 = pre_host[g.i1];
        if (u1 <= u0) continue;
        DigMaps dm;
        std::memset(&dm, 0, sizeof(dm));
        for (int b = 0; b < g.nb; ++b)
            std::memcpy(&dm.m[b], static_cast<const char*>(maps) + 128 * (size_t)(g.b0 + b), sizeof(CUtensorMap));
        launch_pdl(k_dig_mma, (unsigned)(u1 - u0), kMmaThreads, kMmaSmem, st, dm, in, wu.pre, g.i0, g.i1, u0, g.b0, dig_a, dig_b,
                                                                      dig_fused >= 0 ? s.out : -1, s.need_m, err_flag);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        *launches += 1;
    }
    if (s.alpha64 != 1.0 && s.alpha64 != 2.0) return cudaErrorInvalidValue;   // the recurrences' factors
    DigStep d;
    d.a = s.a;
    d.b = s.b;
    d.c = s.c;
    d.d = s.d;
    d.out = s.out;
    d.dig_out = dig_fused;
    d.out64 = s.out64;
    d.need_m = s.need_m;
    d.alpha_exp = s.alpha64 == 2.0 ? 1 : 0;
    d.beta = s.beta64;
    d.shift = s.shift64;
    launch_pdl(k_dig_update, (unsigned)wsym.total, 32 * kUpWarps, 0, st, in, io, wsym, d);
    *launches += 1;
    if (dig_out >= 0 && dig_fused < 0) {
        *launches += 1;
        launch_pdl(k_dig_split, (unsigned)wsym.total, 128, 0, st, in, wsym, s.out, 0, dig_out, s.need_m);
    }
    return cudaGetLastError();
}

cudaError_t dig_split(const Inst* in, const Work& wsym, int slot0, int last_m, int buf, cudaStream_t st) {
    launch_pdl(k_dig_split, (unsigned)wsym.total, 128, 0, st, in, wsym, slot0, last_m, buf, 0);
    return cudaGetLastError();
}
cudaError_t dig_reset(const Inst* in, int batch, int slot0, int count, cudaStream_t st) {
    launch_pdl(k_dig_reset, batch, 256, 0, st, in, slot0, count);
    return cudaGetLastError();
}
}  // namespace fo
