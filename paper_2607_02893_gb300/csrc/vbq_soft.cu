// vbq_soft.cu — the training-time soft-quantised forward (§3.2 differentiable
// bit selection; Alg. 1's weight step): per group of 64 weights, the convex
// combination of its four candidate reconstructions (§3.1: Eq. 1 at 2, 4 and 8
// bits, sign times absmean at 1 bit) under pi = softmax((l + e) / tau), the
// group's expected width sum_k pi_k B_k and its hardened width B_argmax l.
//
// A warp takes 16 consecutive groups at a time, two per 16-byte load (16 lanes
// a group, four weights a lane). max|w| and sum|w| of the 16 groups are
// reduced together across the lanes by a transposing butterfly (8 shuffles per
// quantity for the 16 groups, a balanced tree of depth 6 per group) that
// leaves each group's in a lane of its own; that lane evaluates the group's
// selection and scales and hands the products pi_k s_k to the warp through
// shared memory. The integer decisions of Eq. 1 are those of a float32
// framework: s = max|w| / qmax is a correctly rounded quotient (__fdiv_rn), and
// every code is rint of the correctly rounded quotient w / s, clipped. That
// code is found from t = |w| * fl(1/s), within 2^-16 of the exact quotient for
// quotients up to 127: rint(t) (by adding 1.5 * 2^23) is the code whenever t
// is at least 2^-15 from a half-integer (the correctly rounded quotient,
// within 2^-17 of the exact one, is then on the same side of it); otherwise,
// and for scales outside [2^-125, 2^125] (whose reciprocal is not a normal
// float), the IEEE quotient is taken. At 2 bits (qmax 1, s = max|w|) the code
// is 1 exactly when |w| > s / 2: fl(|w| / s) is above 1/2 as soon as |w|
// exceeds s / 2, since the exact quotient then exceeds 1/2 by more than half
// a float32 spacing. Explicitly rounded operations (no contraction) throughout.
// Bound: HBM, 4 bytes in and 4 out per weight, 16 or 32 in and 5 out per
// group. 14336 x 4096: 280 us (two weights per lane and group, each candidate
// reconstructed on its own: about 70 instructions per weight-pair, issue-bound)
// -> 83 us.
#include <cstdint>
#include <cuda_runtime.h>

#include "vbq_kernels.h"

namespace vbq {
namespace {

constexpr int SQ_THREADS = 256;
constexpr int SQ_WARPS = SQ_THREADS / 32;
constexpr int SQ_BLOCKS = 3;             // resident per SM (80 registers a thread); the grid is one such wave, grid-stride
constexpr int SQ_BATCH = 16;             // groups per warp pass
constexpr int SQ_LOADS = SQ_BATCH / 2;   // two groups per load

// Per-group terms, written by the group's owner lane, read by the warp.
struct __align__(16) GroupTerms {
    float c1, c12, half2, r4;            // pi_1 mean; that plus pi_2 s_2; s_2 / 2; fl(1/s_4), 0 when quotients must be divided out
    float c4, r8, c8, s2;                // pi_4 s_4; fl(1/s_8); pi_8 s_8; the 2-bit scale
    float s4, s8, mean, pad;             // the other scales, the 1-bit magnitude
    float pi0, pi1, pi2, pi3;            // the selection
};

// Whether t = |w| * fl(1/s) may stand in for the quotient (fl(1/s) normal).
__device__ __forceinline__ bool rcp_usable(float s) { return s >= 0x1p-125f && s <= 0x1p125f; }

// clip(rint(fl(a / s)), 0, qmax) for a >= 0; 0 for s = 0 (an all-zero group).
__device__ __forceinline__ float code_by_quotient(float a, float s, float qmax) {
    return s == 0.f ? 0.f : fminf(rintf(__fdiv_rn(a, s)), qmax);
}

// The convex combination for |w| = a, by the quotients themselves, each
// reconstruction s q before its share: with a subnormal scale s q is exact,
// where a rounded pi s times q would not be.
__device__ __noinline__ float combine_by_quotient(float a, const GroupTerms& t) {
    const float q2 = code_by_quotient(a, t.s2, 1.f), q4 = code_by_quotient(a, t.s4, 7.f), q8 = code_by_quotient(a, t.s8, 127.f);
    return __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(t.pi0, t.mean), __fmul_rn(t.pi1, __fmul_rn(t.s2, q2))),
                               __fmul_rn(t.pi2, __fmul_rn(t.s4, q4))),
                     __fmul_rn(t.pi3, __fmul_rn(t.s8, q8)));
}

// One level of the transposing butterfly over 16 lanes: of a lane's N values,
// the half its bit H of the lane index selects stays, the other half goes to
// lane ^ H.
template <int N, int H>
__device__ __forceinline__ void reduce_level(float (&m)[SQ_LOADS], float (&s)[SQ_LOADS], int lane) {
    const bool hi = lane & H;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const float ms = hi ? m[i] : m[i + N / 2], mk = hi ? m[i + N / 2] : m[i];
        const float ss = hi ? s[i] : s[i + N / 2], sk = hi ? s[i + N / 2] : s[i];
        m[i] = fmaxf(mk, __shfl_xor_sync(0xffffffffu, ms, H));
        s[i] = __fadd_rn(sk, __shfl_xor_sync(0xffffffffu, ss, H));
    }
}

__global__ void __launch_bounds__(SQ_THREADS, SQ_BLOCKS) soft_quant_kernel(const float* __restrict__ w,
                                                                const float* __restrict__ logits,
                                                                const float* __restrict__ gumbel, float tau,
                                                                int64_t groups, float* __restrict__ w_soft,
                                                                float* __restrict__ exp_bits,
                                                                uint8_t* __restrict__ hard) {
    __shared__ GroupTerms terms[SQ_WARPS][SQ_BATCH];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int half = lane >> 4, l = lane & 15;          // the lane's group of each load, its four weights
    // after the reduction: the lane's own group (lanes l and l ^ 8 hold the same one)
    const int own = 2 * (((lane & 1) << 2) | (lane & 2) | ((lane >> 2) & 1)) + half;
    const int64_t warp0 = ((int64_t)blockIdx.x * SQ_THREADS + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * SQ_THREADS) >> 5;
    for (int64_t g0 = warp0 * SQ_BATCH; g0 < groups; g0 += nwarps * SQ_BATCH) {
        const int nb = (int)(groups - g0 < SQ_BATCH ? groups - g0 : SQ_BATCH);
        float4 v[SQ_LOADS];
        float m[SQ_LOADS], sm[SQ_LOADS];
#pragma unroll
        for (int k = 0; k < SQ_LOADS; ++k) {
            const int j = 2 * k + half;
            v[k] = j < nb ? __ldcs(reinterpret_cast<const float4*>(w + (g0 + j) * GROUP) + l) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float4 lg = make_float4(0.f, 0.f, 0.f, 0.f), e = lg;
        if (own < nb) {
            lg = reinterpret_cast<const float4*>(logits)[g0 + own];
            if (gumbel) e = reinterpret_cast<const float4*>(gumbel)[g0 + own];
        }
#pragma unroll
        for (int k = 0; k < SQ_LOADS; ++k) {
            const float a = fabsf(v[k].x), b = fabsf(v[k].y), c = fabsf(v[k].z), d = fabsf(v[k].w);
            m[k] = fmaxf(fmaxf(a, b), fmaxf(c, d));
            sm[k] = __fadd_rn(__fadd_rn(a, b), __fadd_rn(c, d));
        }
        reduce_level<8, 1>(m, sm, lane);
        reduce_level<4, 2>(m, sm, lane);
        reduce_level<2, 4>(m, sm, lane);
        const float mx = fmaxf(m[0], __shfl_xor_sync(0xffffffffu, m[0], 8));
        const float sum = __fadd_rn(sm[0], __shfl_xor_sync(0xffffffffu, sm[0], 8));
        {
            // group g0 + own: its selection pi = softmax((l + e) / tau), widths and scales
            const float z0 = __fdiv_rn(__fadd_rn(lg.x, e.x), tau), z1 = __fdiv_rn(__fadd_rn(lg.y, e.y), tau);
            const float z2 = __fdiv_rn(__fadd_rn(lg.z, e.z), tau), z3 = __fdiv_rn(__fadd_rn(lg.w, e.w), tau);
            const float zm = fmaxf(fmaxf(z0, z1), fmaxf(z2, z3));
            const float p0 = expf(__fsub_rn(z0, zm)), p1 = expf(__fsub_rn(z1, zm));
            const float p2 = expf(__fsub_rn(z2, zm)), p3 = expf(__fsub_rn(z3, zm));
            const float S = __fadd_rn(__fadd_rn(p0, p1), __fadd_rn(p2, p3));
            GroupTerms t;
            t.pi0 = __fdiv_rn(p0, S);
            t.pi1 = __fdiv_rn(p1, S);
            t.pi2 = __fdiv_rn(p2, S);
            t.pi3 = __fdiv_rn(p3, S);
            t.mean = __fmul_rn(sum, 1.f / GROUP);                 // a power of two, exact
            t.pad = 0.f;
            t.s2 = mx;                                            // qmax 1
            t.s4 = __fdiv_rn(mx, 7.f);
            t.s8 = __fdiv_rn(mx, 127.f);
            t.c1 = __fmul_rn(t.pi0, t.mean);
            t.c12 = __fmaf_rn(t.pi1, mx, t.c1);
            t.half2 = 0.5f * mx;
            t.c4 = __fmul_rn(t.pi2, t.s4);
            t.c8 = __fmul_rn(t.pi3, t.s8);
            const bool fast = rcp_usable(t.s2) && rcp_usable(t.s4) && rcp_usable(t.s8);
            t.r4 = fast ? __frcp_rn(t.s4) : 0.f;
            t.r8 = fast ? __frcp_rn(t.s8) : 0.f;
            if (own < nb && !(lane & 8)) {
                const int64_t g = g0 + own;
                terms[wib][own] = t;
                if (exp_bits)
                    exp_bits[g] = __fadd_rn(__fadd_rn(__fadd_rn(t.pi0, __fmul_rn(2.f, t.pi1)), __fmul_rn(4.f, t.pi2)),
                                            __fmul_rn(8.f, t.pi3));
                if (hard) {                                       // the first maximum of the logits
                    int k = 0;
                    float best = lg.x;
                    if (lg.y > best) { k = 1; best = lg.y; }
                    if (lg.z > best) { k = 2; best = lg.z; }
                    if (lg.w > best) k = 3;
                    hard[g] = (uint8_t)(1u << k);
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < SQ_LOADS; ++k) {
            const int j = 2 * k + half;
            if (j < nb) {
                const GroupTerms& t = terms[wib][j];
                const float4 A = *reinterpret_cast<const float4*>(&t.c1), B = *reinterpret_cast<const float4*>(&t.c4);
                const float x[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
                const float2 magic = make_float2(12582912.f, 12582912.f), nmagic = make_float2(-12582912.f, -12582912.f);
                const float2 r4 = make_float2(A.w, A.w), r8 = make_float2(B.y, B.y);
                float o[4], worst = 0.f;
#pragma unroll
                for (int i = 0; i < 4; i += 2) {
                    const float2 a = make_float2(fabsf(x[i]), fabsf(x[i + 1]));
                    const float2 k4 = __fadd2_rn(__ffma2_rn(a, r4, magic), nmagic);
                    const float2 k8 = __fadd2_rn(__ffma2_rn(a, r8, magic), nmagic);
                    const float2 d4 = __ffma2_rn(a, r4, make_float2(-k4.x, -k4.y));
                    const float2 d8 = __ffma2_rn(a, r8, make_float2(-k8.x, -k8.y));
                    worst = fmaxf(fmaxf(worst, fmaxf(fabsf(d4.x), fabsf(d4.y))), fmaxf(fabsf(d8.x), fabsf(d8.y)));
                    const float2 base = make_float2(a.x > A.z ? A.y : A.x, a.y > A.z ? A.y : A.x);
                    const float2 c = __ffma2_rn(make_float2(B.z, B.z), k8, __ffma2_rn(make_float2(B.x, B.x), k4, base));
                    o[i] = c.x;
                    o[i + 1] = c.y;
                }
                if (worst > 0.5f - 0x1p-15f || A.w == 0.f) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) o[i] = combine_by_quotient(fabsf(x[i]), t);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) o[i] = x[i] < 0.f ? -o[i] : o[i];        // sign(0) = +1
                __stcs(reinterpret_cast<float4*>(w_soft + (g0 + j) * GROUP) + l, make_float4(o[0], o[1], o[2], o[3]));
            }
        }
        __syncwarp();                    // the terms are read before the next pass rewrites them
    }
}

}  // namespace

cudaError_t launch_soft_quant(const float* w, const float* logits, const float* gumbel, float tau, int64_t N,
                              int64_t K, float* w_soft, float* exp_bits, uint8_t* hard, cudaStream_t s) {
    const int64_t groups = N * (K / GROUP);
    int sms = 0;
    const int err = device_sms(&sms);
    if (err != 0) return (cudaError_t)err;
    const int64_t per_block = (int64_t)SQ_WARPS * SQ_BATCH;
    const int64_t want = (groups + per_block - 1) / per_block;
    const int64_t cap = (int64_t)sms * SQ_BLOCKS;
    const int grid = (int)(want < cap ? want : cap);
    soft_quant_kernel<<<grid, SQ_THREADS, 0, s>>>(w, logits, gumbel, tau, groups, w_soft, exp_bits, hard);
    return cudaGetLastError();
}

}  // namespace vbq
