// vbq_quant.cu — per-group quantisation of a dense FP32 matrix into codes and
// FP16 scales (§3.1), the export step before vbq_pack:
//   b >= 2 (Eq. 1): s = FP16(max|w| / qmax), qmax = 2^(b-1) - 1;
//                   q = clip(round(w / s), -qmax, qmax) with round-half-even
//                   of the exact quotient; u = q + 2^(b-1) (s = 0: every
//                   u = 2^(b-1));
//   b = 1         : s = FP16(mean|w|), the sum of |w| taken as a balanced
//                   fp64 tree over neighbouring weights; u = [w >= 0].
// FP16(v) rounds to nearest even and saturates above 65504. The results are
// those of the fp64 formulas (the library's definition), computed without
// fp64 arithmetic in the common case (fp64 runs at a small fraction of the
// fp32 rate on this GPU):
//   - a code: an estimate k = rint(|w| * (1/s)) is within one of the answer,
//     and the thresholds (k -+ 1/2) s are exact fp32 numbers (2k + 1 has at
//     most 10 significant bits, the FP16 s at most 11), so comparing |w| with
//     them gives the correctly rounded quotient, ties included; an fp64
//     quotient rounds to the same integer (with a 24-bit w and an 11-bit s
//     it cannot land on a half-integer the exact quotient misses);
//   - the scale of Eq. 1: the same argument for max|w| / qmax against the
//     FP16 midpoints (fp64 rounding of the quotient never reaches one);
//   - the 1-bit mean: exact integer arithmetic when the fp64 tree is exact
//     (see one_bit_scale), else the fp64 tree itself.
//
// A warp takes 16 groups at a time, four per 16-byte load and lane: eight
// lanes hold a group, weights 4l .. 4l + 3 and 32 + 4l .. of it in lane l, so
// loads and stores are whole 128- and 32-byte segments and a group's reduction
// is three shuffles for four groups at once. The scale rounding (about 60
// instructions) is done once per 16 groups, a group per lane, instead of once
// per group by every lane.
#include "vbq_kernels.h"

namespace vbq {
namespace {

constexpr int QTHREADS = 256;            // 8 warps per block
constexpr int QLOADS = 4;                // loads of four groups in flight per warp
constexpr int QGROUPS = 4 * QLOADS;      // groups per warp pass
constexpr int64_t QKEEP_BYTES = 64 << 20;   // weights the validation leaves in L2 (129 MB) for the quantisation

// FP16 bits of RN(S * 2^P) (S >= 0 an exact integer below 2^53), values
// above 65504 saturating to 65504: integer round-half-even at the FP16
// quantum of the value's binade (2^-24 in the subnormal range).
__device__ __forceinline__ uint32_t fp16_bits_of_scaled(unsigned long long S, int P) {
    if (S == 0) return 0u;
    const int n = 63 - __clzll((long long)S);           // S in [2^n, 2^(n+1))
    int qe = max(n + P - 10, -24);                       // quantum exponent
    const int r = qe - P;                                // bits below the quantum
    unsigned long long mant;
    if (r <= 0) {
        mant = S << (-r);                                // exact (r >= n - 10 >= -10)
    } else if (r >= n + 2) {
        mant = 0;                                        // below half a quantum
    } else {
        mant = S >> r;
        const unsigned long long rem = S & ((1ull << r) - 1), half = 1ull << (r - 1);
        if (rem > half || (rem == half && (mant & 1))) mant += 1;
    }
    if (mant >= 2048) { mant >>= 1; qe += 1; }           // carry out of the 11-bit significand
    if (mant < 1024) return (uint32_t)mant;              // subnormal (qe == -24) or zero
    const int e = qe + 10;
    if (e > 15) return 0x7BFFu;
    return (uint32_t)(((e + 15) << 10) | (int)(mant - 1024));
}

// FP16 bits of RN(m / qmax) for m >= 0 (or +inf), qmax in {1, 7, 127},
// saturating above 65504. An fp32 estimate gives a candidate within one FP16
// step; the midpoints
// to its neighbours times qmax are exact fp32 numbers (at most 12 + 7
// significant bits), so comparing m with them settles the rounding exactly.
__device__ __forceinline__ uint32_t fp16_bits_of_quotient(float m, int qmax) {
    if (m > 65504.f * (float)qmax) return 0x7BFFu;       // exact product; also m = +inf
    // candidate: m times fl(1 / qmax), within 2^-23 of the quotient, so its
    // FP16 rounding is at most one step off
    const float inv = qmax == 1 ? 1.f : qmax == 7 ? (1.f / 7.f) : (1.f / 127.f);
    uint32_t c = (uint32_t)__half_as_ushort(__float2half_rn(m * inv));
    const float cv = __half2float(__ushort_as_half((uint16_t)c));
    if (c < 0x7BFFu) {
        const float hu = 0.5f * (cv + __half2float(__ushort_as_half((uint16_t)(c + 1))));
        const float tu = hu * (float)qmax;
        if (m > tu || (m == tu && (c & 1u))) return c + 1;
    }
    if (c > 0u) {
        const float hd = 0.5f * (cv + __half2float(__ushort_as_half((uint16_t)(c - 1))));
        const float td = hd * (float)qmax;
        if (m < td || (m == td && (c & 1u))) return c - 1;
    }
    return c;
}

__device__ __forceinline__ uint32_t fp16_bits_sat(double s) {   // s >= 0 (or +inf)
    if (s > 65504.0) return 0x7BFFu;
    return (uint32_t)__half_as_ushort(__double2half(s));
}

// 1 / x to within about 2^-22 relative for a normal x (the hardware
// reciprocal approximation): an estimate only; the callers' exact checks
// absorb its error.
__device__ __forceinline__ float rcp_estimate(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// round-half-even(a / sf) for a >= 0 (finite or +inf) and sf > 0, capped at
// qmax, given k = rint of an estimate of the quotient that is within one of
// the answer: the thresholds (k -+ 1/2) sf are exact, so comparing a with
// them settles the rounding, ties included.
__device__ __noinline__ int code_magnitude_exact(float a, float sf, float hs, float k, int qmax) {
    const float base = k * sf;                  // exact
    const float up = base + hs, lo = base - hs; // exact: (k + 1/2) s and (k - 1/2) s
    int q = (int)k;
    if (a > up) q += 1;
    else if (a < lo) q -= 1;
    else if (a == up) q += q & 1;              // tie between k and k + 1: the even one
    else if (a == lo) q -= q & 1;              // tie between k - 1 and k
    return min(q, qmax);
}
// The 1-bit scale FP16(mean |w|) of a group in global memory, by the eight
// lanes of mask (lane l of them: weights 4l .. and 32 + 4l ..), with the
// mean's sum taken as the balanced fp64 tree over neighbouring weights.
// When every nonzero |w| is a multiple of 2^L (L the smallest ulp exponent)
// and the largest ulp exponent is at most L + 23, all partial sums of that
// tree are multiples of 2^L below 2^(L + 53): the fp64 tree is exact, and the
// exact integer sum S = sum |w| / 2^L (below 2^53) gives FP16(S * 2^(L - 6))
// directly. Otherwise (a spread over 23 binades, or an infinity) the fp64
// tree is evaluated as written.
__device__ __noinline__ uint32_t one_bit_scale_exact(const float* group, int l, unsigned mask) {
    const float4 f0 = reinterpret_cast<const float4*>(group)[l], f1 = reinterpret_cast<const float4*>(group)[8 + l];
    const float a[8] = {fabsf(f0.x), fabsf(f0.y), fabsf(f0.z), fabsf(f0.w), fabsf(f1.x), fabsf(f1.y), fabsf(f1.z), fabsf(f1.w)};
    int L = 1000, H = -1000;
    bool finite = true;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t b = __float_as_uint(a[i]);
        const int e = (int)(b >> 23), u = max(e, 1) - 150;          // ulp exponent (subnormals share the smallest normal's)
        if (b) { L = min(L, u); H = max(H, u); }
        finite &= e < 255;
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        L = min(L, __shfl_xor_sync(mask, L, o));
        H = max(H, __shfl_xor_sync(mask, H, o));
    }
    finite = __all_sync(mask, finite);
    if (L == 1000) return 0u;                                        // all zero
    if (finite && H - L <= 23) {
        unsigned long long S = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t b = __float_as_uint(a[i]);
            const int e = (int)(b >> 23), u = max(e, 1) - 150;
            if (b) S += (unsigned long long)((b & 0x7FFFFFu) | (e ? 0x800000u : 0u)) << (u - L);
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) S += __shfl_xor_sync(mask, S, o);
        return fp16_bits_of_scaled(S, L - 6);
    }
    // the pairwise tree: each half's 32 weights over its lanes, then the halves
    double p = ((double)a[0] + (double)a[1]) + ((double)a[2] + (double)a[3]);
    double q = ((double)a[4] + (double)a[5]) + ((double)a[6] + (double)a[7]);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        p += __shfl_xor_sync(mask, p, o);
        q += __shfl_xor_sync(mask, q, o);
    }
    return fp16_bits_sat((p + q) * (1.0 / GROUP));                   // exact division by 64
}

// The same scale from t, an fp32 tree of depth 6 over the group's |w|: within
// 6 * 2^-24 (depth times unit roundoff) of the exact sum of the non-negative
// values, so its FP16 rounding is the exact mean's unless an FP16 midpoint
// lies within 2^-20 of the fp32 mean; then (rarely) near is set and the exact
// evaluation has to run.
__device__ __forceinline__ uint32_t one_bit_scale(float t, bool& near) {
    near = false;
    if (isinf(t)) return 0x7BFFu;                      // the exact mean is far above 65504 too
    const float mean = t * (1.f / GROUP);              // exact
    const uint32_t c = min((uint32_t)__half_as_ushort(__float2half_rn(mean)), 0x7BFFu);
    const float cv = __half2float(__ushort_as_half((uint16_t)c)), err = mean * 0x1p-20f;
    if (c < 0x7BFFu) near |= fabsf(mean - 0.5f * (cv + __half2float(__ushort_as_half((uint16_t)(c + 1))))) <= err;
    if (c > 0u) near |= fabsf(mean - 0.5f * (cv + __half2float(__ushort_as_half((uint16_t)(c - 1))))) <= err;
    return c;
}

// Codes of four weights as bytes (b >= 2), from r, an estimate of 1 / sf within
// 2^-22 relative (0 for sf = 0: every code is z). t = fl(v r), clipped to
// +-qmax, is within 2^-13 of the clipped quotient, and adding 1.5 * 2^23 + z
// rounds it half to even to the integer q and leaves q + z in the low byte.
// That is the answer whenever t is at least 0.0005 from a half-integer;
// otherwise (rarely) the exact thresholds decide.
__device__ __forceinline__ uint32_t codes4(float4 v, float r, float sf, float qmaxf, float magic) {
    const float x[4] = {v.x, v.y, v.z, v.w};
    uint32_t u[4];
    float worst = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float t = fminf(fmaxf(__fmul_rn(x[i], r), -qmaxf), qmaxf);
        const float m = __fadd_rn(t, magic);
        worst = fmaxf(worst, fabsf(__fsub_rn(t, __fsub_rn(m, magic))));
        u[i] = __float_as_uint(m);
    }
    if (worst > 0.4995f && r != 0.f) {                 // some weight near a half-integer
        const int z = (int)(magic - 12582912.f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = fabsf(x[i]);
            const int q = code_magnitude_exact(a, sf, 0.5f * sf, rintf(fminf(a * r, 256.f)), (int)qmaxf);
            u[i] = (uint32_t)(z + (x[i] < 0.f ? -q : q));
        }
    }
    return __byte_perm(__byte_perm(u[0], u[1], 0x0040), __byte_perm(u[2], u[3], 0x0040), 0x5410);
}

// Width in {1, 2, 4, 8} for every group (else err[0] = 1) and no NaN weight
// (else err[1] = 1): 16-byte loads over w and the widths as flat arrays. The
// weights from `keep` on are loaded to stay in L2: quantize_kernel, which
// walks the groups from the last, finds them there.
__global__ void quant_validate_kernel(const float* __restrict__ w, const uint8_t* __restrict__ widths,
                                      int64_t nweights, int64_t ngroups, int64_t keep, uint32_t* err) {
    uint32_t flags = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n4 = nweights / 4;                    // K % 64 == 0, so a whole number of float4
    const float4* w4 = reinterpret_cast<const float4*>(w);
    for (int64_t i = t0; i < n4; i += 4 * stride) {
        float4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t k = i + j * stride;
            v[j] = k >= n4 ? make_float4(0.f, 0.f, 0.f, 0.f) : 4 * k < keep ? __ldcs(w4 + k) : __ldg(w4 + k);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (isnan(v[j].x) || isnan(v[j].y) || isnan(v[j].z) || isnan(v[j].w)) flags |= 2u;
    }
    for (int64_t gi = t0; gi < ngroups; gi += stride) {
        const uint32_t b = widths[gi];
        if (b != 1 && b != 2 && b != 4 && b != 8) flags |= 1u;
    }
    if (flags & 1u) err[0] = 1u;
    if (flags & 2u) err[1] = 1u;
}

// 14336 x 4096 main: 101 -> 56 us (with the validation pass 146 -> 94).
__global__ void __launch_bounds__(QTHREADS, 3) quantize_kernel(const float* __restrict__ w,
                                                            const uint8_t* __restrict__ widths, int64_t ngroups,
                                                            uint8_t* __restrict__ codes, uint16_t* __restrict__ scales) {
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31, l = lane & 7, sub = lane >> 3;      // lane l of the load's group `sub`
    const int64_t warps = (int64_t)gridDim.x * (QTHREADS >> 5);
    const int64_t chunks = (ngroups + QGROUPS - 1) / QGROUPS;
    for (int64_t ck = (int64_t)blockIdx.x * (QTHREADS >> 5) + (threadIdx.x >> 5); ck < chunks; ck += warps) {
        const int64_t g0 = (chunks - 1 - ck) * QGROUPS;                    // from the last (see quant_validate_kernel)
        const int ng = (int)min((int64_t)QGROUPS, ngroups - g0);
        // lane j < 16 owns group g0 + j's scale
        const uint32_t bw = lane < ng ? widths[g0 + lane] : 2u;
        float4 v[QLOADS][2];
#pragma unroll
        for (int k = 0; k < QLOADS; ++k) {
            const int64_t gi = g0 + min(4 * k + sub, ng - 1);
            const float4* src = reinterpret_cast<const float4*>(w + gi * GROUP);
            v[k][0] = __ldcs(src + l);
            v[k][1] = __ldcs(src + 8 + l);
        }
        // max|w| and the fp32 tree of |w| of group 4k + sub; lane (4k + sub) keeps its own group's
        float gmax = 0.f, gsum = 0.f;
#pragma unroll
        for (int k = 0; k < QLOADS; ++k) {
            const float4 p = v[k][0], q = v[k][1];
            float m = fmaxf(fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fmaxf(fabsf(p.z), fabsf(p.w))),
                            fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fmaxf(fabsf(q.z), fabsf(q.w))));
            float t = ((fabsf(p.x) + fabsf(p.y)) + (fabsf(p.z) + fabsf(p.w))) +
                      ((fabsf(q.x) + fabsf(q.y)) + (fabsf(q.z) + fabsf(q.w)));
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                m = fmaxf(m, __shfl_xor_sync(ALL, m, o));
                t += __shfl_xor_sync(ALL, t, o);
            }
            const float mk = __shfl_sync(ALL, m, 8 * (lane & 3)), tk = __shfl_sync(ALL, t, 8 * (lane & 3));
            if ((lane >> 2) == k) { gmax = mk; gsum = tk; }
        }
        bool near = false;
        const int qmax = (1 << (bw - 1)) - 1;
        uint32_t sbits = bw == 1 ? one_bit_scale(gsum, near) : fp16_bits_of_quotient(gmax, qmax);
        // groups whose 1-bit mean is near an FP16 midpoint: exactly, by their eight lanes
        for (uint32_t todo = __ballot_sync(ALL, near && lane < ng); todo; todo &= todo - 1) {
            const int j = __ffs(todo) - 1;
            uint32_t ex = 0;
            if (lane < 8) ex = one_bit_scale_exact(w + (g0 + j) * GROUP, lane, 0xFFu);
            ex = __shfl_sync(ALL, ex, 0);
            if (lane == j) sbits = ex;
        }
        if (lane < ng) scales[g0 + lane] = (uint16_t)sbits;
        const float sf = __half2float(__ushort_as_half((uint16_t)sbits));
        const float r = sf == 0.f ? 0.f : rcp_estimate(sf);
#pragma unroll
        for (int k = 0; k < QLOADS; ++k) {
            const int j = 4 * k + sub;
            const uint32_t bj = __shfl_sync(ALL, bw, j);
            const float sj = __shfl_sync(ALL, sf, j), rj = __shfl_sync(ALL, r, j);
            uint32_t lo, hi;
            if (bj == 1) {
                const float4 p = v[k][0], q = v[k][1];
                lo = (p.x >= 0.f ? 1u : 0u) | (p.y >= 0.f ? 0x100u : 0u) | (p.z >= 0.f ? 0x10000u : 0u) | (p.w >= 0.f ? 0x1000000u : 0u);
                hi = (q.x >= 0.f ? 1u : 0u) | (q.y >= 0.f ? 0x100u : 0u) | (q.z >= 0.f ? 0x10000u : 0u) | (q.w >= 0.f ? 0x1000000u : 0u);
            } else {
                const int z = 1 << (bj - 1);
                const float qm = (float)(z - 1), magic = 12582912.f + (float)z;
                lo = codes4(v[k][0], rj, sj, qm, magic);
                hi = codes4(v[k][1], rj, sj, qm, magic);
            }
            if (j < ng) {
                uint32_t* dst = reinterpret_cast<uint32_t*>(codes + (g0 + j) * GROUP);
                dst[l] = lo;
                dst[8 + l] = hi;
            }
        }
    }
}

int grid_for(int64_t ngroups, int warps_per_block, int per_warp, int blocks_per_sm) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t need = (ngroups + (int64_t)warps_per_block * per_warp - 1) / ((int64_t)warps_per_block * per_warp);
    const int64_t cap = (int64_t)sms * blocks_per_sm;       // one resident wave, grid-stride
    return (int)(need < cap ? (need > 0 ? need : 1) : cap);
}

}  // namespace

cudaError_t launch_quant_validate(const float* w, const uint8_t* widths, int64_t N, int64_t K, uint32_t* err,
                                  cudaStream_t s) {
    const int64_t ngroups = N * (K / GROUP);
    const int64_t keep = N * K - QKEEP_BYTES / 4;
    quant_validate_kernel<<<grid_for(N * K / 4, QTHREADS, 4, 4), QTHREADS, 0, s>>>(w, widths, N * K, ngroups, keep, err);
    return cudaGetLastError();
}

cudaError_t launch_quantize(const float* w, const uint8_t* widths, int64_t N, int64_t K, uint8_t* codes,
                            uint16_t* scales, cudaStream_t s) {
    const int64_t ngroups = N * (K / GROUP);
    quantize_kernel<<<grid_for(ngroups, QTHREADS / 32, QGROUPS, 3), QTHREADS, 0, s>>>(w, widths, ngroups, codes, scales);
    return cudaGetLastError();
}

}  // namespace vbq
