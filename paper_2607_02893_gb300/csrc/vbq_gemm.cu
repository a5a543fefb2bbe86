// vbq_gemm.cu — batched product Y = X W^T for 2..16 activation rows (§6's
// fused dequantise-and-multiply, several tokens at once) on the tensor cores.
//
// With B activation rows every decoded weight is used B times, so the product
// is a dense contraction over dequantised tiles: mma.sync m16n8k16, bf16
// operands, fp32 accumulators. A tile is 16 items (groups) of one (column,
// width) bucket of a unit:
//
//   A  the items' levels L_b(u), exact in bf16, decoded in registers: lane (g,
//      t) holds 16 weights of item g and of item g + 8, register r = weights p
//      and p + 16 with p = 32 (t / 2) + 8 (t % 2) + r. Any assignment of a
//      group's weights to the MMA's k positions gives the same sum if B uses
//      it too; this one lets every width decode by shifts, one logic operation
//      and one bf16 operation per register.
//   B  the column's activations as they are (bf16), in the same order, 8 batch
//      rows per MMA (two for more than 8; rows >= B are zero), held in registers
//      for all tiles of the column.
//   D  item x batch row, fp32: scaled by the item's FP16 scale and added to the
//      warp's own row sums in shared memory. A warp takes whole columns of a
//      unit (a column has one item per row), so these are plain loads and
//      stores: no shared-memory float additions (compare-and-swap loops on this
//      GPU) and nothing shared between warps until the unit ends.
//   Levels and activations are exact and their products accumulate in fp32;
//   a group whose codes all sit at the zero level gives exactly 0.
//
// Bound: instruction issue and its latencies (8192^2 main at 8 rows: 51% issue,
// ALU pipe, which runs logic and shifts at half rate, 37% busy, tensor pipe
// 15%; 16384 x 8192: 55% issue). Per 32 groups of the main mix and 8 rows a warp
// issues 268 instructions, where fp16 denormal levels, clamped item indexes and
// per-(row, column) slots took 375. Per product in a graph of dependent
// products, before -> now: 14336 x 4096 main 18.6 -> 12.5 us at 8 rows and 34.7
// -> 17.0 at 16; 16384^2 all 1 bit 59 -> 42 and 97 -> 60, all 2 bits 71 -> 46 and
// 106 -> 63, all 4 bits 72 -> 57 and 121 -> 80, all 8 bits 98 -> 95 and 170 -> 134. The error against 64 bits fell
// from 5e-6 to 1e-7 of the result's norm: denormal operands lose their
// alignment in the tensor core's sums, normal bf16 ones do not.
//
// Two blocks of eight consumer warps per SM, persistent over the units; a
// control warp zeroes Y's split-K rows (epoch-tagged flags, see vbq_gemv.cu)
// and streams each next unit's blob into the stage the consumers have left.
// One block's copies, row flushes and start are covered by the other's work
// (and the next launch's blocks by this one's). (The tcgen05 form was built
// and measured slower here: with the levels in tensor memory a thread decodes
// a whole item, a warp runs every width among its 32 items one after another,
// and each 128-item tile costs its warps about 200 instructions of waits,
// fences and issue; 14336 x 4096 main at 8 rows took 25 us.)
#include "vbq_kernels.h"
#include "vbq_deal.h"
#include "vbq_device.cuh"
#include <cuda_bf16.h>

namespace vbq {
namespace {

constexpr int NCWB = 8;                  // consumer warps
constexpr int NCTB = 32 * NCWB;
constexpr int GB_THREADS = 32 * (NCWB + 1);
constexpr int STAGE_BYTES_B = MAX_BLOB_BYTES;
constexpr int GB_BLOCKS = 2;             // resident per SM

// NB = 8 or 16 batch rows.
template <int NB>
struct __align__(16) TablesB {
    float acc[NCWB][NB / 8][RB][8];             // per warp: the unit's row sums, 8 batch rows together
    unsigned long long full;                    // blob landed
    unsigned long long empty;                   // every consumer warp is done with the blob
    unsigned long long sums;                    // clusters: the other slabs' sums of this block's rows landed
    uint32_t consts[12];                        // DecodeConsts
    int abort;
    uint32_t sk_ok;                             // the control warp's split-K flag check, passed on
};
template <int NB>
constexpr size_t gemmb_smem() { return 256 + (size_t)STAGE_BYTES_B + sizeof(TablesB<NB>); }
static_assert(2 * (gemmb_smem<16>() + 1024) <= 228 * 1024, "two blocks per SM");

__device__ __forceinline__ void consumer_sync_b() {
    asm volatile("bar.sync 1, %0;" :: "n"(NCTB) : "memory");
}

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The same with a zero accumulator (the first k-step of a tile).
__device__ __forceinline__ void mma16816_z(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

__device__ __forceinline__ void sts_f32x2(uint32_t addr, float2 v) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" :: "r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void sts_f32x4(uint32_t addr, float4 v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" :: "r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// ---- levels as bf16 pairs -----------------------------------------------------
//
// Every register is made by one logic operation (a field of the codes into the
// low mantissa bits of bf16 128.0) and one exact bf16 operation. Both take two
// constants where an instruction encodes one, so the others sit in registers:
// DecodeConsts, read from shared memory (a constant the compiler can see is
// moved into place before each use).
struct DecodeConsts {
    uint32_t one28;            // bf16 pair 128, 128
    uint32_t minus256;         // bf16 pair -256, -256
    uint32_t q[5];             // bf16 pairs 2^-1 .. 2^-5
    uint32_t add[5];           // bf16 pairs -(2^(8-k) + 1), k = 2 .. 6 (one bit)
};
constexpr uint32_t bf2_pair(uint32_t bf16_bits) { return bf16_bits | (bf16_bits << 16); }

__device__ __forceinline__ uint32_t bf2_fma(uint32_t a, uint32_t b, uint32_t c) {
    const __nv_bfloat162 r = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b),
                                     *reinterpret_cast<const __nv_bfloat162*>(&c));
    return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ uint32_t bf2_add(uint32_t a, uint32_t b) {
    const __nv_bfloat162 r = __hadd2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ uint32_t bf2_const(float v) {
    const __nv_bfloat162 r = __float2bfloat162_rn(v);
    return *reinterpret_cast<const uint32_t*>(&r);
}

// Lane t's 16 weights of the item at pay (p = 32 (t / 2) + 8 (t % 2) + r and
// p + 16, r < 8) as 8 registers. off: the lane's byte offset within an item of
// this width (lane_offset); sh = 8 (t % 2).
template <int W>
__device__ __forceinline__ uint32_t lane_offset(int t) {
    return W <= 1 ? 4u * (t >> 1) : W == 2 ? 16u * (t >> 1) + 4u * (t & 1) : 32u * (t >> 1) + 8u * (t & 1);
}
// 1 bit: bits r and r + 16 of the lane's byte pair brought to a mantissa bit k
// in 1 .. 6 of 128 (128 + u 2^k), then 2u - 1.
__device__ __forceinline__ void levels_1(const DecodeConsts& K, uint32_t pay, int sh, uint32_t (&r)[8]) {
    const uint32_t w = lds_u32(pay) >> sh;
    r[0] = bf2_add(((w << 1) & 0x00020002u) | K.one28, bf2_const(-129.f));
    r[1] = bf2_add((w & 0x00020002u) | K.one28, bf2_const(-129.f));
#pragma unroll
    for (int k = 2; k <= 6; ++k) r[k] = bf2_fma((w & (0x00010001u << k)) | K.one28, K.q[k - 2], K.add[k - 2]);
    r[7] = bf2_add(((w >> 6) & 0x00020002u) | K.one28, bf2_const(-129.f));
}
// 2 bits in two bit planes: interleaved to two-bit fields (even and odd
// weights), a field at bits 2i of each half (128 + u 4^i, i < 3), then u - 2.
__device__ __forceinline__ void levels_2(const DecodeConsts& K, uint32_t pay, int sh, uint32_t (&r)[8]) {
    const uint32_t p0 = lds_u32(pay) >> sh, p1 = lds_u32(pay + 8) >> sh;
    const uint32_t e1 = p1 << 1, o0 = p0 >> 1;
    const uint32_t even = e1 ^ ((p0 ^ e1) & 0x55555555u), odd = p1 ^ ((o0 ^ p1) & 0x55555555u);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t v = h ? odd : even;
        r[h] = bf2_add((v & 0x00030003u) | K.one28, bf2_const(-130.f));
        r[2 + h] = bf2_fma((v & 0x000C000Cu) | K.one28, K.q[1], bf2_const(-34.f));
        r[4 + h] = bf2_fma((v & 0x00300030u) | K.one28, K.q[3], bf2_const(-10.f));
        r[6 + h] = bf2_add(((v >> 6) & 0x00030003u) | K.one28, bf2_const(-130.f));
    }
}
// 4 bits: nibbles of two words side by side, as the low mantissa bits of 128; minus 136.
__device__ __forceinline__ void levels_4(const DecodeConsts& K, uint32_t pay, uint32_t (&r)[8]) {
    const uint32_t a = lds_u32(pay), b = lds_u32(pay + 8);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t v = __byte_perm(a, b, h ? 0x7632 : 0x5410);
#pragma unroll
        for (int i = 0; i < 4; ++i) r[4 * h + i] = bf2_add(((v >> (4 * i)) & 0x000F000Fu) | K.one28, bf2_const(-136.f));
    }
}
// 8 bits: bytes of two words side by side; 128 plus the low seven bits, minus
// 128 (top bit set) or 256 (clear): bf16 -256 with its lowest exponent bit
// flipped is -128.
__device__ __forceinline__ void levels_8(const DecodeConsts& K, uint32_t pay, uint32_t (&r)[8]) {
    const uint2 a = lds_u32x2(pay), b = lds_u32x2(pay + 16);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const uint32_t v = __byte_perm(h < 2 ? a.x : a.y, h < 2 ? b.x : b.y, h & 1 ? 0x7632 : 0x5410);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t u = v >> (8 * i);
            r[2 * h + i] = bf2_add((u & 0x007F007Fu) | K.one28, (u & 0x00800080u) ^ K.minus256);
        }
    }
}
template <int W>
__device__ __forceinline__ void levels(const DecodeConsts& K, uint32_t pay, int sh, uint32_t (&r)[8]) {
    if (W == 0) levels_1(K, pay, sh, r);
    else if (W == 1) levels_2(K, pay, sh, r);
    else if (W == 2) levels_4(K, pay, r);
    else levels_8(K, pay, r);
}

// Lane (g, t)'s B registers of a column at x (batch row g, and g + 8 for NB =
// 16): weights p + r and p + 16 + r side by side, r < 8. (Loaded ahead, while
// the column before is multiplied, they cost registers: no faster for 8 rows,
// 8% slower with spills for 16.)
template <int NB>
__device__ __forceinline__ void load_acts(uint32_t (&xb)[NB], const uint16_t* __restrict__ x, int64_t K, int B, int g, int t) {
#pragma unroll
    for (int n = 0; n < NB / 8; ++n) {
        uint4 lo = make_uint4(0u, 0u, 0u, 0u), hi = lo;
        if (8 * n + g < B) {
            const uint16_t* src = x + (int64_t)(8 * n + g) * K + 32 * (t >> 1) + 8 * (t & 1);
            lo = ldg_input_u32x4(src);
            hi = ldg_input_u32x4(src + 16);
        }
        const uint32_t a[4] = {lo.x, lo.y, lo.z, lo.w}, b[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            xb[8 * n + 2 * i] = __byte_perm(a[i], b[i], 0x5410);
            xb[8 * n + 2 * i + 1] = __byte_perm(a[i], b[i], 0x7632);
        }
    }
}

// Tiles k0, k0 + kstep, ... of one bucket of n items of width index W. pay, sc
// and rw point at the lane's item g of tile 0 (payload plus lane offset,
// scale, row byte); acc at the lane's pair of batch rows of row 0. Lanes past
// the bucket's end decode whatever bytes follow (levels of any bits are
// finite, and the stage is followed by the block's own tables) and add nothing.
template <int NB, int W>
__device__ __forceinline__ void run_tiles(const DecodeConsts& K, const uint32_t (&xb)[NB], uint32_t pay, uint32_t sc, uint32_t rw,
                                          int n, int k0, int kstep, uint32_t acc, int g, int sh) {
    constexpr int BPI = 8 << W;
    pay += k0 * 16 * BPI;
    sc += k0 * 32;
    rw += k0 * 16;
    for (int left = n - 16 * k0; left > 0; left -= 16 * kstep) {
        const uint32_t sa = lds_u16_ordered(sc), sb = lds_u16_ordered(sc + 16), ra = lds_u8(rw), rb = lds_u8(rw + 8);
        uint32_t la[8], lb[8];
        levels<W>(K, pay, sh, la);
        levels<W>(K, pay + 8 * BPI, sh, lb);
        float d[NB / 8][4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const uint32_t a[4] = {la[2 * s], lb[2 * s], la[2 * s + 1], lb[2 * s + 1]};
#pragma unroll
            for (int m = 0; m < NB / 8; ++m) {
                if (s == 0) mma16816_z(d[m], a, xb[8 * m], xb[8 * m + 1]);
                else mma16816(d[m], a, xb[8 * m + 2 * s], xb[8 * m + 2 * s + 1]);
            }
        }
        const float fa = half_bits(sa), fb = half_bits(sb);
        const uint32_t aa = acc + ra * 32, ab = acc + rb * 32;
        if (g < left) {
#pragma unroll
            for (int m = 0; m < NB / 8; ++m) {
                const uint32_t at = aa + m * (RB * 32);
                sts_f32x2(at, __ffma2_rn(f2(d[m][0], d[m][1]), f2(fa, fa), lds_f32x2_ordered(at)));
            }
        }
        if (g + 8 < left) {
#pragma unroll
            for (int m = 0; m < NB / 8; ++m) {
                const uint32_t at = ab + m * (RB * 32);
                sts_f32x2(at, __ffma2_rn(f2(d[m][2], d[m][3]), f2(fb, fb), lds_f32x2_ordered(at)));
            }
        }
        pay += kstep * 16 * BPI;
        sc += kstep * 32;
        rw += kstep * 16;
    }
}

// How a unit's columns are dealt to the 8 warps: a warp takes columns c0, c0 +
// step, ..., and of each every `parts`-th tile from `sub` on (several warps
// share a column only where the unit has fewer columns than warps).
struct Deal {
    int c0, step, parts, sub;
};
__device__ __forceinline__ Deal deal_columns(int cols, int cw) {
    const int lg = cols > 4 ? 0 : cols > 2 ? 1 : cols > 1 ? 2 : 3;
    return Deal{cw >> lg, NCWB >> lg, 1 << lg, cw & ((1 << lg) - 1)};
}

// One warp's share of columns [c_lo, c_lo + cols) of a unit (blob at sblob,
// activations of its slab at x); xb holds the first column's activations. A
// bucket's offsets are read from the header as it begins: held over the unit
// they took 12 registers of the tile loops (16384^2 all 8 bits at 4 rows 89.2 us,
// 87.0; 14336 x 4096 main at 16 rows 17.8, 17.0).
template <int NB>
__device__ __forceinline__ void consume_unit_b(const DecodeConsts& K, uint32_t sblob, int C, int c_lo, int cols, const Deal& dl,
                                               uint32_t (&xb)[NB], const uint16_t* __restrict__ x, int64_t Kx, int B,
                                               uint32_t acc, int lane) {
    const int g = lane >> 2, t = lane & 3, sh = 8 * (t & 1);
    const uint32_t cc = sblob + lds_u16_ordered(sblob + offsetof(UnitHeader, cc16)) * 16;
    const uint32_t my = acc + 8u * t;
    for (int c = c_lo + dl.c0; c < c_lo + cols; c += dl.step) {
        int s[4], e[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            e[w] = (int)lds_u16_ordered(cc + 2 * (w * C + c));
            s[w] = c ? (int)lds_u16_ordered(cc + 2 * (w * C + c) - 2) : 0;
        }
        int done = 0;                    // tiles of the column before this bucket
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int n = e[w] - s[w], first = s[w] + g;
            const uint32_t p16 = lds_u16_ordered(sblob + offsetof(UnitHeader, pay16) + 2 * w);
            const uint32_t s16 = lds_u16_ordered(sblob + offsetof(UnitHeader, sc16) + 2 * w);
            const uint32_t r16 = lds_u16_ordered(sblob + offsetof(UnitHeader, row16) + 2 * w);
            const uint32_t pay = sblob + p16 * 16 + first * (8 << w), sc = sblob + s16 * 16 + first * 2, rw = sblob + r16 * 16 + first;
            const int k0 = (dl.sub - done) & (dl.parts - 1);
            if (w == 0) run_tiles<NB, 0>(K, xb, pay + lane_offset<0>(t), sc, rw, n, k0, dl.parts, my, g, sh);
            else if (w == 1) run_tiles<NB, 1>(K, xb, pay + lane_offset<1>(t), sc, rw, n, k0, dl.parts, my, g, sh);
            else if (w == 2) run_tiles<NB, 2>(K, xb, pay + lane_offset<2>(t), sc, rw, n, k0, dl.parts, my, g, sh);
            else run_tiles<NB, 3>(K, xb, pay + lane_offset<3>(t), sc, rw, n, k0, dl.parts, my, g, sh);
            done += (n + 15) >> 4;
        }
        __syncwarp();                    // the next column's additions follow this one's (other lanes hold its rows)
        if (c + dl.step < c_lo + cols) load_acts<NB>(xb, x + (int64_t)(c + dl.step) * GROUP, Kx, B, g, t);
    }
}

// After a unit: the warps' row sums added in warp order into Y (stored with
// one slab, else added), and set back to zero. Thread ct: row ct / 2, batch
// rows 4 (ct % 2) .. + 3 of each eight.
template <int NB>
__device__ __forceinline__ void flush_rows(TablesB<NB>& T, const LayoutView& L, float* __restrict__ Y, int B, int rb, int ct) {
    const int r = ct >> 1, q = ct & 1;
    const int rows = min(RB, (int)(L.N - (int64_t)rb * RB));
#pragma unroll
    for (int n = 0; n < NB / 8; ++n) {
        const int b0 = 8 * n + 4 * q;
        if (b0 >= B) continue;           // absent batch rows: their sums stay zero
        const uint32_t at = smem_u32(&T.acc[0][n][r][4 * q]);
        float4 v = lds_f32x4_ordered(at);
        sts_zero4(at);
#pragma unroll
        for (int w = 1; w < NCWB; ++w) {
            const uint32_t aw = at + w * (uint32_t)sizeof(T.acc[0]);
            const float4 o = lds_f32x4_ordered(aw);
            sts_zero4(aw);
            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
        }
        if (r < rows) {
            float* y = Y + (int64_t)b0 * L.N + (int64_t)rb * RB + r;
            const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (b0 + k < B) {
                    if (L.S == 1) y[k * L.N] = f[k];
                    else red_global(y + k * L.N, f[k]);
                }
            }
        }
    }
}

// The slabs of a row block as one cluster (CL): block `rank` holds slab rank's
// unit, and owns rows [rank * own, (rank + 1) * own) of the row block. Once
// every block of the cluster is done with its blob (the cluster barrier before
// this), each sends its sums of the others' rows into their stages (st.async,
// counted on their `sums` barriers), adds the S sums of its own rows in slab
// order and stores them: no zeroing, flags or global additions, and the same
// bits on every call. Slab k's sums of a block's row i sit at ((k * own + i) *
// NB) floats. write is false after a wait that ran out.
__host__ __device__ inline int cluster_rows(int S) { return (RB + S - 1) / S; }
__host__ __device__ inline int batch_quads(int B) { return (B + 3) / 4; }      // only these batch rows are exchanged
template <int NB>
__device__ __forceinline__ void flush_cluster(TablesB<NB>& T, uint32_t stage, const LayoutView& L, float* __restrict__ Y, int B,
                                              int rb, int rank, int ct, bool write) {
    const int rows = min(RB, (int)(L.N - (int64_t)rb * RB)), own = cluster_rows(L.S);
    const uint32_t sums = smem_u32(&T.sums);
    const int r = ct >> 1, q = ct & 1, to = r / own, i = r - to * own;
#pragma unroll
    for (int n = 0; n < NB / 8; ++n) {
        if (8 * n + 4 * q >= B) continue;
        const uint32_t at = smem_u32(&T.acc[0][n][r][4 * q]);
        float4 v = lds_f32x4_ordered(at);
#pragma unroll
        for (int w = 1; w < NCWB; ++w) {
            const float4 o = lds_f32x4_ordered(at + w * (uint32_t)sizeof(T.acc[0]));
            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
        }
        if (r < rows) {
            const uint32_t dst = stage + (uint32_t)(((rank * own + i) * NB + 8 * n + 4 * q) * 4);
            if (to == rank) sts_f32x4(dst, v);
            else st_async_f32x4(cluster_addr(dst, to), v, cluster_addr(sums, to));
        }
    }
    consumer_sync_b();
    const int mine = max(0, min(own, rows - rank * own));
    if (mine > 0 && !__all_sync(0xffffffffu, mbar_wait_cluster(sums, 0))) {
        if ((ct & 31) == 0) raise_abort(&T.abort);
        return;
    }
    if (!write) return;
    for (int k = ct; k < mine * batch_quads(B); k += NCTB) {
        const int b4 = k / mine, row = k - b4 * mine;
        const uint32_t at = stage + (uint32_t)((row * NB + 4 * b4) * 4);
        float4 v = lds_f32x4_ordered(at);
        for (int sl = 1; sl < L.S; ++sl) {
            const float4 o = lds_f32x4_ordered(at + (uint32_t)(sl * own * NB * 4));
            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
        }
        float* y = Y + (int64_t)(4 * b4) * L.N + (int64_t)rb * RB + rank * own + row;
        const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * b4 + j < B) y[j * L.N] = f[j];
    }
}

// How a launch's units go to its blocks, each form an instantiation of its own:
// evenly, with left-over units cut (see Shares), or a row block's slabs as a
// cluster.
enum Split : int { SPLIT_EVEN, SPLIT_CUT, SPLIT_CLUSTER };

template <int NB, int SPLIT>
__global__ void __launch_bounds__(GB_THREADS, GB_BLOCKS) gemmb_kernel(LayoutView L, const uint16_t* __restrict__ X,
                                                                      float* __restrict__ Y, int B, Shares sh) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((256u - (smem_u32(smem_raw) & 255u)) & 255u);
    TablesB<NB>& T = *reinterpret_cast<TablesB<NB>*>(base + STAGE_BYTES_B);
    const uint32_t stage = smem_u32(base);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int P = gridDim.x, p = blockIdx.x;
    constexpr bool CL = SPLIT == SPLIT_CLUSTER, CUT = SPLIT == SPLIT_CUT;
    // the block's places in the deal: begin, begin + 1, ..., and perhaps a part of another
    int begin, whole, part_at = -1, part = 0;
    if (CL) {                            // block rb * S + s: unit (rb, s)
        const int rb = p / L.S;
        begin = (p - rb * L.S) * L.nrb + rb;
        whole = 1;
    } else {
        const BlockShare b = block_share(L.units, CUT ? sh : Shares{0, 0, 1, 0}, P, p);
        begin = b.begin;
        whole = b.whole;
        if (CUT) {
            part_at = b.part_at;
            part = b.part;
        }
    }
    const int n_units = whole + (part_at >= 0), rot = CUT ? sh.rot : 0;
    auto place = [&](int j) { return j < whole ? begin + j : part_at; };
    // the block that zeroes Y's rows of place j's row block (under split-K; slab 0 is dealt in order)
    auto owns_zeroing = [&](int j) { return place(j) < L.nrb && (j < whole || part == 0); };
    auto row_block = [&](int j) { return dealt_row_block(place(j), place(j) / L.nrb, L.nrb, rot); };
    const int rb_lane = lane < n_units ? row_block(lane) : 0;      // a division, ahead of the wait
    const int s0 = place(0) / L.nrb, rb0 = dealt_row_block(place(0), s0, L.nrb, rot);

    const uint32_t full = smem_u32(&T.full), empty = smem_u32(&T.empty);
    const uint32_t abort_addr = smem_u32(&T.abort);
    if (tid == 0) {
        mbar_init(full, 1);
        mbar_init(empty, NCWB);
        if (CL) mbar_init(smem_u32(&T.sums), 1);
        T.abort = 0;
        T.sk_ok = 0;
        fence_barrier_init();
        issue_unit(L, s0 * L.nrb + rb0, stage, full);
        if (CL) {
            const int rows = min(RB, (int)(L.N - (int64_t)rb0 * RB)), own = cluster_rows(L.S);
            const int mine = max(0, min(own, rows - s0 * own));
            if (mine > 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                             :: "r"(smem_u32(&T.sums)), "r"((uint32_t)((L.S - 1) * mine * batch_quads(B) * 16)) : "memory");
        }
        T.consts[0] = bf2_pair(0x4300);
        T.consts[1] = bf2_pair(0xC380);
        const uint32_t adds[5] = {0xC282, 0xC204, 0xC188, 0xC110, 0xC0A0};     // -65, -33, -17, -9, -5
        for (int i = 0; i < 5; ++i) {
            T.consts[2 + i] = bf2_pair(0x3F00 - 0x80 * i);
            T.consts[7 + i] = bf2_pair(adds[i]);
        }
    }
    for (int i = tid; i < (int)sizeof(T.acc) / 16; i += GB_THREADS) sts_zero4(smem_u32(&T.acc[0][0][0][0]) + 16 * i);
    {   // the first slab's activations into L2 while waiting for the previous grid
        const int64_t k0 = (int64_t)s0 * L.C * GROUP;
        const int lines = (min(L.C, L.G - s0 * L.C) * GROUP * 2 + 127) / 128;
        for (int q = tid - 32; q >= 0 && q < lines * B; q += GB_THREADS - 32)
            prefetch_l2(X + (int64_t)(q / lines) * L.K + k0 + (int64_t)(q % lines) * 64);
    }
    __syncthreads();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == 0) {
        // ---- control: split-K zeroing, then each next copy into the freed stage ----
        // (whole row blocks are zeroed 4 rows per lane when every batch row of Y
        // starts on a 16-byte boundary)
        if (CL) {
            cluster_arrive();            // see the consumers: every block is done with its blob
            cluster_wait();
            if (lds_volatile(abort_addr) && lane == 0) mbar_wait_bounded(full, 0);
            return;
        }
        const bool vec = (L.N & 3) == 0;
        uint32_t epoch = 0;
        if (L.S > 1) {
            // the call count's load is in flight while the warp zeroes (the zeros
            // do not depend on it; the flags do)
            const unsigned long long count = call_count_raw(L.ctl);
            for (int j = 0; j < n_units; ++j) {
                if (!owns_zeroing(j)) continue;
                const int u = place(j);
                const int rows = min(RB, (int)(L.N - (int64_t)u * RB));
                for (int b = 0; b < B; ++b) {
                    float* yr = Y + (int64_t)b * L.N + (int64_t)u * RB;
                    if (vec && rows == RB) reinterpret_cast<float4*>(yr)[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
                    else
                        for (int r = lane; r < rows; r += 32) yr[r] = 0.f;
                }
            }
            __syncwarp();
            epoch = epoch_of(count);
            // release stores, one unit per lane in parallel: the warp's zeros
            // (ordered by __syncwarp) before each flag
            for (int j = lane; j < n_units; j += 32)
                if (owns_zeroing(j)) st_release_gpu(L.ctl + 2 + place(j), epoch);
        }
        bool dead = false;
        if (L.S > 1) {
            // every row block this block adds into zeroed in this call (flag ==
            // epoch), within the wait limit; a lane per unit, acquire loads
            bool seen = true;
            const unsigned long long t0 = global_ns();
            for (int j = lane; j < n_units && seen; j += 32) {
                if (owns_zeroing(j)) continue;
                const uint32_t* f = L.ctl + 2 + (j == lane ? rb_lane : row_block(j));
                while (!(seen = ld_acquire_gpu(f) == epoch))
                    if (global_ns() - t0 > WAIT_LIMIT_NS) break;
            }
            __syncwarp();                // every lane's later additions after every acquire
            if (!__all_sync(0xffffffffu, seen)) {
                dead = true;
                if (lane == 0) raise_abort(&T.abort);
            }
        }
        // the consumers write Y; they add only after these flags (and this
        // warp's own zeroing), passed on by a release
        if (L.S > 1 && lane == 0) red_release_cta_shared_add(smem_u32(&T.sk_ok), dead ? 0x10000u : 1u);
        int issued = 1;
        for (int j = 0; j + 1 < n_units && !dead; ++j) {
            // A refill's latency is on the block's path (one stage). With narrow units,
            // of few groups for their bytes, its offsets are read before the stage
            // is free (16384^2 all 4 bits at 4 rows 53.3 us, 55.7 otherwise); with
            // 16-column units that loses 1% (8192^2 main 15.1, 15.3).
            const int d = place(j + 1), sl = d / L.nrb, u = sl * L.nrb + dealt_row_block(d, sl, L.nrb, rot);
            const bool early = L.C < MAX_C;
            uint32_t o0 = 0, o1 = 0;
            if (early) { o0 = L.blob_off[u]; o1 = L.blob_off[u + 1]; }
            if (!warp_wait(empty, (uint32_t)j & 1u, abort_addr, 128)) {
                dead = true;
                if (lane == 0) raise_abort(&T.abort);
                break;
            }
            if (lane == 0) {
                if (early) bulk_load(stage, L.blobs + (int64_t)o0 * 16, (o1 - o0) * 16, full);
                else issue_unit(L, u, stage, full);
            }
            ++issued;
        }
        if (L.S > 1 && lane == 0) call_done(L.ctl);      // this block's share of the call count
        // after a wait that ran out, let the last copy land before the block exits
        if (lds_volatile(abort_addr) && lane == 0) mbar_wait_bounded(full, (uint32_t)(issued - 1) & 1u);
    } else {
        // ---- consumers: every unit, whole columns (or a share of one) per warp ----
        const int ct = tid - 32, cw = warp - 1;
        bool dead = false, sk_seen = L.S == 1;
        const uint32_t acc = smem_u32(&T.acc[cw][0][0][0]);
        DecodeConsts K;
        {
            const uint32_t at = smem_u32(T.consts);
            K.one28 = lds_volatile(at);
            K.minus256 = lds_volatile(at + 4);
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                K.q[i] = lds_volatile(at + 8 + 4 * i);
                K.add[i] = lds_volatile(at + 28 + 4 * i);
            }
        }
        for (int j = 0; j < n_units; ++j) {
            const int d = place(j), sj = d / L.nrb, rbj = dealt_row_block(d, sj, L.nrb, rot);
            int cols = min(L.C, L.G - sj * L.C), c_lo = 0;
            if (CUT && j >= whole) {     // a part: its share of the columns
                c_lo = cols * part / sh.parts;
                cols = cols * (part + 1) / sh.parts - c_lo;
            }
            const Deal dl = deal_columns(cols, cw);
            const uint16_t* x = X + (int64_t)sj * L.C * GROUP;
            uint32_t xb[NB];             // the first column's activations, on their way while the blob lands
            if (dl.c0 < cols) load_acts<NB>(xb, x + (int64_t)(c_lo + dl.c0) * GROUP, L.K, B, lane >> 2, lane & 3);
            if (!dead && !warp_wait(full, (uint32_t)j & 1u, abort_addr)) { dead = true; if (lane == 0) raise_abort(&T.abort); }
            if (!dead) {
                consume_unit_b<NB>(K, stage, L.C, c_lo, cols, dl, xb, x, L.K, B, acc, lane);
                __syncwarp();
                if (!CL && lane == 0) mbar_arrive(empty);
            }
            if constexpr (CL) {
                // every warp's sums, and every block of the cluster done with its blob
                cluster_arrive();
                cluster_wait();
                flush_cluster<NB>(T, stage, L, Y, B, rb0, s0, ct, !dead && !lds_volatile(abort_addr));
                return;
            }
            consumer_sync_b();           // every warp's sums
            if (!sk_seen && !dead) {
                // split-K: after the control warp's flag check (bounded wait)
                uint32_t g = 0;
                const unsigned long long w0 = global_ns();
                while ((g = ld_acquire_cta_shared(smem_u32(&T.sk_ok))) == 0u && !lds_volatile(abort_addr) &&
                       global_ns() - w0 < WAIT_LIMIT_NS)
                    __nanosleep(32);
                if (g != 1u) {
                    dead = true;
                    if (lane == 0) raise_abort(&T.abort);
                }
                sk_seen = true;
            }
            if (!dead && !lds_volatile(abort_addr)) flush_rows<NB>(T, L, Y, B, rbj, ct);
            if (j + 1 < n_units) consumer_sync_b();      // the rows are read and zero again
        }
    }
}

template <int NB, int SPLIT>
cudaError_t launch_gemmb(const LayoutView& L, const uint16_t* X, float* Y, int B, cudaStream_t s, int grid, Shares sh) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(GB_THREADS);
    cfg.dynamicSmemBytes = gemmb_smem<NB>();
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = L.S;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = SPLIT == SPLIT_CLUSTER ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, gemmb_kernel<NB, SPLIT>, L, X, Y, B, sh);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// Layouts of narrow units that all have a block at once (two per SM, less what
// clusters leave unused of a GPC's SMs, see unit_plan_fits) run a row block's
// slabs as a cluster for more than 8 rows, and for 5 to 8 where the matrix, and
// a square one on its input (its neighbours on the stream), is small (under
// 50,000 groups, at most 8 slabs): zeroing the rows of Y behind flags and adding
// into them is then on the product's path. Flags -> cluster (us in a graph): at
// 16 rows 768x768 4.8 -> 3.8, 2048x2048 6.3 -> 5.3, 1024x4096 5.8 -> 5.3; four ~131M
// layers at 8 rows 107.7 -> 101.1, at 4 rows 98.6 -> 98.0, at 3 rows 95.9 -> 97.1;
// a ~1B layer (16,384 to 180,224 groups a product) at 4 rows 34.2 -> 36.2, at 6
// rows 35.3 -> 36.7 with all of it as clusters and 38.7 with the smallest alone.
// Otherwise units of 16 columns that would leave some blocks one unit more
// than others are cut in two where both halves of all of them find a block
// (see Shares; half a unit still gives every warp a column): 4096x4096, 128
// units, 7.9 -> 6.6 us at 8 rows and 10.6 -> 8.1 at 16; 14336x4096, 448 units,
// 15.1 -> 12.6 and 20.9 -> 17.6.
template <int NB>
cudaError_t launch_gemm(const LayoutView& L, const uint16_t* X, float* Y, int B, cudaStream_t s) {
    static LaunchPrep prep, prep_cut, prep_cl;
    int sms = 0;
    cudaError_t e = prep.get(gemmb_kernel<NB, SPLIT_EVEN>, gemmb_smem<NB>(), &sms);
    if (e != cudaSuccess) return e;
    constexpr int64_t SMALL = 50000;
    const bool pays = NB == 16 ? L.S <= MAX_CLUSTER
                               : B > 4 && L.S <= 8 && L.N * L.G < SMALL && GROUP * (int64_t)L.G * L.G < SMALL;
    if (pays && L.S > 1 && L.C <= 8 && 4 * (int64_t)L.units <= (L.S <= 8 ? 7 : 5) * (int64_t)sms) {
        if ((e = prep_cl.get(gemmb_kernel<NB, SPLIT_CLUSTER>, gemmb_smem<NB>(), &sms, true)) != cudaSuccess) return e;
        return launch_gemmb<NB, SPLIT_CLUSTER>(L, X, Y, B, s, L.units, Shares{0, 0, 1, 0});
    }
    const int blocks = GB_BLOCKS * sms;
    const Shares sh = plan_shares(L.units, L.nrb, L.S, L.C == 2 * NCWB, blocks);
    if (sh.parts > 1) {
        if ((e = prep_cut.get(gemmb_kernel<NB, SPLIT_CUT>, gemmb_smem<NB>(), &sms)) != cudaSuccess) return e;
        return launch_gemmb<NB, SPLIT_CUT>(L, X, Y, B, s, grid_blocks(L.units, sh, blocks), sh);
    }
    return launch_gemmb<NB, SPLIT_EVEN>(L, X, Y, B, s, grid_blocks(L.units, sh, blocks), sh);
}

}  // namespace

cudaError_t launch_gemm_small(const LayoutView& L, const uint16_t* X, float* Y, int B, cudaStream_t s) {
    return B > 8 ? launch_gemm<16>(L, X, Y, B, s) : launch_gemm<8>(L, X, Y, B, s);
}

cudaError_t read_device_status_gemm(uint32_t* status) {
    cudaError_t e = cudaMemcpyFromSymbol(status, g_device_status, sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    const uint32_t zero = 0;
    return cudaMemcpyToSymbol(g_device_status, &zero, sizeof(uint32_t));
}

}  // namespace vbq
