// vbq_pack.cu — kernels that build the packed layout described in
// vbq_common.cuh (the export step of §6) and unpack it again.
#include "vbq_kernels.h"
#include "vbq_device.cuh"

namespace vbq {
namespace {

__device__ __forceinline__ int width_index(uint32_t b) {
    return b == 1 ? 0 : b == 2 ? 1 : b == 4 ? 2 : b == 8 ? 3 : -1;
}

// Item counts per width of one unit's columns, shared by the two pack kernels.
// Warp rw of a 128-row strip counts its 32 rows' groups of each width per
// column by ballots (cnt); after one block barrier 64 threads, one per (width,
// column), add the strip's four warps and scan over the columns. (One ballot,
// barrier and dependent width load per column took 8 of the counting
// kernel's 31 us.)
struct UnitCounts {
    uint8_t cnt[RB / 32][4][MAX_C];      // groups of warp rw's rows in column c at width w (at most 32)
    uint16_t ce[4][MAX_C];               // column ends: items of width w in columns 0 .. c
};

// Threads 0 .. 63 after the barrier that follows the counting: ce from cnt.
__device__ __forceinline__ void scan_columns(UnitCounts& U, int t, int cols) {
    const int v = t >> 4, c = t & 15;
    int n = 0;
    if (c < cols)
        for (int rw = 0; rw < RB / 32; ++rw) n += U.cnt[rw][v][c];
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
        const int below = __shfl_up_sync(0xffffffffu, n, o, 16);
        if (c >= o) n += below;
    }
    U.ce[v][c] = (uint16_t)n;
}

// width_tasks by a whole warp: when no more column ends meet on an item than
// the masks count, every task but the last spans its full TASK_SPAN items, so
// lane k builds task k by itself; otherwise (an empty column or several) lane
// 0 walks the columns. out, if not null, receives the descriptors.
__device__ __forceinline__ int warp_tasks(const uint16_t* ce, int cols, int w, const UnitHeader* h, TaskDesc* out,
                                          int lane) {
    const int span = w == 0 ? TASK_SPAN1 : TASK_SPAN, maxm = w == 0 ? 1 : 3;
    const int n = ce[cols - 1];
    const bool crowded = lane >= maxm && lane < cols && ce[lane] == ce[lane - maxm] && ce[lane] > 0 && ce[lane] < n;
    if (__any_sync(0xffffffffu, crowded)) {
        int nt = 0;
        if (lane == 0) nt = width_tasks(ce, cols, w, h, out);
        return __shfl_sync(0xffffffffu, nt, 0);
    }
    const int nt = (n + span - 1) / span;
    for (int k = lane; out && k < nt; k += 32) {
        const int i0 = span * k, end = min(i0 + span, n);
        uint32_t m1 = 0, m2 = 0;
        int c0 = 0;
        for (int c = 0; c < cols; ++c) {
            const int e = ce[c], p = e - i0;
            c0 += e <= i0;
            if (e > i0 && e < end) {
                if (w == 0) {
                    if (p & 1) m2 |= 1u << (p >> 1);
                    else m1 |= 1u << (p >> 1);
                } else {                            // a two-bit counter per item
                    m2 ^= m1 & (1u << p);
                    m1 ^= 1u << p;
                }
            }
        }
        TaskDesc d;
        d.x = (uint32_t)(h->sc16[w] * 16 + 2 * i0) | ((uint32_t)c0 << 16) | ((uint32_t)(end - i0 - 1) << 20) |
              ((uint32_t)w << 26);
        d.y = m1;
        d.z = m2;
        d.w = (uint32_t)(h->pay16[w] * 16 + (8 << w) * i0) | ((uint32_t)(h->row16[w] * 16 + i0) << 16);
        out[k] = d;
    }
    return nt;
}

// One block per unit (slab-major numbering), one thread per row: item counts
// per width and the number of warp tasks the unit's column ends give
// (width_tasks), as counts[5u .. 5u + 4]; err set for a width outside
// {1, 2, 4, 8}. Every width of a thread's row is loaded before any is used,
// and each warp counts one width's tasks. Latency-bound (one short wave of
// blocks): 14336 x 4096 32 -> 6.5 us.
__global__ void __launch_bounds__(RB) count_kernel(const uint8_t* __restrict__ widths, int64_t N, int G, int C,
                                                   int nrb, uint32_t* __restrict__ counts, uint32_t* err) {
    __shared__ UnitCounts U;
    __shared__ int n_tasks[4];
    const int u = blockIdx.x, rb = u % nrb, s = u / nrb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row = (int64_t)rb * RB + threadIdx.x;
    const bool valid = row < N;
    const int c0 = s * C, cols = min(C, G - c0);
    uint32_t b[MAX_C];
#pragma unroll
    for (int c = 0; c < MAX_C; ++c) b[c] = valid && c < cols ? widths[row * G + c0 + c] : 0u;
    bool bad = false;
#pragma unroll
    for (int c = 0; c < MAX_C; ++c) {
        if (c < cols) {                             // uniform
            bad |= valid && width_index(b[c]) < 0;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const uint32_t m = __ballot_sync(0xffffffffu, b[c] == (1u << v));
                if (lane == 0) U.cnt[warp][v][c] = (uint8_t)__popc(m);
            }
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) *err = 1u;
    __syncthreads();
    if (threadIdx.x < 64) scan_columns(U, threadIdx.x, cols);
    __syncthreads();
    const int nt = warp_tasks(U.ce[warp], cols, warp, nullptr, nullptr, lane);      // width index = warp
    if (lane == 0) {
        counts[(int64_t)u * 5 + warp] = U.ce[warp][cols - 1];
        n_tasks[warp] = nt;
    }
    __syncthreads();
    if (threadIdx.x == 0) counts[(int64_t)u * 5 + 4] = (uint32_t)(n_tasks[0] + n_tasks[1] + n_tasks[2] + n_tasks[3]);
}

// The batch-1 kernel deals a unit's task k to warp (k + rotation) mod tw of its
// team (tw = 16 or 8) and a block's warps meet at the end of its last unit, so
// the table is written in an order that balances those warps: tasks by
// decreasing cost, each to the least-loaded of 16 bins that still has a
// position (bin b holds positions b, b + 16, ...; the first nt % 16 bins one
// more than the rest, so the positions are exactly 0 .. nt - 1; bins b and
// b + 8 together are a warp's share when tw = 8). The costs are a time per group
// and width (5.33, 7.02, 9.98, 14.0 units for 1, 2, 4, 8 bits, measured on an
// earlier form of the batch-1 kernel) times a task's items: a task costs its full
// span even when shorter, since idle lanes repeat its first item. The kernel's
// costs since (4.09, 5.86, 8.78, 13.1, vbq_plan.cu) give the same times: ~9B layer
// 45.7 us with either, head 36.8, ~131M step 196.4. The order does not change any result: every group has its own slot.
// One warp: lane b < 16 is bin b, and the least-loaded bin is one warp
// reduction (a single thread scanning the bins took about 50 us a unit).
// in: the tasks of widths 8, 4, 2, 1 bits, of which width w has n[w] from off[w].
__device__ __forceinline__ void balance_tasks(const TaskDesc* in, const int* off, const int* n, int nt, TaskDesc* out,
                                              int lane) {
    constexpr int BINS = 16;
    constexpr uint32_t cost_w[4] = {341, 225, 319, 448};     // 64 x 5.33, 32 x 7.02, 32 x 9.98, 32 x 14.0
    constexpr int by_cost[4] = {3, 0, 2, 1};                  // 8, 1, 4, 2 bits
    const int room = lane < BINS ? nt / BINS + (lane < nt % BINS ? 1 : 0) : 0;
    uint32_t load = 0;
    int cnt = 0;
#pragma unroll
    for (int oi = 0; oi < 4; ++oi) {
        const int w = by_cost[oi];
        for (int k = 0; k < n[w]; ++k) {
            const uint32_t key = cnt < room ? (load << 5) | (uint32_t)lane : 0xffffffffu;
            if ((__reduce_min_sync(0xffffffffu, key) & 31u) == (uint32_t)lane && cnt < room) {
                out[lane + BINS * cnt] = in[off[w] + k];
                load += cost_w[w];
                ++cnt;
            }
        }
    }
}

// Four code bytes' lowest bits as a nibble (bit i from byte i): the products'
// bits all fall on distinct positions, so nothing carries.
__device__ __forceinline__ uint32_t gather_bits(uint32_t w) { return (((w & 0x01010101u) * 0x00204081u) >> 21) & 0xFu; }
__device__ __forceinline__ uint32_t gather_bits16(uint4 v) {
    return gather_bits(v.x) | (gather_bits(v.y) << 4) | (gather_bits(v.z) << 8) | (gather_bits(v.w) << 12);
}

// Codes 16q .. 16q + 15 of a group (v, a byte each) into their part of its item.
__device__ __forceinline__ void pack_quarter(uint8_t* item, int w, int q, uint4 v) {
    if (w == 0) {
        reinterpret_cast<uint16_t*>(item)[q] = (uint16_t)gather_bits16(v);
    } else if (w == 1) {
        reinterpret_cast<uint16_t*>(item)[q] = (uint16_t)gather_bits16(v);
        const uint4 hi = make_uint4(v.x >> 1, v.y >> 1, v.z >> 1, v.w >> 1);
        reinterpret_cast<uint16_t*>(item + 8)[q] = (uint16_t)gather_bits16(hi);
    } else if (w == 2) {
        // each pair of code bytes into one byte, then four such bytes together
        reinterpret_cast<uint2*>(item)[q] = make_uint2(__byte_perm(v.x | (v.x >> 4), v.y | (v.y >> 4), 0x6420),
                                                       __byte_perm(v.z | (v.z >> 4), v.w | (v.w >> 4), 0x6420));
    } else {
        reinterpret_cast<uint4*>(item)[q] = v;
    }
}

// One block per unit; its blob is built in shared memory and copied out whole.
// First the item of every (row, column): a group's rank among its column's
// groups of the same width (rows in increasing order). Then four threads per
// group, 16 codes each, in row order, so that both the codes' loads and the
// blob's stores are coalesced (one thread per group read 64 bytes on its own
// and stored items straight to memory). The column ends' tasks are built by a
// warp per width and put into the balanced order by one warp meanwhile.
// err is set for a code >= 2^b, checked here, where the codes pass through
// anyway, instead of in a pass of its own.
// Bound: HBM (the codes in, the blobs out); 14336 x 4096 main 138 + 14 us
// (with the separate check) -> 40 us.
constexpr int SC_THREADS = 4 * RB;

struct __align__(16) ScatterShared {
    uint8_t blob[MAX_BLOB_BYTES];
    TaskDesc tasks[MAX_UNIT_TASKS];
    uint16_t item_of[MAX_C * RB];           // width index << 12 | item
    UnitCounts U;
    int n_tasks[4];
};

__global__ void __launch_bounds__(SC_THREADS) scatter_kernel(const uint8_t* __restrict__ codes,
                                                             const uint8_t* __restrict__ widths,
                                                             const uint16_t* __restrict__ scales,
                                                             const uint32_t* __restrict__ counts,
                                                             LayoutView L, uint8_t* __restrict__ blobs, uint32_t* err) {
    extern __shared__ __align__(16) unsigned char smem[];
    ScatterShared& T = *reinterpret_cast<ScatterShared*>(smem);
    UnitHeader& h = *reinterpret_cast<UnitHeader*>(T.blob);
    const int u = blockIdx.x, rb = unit_rb(L, u), s = unit_slab(L, u);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rows = unit_rows(L, rb), cols = unit_cols(L, s);
    const int64_t g00 = (int64_t)rb * RB * L.G + (int64_t)s * L.C;      // the unit's first group
    constexpr int PER = MAX_C / 4;
    {
        // thread: row r, columns quarter, quarter + 4, ...
        const int r = tid & (RB - 1), quarter = tid >> 7, rw = warp & 3;
        const bool valid = r < rows;
        const int64_t g0 = g00 + (int64_t)r * L.G;
        uint32_t b[PER], rank[PER];
        uint16_t sc[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int c = quarter + 4 * i;
            b[i] = 0;
            sc[i] = 0;
            if (valid && c < cols) {
                b[i] = widths[g0 + c];
                sc[i] = scales[g0 + c];
            }
        }
        if (tid == 0) {
            const uint32_t* n = counts + (int64_t)u * 5;
            h = make_header(n, L.C, (int)n[4]);
        }
        const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int c = quarter + 4 * i;
            rank[i] = 0;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const uint32_t m = __ballot_sync(0xffffffffu, b[i] == (1u << v));
                if (lane == 0 && c < cols) T.U.cnt[rw][v][c] = (uint8_t)__popc(m);
                if (b[i] == (1u << v)) rank[i] = __popc(m & lt);
            }
        }
        __syncthreads();
        if (tid < 64) scan_columns(T.U, tid, cols);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int c = quarter + 4 * i;
            if (!valid || c >= cols) continue;
            const int w = width_index(b[i]) & 3;
            uint32_t item = (c ? T.U.ce[w][c - 1] : 0) + rank[i];
            for (int pw = 0; pw < rw; ++pw) item += T.U.cnt[pw][w][c];
            T.item_of[c * RB + r] = (uint16_t)((w << 12) | item);
            reinterpret_cast<uint16_t*>(T.blob + h.sc16[w] * 16)[item] = sc[i];
            (T.blob + h.row16[w] * 16)[item] = (uint8_t)r;
        }
        if (tid < 64 && (tid & 15) < cols)
            reinterpret_cast<uint16_t*>(T.blob + h.cc16 * 16)[(tid >> 4) * L.C + (tid & 15)] = T.U.ce[tid >> 4][tid & 15];
        // tasks in the order 8, 4, 2, 1 bits: warp w counts width w's, then
        // (behind the barrier, when the offsets are known) builds them
        if (warp < 4) {
            const int nt = warp_tasks(T.U.ce[warp], cols, warp, nullptr, nullptr, lane);
            if (lane == 0) T.n_tasks[warp] = nt;
        }
    }
    __syncthreads();
    int n[4], off[4], nt = 0;
#pragma unroll
    for (int w = 3; w >= 0; --w) {
        n[w] = T.n_tasks[w];
        off[w] = nt;
        nt += n[w];
    }
    if (warp < 4 && nt <= MAX_UNIT_TASKS) {
        warp_tasks(T.U.ce[warp], cols, warp, &h, T.tasks + (warp == 0 ? off[0] : warp == 1 ? off[1] : warp == 2 ? off[2] : off[3]),
                   lane);
        asm volatile("bar.sync 1, 128;" ::: "memory");          // the four task warps
        if (warp == 0) balance_tasks(T.tasks, off, n, nt, reinterpret_cast<TaskDesc*>(T.blob + h.task16 * 16), lane);
    }
    uint32_t over = 0;
    const int total = 4 * rows * cols;
    constexpr int AHEAD = 4;
    for (int base = tid; base < total; base += AHEAD * SC_THREADS) {
        uint4 v[AHEAD];
        uint32_t it[AHEAD];
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
            const int p = base + i * SC_THREADS;
            it[i] = 0xFFFFu;
            if (p < total) {
                const int gi = p >> 2, r = gi / cols, c = gi - r * cols;
                it[i] = T.item_of[c * RB + r];
                v[i] = reinterpret_cast<const uint4*>(codes + (g00 + (int64_t)r * L.G + c) * GROUP)[p & 3];
            }
        }
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
            if (it[i] == 0xFFFFu) continue;
            const int w = (int)(it[i] >> 12);
            pack_quarter(T.blob + h.pay16[w] * 16 + (it[i] & 0xFFFu) * (8u << w), w, tid & 3, v[i]);
            over |= (v[i].x | v[i].y | v[i].z | v[i].w) & (0x01010101u * (0xFFu & ~((1u << (1 << w)) - 1u)));
        }
    }
    if (__any_sync(0xffffffffu, over != 0) && lane == 0) *err = 1u;
    __syncthreads();
    uint4* dst = reinterpret_cast<uint4*>(blobs) + L.blob_off[u];
    for (int i = tid; i < h.size16; i += SC_THREADS) dst[i] = reinterpret_cast<const uint4*>(T.blob)[i];
}

// Four code bytes from the four bits of a nibble (bit i into byte i).
__device__ __forceinline__ uint32_t spread_bits(uint32_t nib) { return (nib * 0x00204081u) & 0x01010101u; }

// Codes 4l .. 4l + 3 of the item of width index w at src (16-byte aligned
// shared memory, 8-byte for one bit), as four bytes.
__device__ __forceinline__ uint32_t item_codes4(const uint8_t* src, int w, int l) {
    if (w == 3) return reinterpret_cast<const uint32_t*>(src)[l];
    if (w == 2) {
        const uint32_t v = reinterpret_cast<const uint16_t*>(src)[l];
        return (v & 0xFu) | ((v & 0xF0u) << 4) | ((v & 0xF00u) << 8) | ((v & 0xF000u) << 12);
    }
    const uint32_t* p = reinterpret_cast<const uint32_t*>(src);
    const int sh = 4 * (l & 7);
    const uint32_t lo = spread_bits((p[l >> 3] >> sh) & 0xFu);
    return w == 0 ? lo : lo | (spread_bits((p[2 + (l >> 3)] >> sh) & 0xFu) << 1);
}

// gridDim.y blocks per unit: the blob into shared memory, the item of every
// (row, column) by one pass over the row bytes, then the groups in row order
// (each block its share, `per` at a time per warp), two at once per warp (16
// lanes, four codes each), so that a warp writes whole 256-byte groups of floats.
// Bound: HBM, by the outputs. (One thread per item wrote 256 bytes on its own:
// 322 us for all outputs of 14336 x 4096, now 54 us.) Small layouts are bound by
// the latency of a warp's groups one after another: see launch_dequant.
constexpr int DQ_THREADS = 256;

__global__ void __launch_bounds__(DQ_THREADS) dequant_kernel(LayoutView L, uint8_t* codes_out,
                                                             uint8_t* widths_out, uint16_t* scales_out,
                                                             float* w_out, int per) {
    __shared__ __align__(16) uint8_t blob[MAX_BLOB_BYTES];
    __shared__ uint16_t item_of[MAX_C * RB];            // width index << 12 | item
    const int u = blockIdx.x, rb = unit_rb(L, u), s = unit_slab(L, u);
    const int rows = unit_rows(L, rb), cols = unit_cols(L, s);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {
        const uint32_t o0 = L.blob_off[u], n16 = L.blob_off[u + 1] - o0;
        const uint4* src = reinterpret_cast<const uint4*>(L.blobs) + o0;
        for (uint32_t i = tid; i < n16; i += DQ_THREADS) reinterpret_cast<uint4*>(blob)[i] = src[i];
    }
    __syncthreads();
    const UnitHeader& h = *reinterpret_cast<const UnitHeader*>(blob);
    const uint16_t* cend = reinterpret_cast<const uint16_t*>(blob + h.cc16 * 16);
    for (int seg = warp; seg < 4 * cols; seg += DQ_THREADS / 32) {
        const int w = seg / cols, c = seg - w * cols;
        const int i0 = c ? cend[w * L.C + c - 1] : 0, i1 = cend[w * L.C + c];
        const uint8_t* row_of = blob + h.row16[w] * 16;
        for (int i = i0 + lane; i < i1; i += 32) item_of[c * RB + row_of[i]] = (uint16_t)((w << 12) | i);
    }
    __syncthreads();
    const int total = rows * cols;
    const int64_t g00 = (int64_t)rb * RB * L.G + (int64_t)s * L.C;
    const int pass = per * (DQ_THREADS / 32);           // groups per block and pass
    for (int base = per * warp + pass * blockIdx.y; base < total; base += pass * gridDim.y) {
        // lane's group, in row order
        const int p = base + lane, pv = min(p, total - 1);
        const int r = pv / cols, c = pv - r * cols;
        const uint32_t m = item_of[c * RB + r], w = m >> 12, it = m & 0xFFFu;
        const uint16_t sbits = reinterpret_cast<const uint16_t*>(blob + h.sc16[w] * 16)[it];
        const uint32_t pay = h.pay16[w] * 16u + it * (8u << w);
        const int64_t g = g00 + (int64_t)r * L.G + c;
        if (lane < per && p < total) {
            if (widths_out) widths_out[g] = (uint8_t)(1u << w);
            if (scales_out) scales_out[g] = sbits;
        }
        if (!codes_out && !w_out) continue;
        const float sf = __half2float(__ushort_as_half(sbits));
        const int nb = min(per, total - base);
        const int l = lane & 15;
#pragma unroll 4
        for (int k = 0; k < nb; k += 2) {
            const int src = k + (lane >> 4);
            const uint32_t pk = __shfl_sync(0xffffffffu, pay | (w << 16), src);
            const float sk = __shfl_sync(0xffffffffu, sf, src);
            const int64_t gk = __shfl_sync(0xffffffffu, g, src);
            if (src >= nb) continue;
            const int wk = (int)(pk >> 16);
            const uint32_t u4 = item_codes4(blob + (pk & 0xFFFFu), wk, l);
            if (codes_out) reinterpret_cast<uint32_t*>(codes_out + gk * GROUP)[l] = u4;
            if (w_out) {
                // L_b(u): 2u - 1 for one bit, u - 2^(b-1) otherwise (small integers: exact)
                const float mul = wk == 0 ? 2.f : 1.f, sub = wk == 0 ? 1.f : (float)(1 << ((1 << wk) - 1));
                float4 f;
                f.x = sk * (mul * (float)(u4 & 0xFFu) - sub);
                f.y = sk * (mul * (float)((u4 >> 8) & 0xFFu) - sub);
                f.z = sk * (mul * (float)((u4 >> 16) & 0xFFu) - sub);
                f.w = sk * (mul * (float)(u4 >> 24) - sub);
                reinterpret_cast<float4*>(w_out + gk * GROUP)[l] = f;
            }
        }
    }
}

}  // namespace

cudaError_t launch_count(const uint8_t* widths, int64_t N, int G, int C, int nrb, int units,
                         uint32_t* counts, uint32_t* err, cudaStream_t s) {
    count_kernel<<<units, RB, 0, s>>>(widths, N, G, C, nrb, counts, err);
    return cudaGetLastError();
}

cudaError_t launch_scatter(const uint8_t* codes, const uint8_t* widths, const uint16_t* scales,
                           const uint32_t* counts, const LayoutView& L, uint8_t* blobs, uint32_t* err,
                           cudaStream_t s) {
    static LaunchPrep prep;
    int sms = 0;
    const cudaError_t e = prep.get(scatter_kernel, sizeof(ScatterShared), &sms);
    if (e != cudaSuccess) return e;
    scatter_kernel<<<L.units, SC_THREADS, sizeof(ScatterShared), s>>>(codes, widths, scales, counts, L, blobs, err);
    return cudaGetLastError();
}

cudaError_t launch_dequant(const LayoutView& L, uint8_t* codes_out, uint8_t* widths_out,
                           uint16_t* scales_out, float* w_out, cudaStream_t s) {
    int sms = 0;
    const int err = device_sms(&sms);
    if (err != 0) return (cudaError_t)err;
    // Codes and weights of a layout with few units are bound by latency: a warp's
    // 32 groups take about 2.5 us, two at a time, and a unit's several passes
    // follow one another. So while blocks are fewer than two per SM a unit's
    // passes go to several blocks, of 16 groups a warp where those all fit (us
    // for the codes: 256 x 2048 7.7 -> 4.0, 768 x 768 4.8 -> 3.6; 2048 x 2048, of
    // 32 groups, 7.8 -> 5.7; 4096 x 4096 24.6 -> 15.4).
    int per = 32, parts = 1;
    if (codes_out || w_out) {
        const int64_t fit = 2 * (int64_t)sms;
        if (L.units * (int64_t)(RB * L.C / 128) <= fit) per = 16;
        while (L.units * (int64_t)parts < fit && per * (DQ_THREADS / 32) * parts < RB * L.C) parts *= 2;
    }
    dequant_kernel<<<dim3(L.units, parts), DQ_THREADS, 0, s>>>(L, codes_out, widths_out, scales_out, w_out, per);
    return cudaGetLastError();
}

}  // namespace vbq
