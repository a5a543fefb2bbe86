// vbq_deal.h — how the batched kernel deals a layout's units to its blocks, and
// which block zeroes each row block's rows of Y under split-K. Plain functions
// of a few integers, so that the host can check them for every layout shape.
#pragma once

#if defined(__CUDACC__)
#define VBQ_HD __host__ __device__
#else
#define VBQ_HD
#endif

namespace vbq {

// How the units are shared out beyond an even contiguous split: every block
// takes `whole` units, and the units from `rest` on, too few for another one
// per block, are cut into `parts` runs of columns, a block each (split-K adds
// them up). Otherwise some blocks run one unit more than their neighbours, half
// an SM's warps alone: 448 units on 304 blocks as one each and 288 halves take
// 12.6 us instead of 15.1 (14336 x 4096, 8 rows). parts 1: the even split.
//
// Units are dealt slab by slab. Under split-K the block that takes a row
// block's slab-0 unit (the first part of it, when cut) zeroes its rows of Y, and
// the others wait for that. A block may only wait for blocks before it: then a
// launch of which only the first blocks have found room (beside another
// stream's kernels) still runs to its end. An even split has that order by
// itself. The parts of the left-over units go to the blocks from 0 on, though,
// so the slabs after the first are dealt `rot` row blocks later: left-over unit
// i is then of row block i mod nrb, zeroed by block (i mod nrb) / whole, which
// is not after its own blocks i * parts and following.
struct Shares {
    int whole, rest, parts, rot;
};

// A block's places in the deal: begin, begin + 1, ... (whole of them), and
// perhaps part `part` of one more (part_at, else -1).
struct BlockShare {
    int begin, whole, part_at, part;
};

VBQ_HD inline BlockShare block_share(int units, const Shares& sh, int blocks, int p) {
    BlockShare b;
    b.part_at = -1;
    b.part = 0;
    if (sh.parts > 1) {
        b.begin = p * sh.whole;
        b.whole = sh.whole;
        const int i = p / sh.parts;
        if (sh.rest + i < units) {
            b.part_at = sh.rest + i;
            b.part = p - i * sh.parts;
        }
    } else {
        const int per = units / blocks, extra = units - per * blocks;
        b.begin = p * per + (p < extra ? p : extra);
        b.whole = per + (p < extra ? 1 : 0);
    }
    return b;
}

// The row block at place d of the deal, which lies in slab d / nrb.
VBQ_HD inline int dealt_row_block(int d, int slab, int nrb, int rot) {
    const int q = d - slab * nrb - (slab > 0 ? rot : 0);
    return q < 0 ? q + nrb : q;
}

// Cut where both halves of every left-over unit find a block (a half of a
// 16-column unit still gives each of the 8 warps a column).
inline Shares plan_shares(int units, int nrb, int slabs, bool wide, int blocks) {
    const int whole = units / blocks, left = units - whole * blocks;
    if (slabs > 1 && wide && left > 0 && 2 * left <= blocks) return Shares{whole, whole * blocks, 2, whole * blocks % nrb};
    return Shares{0, 0, 1, 0};
}
inline int grid_blocks(int units, const Shares& sh, int blocks) {
    if (sh.parts > 1) return sh.whole ? blocks : sh.parts * (units - sh.rest);
    return units < blocks ? units : blocks;
}

}  // namespace vbq
