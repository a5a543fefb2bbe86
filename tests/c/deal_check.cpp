// Host check of the batched kernel's deal (csrc/vbq_deal.h), for layouts of
// every number of row blocks and slabs up to a few hundred units per block
// row: every unit is taken exactly once (a cut one once per part), every row
// block is zeroed by exactly one block, and no block waits for a block after
// it. Prints the first fault of each kind and exits 1.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "vbq_deal.h"

using namespace vbq;

static int faults = 0;
static void fault(const char* what, int nrb, int slabs, int blocks, int at) {
    if (faults++ < 10) std::printf("FAIL %s: %d row blocks, %d slabs, %d blocks, at %d\n", what, nrb, slabs, blocks, at);
}

int main() {
    long cut = 0, cut_with_whole = 0, even = 0;
    for (int sms : {132, 148, 152, 160}) {
        const int resident = 2 * sms;
        for (int slabs = 2; slabs <= 9; ++slabs) {
            for (int nrb = 1; nrb <= 420; ++nrb) {
                const int units = nrb * slabs;
                for (int wide = 0; wide < 2; ++wide) {
                    const Shares sh = plan_shares(units, nrb, slabs, wide != 0, resident);
                    const int blocks = grid_blocks(units, sh, resident);
                    if (blocks < 1 || blocks > resident) fault("grid", nrb, slabs, blocks, 0);
                    (sh.parts > 1 ? sh.whole ? cut_with_whole : cut : even) += 1;
                    // taken: the unit's columns as two halves (1 and 2)
                    std::vector<int> taken((size_t)units, 0), zeroer((size_t)nrb, -1), first((size_t)nrb, blocks);
                    for (int p = 0; p < blocks; ++p) {
                        const BlockShare b = block_share(units, sh, blocks, p);
                        const int n = b.whole + (b.part_at >= 0);
                        if (n < 1) fault("a block without work", nrb, slabs, blocks, p);
                        for (int j = 0; j < n; ++j) {
                            const int d = j < b.whole ? b.begin + j : b.part_at;
                            const int s = d / nrb, rb = dealt_row_block(d, s, nrb, sh.rot);
                            if (d < 0 || d >= units || rb < 0 || rb >= nrb) { fault("out of range", nrb, slabs, blocks, d); continue; }
                            taken[(size_t)(s * nrb + rb)] += j < b.whole ? 3 : 1 << b.part;
                            first[(size_t)rb] = std::min(first[(size_t)rb], p);
                            if (s == 0 && (j < b.whole || b.part == 0)) {
                                if (rb != d) fault("slab 0 is not dealt in order", nrb, slabs, blocks, d);
                                if (zeroer[(size_t)rb] >= 0) fault("zeroed twice", nrb, slabs, blocks, rb);
                                zeroer[(size_t)rb] = p;
                            }
                        }
                    }
                    for (int u = 0; u < units; ++u)
                        if (taken[(size_t)u] != 3) fault("unit not taken once", nrb, slabs, blocks, u);
                    for (int rb = 0; rb < nrb; ++rb) {
                        if (zeroer[(size_t)rb] < 0) fault("never zeroed", nrb, slabs, blocks, rb);
                        if (zeroer[(size_t)rb] > first[(size_t)rb]) fault("waits for a later block", nrb, slabs, blocks, first[(size_t)rb]);
                    }
                }
            }
        }
    }
    std::printf("%ld even, %ld cut, %ld whole and cut: %s\n", even, cut, cut_with_whole, faults ? "FAILED" : "ALL OK");
    return faults || !cut || !cut_with_whole ? 1 : 0;
}
