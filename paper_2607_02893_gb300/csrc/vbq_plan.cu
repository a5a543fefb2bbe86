// vbq_plan.cu — host-side choice of the kernel for a small batch (2..4 rows).
#include "vbq_kernels.h"

namespace vbq {

// Batches of 2..GEMV1_MAX_B rows run on the table kernel (two rows per launch,
// the two-vector variant sharing every lookup address and masked code between
// its rows, plus a one-vector launch for an odd count) or on the tensor cores,
// whichever the layout's width mix makes cheaper. Cost per million groups of
// each width (1, 2, 4, 8 bits), in microseconds, measured on a GB300 on
// 16384 x 16384 matrices of one width: one row on the table kernel, two rows
// on it, and four rows on the tensor cores. The tensor cores take items in
// tiles of 16 from each (column, width) bucket of a unit, so a bucket leaves
// about 6 item slots of its last tile idle (16384 x 16384 of the main mix: 50
// us measured at 4 rows, 55 us modelled). They are charged also where a
// single-width matrix fills its tiles, which keeps two rows of an all-2-bit one
// on the tables: the faster side on small matrices (4096 x 4096 5.9 us, 7.2 on
// the tensor cores), the slower one on large ones (14336 x 4096 12.1, 11.2).
// Narrow units are charged like wide ones, though both sides cost more on them.
// So two rows of a 1- or 2-bit heavy
// matrix stay on the tables (main mix 43 us) and three or four go to the
// tensor cores (64 and 83 us on the tables).
constexpr double COST_ONE[4] = {4.09, 5.86, 8.78, 13.1};
constexpr double COST_PAIR[4] = {8.06, 10.8, 15.9, 24.0};
constexpr double COST_MMA[4] = {9.3, 10.4, 12.7, 20.8};
constexpr double MMA_IDLE_PER_BUCKET = 6.0;

bool tables_for_batch(const LayoutView& L, int B) {
    const double buckets = (double)L.units * L.C;
    double tab = 0.0, mma = 0.0;
    for (int w = 0; w < 4; ++w) {
        if (L.items[w] == 0) continue;
        tab += (double)L.items[w] * ((B / 2) * COST_PAIR[w] + (B % 2) * COST_ONE[w]);
        mma += ((double)L.items[w] + MMA_IDLE_PER_BUCKET * buckets) * COST_MMA[w];
    }
    return tab <= mma;
}

}  // namespace vbq
