"""The batched product's tiles (16 items of one column and width, a warp per
column or several warps on one where a unit has few): buckets of every length
around 16, units of 1 to 16 columns, ragged row blocks and slabs, odd row
counts (rows of Y off the 16-byte grid), one and several slabs per row, against
the oracle within the library's bound, at 2..16 activation rows."""

import numpy as np
import pytest
import torch

import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix, bits_to_i16

pytestmark = pytest.mark.gpu

MAIN, EVEN = (0.69, 0.15, 0.11, 0.05), (0.25, 0.25, 0.25, 0.25)


def _check(m, batches):
    layout = vbq.vbq_pack(*m.device_args("cuda"))
    x = bits_to_i16(m.x_bits).cuda()
    y_ref, a_ref = oracle.gemv(m.codes.cpu().numpy(), m.widths, m.scales, m.x())
    for b in batches:
        y = torch.full((b, m.n), float("nan"), device="cuda")
        for _ in range(2):                       # the second call finds the first one's Y
            vbq.vbq_gemm_small(layout, x[:b].contiguous(), y)
        assert oracle.within_bound(y.cpu().numpy(), y_ref[:b], a_ref[:b]).all(), b


@pytest.mark.parametrize("dist", [MAIN, EVEN, (1.0, 0, 0, 0), (0, 0, 0, 1.0)])
@pytest.mark.parametrize("n,g", [(1, 1), (15, 3), (16, 1), (17, 2), (127, 16), (129, 5)])
def test_few_rows(n, g, dist):
    _check(Matrix(n, 64 * g, dist=dist, seed_path=(98, n, g), batch=16), (2, 5, 8, 9, 16))


# 76 row blocks and more make units of 16, 8, 4, 2 and 1 columns; g past a
# multiple leaves a ragged last slab
@pytest.mark.parametrize("n,g", [(9728, 16), (9729, 19), (4864, 11), (2432, 15), (1217, 6), (640, 9)])
@pytest.mark.parametrize("dist", [MAIN, EVEN])
def test_unit_widths(n, g, dist):
    _check(Matrix(n, 64 * g, dist=dist, seed_path=(98, n, g), batch=16), (8, 13))


# 16-column units cut in two: all of them (few units), or those beyond one per
# block; a ragged last slab whose halves are uneven, odd rows
@pytest.mark.parametrize("n,g", [(12800, 17), (4992, 65), (20001, 47)])
def test_unit_halves(n, g):
    _check(Matrix(n, 64 * g, dist=MAIN, seed_path=(98, n, g), batch=16), (5, 16))


# clusters: every size of a block's own rows (128 rows over S slabs), and row
# blocks so short that some blocks own none; the same bits on every call
@pytest.mark.parametrize("n,g", [(130, 4), (257, 6), (384, 10), (1, 14), (5, 16), (1000, 32), (200, 24), (1024, 64)])
def test_clusters(n, g):
    m = Matrix(n, 64 * g, dist=EVEN, seed_path=(99, n, g), batch=16)
    _check(m, (6, 16))
    layout = vbq.vbq_pack(*m.device_args("cuda"))
    x = bits_to_i16(m.x_bits).cuda()
    ys = [torch.empty((16, n), device="cuda") for _ in range(3)]
    for y in ys:
        vbq.vbq_gemm_small(layout, x, y)
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2])
