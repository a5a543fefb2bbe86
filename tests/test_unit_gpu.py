"""Batch-1 products of small layouts, one unit per block and a row block's slabs
one cluster: cluster sizes from 1 to the largest, ragged rows and slabs, and
layouts just outside the rule (17 slabs, more units than fit at once), against
the oracle within the library's bound; the same bits on every call."""

import numpy as np
import pytest
import torch

import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix, bits_to_i16

pytestmark = pytest.mark.gpu


# (rows, group columns): at most 16 columns and few row blocks pack one column
# per slab, so the group columns are the cluster size
@pytest.mark.parametrize("n,g", [(1, 1), (127, 1), (129, 2), (300, 5), (640, 8), (513, 11), (258, 16), (130, 17),
                                 (2047, 32), (4608, 32), (5000, 33), (1024, 64)])
@pytest.mark.parametrize("dist", [(0.69, 0.15, 0.11, 0.05), (0.0, 1.0, 0.0, 0.0)])
def test_unit_per_block(n, g, dist):
    m = Matrix(n, 64 * g, dist=dist, seed_path=(96, n, g), batch=2)
    layout = vbq.vbq_pack(*m.device_args("cuda"))
    x = bits_to_i16(m.x_bits).cuda()     # K % 64 == 0: every row is 16-byte aligned
    ys = [torch.full((n,), float("nan"), device="cuda") for _ in range(4)]
    for i in range(4):                  # back to back, alternating inputs
        vbq.vbq_gemv(layout, x[i % 2], ys[i])
    torch.cuda.synchronize()
    got = torch.stack(ys).cpu().numpy()
    y_ref, a_ref = oracle.gemv(m.codes.cpu().numpy(), m.widths, m.scales, m.x())
    assert oracle.within_bound(got[:2], y_ref, a_ref).all()
    assert oracle.within_bound(got[2:], y_ref, a_ref).all()
    if g <= 16 and n <= 640:            # one cluster per row block: no atomics, one order of additions
        assert np.array_equal(got[0], got[2]) and np.array_equal(got[1], got[3])
