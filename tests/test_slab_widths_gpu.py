"""Batched products on slabs of 16, 8, 4 and 1 columns, one and several per row,
with ragged row blocks and last slabs, at 2 to 16 activation rows; every output
row against the oracle within the library's bound. 16-column units here are
neither cut nor clusters: stores with one slab per row, flags and additions with
several."""

import pytest
import torch

import layout_ref
import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix, bits_to_i16

pytestmark = pytest.mark.gpu

MAIN, TWO = (0.69, 0.15, 0.11, 0.05), (0.0, 1.0, 0.0, 0.0)


@pytest.mark.parametrize("n,g,c,slabs", [(12801, 16, 16, 1), (13000, 17, 16, 2), (20001, 47, 16, 3), (2100, 60, 8, 8),
                                         (1001, 31, 4, 8), (100, 140, 1, 140), (129, 1, 1, 1)])
@pytest.mark.parametrize("dist", [MAIN, TWO])
def test_slab_widths(n, g, c, slabs, dist):
    m = Matrix(n, 64 * g, dist=dist, seed_path=(93, n, g), batch=16)
    layout = vbq.vbq_pack(*m.device_args("cuda"))
    got_c, got_s, units = layout_ref.check(layout, m.widths)
    assert (got_c, got_s) == (c, slabs)
    if c == 16 and slabs > 1:
        blocks = 2 * layout_ref.sm_count()
        assert units % blocks == 0 or 2 * (units % blocks) > blocks       # not cut
    x = bits_to_i16(m.x_bits).cuda()
    y_ref, a_ref = oracle.gemv(m.codes.numpy(), m.widths, m.scales, m.x())
    for b in (2, 3, 4, 5, 8, 9, 16):
        y = torch.full((b, n), float("nan"), device="cuda")
        for _ in range(2):                       # the second call finds the first one's Y
            vbq.vbq_gemm_small(layout, x[:b].contiguous(), y)
        assert oracle.within_bound(y.cpu().numpy(), y_ref[:b], a_ref[:b]).all(), b
