"""Two rows on layouts packed in narrower slabs than the two-vector table kernel
takes: two or four slabs as one, a last one of fewer, ragged rows and columns,
one and several slabs left, blobs too large to go together; against the oracle
within the library's bound."""

import pytest
import torch

import layout_ref
import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix, bits_to_i16

pytestmark = pytest.mark.gpu

MAIN, ONE, TWO, MIX8 = (0.69, 0.15, 0.11, 0.05), (1.0, 0.0, 0.0, 0.0), (0.1, 0.8, 0.1, 0.0), (0.3, 0.2, 0.2, 0.3)


# rows, group columns, widths, the layout's columns per slab, the kernel's
@pytest.mark.parametrize("n,g,dist,c,wide", [
    (5632, 32, MAIN, 8, 16), (2047, 88, MAIN, 8, 16), (6001, 25, MAIN, 8, 16), (8190, 23, ONE, 8, 16), (10000, 16, MAIN, 8, 16),
    (4000, 16, MAIN, 2, 4), (2600, 30, MAIN, 4, 8), (5000, 17, ONE, 4, 16), (2500, 29, TWO, 4, 8), (3300, 87, MIX8, 8, 8),
    (1300, 127, ONE, 8, 16)])
def test_pair_view(n, g, dist, c, wide):
    m = Matrix(n, 64 * g, dist=dist, seed_path=(89, n, g), batch=3)
    layout = vbq.vbq_pack(*m.device_args("cuda"))
    got = layout_ref.check(layout, m.widths)
    assert (got[0], layout_ref.pair_view(m.widths, got[0])[0]) == (c, wide)
    x = bits_to_i16(m.x_bits).cuda()
    y_ref, a_ref = oracle.gemv(m.codes.numpy(), m.widths, m.scales, m.x())
    for b in (2, 3, 2):
        y = torch.full((b, n), float("nan"), device="cuda")
        for _ in range(2):                       # the second call finds the first one's Y
            vbq.vbq_gemm_small(layout, x[:b].contiguous(), y)
        assert oracle.within_bound(y.cpu().numpy(), y_ref[:b], a_ref[:b]).all(), b
    vbq.vbq_device_status()
