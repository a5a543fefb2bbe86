"""Batched products on 16-column units cut in two: nothing but halves, whole
units followed by a half, left-over units from two slabs, a last slab of one
column (whose first half is empty), even and odd row counts; every output row
against the oracle within the library's bound."""

import pytest
import torch

import layout_ref
import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix, bits_to_i16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,g,whole,wraps", [(4700, 49, 0, True), (4699, 49, 0, True), (17900, 33, 1, False),
                                             (17901, 33, 1, False), (14001, 64, 1, True)])
def test_cut_units(n, g, whole, wraps):
    m = Matrix(n, 64 * g, seed_path=(94, n, g), batch=16)
    layout = vbq.vbq_pack(*m.device_args("cuda"))
    c, slabs, units = layout_ref.check(layout, m.widths)
    blocks = 2 * layout_ref.sm_count()
    left = units % blocks
    assert c == 16 and slabs > 1 and 0 < 2 * left <= blocks       # the units are cut
    assert units // blocks == whole and (left > -(-n // 128)) == wraps
    x = bits_to_i16(m.x_bits).cuda()
    y_ref, a_ref = oracle.gemv(m.codes.numpy(), m.widths, m.scales, m.x())
    for b in (3, 5, 8, 11, 16):
        y = torch.full((b, n), float("nan"), device="cuda")
        for _ in range(2):                       # the second call finds the first one's Y
            vbq.vbq_gemm_small(layout, x[:b].contiguous(), y)
        assert oracle.within_bound(y.cpu().numpy(), y_ref[:b], a_ref[:b]).all(), b
