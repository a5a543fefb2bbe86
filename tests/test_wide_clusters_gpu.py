"""Clusters of more than 8 blocks (one slab of a row block each), which a launch
has to opt in to: batch 1 on 9 to 14 slabs, reached by matrices too heavy in 8
bits for wider slabs (15 and 16 would need more columns than the rule on a
product's neighbours lets through), and batched products on 9 to 16 slabs, where
the 128 rows do not divide evenly among the blocks; last row blocks of a few
rows, some with blocks that own none. Against the oracle within the library's
bound; the same bits on every call."""

import numpy as np
import pytest
import torch

import layout_ref
import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix, bits_to_i16

pytestmark = pytest.mark.gpu


# all groups at 8 bits run the single-width variant, a few others the task tables
@pytest.mark.parametrize("dist", [(0.0, 0.0, 0.0, 1.0), (0.02, 0.02, 0.02, 0.94)])
@pytest.mark.parametrize("n,g,slabs", [(1150, 33, 9), (1000, 40, 10), (897, 44, 11), (1280, 48, 12), (800, 51, 13), (700, 55, 14)])
def test_batch_1(n, g, slabs, dist):
    m = Matrix(n, 64 * g, dist=dist, seed_path=(92, n, g), batch=2)
    layout = vbq.vbq_pack(*m.device_args("cuda"))
    c, s, units = layout_ref.check(layout, m.widths)
    assert s == slabs and layout_ref.runs_unit_per_block(m.widths, c, s, units)
    x = bits_to_i16(m.x_bits).cuda()
    ys = [torch.full((n,), float("nan"), device="cuda") for _ in range(4)]
    h = torch.zeros(n // 2, dtype=torch.int16, device="cuda")
    for i in range(4):                  # back to back, alternating inputs
        if i >= 2 and n % 2 == 0:
            vbq.vbq_gemv_swiglu(layout, x[i % 2], ys[i], h)
        else:
            vbq.vbq_gemv(layout, x[i % 2], ys[i])
    torch.cuda.synchronize()
    got = torch.stack(ys).cpu().numpy()
    y_ref, a_ref = oracle.gemv(m.codes.numpy(), m.widths, m.scales, m.x())
    assert oracle.within_bound(got[:2], y_ref, a_ref).all() and oracle.within_bound(got[2:], y_ref, a_ref).all()
    vbq.vbq_gemv(layout, x[0], ys[1])
    assert torch.equal(ys[0], ys[1])


@pytest.mark.parametrize("n,g,slabs", [(1100, 67, 9), (1030, 80, 10), (850, 83, 11), (897, 90, 12), (700, 99, 13), (770, 112, 14),
                                       (641, 113, 15), (1280, 128, 16)])
def test_batched(n, g, slabs):
    m = Matrix(n, 64 * g, dist=(0.25, 0.25, 0.25, 0.25), seed_path=(91, n, g), batch=16)
    layout = vbq.vbq_pack(*m.device_args("cuda"))
    c, s, units = layout_ref.check(layout, m.widths)
    assert c <= 8 and s == slabs and 4 * units <= 5 * layout_ref.sm_count()      # a cluster per row block from 9 rows on
    x = bits_to_i16(m.x_bits).cuda()
    y_ref, a_ref = oracle.gemv(m.codes.numpy(), m.widths, m.scales, m.x())
    for b in (9, 13, 16):
        ys = [torch.full((b, n), float("nan"), device="cuda") for _ in range(2)]
        for y in ys:
            vbq.vbq_gemm_small(layout, x[:b].contiguous(), y)
        assert oracle.within_bound(ys[0].cpu().numpy(), y_ref[:b], a_ref[:b]).all(), b
        assert torch.equal(ys[0], ys[1])
