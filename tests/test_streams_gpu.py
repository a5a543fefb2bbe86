"""Batched products on two streams at once (their blocks share the SMs, so a
launch may be resident in part for a while): split-K and cut units on both,
results within the library's bound, and no bounded wait that gave up."""

import numpy as np
import pytest
import torch

import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix, bits_to_i16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", [5, 16])
def test_two_streams(b):
    mats = [Matrix(n, 64 * g, seed_path=(97, n, g), batch=16) for n, g in ((4096, 64), (17900, 33))]
    layouts = [vbq.vbq_pack(*m.device_args("cuda")) for m in mats]
    xs = [bits_to_i16(m.x_bits).cuda()[:b].contiguous() for m in mats]
    ys = [torch.full((b, m.n), float("nan"), device="cuda") for m in mats]
    streams = [torch.cuda.Stream(priority=p) for p in (0, -1)]
    torch.cuda.synchronize()
    vbq.vbq_device_status()
    for _ in range(200):
        for layout, x, y, s in zip(layouts, xs, ys, streams):
            vbq.vbq_gemm_small(layout, x, y, stream=s)
    torch.cuda.synchronize()
    vbq.vbq_device_status()
    for m, y in zip(mats, ys):
        y_ref, a_ref = oracle.gemv(m.codes.numpy(), m.widths, m.scales, m.x()[:b])
        assert oracle.within_bound(y.cpu().numpy(), y_ref, a_ref).all()
