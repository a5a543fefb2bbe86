"""The group-batched kernels (vbq_quantize, vbq_soft_quant take 16 groups per
warp pass, several per load) at group counts around a pass: partial loads,
partial passes, and the exact 1-bit mean at every place of a pass."""

import numpy as np
import pytest
import torch

import oracle
import paper_2607_02893_gb300 as vbq
from synth import gen

pytestmark = pytest.mark.gpu

COUNTS = [(1, 1), (1, 2), (1, 3), (3, 5), (1, 16), (1, 17), (31, 1), (11, 47)]


@pytest.mark.parametrize("n,g", COUNTS)
def test_quantize_counts(n, g):
    rng = gen.rng_for((78, n, g))
    w = gen.draw_dense_weights(n, 64 * g, rng)
    widths = rng.choice(np.array([1, 2, 4, 8], np.uint8), size=(n, g))
    # every third group at one bit with a spread over 23 binades: its mean is
    # the fp64 tree over neighbouring weights; every fifth all zero
    flat = w.reshape(-1, 64)
    fw = widths.reshape(-1)
    for i in range(0, len(flat), 3):
        flat[i] *= (2.0 ** rng.integers(-30, 31, size=64)).astype(np.float32)
        fw[i] = 1
    flat[4::5] = 0.0
    codes, scales = vbq.vbq_quantize(torch.from_numpy(w).cuda(), torch.from_numpy(widths).cuda())
    rc, rs = oracle.quantize(w.astype(np.float64), widths)
    assert np.array_equal(scales.cpu().numpy().view(np.uint16), rs.view(np.uint16))
    assert np.array_equal(codes.cpu().numpy(), rc)


@pytest.mark.parametrize("n,g", COUNTS)
@pytest.mark.parametrize("noise", [True, False])
def test_soft_counts(n, g, noise):
    w, lg, gb = gen.draw_soft_inputs(n, 64 * g, gen.rng_for((79, n, g)))
    w.reshape(-1, 64)[2::7] = 0.0                                  # zero groups
    gumbel = gb if noise else None
    guard = torch.full((n * g * 64 + 64,), 7.0, device="cuda")     # nothing is written past the last group
    out = guard[:n * g * 64].view(n, 64 * g)
    ws, eb, hw = vbq.vbq_soft_quant(torch.from_numpy(w).cuda(), torch.from_numpy(lg).cuda(), 0.7,
                                    gumbel=None if gumbel is None else torch.from_numpy(gumbel).cuda(), w_soft=out)
    assert (guard[n * g * 64:] == 7.0).all()
    _, _, hard_ref, _ = oracle.soft_quant_forward(w, lg, gumbel, 0.7)
    assert np.array_equal(hw.cpu().numpy(), hard_ref)
    ok_w, ok_b = oracle.soft_quant_within_bound(ws.cpu().numpy(), eb.cpu().numpy(), w, lg, gumbel, 0.7)
    assert ok_w.all() and ok_b.all()
