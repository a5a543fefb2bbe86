"""Packing and unpacking: codes, widths and scales come back bit for bit, and
the batch-1 product (which runs on the packed task tables) agrees with the
oracle, on shapes and mixes where a unit's tables can go wrong: widths absent
from many columns (several column ends on one item), tasks cut at every
length, one row or one column, ragged row blocks and slabs."""

import numpy as np
import pytest
import torch

import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix, bits_to_i16

pytestmark = pytest.mark.gpu

MIXES = {
    "head": (0.96, 0.025, 0.01, 0.005),          # 2, 4 and 8 bits missing from most columns
    "no1": (0.004, 0.30, 0.30, 0.396),           # 1 bit missing from most columns
    "even": (0.25, 0.25, 0.25, 0.25),
    "main": (0.69, 0.15, 0.11, 0.05),
}


@pytest.mark.parametrize("mix", list(MIXES))
@pytest.mark.parametrize("n,g", [(1, 1), (1, 40), (33, 16), (128 * 80, 16), (128 * 76 + 1, 37), (300, 7), (9728, 3)])
def test_pack_round_trip(mix, n, g):
    m = Matrix(n, 64 * g, dist=MIXES[mix], seed_path=(97, n, g), batch=1)
    codes, widths, scales = m.device_args("cuda")
    layout = vbq.vbq_pack(codes, widths, scales)
    back = {"c": torch.full_like(codes, 255), "b": torch.zeros_like(widths), "s": torch.full_like(scales, -1),
            "w": torch.full((n, 64 * g), float("nan"), device="cuda")}
    vbq.vbq_dequant(layout, back["c"], back["b"], back["s"], back["w"])
    assert torch.equal(back["c"], codes) and torch.equal(back["b"], widths) and torch.equal(back["s"], scales)
    # each output alone gives the same values
    for key, args in (("c", (0,)), ("b", (1,)), ("s", (2,)), ("w", (3,))):
        one = torch.zeros_like(back[key])
        vbq.vbq_dequant(layout, *[one if i in args else None for i in range(4)])
        assert torch.equal(one, back[key])
    wl = widths.long().repeat_interleave(64, 1)
    level = torch.where(wl == 1, 2 * codes.long() - 1, codes.long() - 2 ** (wl - 1))
    s = scales.view(torch.float16).float().repeat_interleave(64, 1)
    assert torch.equal(back["w"], s * level.float())          # an 11-bit times an 8-bit number: exact
    x = bits_to_i16(m.x_bits).cuda()
    y = torch.empty(n, device="cuda")
    vbq.vbq_gemv(layout, x[0], y)
    rows = np.unique(np.r_[0:min(n, 300), max(0, n - 200):n])
    y_ref, a_ref = oracle.gemv(m.codes.cpu().numpy()[rows], m.widths[rows], m.scales[rows], m.x())
    assert oracle.within_bound(y.cpu().numpy()[rows][None], y_ref, a_ref).all()


@pytest.mark.parametrize("b", [1, 2, 4])
def test_code_out_of_range(b):
    # found while the blobs are built: no layout comes back, and the next call is unaffected
    codes = torch.zeros((200, 192), dtype=torch.uint8, device="cuda")
    widths = torch.full((200, 3), b, dtype=torch.uint8, device="cuda")
    scales = torch.zeros((200, 3), dtype=torch.int16, device="cuda")
    codes[199, 191] = 1 << b
    with pytest.raises(vbq.VbqError) as e:
        vbq.vbq_pack(codes, widths, scales)
    assert e.value.name == "VBQ_ERR_CODE_RANGE"
    codes[199, 191] = (1 << b) - 1
    vbq.vbq_pack(codes, widths, scales)
