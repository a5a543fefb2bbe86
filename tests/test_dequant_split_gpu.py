"""Unpacking layouts of few units, whose groups several blocks share: every way
of sharing a unit (1 to 16 columns, passes of 16 and 32 groups a warp), ragged
rows and slabs, each output alone and all together, bit-exact."""

import numpy as np
import pytest
import torch

import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,g", [(1, 1), (127, 1), (129, 2), (300, 7), (256, 32), (768, 32), (2048, 32), (1000, 37),
                                 (130, 200), (4096, 64), (9700, 17)])
@pytest.mark.parametrize("dist", [(0.69, 0.15, 0.11, 0.05), (0.0, 0.0, 0.0, 1.0)])
def test_outputs(n, g, dist):
    m = Matrix(n, 64 * g, dist=dist, seed_path=(95, n, g))
    layout = vbq.vbq_pack(*m.device_args("cuda"))
    ref = (m.codes.numpy(), m.widths, m.scales.view(np.int16), oracle.dequant(m.codes.numpy(), m.widths, m.scales))
    for want in ((1, 0, 0, 0), (0, 1, 1, 0), (0, 0, 0, 1), (1, 1, 1, 1)):
        # one row more than the layout has: nothing is written past its end
        out = [torch.full((n + 1, k), fill, dtype=t, device="cuda") if w else None
               for w, k, t, fill in zip(want, (64 * g, g, g, 64 * g), (torch.uint8, torch.uint8, torch.int16, torch.float32),
                                        (255, 77, -1, float("nan")))]
        vbq.vbq_dequant(layout, *out)
        for o, r, fill in zip(out, ref, (255, 77, -1, None)):
            if o is None:
                continue
            o = o.cpu().numpy()
            assert np.array_equal(o[:n].astype(r.dtype), r)
            assert np.isnan(o[n]).all() if fill is None else (o[n] == fill).all()
