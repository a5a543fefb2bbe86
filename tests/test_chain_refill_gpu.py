"""Chains whose products give a block one, two or three units: the copies of
later units are started after a product's completion count where something waits
for it, and at once where nothing does. Every waits form, several runs, a graph,
and products on the layouts in between; against the oracle within the library's
bound."""

import pytest
import torch

import layout_ref
import oracle
import paper_2607_02893_gb300 as vbq
from vbq_cases import Matrix, bits_to_i16

pytestmark = pytest.mark.gpu

# units per block on 148 to 152 SMs: 1-2 (192 units), 1 (few), 2-3 (440), 1-2 (187)
SHAPES = [(8190, 24, 1), (300, 7, 0), (14001, 64, 2), (2050, 88, 1)]


@pytest.fixture(scope="module")
def products():
    out = []
    for n, g, most in SHAPES:
        m = Matrix(n, 64 * g, seed_path=(90, n, g))
        layout = vbq.vbq_pack(*m.device_args("cuda"))
        assert layout_ref.check(layout, m.widths)[2] // layout_ref.sm_count() == most
        y_ref, a_ref = oracle.gemv(m.codes.numpy(), m.widths, m.scales, m.x())
        out.append((m, layout, bits_to_i16(m.x_bits[0]).cuda(), y_ref[0], a_ref[0]))
    return out


@pytest.mark.parametrize("waits", [None, [0, 0, 0, 0], [1, 2, 1, 2], [0, 1, 0, 1], [1, 0, 2, 0], [0, 0, 1, 2]])
@pytest.mark.parametrize("order", [(0, 1, 2, 3), (2, 0, 3, 1), (3, 2, 1, 0)])
def test_chain(products, waits, order):
    ps = [products[i] for i in order]
    ys = [torch.full((m.n,), float("nan"), device="cuda") for m, *_ in ps]
    chain = vbq.vbq_chain_create([p[1] for p in ps], [p[2] for p in ps], ys, waits)

    def check():
        torch.cuda.synchronize()
        vbq.vbq_device_status()
        for (m, _, _, y_ref, a_ref), y in zip(ps, ys):
            assert oracle.within_bound(y.cpu().numpy()[None], y_ref[None], a_ref[None]).all()
            y.fill_(float("nan"))

    for _ in range(3):
        chain.run()
    check()
    vbq.vbq_gemv(ps[0][1], ps[0][2], ys[0])
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        for _ in range(2):
            chain.run()
    for _ in range(5):
        graph.replay()
    check()
