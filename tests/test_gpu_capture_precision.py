"""A handle used in one precision and then captured in the other: its tables for the second are built inside the capture,
in buffers that outlive the graph, and calls outside do not rely on the graph having run.

Every result has to be the bits of the plain call in that precision.
"""
import numpy as np
import pytest

from workloads import config1_plain

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0712_1695_gb300 as bs  # noqa: E402

bs.build()


@pytest.mark.parametrize("first,second", [(bs.BS_FP32, bs.BS_FP64), (bs.BS_FP64, bs.BS_FP32)])
@pytest.mark.parametrize("nodes", [True, False])
@pytest.mark.parametrize("near_rule", [bs.BS_NEAR_RAY, bs.BS_NEAR_EXACT])
def test_captured_in_the_other_precision(first, second, nodes, near_rule):
    m = config1_plain(9)
    p = dict(far_ratio=2.0, tet_gauss_order=4, n_theta=4, n_phi=8, near_rule=near_rule)
    pts = torch.from_numpy(m.nodes).cuda()
    out = torch.empty_like(pts)

    def call(h, prec):
        return (h.bs_velocity_nodes(out_dev=out, precision=prec, **p) if nodes
                else h.bs_velocity(pts, out_dev=out, precision=prec, **p))

    plain = bs.Mesh(m.nodes, m.tets, m.omega)
    want = call(plain, second).cpu().numpy()
    h = bs.Mesh(m.nodes, m.tets, m.omega)
    many = pts.repeat(8, 1)  # buffers that grow with the points: large enough for either precision
    h.bs_velocity(many, precision=first, **p)
    call(h, first)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call(h, second)
    tol = 1e-6 if near_rule == bs.BS_NEAR_EXACT and second == bs.BS_FP32 else 1e-13  # no table in the capture
    close = lambda v: np.linalg.norm(v - want) <= (tol if near_rule == bs.BS_NEAR_EXACT else 0.0) * np.linalg.norm(want)
    assert np.array_equal(call(h, second).cpu().numpy(), want)  # before the graph has run
    for _ in range(3):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert close(out.cpu().numpy())
    del g
    assert np.array_equal(call(h, second).cpu().numpy(), want)
    larger = dict(p, tet_gauss_order=64, precision=second)  # buffers that the capture allocated give way to larger ones
    assert np.array_equal(h.bs_velocity(pts, out_dev=out, **larger).cpu().numpy(),
                          plain.bs_velocity(pts, **larger).cpu().numpy())
    h.bs_status()
