"""The float32 walk of all lines on a convex mesh on both sides of the rules between its two kernels (8 lines; 64 lines or
three quarters of nodes^(2/3), whichever is more) and between a full and a part-filled GPU: against the float64 walk, RMS error over max
speed <= 1e-5 and ray hits to 0.1%, as the other float32 walk tests.
"""
import numpy as np
import pytest
from gpu_helpers import TOL_FP32_RMS_MAX, rms_over_max

from workloads import config1_plain

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0712_1695_gb300 as bs  # noqa: E402

bs.build()


# 125 and 729 nodes: 64 lines; 4096, more than the GPU takes at once: 192
@pytest.mark.parametrize("n,dirs", [(5, [(1, 1), (1, 7), (2, 4), (8, 8), (5, 13), (32, 32)]), (9, [(8, 8), (5, 13), (16, 16)]),
                                    (16, [(1, 1), (1, 7), (8, 16), (12, 16), (1, 193), (16, 16)])])
def test_both_sides(n, dirs):
    m = config1_plain(n)
    q, _ = np.linalg.qr(np.random.default_rng(8).standard_normal((3, 3)))  # no line along a boundary face
    h = bs.Mesh(np.ascontiguousarray(m.nodes @ q), m.tets, m.omega)
    for n_theta, n_phi in dirs:
        p = dict(far_ratio=np.inf, tet_gauss_order=4, n_theta=n_theta, n_phi=n_phi)
        got = []
        for prec in (bs.BS_FP32, bs.BS_FP64):
            c = torch.zeros((len(m.nodes), 3), dtype=torch.int32, device="cuda")
            got.append((h.bs_velocity_nodes(counts_dev=c, precision=prec, **p).cpu().numpy(), c.cpu().numpy()))
        h.bs_status()
        (v, c), (v64, c64) = got
        assert rms_over_max(v, v64) <= TOL_FP32_RMS_MAX
        assert np.abs(c[:, 2] - c64[:, 2]).sum() <= 1e-3 * c64[:, 2].sum()
