"""The float64 walk far from the origin, where a node's coordinate is more than the two float32 words that the float32 test
of a tet's faces takes of it.

The nodes are multiples of 2^-12, so that the shift is exact and the walk, which takes differences of coordinates alone,
has to give the same numbers as at the origin, to 1e-12, and the same counts.
"""
import numpy as np
import pytest
from gpu_helpers import TOL_FP64_REL_L2, rel_l2

from workloads import config1_plain

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0712_1695_gb300 as bs  # noqa: E402

bs.build()

ALLRAY = dict(far_ratio=np.inf, tet_gauss_order=4, n_theta=8, n_phi=16, precision=bs.BS_FP64)


def _velocity(nodes, tets, omega):
    h = bs.Mesh(nodes, tets, omega)
    c = torch.full((len(nodes), 3), -1, dtype=torch.int32, device="cuda")
    v = h.bs_velocity_nodes(counts_dev=c, **ALLRAY).cpu().numpy()
    h.bs_status()
    return v, c.cpu().numpy()


@pytest.mark.parametrize("shift", [1395864371.0, 89335319757.0, 1429365116108.0])
def test_far_from_the_origin(shift):
    m = config1_plain(7)
    x = np.round(m.nodes * 6 * 2.0**12) / 2.0**12
    v, c = _velocity(x, m.tets, m.omega)
    moved = x + np.array([shift, -shift, shift])
    assert np.array_equal(moved - np.array([shift, -shift, shift]), x)
    w, d = _velocity(moved, m.tets, m.omega)
    assert rel_l2(w, v) <= TOL_FP64_REL_L2
    assert np.array_equal(c, d)
