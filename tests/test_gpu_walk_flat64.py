"""The float64 walk's start tets where float32 sees them worst: meshes flattened 1e4 and 1e5 times, where a gradient formed
as the negative sum of the others cancels.

Against the same rule without the walk (every line against every tet), in float64.  The area coordinates of a tet lose its
aspect, their products its square: 1e-16 aspect^2, as in the other float64 walk tests, which hold 1e-10 at an aspect of
1e3; a half-line that starts in a wrong tet, one in 256 of a node's, moves the field by 1e-5 and more.
"""
import numpy as np
import pytest
from gpu_helpers import rel_l2

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


@pytest.mark.parametrize("axis,flat", [(2, 1e-4), (2, 1e-5), (0, 1e-5)])
@pytest.mark.parametrize("seed", [3, 4, 5])
def test_flat(monkeypatch, axis, flat, seed):
    m = config1_plain(9)
    q, _ = np.linalg.qr(np.random.default_rng(seed).standard_normal((3, 3)))
    scale = np.ones(3)
    scale[axis] = flat
    x = np.ascontiguousarray((m.nodes * scale) @ q)
    v, _ = _velocity(x, m.tets, m.omega)
    monkeypatch.setenv("BS_WALK", "0")
    ref, _ = _velocity(x, m.tets, m.omega)
    assert rel_l2(v, ref) <= 1e-16 / flat**2
