"""The exact near rule at points a few roundings away from the nodes (a copy of the nodes that went through other
arithmetic): displaced by 1 to 400 units in the last place along an edge, in a face's plane and across, on fine and coarse
meshes near to and away from the origin.  There two of a pair's lengths are 1e-13 of the third and their products leave
the float32 range, which the float32 path's two-float geometry has to stand.

Float32 against the same rule evaluated without a table (bs_velocity_noalloc, geometry in float64), which leaves out what
the float32 far sums are off at coordinates of 1e4 spacings: the float32 paths' 1e-5 RMS over the largest speed.
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
from paper_0712_1695_gb300.binding import bs_velocity_noalloc  # noqa: E402

bs.build()


@pytest.mark.parametrize("spacing", [1.0, 0.03, 0.001])
@pytest.mark.parametrize("origin", [0.37, 10.0])
def test_points_beside_nodes(spacing, origin):
    m = config1_plain(6)
    x = origin + m.nodes * (5 * spacing)
    h = bs.Mesh(x, m.tets, m.omega)
    rng = np.random.default_rng(5)
    t = m.tets[rng.permutation(len(m.tets))[:120]]
    a, b, c = x[t[:, 0]], x[t[:, 1]], x[t[:, 2]]
    along, inplane = (b - a) / spacing, (0.4 * b + 0.6 * c - a) / spacing
    across = rng.standard_normal(a.shape)
    pts = [a]
    for ulps in (1, 2, 4, 16, 60, 150, 400):
        for d in (along, inplane, across):
            pts.append(a + ulps * np.spacing(a) * np.sign(d) if ulps < 16 else a + ulps * np.spacing(a.max()) * d)
    pts = np.concatenate(pts)
    p = dict(far_ratio=2.0, tet_gauss_order=4, n_theta=4, n_phi=8, near_rule=bs.BS_NEAR_EXACT)
    dev = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
    v64 = h.bs_velocity(dev, precision=bs.BS_FP64, **p).cpu().numpy()
    v32 = h.bs_velocity(dev, precision=bs.BS_FP32, **p).cpu().numpy()
    h.bs_status()
    assert np.isfinite(v64).all() and np.isfinite(v32).all()
    mesh = [torch.from_numpy(q).cuda() for q in (x, m.tets, m.omega)]
    plain = bs_velocity_noalloc(*mesh, dev, torch.empty_like(dev), precision=bs.BS_FP32, **p).cpu().numpy()
    assert rms_over_max(v32, plain) <= TOL_FP32_RMS_MAX


@pytest.mark.parametrize("distance", [1e8, 1e10, 1e13])
def test_far_outside_the_range_of_the_products(distance):
    """Every pair exact, a point so far away that four lengths multiplied leave the float32 range: as without a table
    (the closed form itself has lost everything but the range to cancellation there)."""
    m = config1_plain(4)
    h = bs.Mesh(m.nodes, m.tets, m.omega)
    p = dict(far_ratio=np.inf, tet_gauss_order=4, n_theta=4, n_phi=8, near_rule=bs.BS_NEAR_EXACT, precision=bs.BS_FP32)
    pts = torch.from_numpy(distance * np.random.default_rng(1).standard_normal((64, 3))).cuda()
    v = h.bs_velocity(pts, **p).cpu().numpy()
    h.bs_status()
    out = torch.empty_like(pts)
    dev = [torch.from_numpy(q).cuda() for q in (m.nodes, m.tets, m.omega)]
    plain = bs_velocity_noalloc(*dev, pts, out, **p).cpu().numpy()
    assert np.array_equal(np.isfinite(v), np.isfinite(plain))
