"""The float64 far sweep pair by pair: one tet, nothing to average over.

Reference: the far rule in numpy's long double.  Each point's error is measured against the sum of its pairs' sizes,
|w_q| / r_q^2: a float64 evaluation rounds the tet's volume and weights (ten products and sums), the distance and the
cross product, 1.1e-16 each: 4e-15 holds it in every point of a tet near the origin, and a sum held in 48 bits does not.
The quadrature point is rounded at the size of the coordinates (four terms, which count three times in r^-3, against the
smallest distance of 2.5 edges).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0712_1695_gb300 as bs  # noqa: E402

bs.build()

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def _rule(order):
    if order == 1:
        return np.full((1, 4), LD(1) / 4), np.ones(1, LD)
    b = (5 - np.sqrt(LD(5))) / 20
    return np.full((4, 4), b) + np.eye(4, dtype=LD) * (1 - 4 * b), np.full(4, LD(1) / 4)


def _reference(x, w, pts, order):
    x, w, pts = x.astype(LD), w.astype(LD), pts.astype(LD)
    e = x[1:] - x[:1]
    vol = abs(e[0] @ np.cross(e[1], e[2])) / 6
    v, size = np.zeros_like(pts), np.zeros(len(pts), LD)
    for b, wq in zip(*_rule(order)):
        d = pts - b @ x
        s = -wq * vol / (4 * PI) * (b @ w)
        r = np.sqrt((d * d).sum(1))
        v += np.cross(d, s) / (r**3)[:, None]
        size += np.sqrt((s * s).sum()) / (r * r)
    return v, size


@pytest.mark.skipif(np.finfo(LD).eps > 1e-18, reason="long double is double here")
@pytest.mark.parametrize("order", [1, 4])
@pytest.mark.parametrize("at,scale", [(0.0, 1.0), (0.7, 0.01), (-40.0, 3.0)])
def test_single_tet(order, at, scale):
    rng = np.random.default_rng(11)
    tets = np.array([[0, 1, 2, 3]], np.int32)
    for _ in range(5):
        x = at + scale * (np.eye(4)[:, :3] + rng.uniform(-0.1, 0.1, (4, 3)))
        w = rng.standard_normal((4, 3))
        d = rng.standard_normal((2000, 3))
        d *= (scale * np.exp(rng.uniform(np.log(2.5), np.log(200.0), 2000)) / np.linalg.norm(d, axis=1))[:, None]
        pts = x.mean(0) + d
        h = bs.Mesh(x, tets, w)
        c = torch.zeros((len(pts), 3), dtype=torch.int32, device="cuda")
        v = h.bs_velocity(torch.from_numpy(pts).cuda(), counts_dev=c, precision=bs.BS_FP64, far_ratio=2.0,
                          tet_gauss_order=order, n_theta=4, n_phi=8).cpu().numpy()
        h.bs_status()
        assert np.all(c.cpu().numpy()[:, 1] == 1)
        ref, size = _reference(x, w, pts, order)
        err = np.sqrt(((v - ref) ** 2).sum(1)) / size
        assert float(err.max()) <= 4e-15 + 1.3e-15 * abs(at) / (2.5 * scale)
