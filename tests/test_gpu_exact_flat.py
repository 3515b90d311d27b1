"""The exact near rule at the nodes of flat meshes (rotated, so that every product rounds; the tets' vertices permuted, so
that each of a tet's edges is the short one in turn), where x is an endpoint of edges much shorter than the longest.

Against the same rule evaluated without a table (bs_velocity_noalloc), and the oracle where its own closed form stands at
such nodes (aspects up to 10).  Float64: a pair's terms are of the size of its longest edge and cancel to that of the
flat direction, squared in the sums over edges, so about 1e-15 aspect^2 of the result is rounding; 1e-14 aspect^2 is asked
for, beside the 1e-12 of the float64 paths.  Float32 (its logarithms and arc tangents lose as much, from 6e-8 on): both
forms round the same pairs to float32, 1e-6 RMS over the largest speed.
"""
import numpy as np
import pytest
from gpu_helpers import TOL_FP64_REL_L2, rel_l2, rms_over_max

from workloads import config1_plain

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0712_1695_gb300 as bs  # noqa: E402
from paper_0712_1695_gb300.binding import bs_velocity_noalloc  # noqa: E402

bs.build()


def _mesh(n, aspect, seed):
    m = config1_plain(n)
    rng = np.random.default_rng(seed)
    x = m.nodes + rng.uniform(-0.1, 0.1, m.nodes.shape) / (n - 1)
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    x = (x * [1.0 / aspect, 1.0, 1.0]) @ q.T
    tets = np.stack([t[rng.permutation(4)] for t in m.tets]).astype(np.int32)
    return np.ascontiguousarray(x), tets, rng.standard_normal(x.shape)


@pytest.mark.parametrize("far_ratio", [2.0, np.inf])
@pytest.mark.parametrize("aspect", [1.0, 10.0, 100.0, 1000.0])
def test_nodes_of_flat_tets(orc, aspect, far_ratio):
    for seed in range(3):
        x, tets, w = _mesh(6, aspect, seed)
        h = bs.Mesh(x, tets, w)
        pts = torch.from_numpy(x).cuda()
        p = dict(far_ratio=far_ratio, tet_gauss_order=4, n_theta=4, n_phi=8, near_rule=bs.BS_NEAR_EXACT)
        v64 = h.bs_velocity(pts, precision=bs.BS_FP64, **p).cpu().numpy()
        v32 = h.bs_velocity(pts, precision=bs.BS_FP32, **p).cpu().numpy()
        h.bs_status()
        assert np.isfinite(v64).all() and np.isfinite(v32).all()
        dev = [torch.from_numpy(a).cuda() for a in (x, tets, w)]
        out = torch.empty_like(pts)
        plain = [bs_velocity_noalloc(*dev, pts, out, precision=q, **p).cpu().numpy() for q in (bs.BS_FP64, bs.BS_FP32)]
        tol = TOL_FP64_REL_L2 + 1e-14 * aspect**2
        assert rel_l2(v64, plain[0]) <= tol
        assert rms_over_max(v32, plain[1]) <= 1e-6
        if aspect <= 10:
            ref = orc.velocity(x, tets, w, x, far_ratio=far_ratio, tet_order=4, n_theta=4, n_phi=8, near_rule=1)
            assert rel_l2(v64, ref) <= tol
