"""Accuracy of queries that leave the ordinary path of the query pipeline: many exact leaves a
point, lists that run full, points on the surface, values next to zero."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2605_19200_gb300 as gwn
from synth import configs
from tests import refgeom as R


def _on_faces(patches, n, seed, off):
    """n points of the patches' surfaces, moved by `off` (relative to 1) in a random direction."""
    rng = np.random.default_rng(seed)
    k = rng.integers(len(patches), size=n)
    q = np.zeros((n, 3))
    for j in np.unique(k):
        at = np.flatnonzero(k == j)
        uv = rng.uniform(0.05, 0.95, (2, len(at)))
        q[at] = R.surface_point_derivs(patches[j], uv[0], uv[1])[0]
    d = rng.normal(size=(n, 3))
    return (q + off * d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("n", [3000, 9000, 160001])
def test_crowded_leaves_take_the_nodes_far_factor(n):
    """More exact pairs than the limit: the leaves' far test is at beta.  The same terms as with
    beta_leaf = beta, up to the order of FP32 sums: 600 terms and partial sums below 1/2 round
    to 600^(1/2) 2^-25 ~ 7e-7 on one standard deviation, 5e-6 on seven; at beta_leaf the values
    differ by 2e-5."""
    patches = configs.cad_3d(seed=9, n_patches=330)[0]
    pts = torch.from_numpy(_on_faces(patches, n, 5, 1e-3)).cuda()
    m = gwn.gwn_build_3d(patches, beta=9.0, beta_leaf=5.5, precision=gwn.PREC_FP32)
    w, _, st = m.query(pts)
    assert m.last_query_stats()["pairs"] > 1.4 * (96 * max(n, 4096) + 65536)
    assert not torch.any(st & gwn.QS_STACK_OVERFLOW)
    wb, _, _ = m.query(pts, beta_leaf=9.0)
    assert float((w - wb).abs().max()) <= 5e-6
