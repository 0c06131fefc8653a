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


def _cube():
    """A closed cube: its winding number is 0 outside."""
    from synth import geometry as G
    out = []
    for ax in range(3):
        a, b = np.zeros(3), np.zeros(3)
        a[(ax + 1) % 3] = b[(ax + 2) % 3] = 1
        for s in (0, 1):
            o = np.zeros(3)
            o[ax] = s
            out.append(G.planar_patch(o, a, b) if s else G.planar_patch(o, b, a))
    return out


# values outside the cube, all of them truncation and rounding, in the order of sums that queries
# of a handful of points keep: (order, points, mode) -> values
_OUTSIDE = {
    (2, 7, gwn.MODE_BVH): [-2.60828383e-05, -5.96280097e-06, 1.08491986e-05, 2.28533008e-05, 6.47999987e-05,
                           -7.4230461e-06, -1.07851747e-05],
    (3, 1, gwn.MODE_BVH): [0.000139282085],
    (3, 7, gwn.MODE_BVH): [1.36382878e-05, 9.608455e-06, 8.14069062e-06, 2.05226243e-05, -8.98176804e-05,
                           -6.27432019e-06, -1.46380626e-06],
    (2, 7, gwn.MODE_DIRECT): [2.92038749e-09, -2.00088834e-09, 2.31011654e-10, 3.81987775e-11, 3.97267286e-09,
                              3.53975338e-09, 6.34463504e-09],
}


@pytest.mark.parametrize("order,n,mode", list(_OUTSIDE))
def test_few_points_keep_their_values(order, n, mode):
    """Values next to 0, pinned to 2e-5 of their norm (the bound an FP32 output is held to)."""
    b, bl = {2: (6.0, 3.25), 3: (4.5, 3.0)}[order]
    m = gwn.gwn_build_3d(_cube(), beta=b, beta_leaf=bl, order=order)
    r = np.random.default_rng(n + order)
    d = r.normal(size=(n, 3))
    d /= np.max(np.abs(d), axis=1, keepdims=True)
    q = (0.5 + d * r.uniform(0.55, 1.0, (n, 1))).astype(np.float32)
    ref = np.array(_OUTSIDE[order, n, mode])
    w = np.stack([m.query(torch.from_numpy(q).cuda(), mode=mode)[0].cpu().numpy() for _ in range(5)])
    off = np.linalg.norm(w - ref, axis=1) / np.linalg.norm(ref)
    assert np.median(off) <= 2e-5  # pairs' sums are atomic: one run's order may differ


def _octants(shape, c, r, ccw, half=False):
    """Curves that show c at 45 degrees each: a square with halved sides, a circle of eight arcs, or
    the upper half of them."""
    from synth import geometry as G
    n = 4 if half else 8
    if shape == "circle":
        out = [G.arc(c, r, 0.25 * np.pi * k, 0.25 * np.pi * (k + 1)) for k in range(n)]
    else:
        v = np.array([[1, 0], [1, 1], [0, 1], [-1, 1], [-1, 0], [-1, -1], [0, -1], [1, -1], [1, 0]], dtype=float)
        out = [G.polyline(c + r * v[k:k + 2], closed=False) for k in range(n)]
    return out if ccw else [x.reversed() for x in out]


@pytest.mark.parametrize("ccw", [True, False])
@pytest.mark.parametrize("shape", ["square", "circle"])
def test_leaves_of_45_degrees(shape, ccw):
    """FP64 traversal, direct sum (32 copies: whole groups in each lane) and repair at the centre: whole
    and half turns to rounding (the sums' 2^-52 per leaf, 1e-12 for 256 of them)."""
    rng = np.random.default_rng(2)
    sgn = 1.0 if ccw else -1.0
    for k in range(12):
        c = np.zeros(2) if k == 0 else rng.uniform(-1, 1, 2)
        r = 1.0 if k == 0 else float(np.exp(rng.uniform(-1, 1)))
        q = torch.from_numpy(c[None]).cuda()
        for copies in (1, 32):
            curves = [x for x in _octants(shape, c, r, ccw) for _ in range(copies)]
            m = gwn.gwn_build_2d(curves, max_aabb_frac=0.0, beta=1e9)
            for mode in (gwn.MODE_BVH, gwn.MODE_DIRECT):
                w, _, _ = m.query(q, precision=gwn.PREC_FP64, mode=mode)
                assert abs(float(w[0]) - sgn * copies) <= 1e-12 * copies
        for kw in (dict(), dict(beta_repair=1e9)):  # a half turn goes to the repair
            m = gwn.gwn_build_2d(_octants(shape, c, r, ccw, half=True), max_aabb_frac=0.0, beta=1e9, **kw)
            w, _, st = m.query(q)
            assert int(st[0]) & gwn.QS_REPAIRED
            assert abs(float(w[0]) - 0.5 * sgn) <= 1e-12


def test_fp64_sums_stay_finite_far_away():
    """FP64 direct sum and traversal (every leaf exact) 1e35 to 1e70 away: outside a closed loop of 48
    leaves.  A leaf's end points round to the same vector there, and its cross product is at most the
    rounding of a fused one, 2^-53 of the dot product: 48 x 2^-53 / (2 pi) = 8.5e-16."""
    from synth import geometry as G
    curves = [G.arc((0, 0), 1.0, np.pi * k / 24, np.pi * (k + 1) / 24) for k in range(48)]
    m = gwn.gwn_build_2d(curves, max_aabb_frac=0.0, beta=1e100)
    d = np.array([[1.0, 0.3], [-0.4, 1.0], [-1.0, -1.0]])
    q = np.concatenate([10.0 ** e * d for e in (35, 38, 40, 50, 70)])
    for mode in (gwn.MODE_BVH, gwn.MODE_DIRECT):
        w, _, _ = m.query(torch.from_numpy(q).cuda(), precision=gwn.PREC_FP64, mode=mode)
        assert float(w.abs().max()) <= 1e-15


@pytest.mark.parametrize("n", [40, 2049, 20001])
def test_direct_sum_on_the_surface(oracle_lib, n):
    """Points 1e-5 off the faces have two or more near-band pairs each: the FP32 direct sum without repair
    keeps the FP32 path's bound."""
    patches = configs.cad_3d(seed=5, n_patches=60)[0]
    q = _on_faces(patches, n, 11, 1e-5)
    m = gwn.gwn_build_3d(patches, beta=6.0)
    w, _, st = m.query(torch.from_numpy(q).cuda(), mode=gwn.MODE_DIRECT, precision=gwn.PREC_FP32)
    bad = (st & (gwn.QS_UNRESOLVED | gwn.QS_STACK_OVERFLOW)) != 0
    assert int(bad.sum()) <= n // 1000  # a point may lie on a trimming curve
    idx = np.unique(np.r_[0, n - 1, np.random.default_rng(1).integers(0, n, 400)])
    w_ref, _ = oracle_lib.gwn3d(patches, q[idx].astype(np.float64))
    ok = np.isfinite(w_ref) & ~bad.cpu().numpy()[idx]
    assert ok.mean() > 0.95 and np.max(np.abs(w.cpu().numpy()[idx][ok] - w_ref[ok])) <= 1e-4


@pytest.mark.parametrize("n", [3, 40, 5000, 40000])
def test_near_band_on_the_surface(oracle_lib, n):
    """Points 1e-5 off the faces have two or more near-band pairs each: the traversal without repair and the
    no-alloc call evaluate them all (flagged where a list is full), within the FP32 path's bound."""
    patches = configs.cad_3d(seed=5, n_patches=60)[0]
    q = _on_faces(patches, n, 12, 1e-5)
    m = gwn.gwn_build_3d(patches, beta=6.0, beta_leaf=4.0)
    pts = torch.from_numpy(q).cuda()
    out = (torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"),
           torch.empty(n, dtype=torch.int32, device="cuda"))
    idx = np.unique(np.r_[0, n - 1, np.random.default_rng(1).integers(0, n, 400)])
    w_ref, _ = oracle_lib.gwn3d(patches, q[idx].astype(np.float64))
    ok = np.isfinite(w_ref)
    assert ok.mean() > 0.95
    for w, _, st in (m.query(pts, precision=gwn.PREC_FP32), gwn.api.gwn_query_noalloc(m, pts, out)):
        assert int(((st & gwn.QS_STACK_OVERFLOW) != 0).sum()) == 0
        good = ok & ((st & gwn.QS_UNRESOLVED) == 0).cpu().numpy()[idx]
        assert np.max(np.abs(w.cpu().numpy()[idx][good] - w_ref[good])) <= 1e-4


@pytest.mark.parametrize("n,side", [(5, 6), (4000, 6), (5003, 6), (290001, 20), (1 << 20, 64)])
def test_pair_count(n, side):
    """Every leaf exact for every point: the statistics count n pairs a leaf, and those of the points that
    are evaluated again, without the list's padding and beyond 2^32."""
    from synth import geometry as G
    patches = [G.planar_patch((i, j, 0), (0.9, 0, 0), (0, 0.9, 0)) for i in range(side) for j in range(side)]
    m = gwn.gwn_build_3d(patches, max_aabb_frac=0.0, beta=1e4, beta_leaf=1e4, precision=gwn.PREC_FP32)
    nl = m.info()["n_leaves"]
    g = torch.Generator(device="cuda").manual_seed(1)
    q = torch.rand(n, 3, generator=g, device="cuda") * torch.tensor([side, side, 1.0], device="cuda")
    q[:, 2] += 2.0
    m.query(q)
    s = m.last_query_stats()
    assert s["pairs"] == nl * (n + s["overflow"])
    assert n < (1 << 20) or s["pairs"] > 2 ** 32


def test_small_queries_keep_a_small_workspace():
    """A 64-point query of a model of 14,400 leaves: the FP64 repair's two pair lists (67 MB) and the
    FP32 lists (4 million pairs, 34 MB) are most of its scratch, not a list of every leaf for every point."""
    from synth import geometry as G
    patches = [G.planar_patch((i, j, 0), (0.9, 0, 0), (0, 0.9, 0)) for i in range(120) for j in range(120)]
    m = gwn.gwn_build_3d(patches, max_aabb_frac=0.0, beta=6.0, beta_leaf=4.0)
    q = torch.rand(64, 3, device="cuda")
    out = (torch.empty(64, dtype=torch.float64, device="cuda"), None, None)
    small = gwn.gwn_build_3d(patches[:40], max_aabb_frac=0.0, beta=6.0, beta_leaf=4.0)
    gwn.gwn_query(small, q, out=out)  # loads the kernels
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    gwn.gwn_query(m, q, out=out)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 128 << 20


@pytest.mark.parametrize("call", ["direct", "noalloc"])
@pytest.mark.parametrize("kind", ["cad", "round"])
def test_two_runs_give_the_same_bits(call, kind):
    """The FP32 direct sum and the no-alloc call at points next to the faces, where each point has several
    near pairs whose order in the lists differs from run to run."""
    patches = configs.cad_3d(seed=5, n_patches=60)[0] if kind == "cad" else configs.sphere_3d(cells=2, n_queries=1)[0]
    n = 20001
    pts = torch.from_numpy(np.concatenate([_on_faces(patches, n // 2, 11, 1e-5), _on_faces(patches, n - n // 2, 12, 1e-3)])).cuda()
    m = gwn.gwn_build_3d(patches, beta=6.0, beta_leaf=4.0)

    def run():
        if call == "direct":
            return m.query(pts, mode=gwn.MODE_DIRECT, precision=gwn.PREC_FP32)
        return gwn.api.gwn_query_noalloc(m, pts, (torch.empty(n, dtype=torch.float64, device="cuda"), None,
                                                  torch.empty(n, dtype=torch.int32, device="cuda")))
    w, _, st = run()
    assert int((st & gwn.QS_NEAR).ne(0).sum()) > n // 8
    for _ in range(5):
        w2, _, st2 = run()
        assert torch.equal(w, w2) and torch.equal(st, st2)


@pytest.mark.parametrize("n", [1, 16, 17, 200, 4097])
@pytest.mark.parametrize("local_ratio", [0.0, 64.0])
def test_small_queries_of_round_parts(oracle_lib, n, local_ratio):
    """Curves of high degree (circular trims) on the small-query paths, with and without packet local
    expansions (at 64 packet radii their remainder, 64^-3 of a term, is far below the bound)."""
    from synth import geometry as G
    patches = configs.sphere_3d(cells=2, n_queries=1)[0]
    lo, hi = G.shape_bbox_3d(patches)
    q = np.concatenate([_on_faces(patches, (n + 1) // 2, n, 1e-2),
                        np.random.default_rng(n).uniform(lo, hi, (n // 2, 3)).astype(np.float32)])
    m = gwn.gwn_build_3d(patches, beta=6.0, beta_leaf=4.0)
    w, lab, _ = m.query(torch.from_numpy(q).cuda(), local_ratio=local_ratio)
    idx = np.unique(np.r_[0, n - 1, np.random.default_rng(1).integers(0, n, 200)])
    w_ref, _ = oracle_lib.gwn3d(patches, q[idx].astype(np.float64))
    ok = np.isfinite(w_ref)
    assert np.max(np.abs(w.cpu().numpy()[idx][ok] - w_ref[ok])) <= 1e-4
    assert torch.equal(lab, torch.round(w).int())


def test_values_do_not_depend_on_earlier_queries():
    """A crowded query before and after a larger one on the same model: the same terms, up to FP32 sums (5e-6,
    as above); with its leaves at another factor it would differ by 2e-5."""
    patches = configs.cad_3d(seed=9, n_patches=330)[0]
    m = gwn.gwn_build_3d(patches, beta=9.0, beta_leaf=5.5, precision=gwn.PREC_FP32)
    pts = torch.from_numpy(_on_faces(patches, 9000, 5, 1e-3)).cuda()
    before = m.query(pts)[0].clone()
    m.query(torch.from_numpy(_on_faces(patches, 120000, 6, 1e-3)).cuda())
    assert float((m.query(pts)[0] - before).abs().max()) <= 5e-6


def test_concurrent_callers():
    """Two threads with a stream each, on a model they share and on one of their own, over the paths that
    keep state in the workspace: values as alone, to the rounding of FP32 sums (as above: 5e-6)."""
    import threading
    models = [gwn.gwn_build_3d(configs.cad_3d(seed=9, n_patches=k)[0], beta=9.0, beta_leaf=5.5) for k in (330, 60, 100)]
    patches = configs.cad_3d(seed=9, n_patches=330)[0]
    pts = [torch.from_numpy(_on_faces(patches, n, n, 1e-3)).cuda() for n in (9, 900, 9000, 40000)]
    ref = {(j, k): models[j].query(p)[0] for j in range(3) for k, p in enumerate(pts)}
    torch.cuda.synchronize()
    bad = []

    def work(own):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for r in range(6):
                for k, p in enumerate(pts):
                    for j in (0, own):
                        w, _, _ = models[j].query(p)
                        stream.synchronize()
                        d = float((w - ref[j, k]).abs().max())
                        if not d <= 5e-6:
                            bad.append((j, k, d))

    threads = [threading.Thread(target=work, args=(own,)) for own in (1, 2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
