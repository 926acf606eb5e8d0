"""Surfel attributes on the GPU (pe_point_attributes) against the brute-force
oracle: radii bit-exact (same neighbour lists: FP32 squared distances in one
order, ties by index; FP64 sums in list order), PCA normals within 1e-6 rad
wherever the normal is well defined (the two smallest covariance eigenvalues
apart by at least 10 % of the middle one), orientation exact where the
reference is not near perpendicular.  At the composite workload's full size
(1M points) a sample of points is checked one by one."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import scenes  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _gpu(pos, k_r, k_n, ref=None):
    from paper_2408_15583_gb300 import api
    p = torch.from_numpy(np.ascontiguousarray(pos, np.float32)).to(DEV)
    rf = None if ref is None else torch.from_numpy(np.ascontiguousarray(ref, np.float32)).to(DEV)
    r, n = api.point_attributes(p, k_r, k_n, rf)
    api.stream_check()
    return r.cpu().numpy(), n.cpu().numpy()


def _clouds():
    rng = np.random.default_rng(7)
    line = np.zeros((400, 3), np.float32)
    line[:, 0] = np.sort(rng.random(400)).astype(np.float32)          # collinear
    dup = np.concatenate([rng.random((300, 3)), rng.random((300, 3))[:100]])
    dup = np.concatenate([dup, dup[:60]]).astype(np.float32)           # exact duplicates
    return {
        "sphere": (scenes.sphere(6000, 1.0).pos, scenes.sphere(6000, 1.0).nrm),
        "octar": (scenes.octar(6000, 2.0, seed=3).pos, scenes.octar(6000, 2.0, seed=3).nrm),
        "noisy_composite": (scenes.composite(8000, seed=3, pca=False).pos,
                            scenes.composite(8000, seed=3, pca=False).nrm),
        "uniform": (rng.random((3000, 3)).astype(np.float32), None),
        "line": (line, None),
        "duplicates": (dup, None),
        "minimal": (rng.random((17, 3)).astype(np.float32), None),
    }


@pytest.mark.parametrize("name", list(_clouds().keys()))
def test_radius_bitexact_and_normals_vs_oracle(name):
    pos, ref = _clouds()[name]
    _check(pos, ref, 8, 16, name != "line")


@pytest.mark.parametrize("k_r,k_n", [(31, 32), (1, 3), (31, 3), (1, 32)])
@pytest.mark.parametrize("cloud", ["octar", "uniform", "exactly_k"])
def test_neighbour_count_limits(k_r, k_n, cloud):
    # the smallest and largest neighbour counts the ABI accepts, and a cloud
    # of exactly max(k_r + 1, k_n) points (every list is the whole cloud)
    rng = np.random.default_rng(k_r * 100 + k_n)
    if cloud == "exactly_k":
        pos, ref = rng.random((max(k_r + 1, k_n), 3)).astype(np.float32), None
    else:
        pos, ref = _clouds()[cloud]
    _check(pos, ref, k_r, k_n, cloud != "exactly_k" and k_n > 3)


def _check(pos, ref, k_r, k_n, most_defined):
    r, n = _gpu(pos, k_r, k_n, ref)
    ro, no, w, _ = oracle.point_attributes(pos, k_r, k_n, ref=ref)
    assert np.array_equal(r, ro), f"{np.flatnonzero(r != ro)[:10]}"
    good = (w[:, 1] - w[:, 0]) > 0.1 * np.maximum(w[:, 1], 1e-300)
    if most_defined:
        assert good.mean() > 0.5
    # angle from atan2(|a x b|, |a . b|): acos of a dot product near 1 would
    # turn the FP32 rounding of the output into ~1e-4 rad
    n64 = n.astype(np.float64)
    ang = np.arctan2(np.linalg.norm(np.cross(n64, no), axis=1), np.abs((n64 * no).sum(1)))
    assert ang[good].max(initial=0.0) < 1e-6
    # orientation: the same side wherever the reference direction decides it
    if ref is not None:
        firm = good & (np.abs((no * ref).sum(1)) > 1e-3)
    else:
        lo, hi = pos.astype(np.float64).min(0), pos.astype(np.float64).max(0)
        firm = good & (np.abs((no * (pos - 0.5 * (lo + hi))).sum(1)) > 1e-3)
    assert np.all((n.astype(np.float64) * no).sum(1)[firm] > 0)
    assert np.allclose(np.linalg.norm(n, axis=1), 1.0, atol=1e-6)


def test_full_size_sampled():
    # the composite workload's 1M noisy points; 2000 sampled points checked
    # against brute force over the whole cloud
    sc = scenes.composite(1_000_000, pca=False)
    pos = sc.pos
    r, _ = _gpu(pos, 8, 16, sc.nrm)
    q = np.random.default_rng(11).choice(pos.shape[0], 2000, replace=False)
    idx, d2 = oracle.knn(pos, 9, queries=q)
    assert np.array_equal(r[q], oracle.knn_radius(idx, d2, q, 8))


def test_argument_errors():
    from paper_2408_15583_gb300 import api
    p = torch.zeros(10, 3, device=DEV)
    with pytest.raises(RuntimeError):
        api.point_attributes(p, 8, 16)            # fewer points than neighbours
    with pytest.raises(RuntimeError):
        api.point_attributes(torch.zeros(100, 3, device=DEV), 8, 40)   # k_n > 32


@pytest.mark.parametrize("k_r,k_n", [(8, 16), (31, 32), (4, 3)])
def test_nan_points_have_no_neighbours(k_r, k_n):
    """A point with a NaN coordinate gets NaN and is nobody's neighbour: the other
    points' radii are those of the cloud without it, their normals too (one FP32
    rounding of a unit vector's component, 2^-24, and as much for the order of
    the sums).  3000 and 3005 points take the same grid."""
    rng = np.random.default_rng(k_r + k_n)
    clean = rng.random((3000, 3)).astype(np.float32)
    bad = np.sort(rng.choice(3005, 5, replace=False))
    pos = np.zeros((3005, 3), np.float32)
    good = np.setdiff1d(np.arange(3005), bad)
    pos[good] = clean
    pos[bad] = rng.random((5, 3)).astype(np.float32)
    for row, axes in zip(bad, ([0], [1], [2], [0, 1], [0, 1, 2])):
        pos[row, axes] = np.nan
    r, n = _gpu(pos, k_r, k_n)
    rc, nc = _gpu(clean, k_r, k_n)
    assert np.isnan(r[bad]).all() and np.isnan(n[bad]).all()
    assert np.array_equal(r[good], rc)
    assert np.abs(n[good] - nc).max() <= 2.0 ** -23


# 40 points of which all but `finite` are NaN: a point's normal needs k_n = 16
# points, its radius k_r = 8 others
@pytest.mark.parametrize("finite", [1, 8, 9, 15, 16])
def test_too_few_points_besides_nan(finite):
    rng = np.random.default_rng(finite)
    pos = np.full((40, 3), np.nan, np.float32)
    keep = np.sort(rng.choice(40, finite, replace=False))
    pos[keep] = rng.random((finite, 3)).astype(np.float32)
    r, n = _gpu(pos, 8, 16)
    rest = np.setdiff1d(np.arange(40), keep)
    assert np.isnan(r[rest]).all() and np.isnan(n[rest]).all()
    if finite >= 9:
        idx, d2 = oracle.knn(pos[keep], 9)
        assert np.array_equal(r[keep], oracle.knn_radius(idx, d2, np.arange(finite), 8))
    else:
        assert np.isnan(r[keep]).all()
    assert np.isnan(n).all() if finite < 16 else np.isfinite(n[keep]).all()


# neighbourhoods whose two smallest axes coincide (collinear, lattice, coincident
# points), where the last bit of a sum picks the axis, and ordinary ones; many
# points to a cell
@pytest.mark.parametrize("name", ["line", "lattice", "coincident", "cube", "octar"])
def test_the_same_call_gives_the_same_bits(name):
    rng = np.random.default_rng(5)
    pos = {
        "line": lambda: np.outer(rng.random(20000), [0.3, 0.5, 0.8]),
        "lattice": lambda: np.stack(np.meshgrid(*[np.arange(27) * 0.1] * 3), -1).reshape(-1, 3),
        "coincident": lambda: np.repeat(rng.random((400, 3)), 40, axis=0),
        "cube": lambda: rng.random((20000, 3)),
        "octar": lambda: scenes.octar(20000, 2.0, seed=3).pos,
    }[name]().astype(np.float32)
    pos = rng.permutation(pos)
    first = _gpu(pos, 8, 16)
    for _ in range(6):
        again = _gpu(pos, 8, 16)
        for a, b in zip(first, again):
            assert np.array_equal(a.view(np.uint32), b.view(np.uint32))


# little-endian floats: neighbours' distances from the origin along an axis, found
# by search, whose mean lies within 2^-44 of a boundary between two floats
_NEAR_A_ROUNDING_BOUNDARY = [
    "4519983e0f4da63e700af53e87132e3fe268843fc5278c3fd87b9f3f1f9db93f",
    "ea1f083f38ec113fd3f61e3fd6542a3f6ca43a3f41d9603f3d7c913f65d4d43f",
    "bc86b53ee0e3b63e6a60e73ec6f9643f20086e3fc6b38c3fa635913f25caa53f",
    "003f8b3eb073a83e2a50d53e56fb003fb3ac1e3f12514f3faaae8f3fec7ed13f",
    "c410933eb69b0d3f7d15123f4d5b1c3f38dc2c3f32ff353fb49a6a3f7a1eae3f",
    "ffea8c3e72ca323ff3746f3f62f8863f287c933ff00d983f5a729a3f1cfebc3f",
    "79abbe3ed647103f42b1393fd9ad533f2a787c3fb6bd913f5325943f9148b83f",
    "052dd33eb2d1223f6e2f353fa096553fd695743f9d95813fce17923fff9dd73f",
    "ec58883ec0888e3e260aa83ea33fbe3eec7cce3e0d8edd3e95e8e93e974cfd3e392cff3efe64013f"
    "7e26093f24992a3f7d1b333fdd53363f9b2d433ff4f7433f557e4e3fb1d94e3fe07a513fd3c2623f"
    "8b88723f1471753fc900773f269d843f56668c3fee708e3f2aa98e3fa118953f1e16993fbd039d3f"
    "3f81a13f",
    "4847863e14d48d3e82d2a73ec312bb3e8977c53e4cafd23e5e36053f45481b3fd2d8213f3815243f"
    "28b0263f65262f3f09f03a3fc6b63c3fb173493f2f715d3f49d8633f9cba643f3fd5683f16f9683f"
    "1b606b3f490a783f8684783fba98843f74cb873fbbc88d3f7ce78e3f442a903f4f6f923f60319b3f"
    "6062d43f",
]


@pytest.mark.parametrize("case", range(len(_NEAR_A_ROUNDING_BOUNDARY)))
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_radius_is_the_rounded_fp64_mean(case, axis):
    x = np.frombuffer(bytes.fromhex(_NEAR_A_ROUNDING_BOUNDARY[case]), "<f4")
    k = len(x)
    pos = np.zeros((k + 1, 3), np.float32)
    pos[1:, axis] = x
    idx, d2 = oracle.knn(pos, k + 1)
    from paper_2408_15583_gb300 import api
    r, _ = api.point_attributes(torch.from_numpy(pos).to(DEV), k, 3, normal=False)
    api.stream_check()
    assert np.array_equal(r.cpu().numpy(), oracle.knn_radius(idx, d2, np.arange(k + 1), k))


@pytest.mark.parametrize("shells", [2, 4, 5])
def test_normals_of_nearly_isotropic_neighbourhoods(shells):
    """Six points per shell on the axes at a, b, c, neighbouring floats: the axis is
    z, with eigenvalues 1e-7 apart.  FP64 sums leave some 1e-16 of the moments, so
    1e-9 of the axis; 32 roundings of 2^-53 would leave 2e-8 at the very most of a
    component whose cross moments are all of one sign (they are not), so 2^-27."""
    rng = np.random.default_rng(shells)
    worst = 0.0
    for _ in range(20):
        a = (0.5 + rng.random(shells)).astype(np.float32)
        b = np.nextafter(a, np.float32(0))
        c = np.nextafter(b, np.float32(0))
        z = np.zeros_like(a)
        pos = np.concatenate([np.stack(r, 1) for s in (np.float32(1), np.float32(-1))
                              for r in ((s * a, z, z), (z, s * b, z), (z, z, s * c))])
        _, n = _gpu(pos, 1, 6 * shells)
        worst = max(worst, float(np.abs(n[:, :2]).max()))
    assert worst < 2.0 ** -27
