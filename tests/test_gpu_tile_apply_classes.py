"""The FP32 apply on tiles in its two widest classes (161 to 256 tiles, one a thread;
257 to 512, two), which the stars of the structured meshes reach in 2D at P5 alone:
cones over triangulated spheres and wheels of eight triangles put one vertex of
high valence in the middle.  In 3D their partial sums lie behind the block instead
of over it.

Reference and tolerance as the other saddle applies: numpy's LU solves of the
exported blocks, 2e-4 with FP32 factors; in FP64 about kappa eps_64, with 1e-10 as
there.  The streamed apply takes the same levels, where one or a few pressures give
it more groups of threads than columns."""
import numpy as np
import pytest
from scipy.spatial import ConvexHull

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu


def cone(n):
    """Tetrahedra from the origin to the hull of n points spread over the sphere."""
    i = np.arange(n) + 0.5
    z, t = 1 - 2 * i / n, np.pi * (1 + 5**0.5) * i
    s = np.sqrt(1 - z * z)
    pts = np.stack([s * np.cos(t), s * np.sin(t), z], 1)
    tri = ConvexHull(pts).simplices + 1
    return np.vstack([np.zeros(3), pts]), np.hstack([np.zeros((len(tri), 1), int), tri]).astype(np.int32)


def wheel(n):
    t = 2 * np.pi * np.arange(n) / n
    k = np.arange(n)
    return (np.vstack([np.zeros(2), np.stack([np.cos(t), np.sin(t)], 1)]),
            np.stack([0 * k, k + 1, (k + 1) % n + 1], 1).astype(np.int32))


CASES = {
    "3d_one": (cone(17), 2, [2], 160, 256),
    "3d_two": (cone(24), 2, [2], 256, 512),
    "2d_one": (wheel(8), 4, [4, 2], 160, 256),
    "2d_two": (wheel(9), 4, [4, 2], 256, 512),
}


def check(name, precision):
    (v, c), k, sched, above, most = CASES[name]
    h = P.StokesMG(v, c, 1, P.TH, k, hierarchy=P.HIER_EXPLICIT, schedule=sched, precision=precision, lmax_override=[1.0] * 8)
    n = h.info()["n_free"][0]
    off, dofs = h.patches(0)
    _, comp, _ = h.level_dofs(0)
    n4 = max(-(-int((comp[dofs[a:b]] == 0).sum()) // 4) for a, b in zip(off, off[1:]))
    assert above < n4 * (n4 + 1) // 2 <= most
    flat = h.patch_matrices(0)
    r = np.random.default_rng(k).standard_normal(n)
    want, mult, pos, kappa = np.zeros(n), np.bincount(dofs, minlength=n), 0, 1.0
    for a, b in zip(off, off[1:]):
        d = dofs[a:b]
        K = flat[pos:pos + len(d)**2].reshape(len(d), len(d))
        pos += len(d)**2
        want[d] += np.linalg.solve(K, r[d]) / mult[d]
        kappa = max(kappa, np.linalg.cond(K))
    z = h.asm(0, torch.tensor(r, device="cuda"), precision).cpu().numpy()
    h.close()
    tol = 2e-4 if precision == P.MIXED else max(1e-10, 10 * kappa * np.finfo(np.float64).eps)
    assert np.abs(z - want).max() <= tol * np.abs(want).max()


@pytest.mark.parametrize("name", sorted(CASES))
def test_apply_matches_patch_solves(name):
    check(name, P.MIXED)


@pytest.mark.parametrize("precision", [P.FP64, P.MIXED])
@pytest.mark.parametrize("name", sorted(CASES))
def test_streamed_apply_matches_patch_solves(name, precision, monkeypatch):
    monkeypatch.setenv("STOKES_NO_BULK_APPLY", "1")
    check(name, precision)


@pytest.mark.parametrize("precision", [P.FP64, P.MIXED])
@pytest.mark.parametrize("name", ["sv_p2_level", "3d"])
def test_uneven_levels(name, precision, monkeypatch):
    """Over 1216 patches, most of them far smaller than the largest: the row-wise
    bulk-copy apply, in FP32 too, against the streamed one (the same factors, rounded
    the same; the sums of up to 3 * 95 terms in another order)."""
    (v, c), nref, fam, k, sched, level = {"sv_p2_level": (W.delaunay_disk_mesh(0, h=0.16), 1, P.SV, 3, [3, 2], 1),
                                          "3d": (cone(13), 3, P.TH, 2, [2], 0)}[name]
    z = []
    for stream in (False, True):
        if stream:
            monkeypatch.setenv("STOKES_NO_BULK_APPLY", "1")
        h = P.StokesMG(v, c, nref, fam, k, barycentric=fam == P.SV, hierarchy=P.HIER_EXPLICIT, schedule=sched,
                       precision=precision, lmax_override=[1.0] * 8)
        off, dofs = h.patches(level)
        _, comp, _ = h.level_dofs(level)
        n4 = np.array([-(-int((comp[dofs[a:b]] == 0).sum()) // 4) for a, b in zip(off, off[1:])])
        t = n4 * (n4 + 1) // 2
        assert len(t) > 1216 and t.mean() < 0.4 * t.max() and t.max() > 64
        r = np.random.default_rng(3).standard_normal(len(comp))
        z.append(h.asm(level, torch.tensor(r, device="cuda"), precision).cpu().numpy())
        h.close()
    eps = 2.0**-24 if precision == P.MIXED else 2.0**-53
    assert np.abs(z[0] - z[1]).max() <= 600 * eps * np.abs(z[1]).max()
