"""Patch inverses on both sides of the rule that takes stars of 80 nodes and more to the
tiled inversion: P5 on 24 x 24 (pivot pairs) and 40 x 40 (tiles), the P5 level under P8,
few such stars among smaller ones (P4 on the disk) and beside larger ones (P5 on the
disk).  One FP64 sweep against numpy's LU solves of the exported blocks of some
DoFs' patches, to about kappa eps_64 as the other checks."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu

CASES = {
    "p5_24": (W.unit_square_mesh(6), 2, 5, [5, 2], 0),
    "p5_40": (W.unit_square_mesh(5), 3, 5, [5, 2], 0),
    "p5_under_p8": (W.unit_square_mesh(7), 2, 8, [8, 5, 2], 1),
    "p4_disk": (W.delaunay_disk_mesh(0, h=0.25), 2, 4, [4, 2], 0),
    "p5_disk": (W.delaunay_disk_mesh(0, h=0.3), 1, 5, [5, 2], 0),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_sweep_matches_patch_solves(name):
    (v, c), nref, k, sched, level = CASES[name]
    h = P.StokesMG(v, c, nref, P.TH, k, hierarchy=P.HIER_EXPLICIT, schedule=sched, precision=P.FP64, lmax_override=[1.0] * 8)
    off, dofs = h.patches(level)
    n = h.info()["n_free"][level]
    K = h.get_csr(level)
    r = np.random.default_rng(k).standard_normal(n)
    z = h.asm(level, torch.tensor(r, device="cuda"), P.FP64).cpu().numpy()
    h.close()
    mult = np.bincount(dofs, minlength=n)
    size = np.diff(off)
    # the pressures (one patch each at a vertex) of the smallest and largest patches and some between
    owner = {}
    for i in range(len(size)):
        for j in dofs[off[i]:off[i + 1]]:
            owner.setdefault(int(j), []).append(i)
    single = [(j, i[0]) for j, i in owner.items() if len(i) == 1]
    single.sort(key=lambda s: size[s[1]])
    take = [single[int(t)] for t in np.linspace(0, len(single) - 1, 60)]
    scale = np.abs(z).max()
    for j, i in take:
        d = dofs[off[i]:off[i + 1]]
        A = K[d][:, d].toarray()
        x = np.linalg.solve(A, r[d])
        tol = max(1e-10, 10 * np.linalg.cond(A) * np.finfo(np.float64).eps)
        assert abs(z[j] - x[np.searchsorted(d, j)] / mult[j]) <= tol * max(scale, np.abs(x).max()), (j, i)
