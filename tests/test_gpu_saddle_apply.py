"""The saddle applies (one ASM sweep, Eq. 3.4) on every level of small
hierarchies whose patches cover their edges: one row group or tile to several
per thread, row counts of every remainder of the 16-byte vectors, one pressure
column to more than a warp's, two and three components, both precisions.  Once
with the bulk-copy applies (the FP32 one on tiles) on the levels that they take,
once with them switched off, so that every level takes the streamed one.

Reference: z = sum_i I_i^T W_i K_i^-1 I_i r with numpy's LU solves of the
exported patch blocks.  The two sides factor the blocks differently and agree
to about kappa eps_64 (kappa: the largest block condition number), FP32 factors
and sums to 2e-4 as the other mixed checks."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu

CASES = {
    "th_p2": (W.unit_square_mesh(2), 1, P.TH, 2, [2], False),
    "th_p3": (W.unit_square_mesh(3), 1, P.TH, 3, [3, 2], False),
    "th_p5": (W.unit_square_mesh(2), 1, P.TH, 5, [5, 2], False),
    "th_p8": (W.unit_square_mesh(2), 1, P.TH, 8, [8, 5, 2], False),
    "sv_p4": (W.delaunay_disk_mesh(0, h=0.5), 1, P.SV, 4, [4, 2], True),
    "th3d_p3": (W.kuhn_cube_mesh(2), 1, P.TH, 3, [3, 2], False),
}


@pytest.mark.parametrize("precision", [P.FP64, P.MIXED])
@pytest.mark.parametrize("bulk", [True, False])
@pytest.mark.parametrize("name", sorted(CASES))
def test_apply_matches_patch_solves(name, bulk, precision, monkeypatch):
    if not bulk:
        monkeypatch.setenv("STOKES_NO_BULK_APPLY", "1")
    (v, c), nref, fam, k, sched, bary = CASES[name]
    h = P.StokesMG(v, c, nref, fam, k, barycentric=bary, hierarchy=P.HIER_EXPLICIT, schedule=sched,
                   precision=precision)
    n_free = h.info()["n_free"]
    for li in range(len(n_free) - 1):
        off, dofs = h.patches(li)
        flat = h.patch_matrices(li)
        r = np.random.default_rng(li).standard_normal(n_free[li])
        want, mult, kappa, pos = np.zeros(n_free[li]), np.bincount(dofs, minlength=n_free[li]), 1.0, 0
        for i in range(len(off) - 1):
            d = dofs[off[i]:off[i + 1]]
            K = flat[pos:pos + len(d) ** 2].reshape(len(d), len(d))
            pos += len(d) ** 2
            want[d] += np.linalg.solve(K, r[d]) / mult[d]
            kappa = max(kappa, np.linalg.cond(K))
        z = h.asm(li, torch.tensor(r, device="cuda"), precision).cpu().numpy()
        tol = max(1e-10, 10 * kappa * np.finfo(np.float64).eps) if precision == P.FP64 else 2e-4
        assert np.abs(z - want).max() <= tol * np.abs(want).max(), (name, li)
    h.close()
