"""FBF's scalar patch inverses from the tiled SPD sweep: blocks of one tile to
forty, both launch classes, both precisions; and with a negative viscosity in one
cell, whose indefinite blocks the sweep hands over to the pivoted inversion.

Reference: one ASM sweep z = sum_i I_i^T W_i A_i^-1 I_i r with numpy's LU solves of
the exported blocks, to 10 kappa eps_64 (at least 1e-10), or 2e-4 with FP32
inverses, as the saddle applies are checked."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("negative", [False, True])
@pytest.mark.parametrize("precision", [P.FP64, P.MIXED])
@pytest.mark.parametrize("k,sched", [(3, [3, 2]), (4, [4, 2]), (5, [5, 2])])
def test_apply_matches_patch_solves(k, sched, precision, negative):
    v, c = W.delaunay_disk_mesh(0, h=0.5)
    args = dict(barycentric=True, hierarchy=P.HIER_EXPLICIT, schedule=sched, fbf=True)
    nc = P.StokesMG(v, c, 1, P.SV, k, host_only=1, **args).n_cells()
    nu = W.cell_viscosity(nc, 1)
    if negative:
        nu[nc // 2] = -0.4
    h = P.StokesMG(v, c, 1, P.SV, k, nu_cell=nu, precision=precision, lmax_override=[1.0] * 8, **args)
    n_free = h.info()["n_free"]
    indefinite = False
    for li in range(len(n_free) - 1):
        off, dofs = h.patches(li)
        flat = h.patch_matrices(li)
        r = np.random.default_rng(li).standard_normal(n_free[li])
        want, mult, kappa, pos = np.zeros(n_free[li]), np.bincount(dofs, minlength=n_free[li]), 1.0, 0
        for i in range(len(off) - 1):
            d = dofs[off[i]:off[i + 1]]
            A = flat[pos:pos + len(d) ** 2].reshape(len(d), len(d))
            pos += len(d) ** 2
            want[d] += np.linalg.solve(A, r[d]) / mult[d]
            kappa = max(kappa, np.linalg.cond(A))
            indefinite |= np.linalg.eigvalsh(A).min() < 0
        z = h.asm(li, torch.tensor(r, device="cuda"), precision).cpu().numpy()
        tol = max(1e-10, 10 * kappa * np.finfo(np.float64).eps) if precision == P.FP64 else 2e-4
        assert np.abs(z - want).max() <= tol * np.abs(want).max(), li
    assert indefinite == negative
    h.close()
