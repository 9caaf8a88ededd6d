"""The tiled inversion of a level whose patches take more scratch than one launch
may: P5 on 192 x 192, 37,249 stars, in two parts.  The mesh is uniform, so one
sweep over a constant residual gives the same values at every lattice position
of a cell, away from the boundary: the first part's against the last one's, to the
2e-4 of the other mixed checks."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu


def test_both_parts_invert_the_same_stars():
    n, k = 192, 5
    v, c = W.unit_square_mesh(6)
    h = P.StokesMG(v, c, 5, P.TH, k, hierarchy=P.HIER_EXPLICIT, schedule=[5, 2], precision=P.MIXED,
                   lmax_override=[1.0] * 8)
    xyz, comp, _ = h.level_dofs(0)
    z = h.asm(0, torch.ones(len(comp), dtype=torch.float64, device="cuda"), P.MIXED).cpu().numpy()
    h.close()
    # pressures of P4 lie on another lattice: the velocity components alone
    for a in (0, 1):
        own = comp == a
        at = np.rint(xyz[own] * n * k).astype(int)
        inner = ((at > 2 * k) & (at < (n - 2) * k)).all(1)
        key = (at[inner] % k) @ [k, 1]
        val = z[own][inner]
        lo, hi = np.full(k * k, np.inf), np.full(k * k, -np.inf)
        np.minimum.at(lo, key, val)
        np.maximum.at(hi, key, val)
        assert ((hi - lo) <= 2e-4 * np.abs(z[own]).max()).all()
