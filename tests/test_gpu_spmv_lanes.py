"""The FP32 residual on levels whose operator product takes 32, 16 and 8 lanes per
node (short rows on few nodes, long rows on few and on more), in 2D, 3D and on the
Alfeld split, against the FP64 product of the same handle: a row's sum rounds at
most its number of entries times, 2^-24 of the sum of magnitudes each."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu

CASES = {
    "p4_16": (W.unit_square_mesh(8), 1, P.TH, 4, [4, 2], 32),
    "p4_32": (W.unit_square_mesh(8), 2, P.TH, 4, [4, 2], 16),
    "p3_64": (W.unit_square_mesh(8), 3, P.TH, 3, [3, 2], 8),
    "p7_32": (W.unit_square_mesh(8), 2, P.TH, 7, [7, 4, 2], 16),
    "sv_p4": (W.delaunay_disk_mesh(0, h=0.5), 1, P.SV, 4, [4, 2], 32),
    "3d_p2": (W.kuhn_cube_mesh(2), 2, P.TH, 2, [2], 32),
    "3d_p3": (W.kuhn_cube_mesh(2), 2, P.TH, 3, [3, 2], 32),
    "3d_p2_16": (W.kuhn_cube_mesh(4), 2, P.TH, 2, [2], 16),
    "p2_32": (W.unit_square_mesh(8), 2, P.TH, 2, [2], 8),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_residual(name):
    (v, c), nref, fam, k, sched, lanes = CASES[name]
    h = P.StokesMG(v, c, nref, fam, k, barycentric=fam == P.SV, hierarchy=P.HIER_EXPLICIT, schedule=sched,
                   precision=P.MIXED, lmax_override=[1.0] * 8)
    for level in range(len(h.info()["n_free"])):
        K = h.get_csr(level)
        n = K.shape[0]
        _, comp, _ = h.level_dofs(level)
        groups = int(((comp == 0) | (comp == v.shape[1])).sum())
        if level == 0:
            g = groups * n / K.nnz
            want = 8 if K.nnz <= 20 * n else 32 if g * v.shape[1] <= 800 else 16 if g <= 1600 else 8
            assert want == lanes
        b, x = np.random.default_rng(level).standard_normal((2, n)).astype(np.float32).astype(np.float64)
        r = [h.residual(level, torch.tensor(b, device="cuda"), torch.tensor(x, device="cuda"), p).cpu().numpy()
             for p in (P.MIXED, P.FP64)]
        size = abs(b) + abs(K) @ abs(x)
        # the entries' own rounding, their products and the sums
        assert (np.abs(r[0] - r[1]) <= (np.diff(K.indptr) + 3) * 2.0**-24 * size).all()
    h.close()
