"""The batched FGMRES's orthogonalisation at every width (8, 16, 32, 64) over
a whole restart cycle: 40 iterations of the lightly smoothed default cycle pass
through every unrolling of its multi-dots and a restart.  One column is zero
(its basis stays zero) and one repeats another.

Every column's true residual has to meet the tolerance that the iteration
stopped at: the estimate follows the true residual as long as the basis is
orthogonal to machine precision, so a factor of two is generous.  Columns of a
batch are independent, so a repeated column gives the same bits."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [3, 16, 21, 64])
def test_columns_meet_the_tolerance_through_a_restart(nrhs):
    v, c = W.unit_square_mesh(2)
    h = P.StokesMG(v, c, 2, P.TH, 3, hierarchy=P.HIER_EXPLICIT, schedule=[3, 2], precision=P.MIXED, cheb_lo=0.02,
                   cheb_hi=4.0)
    n = h.info()["n_free"][0]
    K = h.get_csr(0)
    _, comp, _ = h.level_dofs(0)
    B = np.random.default_rng(nrhs).standard_normal((nrhs, n))
    B[:, comp == 2] -= B[:, comp == 2].mean(1, keepdims=True)
    B[1] = 0.0
    B[2] = B[0]
    tol = 1e-12
    X, its, rel = h.fgmres_batched(torch.tensor(B, device="cuda"), P.BATCH_3XTF32, tol=tol)
    X = X.cpu().numpy()
    assert its > 30                       # through the restart
    assert not X[1].any() and np.array_equal(X[2], X[0])
    for q in range(nrhs):
        nb = np.linalg.norm(B[q])
        assert np.linalg.norm(B[q] - K @ X[q]) <= 2 * tol * nb + 1e-13 * abs(K).max() * np.linalg.norm(X[q])
    h.close()
