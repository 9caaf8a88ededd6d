"""The FP32 residual on a level with enough rows for the operator product's
four-lane groups (over a million nodes; the smaller ones, with eight lanes, are
checked with every level's residual elsewhere), against the exported operator in
FP64: a row sums at most 122 FP32 products here, sqrt(122) 2^-24 of the row's
largest partial sums, with a factor of ten for their spread."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu


def test_four_lane_residual():
    w = W.workload("th_p4_256x256")
    h = P.StokesMG(w.verts, w.cells, w.n_refine, w.family, w.k, hierarchy=P.HIER_EXPLICIT, schedule=w.schedule,
                   precision=P.MIXED, lmax_override=[1.0] * 6)
    n = h.info()["n_free"][0]
    g = np.random.default_rng(0)
    b, x = g.standard_normal((2, n))
    r = h.residual(0, torch.tensor(b, device="cuda"), torch.tensor(x, device="cuda"), P.MIXED).cpu().numpy()
    K = h.get_csr(0)
    h.close()
    want = b - K @ x
    scale = abs(b) + abs(K) @ abs(x)
    assert (np.abs(r - want) <= 10 * np.sqrt(122) * 2.0**-24 * scale).all()
