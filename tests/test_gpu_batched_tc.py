"""The tensor-core patch GEMM at the edges of its tiles: patches of one to five
128-row tiles (81, 141, 315 and 540 DoFs and the smaller ones of their
boundaries), every accumulator width, both modes, and a level with more patches
per CTA than the list in shared memory holds.

Reference: the single-vector mixed V-cycle, to the tolerances of the batched
V-cycle's other checks (1e-4 for 3xTF32, which is FP32 accurate; 2e-2 for TF32)."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu

TOL = {P.BATCH_3XTF32: 1e-4, P.BATCH_TF32: 2e-2}
CASES = {
    "th_p3": (W.unit_square_mesh(3), 1, 3, [3, 2]),
    "th_p4": (W.unit_square_mesh(3), 1, 4, [4, 2]),
    "th_p6": (W.unit_square_mesh(2), 1, 6, [6, 4, 2]),
    "th3d_p3": (W.kuhn_cube_mesh(2), 1, 3, [3, 2]),
}


def _check(h, nrhs, mode):
    n = h.info()["n_free"][0]
    R = torch.randn(nrhs, n, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(nrhs))
    Z, Z1 = h.vcycle_batched(R, mode), h.vcycle(R)
    err = (Z - Z1).abs().amax(1) / Z1.abs().amax(1)
    assert err.max().item() < TOL[mode], (nrhs, mode)


@pytest.mark.parametrize("name", sorted(CASES))
def test_tiles_and_widths(name):
    (v, c), nref, k, sched = CASES[name]
    h = P.StokesMG(v, c, nref, P.TH, k, hierarchy=P.HIER_EXPLICIT, schedule=sched, precision=P.MIXED)
    for nrhs in (3, 16, 17, 64):
        for mode in (P.BATCH_3XTF32, P.BATCH_TF32):
            _check(h, nrhs, mode)
    h.close()


def test_more_patches_than_the_list_holds():
    v, c = W.unit_square_mesh(9)
    h = P.StokesMG(v, c, 5, P.TH, 3, hierarchy=P.HIER_EXPLICIT, schedule=[3, 2], precision=P.MIXED, batch_tune=0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert h.info()["n_patches"][0] > 513 * sms
    _check(h, 5, P.BATCH_3XTF32)
    h.close()
