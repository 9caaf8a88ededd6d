"""An FBF handle's setup captures the graph of its solves alone; the one-vector V-cycle
captures its own on the first call, or runs as plain launches inside a capture of the
caller's: the same bits each way."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [P.FP64, P.MIXED])
def test_vcycle_first_call(precision):
    v, c = W.delaunay_disk_mesh(0, h=0.5)

    def handle(**kw):
        return P.StokesMG(v, c, 1, P.SV, 3, barycentric=True, hierarchy=P.HIER_EXPLICIT, schedule=[3, 2], fbf=True,
                          precision=precision, **kw)

    plain, lazy, captured = handle(use_graph=0), handle(), handle()
    r = torch.randn(plain.info()["n_free"][0], dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    want = plain.vcycle(r)
    assert torch.equal(lazy.vcycle(r), want) and torch.equal(lazy.vcycle(2 * r), plain.vcycle(2 * r))
    x = r.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        z = captured.vcycle(x)
    for s in (1.0, 2.0):
        x.copy_(s * r)
        g.replay()
        assert torch.equal(z, plain.vcycle(s * r))
    assert torch.equal(captured.vcycle(r), want)
    # a failed or missing graph would show in the solves too
    f = torch.tensor(W.nodal_forcing(lazy.nodes()[0].shape[0], 2, 1), device="cuda")
    assert torch.equal(lazy.solve(f, None, tol=1e-8)[0], plain.solve(f, None, tol=1e-8)[0])
    del g
    for h in (plain, lazy, captured):
        h.close()
