"""The batched orthogonalisation where a column's Krylov space has closed: the new
vector lies in the span of the basis to about eps, and the norm of what is left of
it cannot come from a difference of squares.  The basis vector still has length one
(or is zero with a zero norm), and w = V h + |.| v holds to a few ulp of the largest
terms, next to columns with ordinary remainders.

Called through the library's internal entry points, one step after another as the
solver does."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu

STEPS = ["_ZN4sbat8col_dotsEiiiPKdxS1_PdS2_iP11CUstream_st", "_ZN4sbat15col_update_dotsEiiiPKdxS1_PdS2_S2_S2_P11CUstream_st",
         "_ZN4sbat13col_normaliseEiiiPKdxS1_S1_PdS2_P11CUstream_st", "_ZN4sbat10col_givensEiiiiPdS0_PKdS0_S0_S0_S0_S0_P11CUstream_st"]


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("n", [40, 1000, 30011])
@pytest.mark.parametrize("nb", [1, 6, 13, 24])
def test_unit_vectors_and_arnoldi_relation(n, nb):
    dots, update, normalise, givens = (getattr(P._binding.lib(), s) for s in STEPS)
    m, ldh = 16, 40
    i, ll, none = ctypes.c_int, ctypes.c_longlong, ctypes.c_void_p(0)
    g = torch.Generator(device="cuda").manual_seed(nb)
    V = torch.randn(m, n, nb, dtype=torch.float64, device="cuda", generator=g)
    V[:4, :, 0] = n**-0.5
    V = torch.linalg.qr(V)[0]
    V[:4, :, 0] = n**-0.5
    V = torch.cat([V.permute(2, 1, 0), torch.zeros(1, n, m, dtype=torch.float64, device="cuda")]).contiguous()
    # column c: a random element of the span and a remainder of size rest[c]
    rest = torch.tensor([0, 0, 0, 0, 1e-17, 1e-16, 1e-16, 1e-15, 1e-14, 1e-12, 1e-8, 1e-4, 1, 1e4, 0, 0],
                        dtype=torch.float64, device="cuda")
    a = torch.randn(nb, m, dtype=torch.float64, device="cuda", generator=g)
    a[:, -2:] = 0.0
    a[1:, :4] = 0.0                 # multiples of a constant vector: what the first pass leaves of them is in the span too
    W0 = torch.einsum("bnm,bm->nm", V[:nb], a) + rest / n**0.5 * torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g)
    W = W0.clone(memory_format=torch.contiguous_format)
    partial = torch.empty(608 * 33 * m, dtype=torch.float64, device="cuda")
    new = lambda *k: torch.zeros(*k, dtype=torch.float64, device="cuda")
    h, h2, hn, H, cs, sn, gg, res = new(32, m), new(33, m), new(m), new(m, ldh, ldh), new(m, ldh), new(m, ldh), new(m, ldh + 1), new(m)
    ld = ll(n * m)
    dots(i(n), i(m), i(nb), _p(V), ld, _p(W), _p(partial), _p(h), i(0), none)
    update(i(n), i(m), i(nb), _p(V), ld, _p(h), _p(W), _p(partial), _p(h2), _p(h), none)
    normalise(i(n), i(m), i(nb), _p(V), ld, _p(h2), _p(W), _p(V[nb]), _p(hn), none)
    givens(i(nb - 1), i(m), i(ldh), i(n), _p(V[nb]), _p(H), _p(h), _p(hn), _p(cs), _p(sn), _p(gg), _p(res), none)
    torch.cuda.synchronize()
    norm = V[nb].norm(dim=0)
    assert ((norm == 0) == (hn == 0)).all() and (hn >= 0).all()
    assert (norm[-2:] == 0).all() and (norm[10:14] > 0).all()
    assert ((norm - 1).abs()[norm > 0] <= 1e-12).all(), norm
    # nb + 2 roundings of numbers up to |w|, once per pass
    left = (W0 - torch.einsum("bnm,bm->nm", V, torch.cat([h[:nb], hn[None]]))).norm(dim=0)
    assert (left <= 4 * (nb + 2) * 2.0**-52 * W0.norm(dim=0)).all()
