"""The bounded waits of the tensor-core patch GEMM at a timeout: a warp whose
lanes reach the limit at different polls gives up as one (a lane that went on
alone would wait for the others in the next warp-wide instruction); the GEMM
reports a timeout whichever role it comes from, waits for its copies and MMAs in
flight, gives its tensor memory back, and the next launch is right."""
import pytest

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2407_07253_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("polls", [0, 1, 64, 4096])
def test_a_warp_gives_up_as_one(polls):
    assert P._binding.selftest_bounded_wait(polls) == 2


def test_the_gemm_reports_a_timeout_and_leaves_the_device_usable():
    for _ in range(3):
        assert P._binding.selftest_bounded_wait(0) == 2
    assert float((torch.ones(4, device="cuda") * 2).sum()) == 8.0
