"""The bounded wait of the CTAs that share a frame (256^2 and 512^2, few
frames): with a bound of no cycles a CTA that is not the last to arrive gives
up at its first look. The kernel returns, the status says so once, and the plan
works again."""

import pytest

from paper_1705_04298_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fwr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04298_gb300 import fwr as m
    m.load()
    return m


@pytest.mark.parametrize("N,n,F", [(256, 128, 1), (256, 101, 60), (512, 200, 1), (512, 200, 19)])
def test_a_wait_that_runs_out_is_reported_and_cleared(fwr, N, n, F):
    mask = synth.pupil_mask(n)
    s = torch.randn((F, 2, n, n), device="cuda") * torch.tensor(mask, device="cuda")
    plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=N)
    ref = plan.reconstruct(s, 3).clone()
    untouched = torch.full_like(ref, -7.0)
    out = untouched.clone()
    plan.set_team_wait(0)
    plan.reconstruct(s, 3, out)
    torch.cuda.synchronize()
    assert not torch.equal(out, ref)
    # until the status is read: nothing is written, whatever the bound
    plan.set_team_wait(4e9)
    out = untouched.clone()
    plan.reconstruct(s, 3, out)
    torch.cuda.synchronize()
    assert torch.equal(out, untouched)
    # the one-CTA kernel has no waits
    plan.set_ctas(1000)
    plan.reconstruct(s, 3, out)
    assert torch.equal(out, ref)
    plan.set_ctas(0)
    assert plan.status() == "FWR_ERR_TIMEOUT"
    assert plan.status() == "FWR_OK"
    for _ in range(2):
        out = untouched.clone()
        plan.reconstruct(s, 3, out)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    assert plan.status() == "FWR_OK"


def test_the_timeout_is_reported_before_nonfinite_slopes(fwr):
    s = torch.randn((1, 2, 128, 128), device="cuda")
    plan = fwr.Plan(synth.pupil_mask(128), 2.0, fwr.LSQ)
    s[0, 0, 64, 64] = float("nan")
    plan.reconstruct(s, 1)
    plan.set_team_wait(0)
    plan.reconstruct(s, 1)
    assert plan.status() == "FWR_ERR_TIMEOUT"


def test_team_wait_values(fwr):
    plan = fwr.Plan(synth.pupil_mask(128), 2.0, fwr.LSQ)
    for bad in (-1.0, float("nan"), 2e15):
        with pytest.raises(fwr.FwrError, match="ARG"):
            plan.set_team_wait(bad)
    with pytest.raises(fwr.FwrError, match="UNSUPPORTED"):
        fwr.Plan(synth.pupil_mask(40), 3.2, fwr.LSQ).set_team_wait(1e6)
