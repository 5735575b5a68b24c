"""Few frames on 256^2 and 512^2 grids: the slab kernel with a team of CTAs per
frame gives bitwise the phase of the same kernel with one CTA per frame (an
explicit persistent-grid size, FWR_OPT_CTAS, keeps that one)."""

import numpy as np
import pytest

import oracle
from paper_1705_04298_gb300 import synth
from parity_check import FP32_RMS, within

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fwr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04298_gb300 import fwr as m
    m.load()
    return m


def frames(n, F, seed):
    sl, _, mask = synth.batch(n, min(F, 3), seed, 0.05)
    s = torch.tensor(sl, dtype=torch.float32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = s.repeat((F + len(sl) - 1) // len(sl), 1, 1, 1)[:F]
    noise = 0.1 * torch.randn(s.shape, generator=g, device="cuda")
    return (s + noise * torch.tensor(mask, device="cuda")).contiguous(), mask


# every team size of both grids' tables, ragged waves, more than one wave
@pytest.mark.parametrize("N,n,F", [(256, 128, 1), (256, 101, 19), (256, 200, 38), (256, 70, 76), (256, 128, 160),
                                   (512, 200, 1), (512, 131, 10), (512, 200, 19), (512, 170, 25), (512, 256, 38),
                                   (512, 200, 50), (512, 200, 64), (512, 200, 76)])
def test_teams_match_one_cta_per_frame(fwr, N, n, F):
    s, mask = frames(n, F, 40 + n)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    plan = fwr.Plan(mask, 1.0, fwr.WIENER, 0.01, 0.6, 100.0, grid=N)
    ext = torch.randn((F, 2, N, N), device="cuda") if F <= 19 else None
    for periodic, k, hud, warm in ((0, 2, False, False), (1, 1, True, False), (2, 0, False, True)):
        if warm and ext is None:
            continue
        plan.set_periodic(periodic)
        plan.set_extension(fwr.EXT_HUDGIN if hud else fwr.EXT_ZERO)
        kw = {"ext_init": ext} if warm else {}
        plan.set_ctas(sms)
        ref = plan.reconstruct(s, k, **kw).clone()
        plan.set_ctas(0)
        out = torch.full_like(ref, float("nan"))
        for _ in range(2):  # the team's counters are zero again after a launch
            plan.reconstruct(s, k, out, **kw)
            torch.cuda.synchronize()
            assert torch.equal(out, ref), (periodic, k)
    assert plan.status() == "FWR_OK"


def test_teams_replay_from_a_cuda_graph(fwr):
    s, mask = frames(128, 5, 3)
    plan = fwr.Plan(mask, 2.0, fwr.LSQ)
    ref = plan.reconstruct(s, 3).clone()
    out = torch.full_like(ref, float("nan"))
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        plan.reconstruct(s, 3, out, stream=stream)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


def test_teams_report_nonfinite_slopes(fwr):
    s, mask = frames(128, 2, 9)
    plan = fwr.Plan(mask, 2.0, fwr.LSQ)
    s[1, 0, 64, 64] = float("inf")
    plan.reconstruct(s, 1)
    assert plan.status() == "FWR_ERR_NONFINITE"
    assert plan.status() == "FWR_OK"


# a white warm start reaches every bin pair of the 256^2 spectral step: the
# self-paired columns 0 and 128, their self-paired bins, every fill mode
@pytest.mark.parametrize("n,k,periodic", [(128, 1, 0), (101, 2, 1), (160, 1, 2), (77, 0, 0)])
@pytest.mark.parametrize("shape", [0, 1])
def test_256_every_bin(fwr, n, k, periodic, shape):
    s, mask = frames(n, 1, 60 + n)
    plan = fwr.Plan(mask, 1.0, fwr.WIENER, 0.01, 0.6, 100.0, periodic, grid=256)
    plan.set_shape(shape)
    ext = np.random.default_rng(n).standard_normal((1, 2, 256, 256)).astype(np.float32)
    ph = plan.reconstruct(s, k, ext_init=torch.tensor(ext, device="cuda"))
    assert plan.status() == "FWR_OK"
    ref, _ = oracle.reconstruct(s[0].cpu().double().numpy(), mask, 1.0, k, oracle.FILTER_WIENER, 0.01, 0.6, 100.0, periodic,
                                ext_init=ext[0].astype(np.float64), N=256)
    assert within(ph[0].cpu().numpy(), ref, FP32_RMS, where="n=%d" % n)


def test_256_largest_pupil(fwr):
    """209 lenslets across are the most that 256^2 takes; the largest runs."""
    with pytest.raises(fwr.FwrError, match="UNSUPPORTED"):
        fwr.Plan(synth.pupil_mask(210), 1.0, fwr.WIENER, 0.01, 0.6, 100.0, grid=256)
    s, mask = frames(209, 1, 5)
    plan = fwr.Plan(mask, 1.0, fwr.WIENER, 0.01, 0.6, 100.0, grid=256)
    ph = plan.reconstruct(s, 1)
    ref, _ = oracle.reconstruct(s[0].cpu().double().numpy(), mask, 1.0, 1, oracle.FILTER_WIENER, 0.01, 0.6, 100.0,
                                N=256)
    assert within(ph[0].cpu().numpy(), ref, FP32_RMS, where="n=209")
