"""The FP64 path with a cluster of CTAs per frame (few frames on 32^2 and 64^2):
against the FP64 oracle, and against the one-CTA kernel (kept by an explicit
persistent-grid size), whose arithmetic orders its sums differently."""

import numpy as np
import pytest

import oracle
from paper_1705_04298_gb300 import synth
from parity_check import FP64_MAX, FP64_RMS, within

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fwr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04298_gb300 import fwr as m
    m.load()
    return m


# one frame, more frames than run at once, pupils from a corner of the grid to all of it
@pytest.mark.parametrize("N,n,F", [(32, 16, 1), (32, 30, 37), (32, 9, 2), (64, 31, 1), (64, 62, 40), (64, 40, 3)])
@pytest.mark.parametrize("periodic,k,start", [(0, 3, "zero"), (1, 2, "hudgin"), (2, 1, "warm"), (0, 0, "zero")])
def test_cluster_against_oracle(fwr, N, n, F, periodic, k, start):
    base, _, mask = synth.batch(n, 2, 70 + N + n, 0.05)
    r0p, L0p = synth.pitch_units(n, 0.15, 25.0)
    plan = fwr.Plan(mask, 1.0, fwr.WIENER, 0.05 ** 2, r0p, L0p, periodic, grid=N)
    if start == "hudgin":
        plan.set_extension(fwr.EXT_HUDGIN)
    s = torch.tensor(base, dtype=torch.float64, device="cuda").repeat(F // 2 + 1, 1, 1, 1)[:F].contiguous()
    kw, ext = {}, [None, None]
    if start == "warm":
        e = np.random.default_rng(N + n).standard_normal((2, 2, N, N))
        kw["ext_init"] = torch.tensor(e, device="cuda").repeat(F // 2 + 1, 1, 1, 1)[:F].contiguous()
        ext = [e[0], e[1]]
    elif start == "hudgin":
        ext = ["hudgin", "hudgin"]
    ph = plan.reconstruct_f64(s, k, **kw)
    assert plan.status() == "FWR_OK"
    for f in {0, F - 1}:
        ref, _ = oracle.reconstruct(base[f % 2], mask, 1.0, k, oracle.FILTER_WIENER, 0.05 ** 2, r0p, L0p, periodic,
                                    ext_init=ext[f % 2], N=N)
        assert within(ph[f].cpu().numpy(), ref, FP64_RMS, FP64_MAX, where="N=%d f=%d" % (N, f))
    for f in range(2, F):
        assert torch.equal(ph[f], ph[f % 2])
    plan.set_ctas(65536)
    one = plan.reconstruct_f64(s, k, **kw)
    assert within(ph[0].cpu().numpy(), one[0].cpu().numpy(), FP64_RMS, FP64_MAX)


def test_cluster_reports_nonfinite_slopes(fwr):
    mask = synth.pupil_mask(16)
    plan = fwr.Plan(mask, 2.0, fwr.LSQ)
    s = torch.zeros((3, 2, 16, 16), dtype=torch.float64, device="cuda")
    s[2, 1, 8, 8] = float("nan")
    plan.reconstruct_f64(s, 1)
    assert plan.status() == "FWR_ERR_NONFINITE"
    assert plan.status() == "FWR_OK"
