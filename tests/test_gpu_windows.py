"""Window grids (even, no power of two) of every size class of their kernel:
odd and even half-lengths, two to four threads per line, against the FP64 oracle; and the same
bits for a frame whatever the batch."""

import numpy as np
import pytest

import oracle
from paper_1705_04298_gb300 import synth
from parity_check import FP32_MAX, FP32_RMS, FP64_MAX, FP64_RMS, within

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fwr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04298_gb300 import fwr as m
    m.load()
    return m


@pytest.mark.parametrize("N,n,k,periodic,precision", [
    (18, 16, 2, 0, "fp32"), (18, 11, 1, 1, "fp64"), (20, 14, 3, 0, "fp64"), (26, 24, 2, 2, "fp32"),
    (34, 29, 2, 0, "fp32"), (36, 30, 1, 1, "fp32"), (44, 40, 2, 0, "fp32"), (50, 45, 2, 0, "fp64"),
    (56, 50, 1, 0, "fp32"), (58, 56, 2, 1, "fp32"), (60, 51, 2, 0, "fp32"), (62, 60, 2, 0, "fp32"),
    (62, 60, 1, 0, "fp64")])
def test_window_sizes(fwr, N, n, k, periodic, precision):
    dt = torch.float64 if precision == "fp64" else torch.float32
    tol, mx = (FP64_RMS, FP64_MAX) if precision == "fp64" else (FP32_RMS, FP32_MAX)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    F = 3 * sms + 7  # the other number of threads per line on the smaller grids
    base, _, mask = synth.batch(n, 2, 600 + N, 0.05)
    r0p, L0p = synth.pitch_units(n, 0.15, 25.0)
    plan = fwr.Plan(mask, 1.0, fwr.WIENER, 0.05 ** 2, r0p, L0p, periodic, grid=N)
    call = plan.reconstruct_f64 if precision == "fp64" else plan.reconstruct
    s = torch.tensor(base, dtype=dt, device="cuda").repeat(F // 2 + 1, 1, 1, 1)[:F].contiguous()
    few = call(s[:2].contiguous(), k).clone()
    many = call(s, k)
    assert plan.status() == "FWR_OK"
    for f in range(2):
        ref, _ = oracle.reconstruct(base[f], mask, 1.0, k, oracle.FILTER_WIENER, 0.05 ** 2, r0p, L0p, periodic, N=N)
        assert within(few[f].cpu().numpy(), ref, tol, where="N=%d f=%d" % (N, f))
    assert torch.equal(many, few.repeat(F // 2 + 1, 1, 1)[:F])
    # warm start and extended slopes
    ext0 = torch.tensor(np.random.default_rng(N).standard_normal((1, 2, N, N)), dtype=dt, device="cuda")
    ext = torch.empty_like(ext0)
    ph = call(s[:1].contiguous(), k, ext_init=ext0, ext_out=ext)
    assert torch.equal(ph, call(s[:1].contiguous(), k, ext_init=ext0))
    ref, ref_ext = oracle.reconstruct(base[0], mask, 1.0, k, oracle.FILTER_WIENER, 0.05 ** 2, r0p, L0p, periodic,
                                      ext_init=ext0[0].cpu().double().numpy(), N=N)
    assert within(ph[0].cpu().numpy(), ref, tol, where="N=%d warm" % N)
    assert within(ext[0].cpu().double().numpy(), ref_ext, 10 * tol, 10 * mx,
                  where="N=%d ext" % N)
