"""Warm starts: where Eq. PC precedes the first transform it replaces the last
column of the x slopes and the last row of the y slopes, so what a warm start
holds there does not reach the result (it may be anything, NaN included)."""

import numpy as np
import pytest

import oracle
from paper_1705_04298_gb300 import synth
from parity_check import FP32_RMS, FP64_RMS, within

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fwr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04298_gb300 import fwr as m
    m.load()
    return m


# window grids with odd and even N/2; 128^2 pupils of the generic kernel, and of
# the fused and the cluster kernel (many and few frames)
@pytest.mark.parametrize("N,n,F,precision", [(46, 40, 2, "fp32"), (20, 14, 3, "fp32"), (46, 40, 500, "fp32"),
                                             (26, 20, 2, "fp64"), (128, 110, 2, "fp32"), (128, 91, 2, "fp32"),
                                             (128, 91, 60, "fp32"), (128, 40, 2, "fp32"), (128, 40, 60, "fp32"),
                                             (32, 16, 2, "fp32"), (32, 16, 2, "fp64"), (64, 31, 130, "fp64")])
@pytest.mark.parametrize("k,periodic", [(2, 0), (0, 1)])
@pytest.mark.parametrize("value", [float("nan"), 1e30])
def test_fill_cells_of_a_warm_start_are_replaced(fwr, N, n, F, precision, k, periodic, value):
    dt = torch.float64 if precision == "fp64" else torch.float32
    s, _, mask = synth.batch(n, 1, 70 + n, 0.05)
    plan = fwr.Plan(mask, 1.0, fwr.WIENER, 0.01, 0.6, 100.0, periodic, grid=N)
    call = plan.reconstruct_f64 if precision == "fp64" else plan.reconstruct
    ext = np.random.default_rng(N + n).standard_normal((2, N, N)).astype(np.float32).astype(np.float64)
    ref, _ = oracle.reconstruct(s[0].astype(np.float32).astype(np.float64), mask, 1.0, k, oracle.FILTER_WIENER, 0.01,
                                0.6, 100.0, periodic, ext_init=ext, N=N)
    ext[0, :, N - 1] = ext[1, N - 1, :] = value
    e = torch.tensor(ext, dtype=dt, device="cuda").repeat(F, 1, 1, 1).contiguous()
    x = torch.tensor(s, dtype=torch.float32, device="cuda").to(dt).repeat(F, 1, 1, 1).contiguous()
    ph = call(x, k, ext_init=e)
    assert plan.status() == "FWR_OK"
    assert within(ph[F - 1].cpu().numpy(), ref, FP64_RMS if precision == "fp64" else FP32_RMS, where="N=%d" % N)
    assert torch.equal(ph[0], ph[F - 1])
