"""Window grids: a frame's phase is the same bits in a batch of any size (many
frames take other numbers of threads per line, so other instantiations of the
kernel), for every number of sums per thread."""

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
    g = torch.Generator(device="cuda").manual_seed(seed)
    mask = synth.pupil_mask(n)
    return torch.randn((F, 2, n, n), generator=g, device="cuda") * torch.tensor(mask, device="cuda"), mask


# 3 to 7 sums per thread in the two-thread form (18 .. 48), 3 or 4 in the other
@pytest.mark.parametrize("N", [18, 22, 24, 28, 30, 38, 40, 46, 48, 54])
@pytest.mark.parametrize("filt,k", [("WIENER", 0), ("LSQ", 2)])
def test_window_frames_are_the_same_bits_in_any_batch(fwr, N, filt, k):
    n = N - 6
    F = 3 * torch.cuda.get_device_properties(0).multi_processor_count + 7
    s, mask = frames(n, F, N)
    plan = fwr.Plan(mask, 1.0, getattr(fwr, filt), 0.01, 0.6, 100.0, grid=N)
    many = plan.reconstruct(s, k)
    few = torch.cat([plan.reconstruct(s[f:f + 4].contiguous(), k) for f in (0, F - 4)])
    assert torch.equal(torch.cat((many[:4], many[F - 4:])), few)
    assert plan.status() == "FWR_OK"
    ref, _ = oracle.reconstruct(s[0].cpu().double().numpy(), mask, 1.0, k, getattr(oracle, "FILTER_" + filt), 0.01, 0.6,
                                100.0, N=N)
    assert within(few[0].cpu().numpy(), ref, FP32_RMS, where="N=%d" % N)
