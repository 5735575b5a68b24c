"""The 128^2 path with a cluster of CTAs per frame (few frames): bitwise the
one-CTA kernel's phase (kept by an explicit persistent-grid size)."""

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


# both cluster sizes, more frames than run at once, the smallest and largest
# pupils (85 across is the most whose arithmetic this is), odd sizes
@pytest.mark.parametrize("n,F", [(40, 1), (7, 3), (64, 7), (40, 8), (33, 19), (61, 30), (2, 1)])
@pytest.mark.parametrize("periodic,k,start", [(0, 3, "zero"), (1, 2, "hudgin"), (2, 1, "warm"), (0, 0, "zero")])
def test_cluster_matches_one_cta(fwr, n, F, periodic, k, start):
    s, mask = frames(n, F, n + F)
    plan = fwr.Plan(mask, 1.0, fwr.WIENER, 0.01, 0.6, 100.0, periodic, grid=128)
    plan.set_extension(fwr.EXT_HUDGIN if start == "hudgin" else fwr.EXT_ZERO)
    kw = {}
    if start == "warm":
        kw["ext_init"] = torch.randn((F, 2, 128, 128), device="cuda")
    plan.set_ctas(65536)
    ref = plan.reconstruct(s, k, **kw).clone()
    plan.set_ctas(0)
    out = torch.full_like(ref, float("nan"))
    for _ in range(2):
        plan.reconstruct(s, k, out, **kw)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    assert plan.status() == "FWR_OK"


def test_cluster_replays_from_a_cuda_graph(fwr):
    s, mask = frames(40, 2, 3)
    plan = fwr.Plan(mask, 3.2, fwr.LSQ)
    ref = plan.reconstruct(s, 2).clone()
    out = torch.full_like(ref, float("nan"))
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        plan.reconstruct(s, 2, out, stream=stream)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


def test_cluster_on_two_streams(fwr):
    """Nothing is shared between launches: two plans on two streams at once."""
    s, mask = frames(40, 4, 8)
    plans = [fwr.Plan(mask, 3.2, fwr.LSQ) for _ in range(2)]
    ref = plans[0].reconstruct(s, 5).clone()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = [[torch.empty_like(ref) for _ in range(8)] for _ in range(2)]
    for i in range(8):
        for j in range(2):
            plans[j].reconstruct(s, 5, outs[j][i], stream=streams[j])
    torch.cuda.synchronize()
    for o in outs[0] + outs[1]:
        assert torch.equal(o, ref)


def test_cluster_reports_nonfinite_slopes(fwr):
    s, mask = frames(40, 3, 9)
    plan = fwr.Plan(mask, 3.2, fwr.LSQ)
    s[1, 1, 20, 20] = float("nan")
    plan.reconstruct(s, 1)
    assert plan.status() == "FWR_ERR_NONFINITE"
    assert plan.status() == "FWR_OK"


@pytest.mark.parametrize("n", [82, 83, 98, 99, 100, 101, 126])
def test_largest_pupils(fwr, n):
    """Pupils around the limits of the fused kernel's shared memory (82 with all
    tables, 100 with the coefficients in tensor memory): one frame by the
    cluster kernel and many by the fused one with the same bits up to 100, the
    basic kernel beyond; against the FP64 oracle; the extended slopes; and what
    needs all tables stays refused."""
    F = torch.cuda.get_device_properties(0).multi_processor_count + 5
    s, mask = frames(n, F, n)
    plan = fwr.Plan(mask, 1.0, fwr.WIENER, 0.01, 0.6, 100.0, grid=128)
    many = plan.reconstruct(s, 2)
    ext = torch.empty((2, 2, 128, 128), device="cuda")
    two = plan.reconstruct(s[:2].contiguous(), 2, ext_out=ext)
    one = plan.reconstruct(s[:1].contiguous(), 2)
    assert plan.status() == "FWR_OK"
    if n <= 100:
        assert torch.equal(one[0], many[0])
    for f in range(2):
        ref, ref_ext = oracle.reconstruct(s[f].cpu().double().numpy(), mask, 1.0, 2, oracle.FILTER_WIENER, 0.01, 0.6,
                                          100.0, N=128)
        for got in (many[f], two[f]) if f else (many[f], two[f], one[0]):
            assert within(got.cpu().numpy(), ref, FP32_RMS, where="n=%d f=%d" % (n, f))
        assert within(ext[f].cpu().double().numpy(), ref_ext, 10 * FP32_RMS, where="n=%d ext" % n)
    plan.set_extension(fwr.EXT_HUDGIN)
    if n <= 82:
        plan.reconstruct(s[:1].contiguous(), 1)
    else:
        with pytest.raises(fwr.FwrError, match="UNSUPPORTED"):
            plan.reconstruct(s[:1].contiguous(), 1)
