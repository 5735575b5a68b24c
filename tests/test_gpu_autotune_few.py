"""What the tuner chooses for one number of frames leaves calls of fewer frames
on the paths that share a frame between SMs."""

import json

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


def test_caps_that_no_launch_reaches_are_not_chosen(fwr):
    """100 frames on 128^2 are 100 CTAs whether the cap is 114 or none."""
    F = 100
    s = torch.randn((F, 2, 40, 40), device="cuda")
    out = torch.empty((F, 128, 128), device="cuda")
    for _ in range(6):
        plan = fwr.Plan(synth.pupil_mask(40), 3.2, fwr.LSQ)
        assert plan.autotune(s, 1, out, None)[1] in (0, 76)


def tuned(fwr, path, N, n, F, **changed):
    """A plan tuned from a cache entry of F frames with other values."""
    mask = synth.pupil_mask(n)
    s = torch.randn((F, 2, n, n), device="cuda")
    out = torch.empty((F, N, N), device="cuda")
    fwr.Plan(mask, 1.0, fwr.LSQ, grid=N).autotune(s, 1, out, path)
    e = json.loads(path.read_text().splitlines()[0])
    e.update(changed)
    path.write_text(json.dumps(e) + "\n")
    plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=N)
    assert plan.autotune(s, 1, out, path) == (e["shape"], e["ctas"])
    return plan, mask


def test_fewer_frames_than_tuned_keep_their_path(fwr, tmp_path):
    """On 32^2 the FP64 kernels for few and for many frames differ in rounding,
    which tells them apart; on 256^2 only their times do."""
    plan, mask = tuned(fwr, tmp_path / "a", 32, 16, 200, ctas=76)
    s = torch.randn((3, 2, 16, 16), device="cuda", dtype=torch.float64)
    fresh = fwr.Plan(mask, 1.0, fwr.LSQ, grid=32)
    few = fresh.reconstruct_f64(s, 3).clone()
    fresh.set_ctas(76)
    assert not torch.equal(fresh.reconstruct_f64(s, 3), few)
    assert torch.equal(plan.reconstruct_f64(s, 3), few)
    plan.set_ctas(76)  # the caller's own value holds for every call
    assert not torch.equal(plan.reconstruct_f64(s, 3), few)


@pytest.mark.parametrize("N,n,changed", [(256, 128, {"ctas": 76}), (256, 128, {"shape": 1}), (128, 40, {"ctas": 76})])
def test_fewer_frames_than_tuned_keep_their_speed(fwr, tmp_path, N, n, changed):
    """One frame takes 142 us by a team of CTAs and 398 by one (256^2), 16 and
    41 us on 128^2: with the tuned plan no more than 1.5 times the fresh plan's."""
    plan, mask = tuned(fwr, tmp_path / "a", N, n, 200, **changed)
    s = torch.randn((1, 2, n, n), device="cuda")
    out = torch.empty((1, N, N), device="cuda")

    def best(p):
        times = []
        for _ in range(30):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(8):
                p.reconstruct(s, 5, out)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    assert best(plan) <= 1.5 * best(fwr.Plan(mask, 1.0, fwr.LSQ, grid=N))


def test_cache_entries_of_other_kernels_are_not_taken(fwr, tmp_path):
    """A line without the kernels' revision in its key (an earlier library's,
    timed on other kernels) is not applied; the call times its own."""
    F, n = 8, 40
    mask = synth.pupil_mask(n)
    s = torch.randn((F, 2, n, n), device="cuda")
    out = torch.empty((F, 128, 128), device="cuda")
    cache = tmp_path / "a"
    fwr.Plan(mask, 1.0, fwr.LSQ, grid=128).autotune(s, 1, out, cache)
    e = json.loads(cache.read_text())
    e["key"] = "|".join(p for p in e["key"].split("|") if not p.startswith("kern"))
    e["ctas"] = 5
    cache.write_text(json.dumps(e) + "\n")
    plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=128)
    assert plan.autotune(s, 1, out, cache)[1] == 0
    assert len(cache.read_text().splitlines()) == 2
