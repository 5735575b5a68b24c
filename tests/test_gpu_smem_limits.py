"""A kernel's shared-memory limit belongs to the function on the device, not
to a plan, batch or network: objects of different sizes that share a kernel
run in any order and from several threads."""

import threading

import numpy as np
import pytest

from oracle import unet
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


def slopes(n, F, seed):
    mask = synth.pupil_mask(n)
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((F, 2, n, n), generator=g, device="cuda") * torch.tensor(mask, device="cuda"), mask


def at_once(calls, times):
    """Each of `calls` `times` times in a thread of its own; the first error is raised."""
    errors = []
    start = threading.Barrier(len(calls))

    def work(call):
        try:
            start.wait()
            for _ in range(times):
                call()
        except Exception as e:  # noqa: BLE001  (re-raised below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def net_problem(fwr, w, F):
    n = 40
    s, mask = slopes(n, F, w)
    plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=128)
    net = fwr.Net(w, F, unet.init_params(w, w))
    return plan, net, s, torch.randn((F, 2, 128, 128), device="cuda")


def test_gradients_of_two_networks_from_two_threads(fwr):
    """The layers of a backward pass need different sizes of one kernel."""
    runs = []
    for w in (16, 32):
        plan, net, s, e = net_problem(fwr, w, 4)
        runs.append((plan, net, s, e, net.gradients(plan, s, e), torch.cuda.Stream()))
    torch.cuda.synchronize()

    def call(plan, net, s, e, ref, stream):
        loss, g = net.gradients(plan, s, e, stream=stream)
        assert loss == ref[0] and np.array_equal(g, ref[1])

    at_once([lambda r=r: call(*r) for r in runs], 300)


def test_few_frames_of_several_pupils_from_several_threads(fwr):
    """256^2 plans of different pupils need different sizes of one kernel."""
    runs = []
    for n in (205, 70, 40, 180, 30, 100, 60, 50):
        s, mask = slopes(n, 1, n)
        plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=256)
        ref = plan.reconstruct(s, 0).clone()
        runs.append((plan, s, ref, torch.empty_like(ref), torch.cuda.Stream()))
    torch.cuda.synchronize()

    def call(plan, s, ref, out, stream):
        plan.reconstruct(s, 0, out, stream=stream)
        with torch.cuda.stream(stream):
            assert torch.equal(out, ref)

    at_once([lambda r=r: call(*r) for r in runs], 1500)


@pytest.mark.parametrize("shape", [1, 2])
def test_static_scratch_after_a_smaller_plan(fwr, shape):
    s, mask = slopes(200, 2, 5)
    plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=256)
    plan.set_shape(shape)
    ref = plan.reconstruct_static(s, 1, ctas=2).clone()
    small, smask = slopes(60, 2, 6)
    other = fwr.Plan(smask, 1.0, fwr.LSQ, grid=256)
    other.set_shape(shape)
    other.set_ctas(2)
    other.reconstruct(small, 1)
    assert torch.equal(plan.reconstruct_static(s, 1, ctas=2), ref)


@pytest.mark.parametrize("conv", ["NET_CONV_AUTO", "NET_CONV_SIMT"])
def test_network_after_a_narrower_one(fwr, conv):
    plan, net, s, e = net_problem(fwr, 32, 2)
    net.set_conv(getattr(fwr, conv))
    ref = net.forward(plan, s).clone()
    loss, g = net.gradients(plan, s, e)
    fwr.Net(16, 2).close()
    fwr.Net(4, 2).close()
    assert torch.equal(net.forward(plan, s), ref)
    loss2, g2 = net.gradients(plan, s, e)
    assert loss == loss2 and np.array_equal(g, g2)


@pytest.mark.parametrize("shape", [1, 2])
def test_batch_after_a_smaller_one(fwr, shape):
    def batch(n):
        s, mask = slopes(n, 2, n)
        plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=256)
        out = torch.empty((2, 256, 256), device="cuda")
        b = fwr.Batch([plan], [0, 0], 1)
        b.set_shape(shape)
        return b, s, out, fwr.Batch.pointer_table(list(s)), fwr.Batch.pointer_table(list(out))

    b, s, out, sp, pp = batch(200)
    b.run(sp, pp)
    torch.cuda.synchronize()
    ref = out.clone()
    batch(60)
    out.zero_()
    b.run(sp, pp)
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


def test_generic_kernel_of_several_pupils_from_several_threads(fwr):
    """128^2 pupils above 100 lenslets run the generic kernel, whose size
    depends on the pupil."""
    runs = []
    for n in (126, 101, 110, 103):
        s, mask = slopes(n, 1, n)
        plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=128)
        ref = plan.reconstruct(s, 0).clone()
        runs.append((plan, s, ref, torch.empty_like(ref), torch.cuda.Stream()))
    torch.cuda.synchronize()

    def call(plan, s, ref, out, stream):
        plan.reconstruct(s, 0, out, stream=stream)
        with torch.cuda.stream(stream):
            assert torch.equal(out, ref)

    at_once([lambda r=r: call(*r) for r in runs], 2000)
