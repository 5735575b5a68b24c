"""Gradients of a few images through the CUDA-core backward kernels (channel
counts that are no multiples of 16): few rows are spread over many CTAs whose
copies and staging warps have no work of their own."""

import numpy as np
import pytest

import oracle
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


def problem(fwr, w, F):
    """Integer inputs and weights of +-1: exact activations, so the FP64
    reference's gradient is that of the same network."""
    rng = np.random.default_rng(100 * w + F)
    parts = []
    for name, ci, co, k in unet.layer_specs(w):
        m = np.zeros((co, k * k * ci))
        for row in m:
            row[rng.choice(len(row), min(4, len(row)), replace=False)] = rng.choice((-1.0, 1.0), min(4, len(row)))
        parts += [m.ravel(), np.zeros(co)]
    params = np.concatenate(parts)
    mask = synth.pupil_mask(40)
    sl = rng.integers(-8, 9, (F, 2, 40, 40)) * (0.25 * mask)
    ext = rng.standard_normal((F, 2, 128, 128)).astype(np.float32)
    plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=128)
    net = fwr.Net(w, F, params)
    return plan, net, torch.tensor(sl, dtype=torch.float32, device="cuda"), torch.tensor(ext, device="cuda"), sl, ext, \
        params, mask


def bf16(x):
    return torch.tensor(np.asarray(x)).to(torch.bfloat16).double().numpy()


# FP32 sums of 14 layers, 8e-8 to 2e-7 of a layer's gradient: 1e-6
@pytest.mark.parametrize("w,F", [(1, 1), (1, 5), (2, 3), (3, 1), (3, 10), (5, 2), (7, 1), (12, 3), (20, 1)])
def test_gradients_match_reference(fwr, w, F):
    plan, net, s, e, sl, ext, params, mask = problem(fwr, w, F)
    loss, g = net.gradients(plan, s, e)
    off = oracle.pupil_offset(40, 128)
    x = bf16(np.stack([unet.net_input(v, mask, off) for v in sl]))
    t, lm = (np.stack(v) for v in zip(*(unet.net_target(v.astype(np.float64), mask, off) for v in ext)))
    out, cache = unet.forward(params, x, w, store=bf16)
    ref_loss, dout = unet.loss_and_grad(out, t, lm)
    ref = unet.backward(params, cache, dout, w)
    assert abs(loss - ref_loss) <= 1e-5 * ref_loss
    at = 0
    for name, ci, co, k in unet.layer_specs(w):
        m = co * k * k * ci + co
        a, b = g[at:at + m], ref[at:at + m]
        at += m
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b), name


def test_one_image_of_a_narrow_network_takes_no_longer_than_of_a_wide_one(fwr):
    """488 us at width 3 against 434 at width 16, where the tensor cores do the
    backward pass; 640 while one image's rows went to one CTA per layer."""
    def best(w):
        plan, net, s, e = problem(fwr, w, 1)[:4]
        times = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                net.gradients(plan, s, e)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    assert best(3) <= 1.35 * best(16)
