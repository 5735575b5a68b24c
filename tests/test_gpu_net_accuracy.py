"""Rounding error of the network's gradients. With integer inputs and weights of
+-1 every activation is exact, so the FP64 reference network's gradient differs
by the loss's and the backward pass's FP32 rounding alone."""

import numpy as np
import pytest

import oracle
from oracle import unet
from paper_1705_04298_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def bf16(x):
    return torch.tensor(np.asarray(x)).to(torch.bfloat16).double().numpy()


def layer_errors(fwr, F, seed, w=16, n=40):
    rng = np.random.default_rng(1000 * seed + F)
    params = []
    for name, ci, co, k in unet.layer_specs(w):
        m = np.zeros((co, k * k * ci))
        for row in m:
            row[rng.choice(k * k * ci, 4, replace=False)] = rng.choice((-1.0, 1.0), 4)
        params += [m.ravel(), np.zeros(co)]
    params = np.concatenate(params)
    mask = synth.pupil_mask(n)
    sl = rng.integers(-8, 9, (F, 2, n, n)) * (0.25 * mask)
    ext = rng.standard_normal((F, 2, 128, 128)).astype(np.float32)
    plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=128)
    _, g = fwr.Net(w, F, params).gradients(plan, torch.tensor(sl, dtype=torch.float32, device="cuda"),
                                           torch.tensor(ext, device="cuda"))
    off = oracle.pupil_offset(n, 128)
    x = bf16(np.stack([unet.net_input(s, mask, off) for s in sl]))
    t, lm = (np.stack(v) for v in zip(*(unet.net_target(e.astype(np.float64), mask, off) for e in ext)))
    out, cache = unet.forward(params, x, w, store=bf16)
    ref = unet.backward(params, cache, unet.loss_and_grad(out, t, lm)[1], w)
    errors, at = [], 0
    for name, ci, co, k in unet.layer_specs(w):
        m = co * k * k * ci + co
        errors.append(np.linalg.norm(g[at:at + m] - ref[at:at + m]) / np.linalg.norm(ref[at:at + m]))
        at += m
    return errors


# the bound: the error of scalar FP32 sums (one thread per weight) on 3 images,
# mean over layers; on 6 they had 9.3e-8
@pytest.mark.parametrize("F", [3, 6])
def test_gradients_are_no_less_accurate_than_scalar_sums(F):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04298_gb300 import fwr
    assert np.mean([layer_errors(fwr, F, seed)[:14] for seed in range(1, 7)]) <= 8.2e-8
