"""The FP64 path's rounding error after ten iterations, against the same
equations in numpy's long double (64 or more bits of significand)."""

import numpy as np
import pytest

import oracle
from paper_1705_04298_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REAL, COMPLEX = np.longdouble, np.clongdouble
PI = REAL("3.14159265358979323846264338327950288")


def reference(s, mask, N, iters):
    """Phase (LSQ filter, Eq. PC before each transform) of one frame."""
    n = len(mask)
    off = oracle.pupil_offset(n, N)
    k = np.arange(N)
    turns = (np.outer(k, k) % N).astype(REAL) / N
    F = (np.cos(2 * PI * turns) - 1j * np.sin(2 * PI * turns)).astype(COMPLEX)
    u = np.where(k < N // 2, k, k - N).astype(REAL) / N
    a = np.cos(2 * PI * u) - 1 + 1j * np.sin(2 * PI * u)
    sinc = np.ones(N, REAL)
    sinc[1:] = np.sin(PI * u[1:]) / (PI * u[1:])
    t = sinc * (np.cos(PI * u) + 1j * np.sin(PI * u))
    t[N // 2] = 0
    gx, gy = t[:, None] * a[None, :], a[:, None] * t[None, :]
    g2 = (gx * gx.conj() + gy * gy.conj()).real
    ok = g2 >= 1e-14
    lsq = np.where(ok, 1 / np.where(ok, g2, 1), 0)
    inside = np.zeros((N, N), bool)
    inside[off:off + n, off:off + n] = mask
    meas = np.zeros((2, N, N), REAL)
    meas[:, off:off + n, off:off + n] = s
    x = np.where(inside, meas, 0)
    for it in range(iters + 1):
        x[0, :, N - 1] = -x[0, :, :N - 1].sum(1)
        x[1, N - 1, :] = -x[1, :N - 1, :].sum(0)
        p = (gx.conj() * (F @ x[0] @ F) + gy.conj() * (F @ x[1] @ F)) * lsq / (REAL(N) * N)
        if it == iters:
            return (F.conj() @ p @ F.conj()).real
        x = np.where(inside, meas, np.stack([(F.conj() @ (g * p) @ F.conj()).real for g in (gx, gy)]))


# the bounds: what the direct sums (46^2, 26^2) and the one-CTA kernel (32^2)
# had with twiddles from cos and sin of 2 pi j / N, 1.9e-15, 2.2e-15 and 1.1e-15
@pytest.mark.parametrize("N,n,most", [(46, 40, 1.9e-15), (26, 20, 2.2e-15), (32, 16, 1.1e-15)])
def test_rounding_error_of_ten_iterations(N, n, most):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04298_gb300 import fwr
    sl, _, mask = synth.batch(n, 4, 900 + N, 0.05)
    plan = fwr.Plan(mask, 1.0, fwr.LSQ, grid=N)
    ph = plan.reconstruct_f64(torch.tensor(sl, device="cuda"), 10).cpu().numpy()
    errors = []
    for f in range(len(sl)):
        ref = reference(sl[f].astype(REAL), mask, N, 10)
        d = ph[f] - ref
        d -= d.mean()
        errors.append(float(np.sqrt((d * d).sum() / ((ref - ref.mean()) ** 2).sum())))
    assert np.mean(errors) <= most, errors
