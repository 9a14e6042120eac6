"""The FP64 step size where the symbol of L_h is almost all s mu (large s, small
eps): for a field so small that the nonlinear terms vanish, the first step from
u0 = 0 is alpha = (r, d) / (L d, d) with L the linear part of N_h, here from sums
of positive terms over the spectrum.

Tolerance 1e-13: both sums are of positive terms, each within a few eps64.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01475_gb300 import Solver  # noqa: E402


# 2D (adjacent pairs of lines) and 3D (mirrored pairs and not)
@pytest.mark.parametrize("shape", [(128, 128), (64, 32, 32), (8, 8, 64)])
@pytest.mark.parametrize("order", [4, 6])
@pytest.mark.parametrize("s,eps", [(0.1, 0.1), (1.0, 1e-4), (1e4, 1e-4), (1e8, 1e-8)])
def test_first_step(shape, order, s, eps):
    h, lam = 2 * np.pi / 64, 1e-3
    f = np.random.default_rng(5).standard_normal(shape)
    f = 1e-60 * (f - f.mean())  # the mean, whose symbol is 1, would outweigh the rest
    S = Solver(order, shape, h, 4.0, s, eps, lam, tol=0.0, max_iter=1)
    S.set_history(4)
    zero = torch.zeros(shape, dtype=torch.float64, device="cuda")
    S.solve(torch.from_numpy(f).cuda(), zero.clone(), zero if order == 6 else None, allow_noconv=True)
    alpha = S.history()[0][0]
    mu = np.zeros(shape, dtype=np.longdouble)
    for a, n in enumerate(shape):
        sn = np.sin(np.pi * np.arange(n, dtype=np.longdouble) / n)
        mu = mu + (4 / np.longdouble(h) ** 2 * sn * sn).reshape([-1 if b == a else 1 for b in range(len(shape))])
    r2 = np.abs(np.fft.fftn(f * 1e60)).astype(np.longdouble) ** 2
    if order == 4:
        lin = 1 + np.longdouble(s) * np.longdouble(eps) ** 2 * mu ** 2
    else:
        r2, mu = r2.ravel()[1:], mu.ravel()[1:]  # without the mean
        lin = np.longdouble(s) * lam + 1 / mu + np.longdouble(s) * np.longdouble(eps) ** 2 * mu ** 2
    L = lin + np.longdouble(s) * mu
    ref = (r2 / L).sum() / (lin * r2 / L ** 2).sum()
    assert abs(alpha - ref) <= 1e-13 * ref
