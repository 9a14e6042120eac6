"""The general-p line search at a root where Newton's method is slow: for 2 < p < 3
q' is not Lipschitz where vertex gradients vanish.  f is chosen so that the first
direction is d = -u0 / a with a = (L_h u0, u0) / (N_h[u0], u0): then the root of
q(alpha) = (N_h[u0 + alpha d] - f, d) is a, where u0 + a d = 0 and every gradient
vanishes.

Tolerance 1e-12: q's sums and the direction carry a few eps64, times up to about 200
for the ratio of the p-term to the linear terms.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01475_gb300 import Solver, synthetic  # noqa: E402


@pytest.mark.parametrize("shape", [(64, 64), (16, 16, 32)])
@pytest.mark.parametrize("p", [2.1, 2.2, 2.5, 3.0, 3.5, 5.0])
@pytest.mark.parametrize("s,eps", [(10.0, 0.01), (100.0, 0.1)])
def test_root_at_vanishing_gradients(oracle, shape, p, s, eps):
    h = 2 * np.pi / shape[-1]
    P = oracle.Problem(4, h, p, s, eps)
    u = synthetic.fourier_field(shape, 2 * np.pi, 4, 3, nmodes=12)
    mu = np.zeros(shape)
    for a, n in enumerate(shape):
        sn = 4 / h ** 2 * np.sin(np.pi * np.arange(n) / n) ** 2
        mu = mu + sn.reshape([-1 if b == a else 1 for b in range(len(shape))])
    Lu = np.fft.ifftn(np.fft.fftn(u) * (1 + s * mu + s * eps ** 2 * mu ** 2)).real
    Nu = oracle.N4(u, P)
    root = (Lu * u).sum() / (Nu * u).sum()
    S = Solver(4, shape, h, p, s, eps, tol=0.0, max_iter=1)
    S.set_history(2)
    S.solve(torch.from_numpy(Nu - Lu / root).cuda(), torch.from_numpy(u).cuda(), allow_noconv=True)
    alpha = S.history()[0][0]
    assert abs(alpha - root) <= 1e-12 * root
