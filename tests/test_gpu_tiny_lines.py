"""FP64 transform passes at the lower end of the exponent range: a solve of L_h is
linear, so r 2^-k has to give d 2^-k, down to values whose smaller ones are subnormal.

Tolerance: 1e-12 relative L-infinity as for every FP64 output of the parity tests,
plus 2^-1022, below which results are taken as zero, for each of the N values that the
passes add up.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01475_gb300 import Solver  # noqa: E402


# lines in one warp and in several, radix 4 and 8, adjacent and mirrored pairs
@pytest.mark.parametrize("shape", [(8, 8), (64, 64), (512, 1024), (16, 32, 64), (256, 128, 64)])
@pytest.mark.parametrize("order", [4, 6])
@pytest.mark.parametrize("k", [940, 960, 985, 990])
def test_precond_scaled(oracle, shape, order, k):
    P = oracle.Problem(order, 0.3, 4.0, 0.05, 0.1, 1.0)
    r = np.random.default_rng(k).standard_normal(shape)
    small = np.ldexp(r, -k)
    S = Solver(order, shape, 0.3, 4.0, P.s, P.eps, P.lam)
    d = torch.empty(shape, dtype=torch.float64, device="cuda")
    S.precond_solve(torch.from_numpy(small).cuda(), d)
    ref = oracle.precond4(r, P) if order == 4 else oracle.precond6(r, P)
    err = np.max(np.abs(np.ldexp(d.cpu().numpy(), k) - ref))
    assert err <= 1e-12 * np.max(np.abs(ref)) + r.size * 2.0 ** (k - 1022)
