"""FP64 residuals and solves of fields far below one, on grids large enough for
the fixed-point variant's scan (2^18 cells): no value may be taken for zero,
and a solve from u0 = 0 must know its first iterate's scale.

Tolerance 1e-12 relative L-infinity, as for every FP64 output of the parity
tests; u and f scale together, so it is relative at every magnitude.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01475_gb300 import Solver, synthetic  # noqa: E402

SHAPES = [(512, 512), (64, 64, 64)]


def dev(a):
    return torch.from_numpy(a).cuda()


# across the FP32 range's end (2^-126), where squares leave it (2^-70), at the
# largest scale of the variant (2^-145) and far below it
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("exponent", [-30, -42, -72, -125, -130, -148, -400, 62, 130])
def test_residual(oracle, shape, exponent):
    h = 2 * np.pi / shape[-1]
    P = oracle.Problem(4, h, 4.0, 0.1, 0.1)
    u = np.ldexp(np.random.default_rng(3).standard_normal(shape), exponent)
    f = np.ldexp(np.random.default_rng(4).standard_normal(shape), exponent)
    S = Solver(4, shape, h, 4.0, P.s, P.eps)
    r = torch.empty(shape, dtype=torch.float64, device="cuda")
    l2, linf = S.residual(dev(u), dev(f), None, r)
    ref = oracle.residual4(u, f, P)
    assert np.max(np.abs(r.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))
    assert abs(linf - np.max(np.abs(ref))) <= 1e-12 * linf


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("exponent", [-20, -66, -110])
def test_solve_from_zero(oracle, shape, exponent):
    h = 2 * np.pi / shape[-1]
    P = oracle.Problem(4, h, 4.0, 0.01, 0.1)
    f = np.ldexp(synthetic.fourier_field(shape, 2 * np.pi, 6, 11, nmodes=12), exponent)
    iters = 3
    S = Solver(4, shape, h, 4.0, P.s, P.eps, tol=0.0, max_iter=iters)
    u = dev(np.zeros(shape))
    S.solve(dev(f), u, allow_noconv=True)
    _, info = oracle.psd_solve(P, f, np.zeros(shape), tol=0.0, kmax=iters, record=True)
    ref = info["u"][iters]
    assert np.max(np.abs(u.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))
