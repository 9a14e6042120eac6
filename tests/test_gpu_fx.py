"""FP64 transform passes in block fixed point on the GPU: every line length on
every axis (one, several and part of a warp per line pair; full and narrowed
tiles) against the oracle's preconditioner, and lines that are zero, tiny or
not finite.

Tolerance 1e-12 relative L-infinity, as for every FP64 output of the parity
tests (rounding of a few eps64 per pass, relative to the largest value).
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01475_gb300 import Solver  # noqa: E402

SHAPES = [(8, 8), (8, 1024), (1024, 8), (512, 16), (16, 512), (128, 32), (32, 128), (8, 8, 1024), (8, 1024, 8),
          (1024, 8, 8), (512, 8, 16), (16, 512, 8), (8, 16, 512), (64, 32, 16), (128, 64, 8), (8, 128, 256)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("order", [4, 6])
def test_precond_every_length(oracle, shape, order):
    rng = np.random.default_rng(sum(shape) + order)
    h = 2 * np.pi / 64
    P = oracle.Problem(order, h, 4.0, 0.05, 0.1, 1.0)
    r = rng.standard_normal(shape)
    S = Solver(order, shape, h, 4.0, P.s, P.eps, P.lam)
    d = torch.empty(shape, dtype=torch.float64, device="cuda")
    S.precond_solve(torch.from_numpy(r).cuda(), d)
    ref = oracle.precond4(r, P) if order == 4 else oracle.precond6(r, P)
    assert np.max(np.abs(d.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))


def test_precond_zero_scaled_and_nonfinite_lines():
    shape = (16, 32, 64)
    S = Solver(4, shape, 0.1, 4.0, 0.05, 0.1)
    r = torch.zeros(shape, dtype=torch.float64, device="cuda")
    d = torch.full_like(r, 7.0)
    S.precond_solve(r, d)
    assert torch.all(d == 0)
    # the solve is linear: powers of two scale every intermediate exactly
    r[3, 5, 7], r[8, 1, 2] = 1.0, -0.3
    S.precond_solve(r, d)
    e = torch.empty_like(d)
    for scale in (2.0 ** -600, 2.0 ** 600):
        S.precond_solve(r * scale, e)
        assert torch.equal(e, d * scale)
    r[1, 1, 1] = float("nan")
    S.precond_solve(r, d)
    assert torch.isnan(d).all()
