"""The 3D FP32 warp marches on grids of several strips with a short last one, of one
warp and several per block, of shares that end inside a column: residuals against
the oracle, element by element, and the iteration counts of mixed solves, whose inner
residuals and line searches they are (the FP64 outer residual would hide a wrong
operator in a higher count).

Tolerance of a residual: about 60 terms, each with a rounding of 2^-24 of at most
144 s eps^2 / h^4 max|u| (Laplacian sums), max|u|, or 6 s max|g|^{p-1} / h (fluxes).
Iterations: the mixed solve reduces the residual at the rate of the FP64 one; an
outer step restarts its inner solve, which ends by a rule on the preconditioned
norm, so it is given twice the FP64 count and 10 more.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01475_gb300 import PSD_FP64, PSD_MIXED, Solver, synthetic  # noqa: E402

SHAPES = [(8, 8, 32), (16, 64, 64), (32, 16, 128), (64, 8, 256), (8, 8, 1024), (8, 512, 64)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("p", [3.0, 4.0, 5.0, 6.0])
def test_residual_f32(oracle, shape, p):
    h = 2 * np.pi / 64
    P = oracle.Problem(4, h, p, 0.05, 0.15)
    rng = np.random.default_rng(sum(shape))
    u, f = (0.05 * rng.standard_normal(shape)).astype(np.float32), rng.standard_normal(shape).astype(np.float32)
    S = Solver(4, shape, h, p, P.s, P.eps, precision=PSD_MIXED)
    r = torch.empty(shape, dtype=torch.float32, device="cuda")
    S.residual_f32(torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda(), r)
    v = u.astype(np.float64)
    ref = oracle.residual4(v, f.astype(np.float64), P)
    g = np.sqrt(np.max(sum(c * c for c in oracle.vgrad(v, h))))
    term = max(144 * P.s * P.eps ** 2 / h ** 4, 1.0) * np.max(np.abs(v)) + 6 * P.s * g ** (p - 1) / h + np.max(np.abs(f))
    assert np.max(np.abs(r.cpu().numpy() - ref)) <= 60 * 2.0 ** -24 * term


@pytest.mark.parametrize("shape", [(8, 8, 32), (16, 64, 64), (32, 16, 128), (8, 8, 1024)])
@pytest.mark.parametrize("p", [3.0, 4.0, 5.0, 6.0])
def test_mixed_iterations(shape, p):
    h = 2 * np.pi / 64
    f = torch.from_numpy(synthetic.fourier_field(shape, 2 * np.pi, 4, 31, nmodes=12)).cuda()
    infos = []
    for prec in (PSD_FP64, PSD_MIXED):
        S = Solver(4, shape, h, p, 0.02, 0.1, precision=prec, tol=1e-10, max_iter=5000, max_outer=60)
        u = torch.zeros_like(f)
        infos.append(S.solve(f, u))
    assert infos[1]["status"] == 0 and infos[1]["iters"] <= 2 * infos[0]["iters"] + 10
