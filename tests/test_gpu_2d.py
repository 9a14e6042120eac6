"""The 2D marching kernels (a warp per strip of cells, periodic wrap inside the
strip): residuals and PSD iterates against the oracle on grids of one strip,
of several with a short last one, narrower than a strip and at the widths
where a lane takes two cells (FP32), for every vertex-factor kind and mode.

FP64 tolerance 1e-12 relative L-infinity as in the parity tests; FP32 residuals:
each value sums about 30 terms of at most 64 s eps^2 / h^4 max|u|, with
rounding 2^-24 each: 30 2^-24 of the largest term.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01475_gb300 import PSD_MIXED, Solver, synthetic  # noqa: E402

SHAPES = [(8, 8), (64, 16), (16, 32), (8, 64), (32, 128), (16, 256), (256, 8), (8, 512), (8, 1024), (1024, 32)]


def dev(a):
    return torch.from_numpy(a).cuda()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("p", [3.0, 4.0, 6.0, 5.0])
def test_residual_and_iterates(oracle, shape, p):
    h = 2 * np.pi / 64
    P = oracle.Problem(4, h, p, 0.05, 0.15)
    rng = np.random.default_rng(shape[0] + 3 * shape[1])
    u, f = 0.3 * rng.standard_normal(shape), rng.standard_normal(shape)
    S = Solver(4, shape, h, p, P.s, P.eps, tol=0.0, max_iter=3)
    r = torch.empty(shape, dtype=torch.float64, device="cuda")
    l2, linf = S.residual(dev(u), dev(f), None, r)
    ref = oracle.residual4(u, f, P)
    assert np.max(np.abs(r.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))
    assert abs(l2 - oracle.norm2(ref, h)) <= 1e-12 * l2 and abs(linf - np.max(np.abs(ref))) <= 1e-12 * linf
    x = dev(np.zeros(shape))
    fs = synthetic.fourier_field(shape, 2 * np.pi, 3, 9, nmodes=8)
    S.solve(dev(fs), x, allow_noconv=True)
    _, info = oracle.psd_solve(P, fs, np.zeros(shape), tol=0.0, kmax=3, record=True)
    assert np.max(np.abs(x.cpu().numpy() - info["u"][3])) <= 1e-12 * np.max(np.abs(info["u"][3]))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("offset", [0, 1])  # offset 1: float32 arrays aligned to 4 bytes only
def test_residual_f32(oracle, shape, offset):
    h = 2 * np.pi / 64
    P = oracle.Problem(4, h, 4.0, 0.05, 0.15)
    rng = np.random.default_rng(shape[0] + shape[1])
    u, f = (0.3 * rng.standard_normal(shape)).astype(np.float32), rng.standard_normal(shape).astype(np.float32)
    n = u.size
    buf = torch.zeros(3, n + 2, dtype=torch.float32, device="cuda")
    ut, ft, rt = (b[offset:offset + n].view(shape) for b in buf)
    ut.copy_(dev(u))
    ft.copy_(dev(f))
    S = Solver(4, shape, h, 4.0, P.s, P.eps, precision=PSD_MIXED)
    S.residual_f32(ut, ft, rt)
    ref = oracle.residual4(u.astype(np.float64), f.astype(np.float64), P)
    term = max(64.0 * P.s * P.eps ** 2 / h ** 4, 1.0) * np.max(np.abs(u)) + np.max(np.abs(ref))
    assert np.max(np.abs(rt.cpu().numpy() - ref)) <= 30 * 2.0 ** -24 * term


@pytest.mark.parametrize("shape", [(8, 16), (64, 64), (32, 256), (16, 1024)])
@pytest.mark.parametrize("p", [3.0, 4.0, 6.0])
def test_mixed_solve(oracle, shape, p):
    """The FP32 kernels with a base iterate (inner residual and line search)."""
    h = 2 * np.pi / max(shape)
    P = oracle.Problem(4, h, p, 0.01, 0.15)
    f = synthetic.fourier_field(shape, 2 * np.pi, 3, 21, nmodes=8)
    S = Solver(4, shape, h, p, P.s, P.eps, precision=PSD_MIXED, tol=1e-10, max_iter=5000, max_outer=60)
    u = dev(np.zeros(shape))
    S.solve(dev(f), u)
    r = oracle.residual4(u.cpu().numpy(), f, P)
    assert oracle.norm2(r, h) < 1e-10 * 1.05
