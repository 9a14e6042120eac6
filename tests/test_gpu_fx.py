"""Fixed-point FP64 kernels on the GPU.  Transform passes: every line length on
every axis (one, several and part of a warp per line pair; full and narrowed
tiles) against the oracle's preconditioner, and lines that are zero, tiny or
not finite.  p = 4 stencils in 3D: residuals and PSD iterates on the smallest
column tiles, on several and on grids large enough for the initial scan, with
smooth data (the fixed-point variant), with gradients steeper than its rule
allows (the FP64 variant) and with an offset much larger than the gradients.

Tolerance 1e-12 relative L-infinity, as for every FP64 output of the parity
tests (rounding of a few eps64 per pass, relative to the largest value).
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01475_gb300 import Solver, synthetic  # noqa: E402

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


# Middle passes on mirrored pairs of lines with several outer pairs per block row,
# at radix 4 and 8 and at 512-point lines of four columns per block.
@pytest.mark.parametrize("shape", [(512, 64, 32), (256, 32, 64), (16, 256, 256), (64, 8, 8)])
@pytest.mark.parametrize("order", [4, 6])
def test_precond_mirrored_lines(oracle, shape, order):
    test_precond_every_length(oracle, shape, order)


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


FIELDS = {"smooth": (1.0, 0.0, 0.0), "rough": (0.0, 0.3, 0.0), "steep": (0.0, 40.0, 0.0), "offset": (0.1, 0.0, 100.0)}


def _field(shape, kind, seed):
    smooth, noise, offset = FIELDS[kind]
    u = np.full(shape, offset)
    if smooth:
        u += smooth * synthetic.fourier_field(shape, 2 * np.pi, 4, seed, nmodes=12)
    if noise:
        u += noise * np.random.default_rng(seed).standard_normal(shape)
    return u


@pytest.mark.parametrize("shape", [(8, 8, 32), (16, 8, 64), (64, 64, 64), (16, 128, 128)])
@pytest.mark.parametrize("kind", sorted(FIELDS))
@pytest.mark.parametrize("order", [4, 6])
def test_residual_variants(oracle, shape, kind, order):
    h = 2 * np.pi / shape[-1]
    P = oracle.Problem(order, h, 4.0, 0.1, 0.1, 0.7)
    u, f = _field(shape, kind, 3), _field(shape, "smooth", 4)
    g = _field(shape, "smooth", 5) if order == 6 else None
    if order == 6:
        u += g.mean() - u.mean()
    S = Solver(order, shape, h, 4.0, P.s, P.eps, P.lam)
    r = torch.empty(shape, dtype=torch.float64, device="cuda")
    S.residual(torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda(), None if g is None else torch.from_numpy(g).cuda(), r)
    ref = oracle.residual4(u, f, P) if order == 4 else oracle.residual6(u, f, g, P)
    # the residual of a large offset cancels: its rounding is that of the terms
    scale = max(np.max(np.abs(ref)), np.max(np.abs(u)) * (1.0 + 64.0 * P.s * P.eps ** 2 / h ** 4))
    assert np.max(np.abs(r.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref)) + 1e-15 * scale


@pytest.mark.parametrize("shape", [(8, 8, 32), (16, 16, 64), (64, 64, 64)])
@pytest.mark.parametrize("kind", ["smooth", "rough", "steep"])
@pytest.mark.parametrize("order", [4, 6])
def test_iterates_variants(oracle, shape, kind, order):
    h = 2 * np.pi / shape[-1]
    P = oracle.Problem(order, h, 4.0, 0.1, 0.1, 0.7)
    u0, f = _field(shape, kind, 6), _field(shape, "smooth", 7)
    g = _field(shape, "smooth", 8) if order == 6 else None
    if order == 6:
        u0 += g.mean() - u0.mean()
    iters = 3
    S = Solver(order, shape, h, 4.0, P.s, P.eps, P.lam, tol=0.0, max_iter=iters)
    u = torch.from_numpy(u0).cuda()
    S.solve(torch.from_numpy(f).cuda(), u, None if g is None else torch.from_numpy(g).cuda(), allow_noconv=True)
    _, info = oracle.psd_solve(P, f, u0, g=g, tol=0.0, kmax=iters, record=True)
    ref = info["u"][iters]
    assert np.max(np.abs(u.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))
