"""The scan that bounds u and its gradients before a fixed-point residual: one
point that stands out of a small field, at the corners and seams of the scan's rows,
planes and chunks.  A point that the scan missed would overflow the fixed-point
range.  The values are small enough for the fixed-point variant's rule.

Tolerance 1e-12 relative L-infinity, as for every FP64 output of the parity tests.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1607_01475_gb300 import Solver, synthetic  # noqa: E402


# one, four and eight rows per thread; eight rows that are the whole axis
@pytest.mark.parametrize("shape", [(512, 512), (1024, 1024), (64, 64, 64), (128, 128, 128), (128, 256, 128), (1024, 8, 512)])
@pytest.mark.parametrize("offset", [0, 1])  # 1: u aligned to 8 bytes only
def test_outstanding_point(oracle, shape, offset):
    h = 2 * np.pi / shape[-1]
    P = oracle.Problem(4, h, 4.0, 0.1, 0.1)
    base = 0.01 * synthetic.fourier_field(shape, 2 * np.pi, 4, 3, nmodes=6)
    S = Solver(4, shape, h, 4.0, P.s, P.eps)
    buf = torch.zeros(base.size + 2, dtype=torch.float64, device="cuda")
    u = buf[offset:offset + base.size].view(shape)
    f, r = torch.zeros(shape, dtype=torch.float64, device="cuda"), torch.empty(shape, dtype=torch.float64, device="cuda")
    for at in (tuple(0 for _ in shape), tuple(n - 1 for n in shape), tuple(n // 2 - 1 for n in shape),
               tuple((7, 8, 3)[k] % n for k, n in enumerate(shape[::-1]))[::-1]):
        x = base.copy()
        x[at] += 0.3
        u.copy_(torch.from_numpy(x))
        S.residual(u, f, None, r)
        ref = oracle.residual4(x, np.zeros(shape), P)
        assert np.max(np.abs(r.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))
