"""The least-squares step near the ends of the FP32 range: values just inside and
outside the range in which its sums run as compensated FP32 pairs."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _context_apply(n, R, V, F, alpha, rho):
    from test_gpu_least_squares import _context
    ctx = _context(n, 1)
    a, s = ctx.apply(0, R, V, F, alpha, rho=rho)
    return a, float(s[0]), ctx.status()


def _reference(R, V, F, rho, alpha):
    F, V, R = F.double(), V.double(), R.double()
    sf, sr = float(F.abs().max()), float(R.abs().max())
    F, R = F / sf, R / sr
    a = torch.linalg.solve(F @ F.T, F @ R)
    s = torch.sqrt(((a @ F - R) ** 2).sum() / (R ** 2).sum())
    a = a * (sr / sf)
    return a, float(s), rho.double() - alpha * (a @ V)


@pytest.mark.parametrize("size", [1.1e18, 5e17, 9e16, 6e16])
def test_gram_below_the_upper_end(size):
    """64 columns (one slice of the points, four steps a lane) of values up to 2^60:
    a lane's sum and the sum over its warp stay finite."""
    n = (52, 50, 50)
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(8)
    F = torch.where(torch.rand(64, ng, generator=gen, device="cuda") < 0.5, -size, size)
    F *= 1.0 - 2.0 ** -8 * torch.rand(64, ng, generator=gen, device="cuda")
    R = F[5] * 0.25 + F[7] * torch.rand(ng, generator=gen, device="cuda")
    V = torch.randn(64, ng, generator=gen, device="cuda")
    rho = torch.rand(ng, generator=gen, device="cuda")
    a_ref, s_ref, rho_ref = _reference(R, V, F, rho, 0.5)
    out = rho.clone()[None]
    a, s, status = _context_apply(n, R[None].contiguous(), V[:, None].contiguous(), F[:, None].contiguous(), 0.5, out)
    assert status == 0
    # random columns: condition below 2; 64 sums of products rounded to 2^-48
    tol = 2.0 * 64 * 2.0 ** -48
    assert float((a - a_ref).abs().max()) <= tol * max(1.0, float(a_ref.abs().max()))
    assert abs(s - s_ref) <= tol * s_ref
    assert float((out[0].double() - rho_ref).abs().max()) <= 2.0 ** -23 * float(rho_ref.abs().max())
