"""The least-squares step near the ends of the FP32 range and over long sums: values
just inside and outside the range in which its sums run as compensated FP32 pairs,
coefficients, residuals and densities far below 1, and constant data over many steps of a lane, where rounding errors do not
average out."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _apply(R, V, F, alpha, rho=None, w=0.125):
    from paper_2211_07894_gb300 import binding
    K, n = F.shape
    coef = torch.empty(K, dtype=torch.float64, device="cuda")
    srel = torch.empty(1, dtype=torch.float64, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    code = binding.lrdm_apply_static(R.data_ptr(), V.data_ptr(), F.data_ptr(), binding.DTYPE_F32, K, n, w, alpha,
                                     1e-12, rho.data_ptr() if rho is not None else 0, coef.data_ptr(),
                                     srel.data_ptr(), status.data_ptr())
    assert code == 0
    torch.cuda.synchronize()
    return coef, float(srel), int(status)


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


@pytest.mark.parametrize("f,r,v", [(1e-30, 1e-30, 1.0), (1.0, 1e-32, 1e30), (1e25, 1e-18, 1e30), (1e20, 1e-20, 1e35),
                                   (1e-3, 1e-28, 1.0), (1.0, 1.0, 1e-37)])
@pytest.mark.parametrize("n", [68921, 68880])
def test_update_far_below_one(f, r, v, n):
    """Coefficients of r / f and residuals of size r: s_rel keeps the accuracy it has
    at size 1, the density its FP32 rounding."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    K = 5
    F = torch.randn(K, n, generator=gen, device="cuda") * f
    R = torch.randn(n, generator=gen, device="cuda") * r
    V = torch.randn(K, n, generator=gen, device="cuda") * v
    size = v * r / f
    for alpha in (0.5, 0.0):
        rho = torch.rand(n, generator=gen, device="cuda") * size
        a_ref, s_ref, rho_ref = _reference(R, V, F, rho, alpha)
        if alpha == 0.0:
            rho_ref = a_ref @ V.double()
        out = rho.clone()
        a, s, status = _apply(R, V, F, alpha, out)
        assert status == 0
        tol = 2.0 * 8 * 2.0 ** -48                # as for data of size 1
        assert float((a - a_ref).abs().max()) <= tol * max(r / f, float(a_ref.abs().max()))
        assert abs(s - s_ref) <= tol * s_ref
        # FP32 rounding, the coefficients' error, half the spacing of the denormals
        err = (out.double() - rho_ref).abs()
        assert bool((err <= 2.0 ** -23 * rho_ref.abs() + 2.0 ** -35 * float(rho_ref.abs().max()) + 2.0 ** -149).all())


# 128 steps of every lane with one vector (eight slices): 128 * 128 * 304 * 8 points
@pytest.mark.parametrize("c,d", [(0.7, 0.3), (1.1, 1.9), (0.37, 1.21), (1.7, 0.69)])
def test_constant_columns(c, d):
    """<f, R> / <f, f> of constant f and R.  A lane's pair is
    renormalised at every step and summed over 64 steps at a time: an emulation of
    one lane stays below 6e-14 for either sum, one running pair of 128 steps
    reaches 2e-12."""
    n = 128 * 128 * 304 * 8
    F = torch.full((1, n), c, device="cuda")
    R = torch.full((n,), d, device="cuda")
    a, s, status = _apply(R, F, F, 0.5)
    want = float(np.float64(np.float32(d)) / np.float64(np.float32(c)))
    assert status == 0
    assert abs(float(a[0]) - want) <= 1e-13 * want
    assert s <= 1e-12


@pytest.mark.parametrize("n", [(137, 136, 135), (137, 137, 137)])
def test_second_segment_against_fp64(n):
    """64 directions (one slice): a lane's points outgrow one segment (2.5 million
    points)."""
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n[0])
    F = torch.randn(64, ng, generator=gen, device="cuda")
    V = torch.randn(64, ng, generator=gen, device="cuda")
    R = torch.randn(ng, generator=gen, device="cuda")
    rho = torch.rand(ng, generator=gen, device="cuda")
    a_ref, s_ref, rho_ref = _reference(R, V, F, rho, 0.5)
    out = rho.clone()[None]
    a, s, status = _context_apply(n, R[None], V[:, None].contiguous(), F[:, None].contiguous(), 0.5, out)
    assert status == 0
    tol = 2.0 * 64 * 2.0 ** -48
    assert float((a - a_ref).abs().max()) <= tol * max(1.0, float(a_ref.abs().max()))
    assert abs(s - s_ref) <= tol * s_ref
    assert float((out[0].double() - rho_ref).abs().max()) <= 2.0 ** -23 * float(rho_ref.abs().max())
