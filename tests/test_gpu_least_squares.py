"""The least-squares step (lrdm_apply) at the edges of its forms: FP32 data above
and below the length where it is summed in FP32 pairs, lengths that are and are
not multiples of the vector width, task groups of four directions filled and
ragged, values beyond the range of the pairs, and a singular matrix."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _context(n, kmax):
    from paper_2211_07894_gb300 import Context
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    psi = torch.linalg.qr(torch.randn(ng, 8, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    eps = torch.linspace(-1, 1, 8, device="cuda", dtype=torch.float64)
    return Context([dict(n=n, h=(0.5,) * 3, psi=[psi.float().contiguous()], eps=[eps], n_electrons=8.0, kT=0.01,
                         g=2.0, rho_floor=1e-3, k_max=kmax)], prec="fp32", io_dtype=torch.float32, k_max=kmax)


def _reference(F, V, R, rho, alpha):
    w = 0.125
    F, V, R = F.double(), V.double(), R.double()
    a = torch.linalg.solve(w * (F @ F.T), w * (F @ R))
    res = a @ F - R
    return a, torch.sqrt((res ** 2).sum() / (R ** 2).sum()), rho.double() - alpha * (a @ V)


# 68,921 points: scalar loads, FP32 pairs; 68,880: vector loads, FP32 pairs;
# 59,319 and 13,824: FP64 sums
@pytest.mark.parametrize("n", [(41, 41, 41), (42, 40, 41), (39, 39, 39), (24, 24, 24)])
@pytest.mark.parametrize("K", [1, 3, 4, 7, 15, 16, 17, 40, 64])
def test_apply_against_fp64(n, K):
    ctx = _context(n, 1)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(100 * K + n[0])
    ng = int(np.prod(n))
    for scale in (1.0, 1e22, 1e-18):
        F = (torch.randn(K, 1, ng, generator=gen, device="cuda") * scale).contiguous()
        V = torch.randn(K, 1, ng, generator=gen, device="cuda")
        R = torch.randn(1, ng, generator=gen, device="cuda") * scale
        rho = torch.rand(1, ng, generator=gen, device="cuda")
        out = rho.clone()
        a, s = ctx.apply(0, R, V, F, 0.5, rho=out)
        a_ref, s_ref, rho_ref = _reference(F[:, 0], V[:, 0], R[0], rho[0], 0.5)
        # random columns: condition below 2; pairs round to 2^-48 a product and
        # the sums of K terms to K 2^-48 at most
        tol = 2.0 * max(K, 8) * 2.0 ** -48
        assert float((a - a_ref).abs().max()) <= tol * max(1.0, float(a_ref.abs().max()))
        assert abs(float(s[0] - s_ref)) <= tol * float(s_ref)
        assert float((out[0].double() - rho_ref).abs().max()) <= 2.0 ** -23 * float(rho_ref.abs().max())
        assert ctx.status() == 0


@pytest.mark.parametrize("n", [(41, 41, 41), (24, 24, 24)])
def test_apply_singular_and_nonfinite(n):
    ctx = _context(n, 1)
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    F = torch.randn(3, 1, ng, generator=gen, device="cuda")
    F[2] = F[0]
    V = torch.randn(3, 1, ng, generator=gen, device="cuda")
    R = (0.7 * F[0] - 0.2 * F[1]).contiguous()
    a, s = ctx.apply(0, R, V, F, 0.5)
    assert ctx.status() == 6                                  # pseudo-inverse used
    want = torch.tensor([0.35, -0.2, 0.35], dtype=torch.float64, device="cuda")
    assert float((a - want).abs().max()) < 1e-6               # R is rounded to FP32
    F[1, 0, ng // 2] = float("inf")
    a, s = ctx.apply(0, R, V, F, 0.5)
    assert ctx.status() == 8 and float(a.abs().max()) == 0.0
