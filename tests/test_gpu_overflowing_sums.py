"""Results beyond the FP32 range: where the density response overflows FP32 the
answer is the infinity of its sign, as an FP32 or FP64 sum gives it, and no other
point is affected."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, H, KT, NS = (12, 11, 10), 0.5, 0.02, 4


def inputs():
    """Columns of size 100, so that the last product alone leaves the range."""
    rng = np.random.default_rng(6)
    ng = int(np.prod(N))
    psi = 100.0 * np.linalg.qr(rng.standard_normal((ng, NS)))[0] / H ** 1.5
    x = np.arange(N[0]) * (2 * np.pi / N[0])
    v = np.broadcast_to(np.cos(x)[:, None, None], N).reshape(-1) + 0.3 * rng.standard_normal(ng)
    return psi, np.linspace(-0.01, 0.01, NS), v


def _forward(kind, prec, scale):
    from paper_2211_07894_gb300 import Context, KpContext
    io = torch.float64 if prec == "fp64" else torch.float32
    psi, eps, v = inputs()
    psi = torch.as_tensor(psi, dtype=io, device="cuda")
    eps = torch.as_tensor(eps, device="cuda")
    v = torch.as_tensor(v[None] * scale, dtype=io, device="cuda")
    rho = torch.ones(1, psi.shape[0], device="cuda", dtype=io)
    if kind == "kp":
        ctx = KpContext(N, (H,) * 3, [psi], [torch.zeros_like(psi)], [eps], [1.0], float(NS), KT, rho=rho[0],
                        prec=prec, io_dtype=io, k_max=1)
        return ctx.gateaux(v)[0][0].double()
    ctx = Context([dict(n=N, h=(H,) * 3, psi=[psi], eps=[eps], n_electrons=float(NS), kT=KT, g=2.0, rho=[rho[0]],
                        k_max=1)], prec=prec, io_dtype=io, k_max=1)
    return ctx.gateaux([v[None]])[0][0][0, 0].double()


@pytest.mark.parametrize("kind,prec", [("real", "fp32"), ("kp", "fp32"), ("kp", "tf32"), ("kp", "bf16x3")])
def test_overflow_is_infinite(kind, prec):
    top = float(torch.finfo(torch.float32).max)
    unit = _forward(kind, "fp64", 1.0)
    # the largest response at 1.5 times the FP32 range: below 0.3 of it no partial
    # sum leaves it, and above it none goes the other way
    scale = 1.5 * top / float(unit.abs().max())
    ref = unit * scale
    got = _forward(kind, prec, scale)
    over, under = ref.abs() > 1.1 * top, ref.abs() < 0.3 * top
    assert int(over.sum()) > 0 and int(under.sum()) > 0
    assert bool((got[over] == torch.sign(ref[over]) * float("inf")).all())
    # operands of 11 bits at worst: a hundredth of the largest value
    assert float((got[under] - ref[under]).abs().max()) <= 0.02 * top
