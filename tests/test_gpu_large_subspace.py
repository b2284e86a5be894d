"""A k-point subspace of 32,768 complex states: 65,536 rows of the stacked
operand, more than a grid's second dimension can count."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, H, KT = (4, 4, 4), 0.5, 0.01


def _forward(psi, eps, V):
    from paper_2211_07894_gb300 import KpContext
    ctx = KpContext(N, (H,) * 3, [psi[0]], [psi[1]], [eps], [1.0], 16.0, KT, rho_floor=1e-3, prec="fp32",
                    io_dtype=torch.float32, k_max=1)
    F, dmu = ctx.gateaux(V)
    out = F[0].double().clone(), dmu.clone()
    ctx.close()
    return out


def test_rows_beyond_65535():
    """Sixteen states that count, at both ends of the subspace; the others are zero
    columns at eigenvalues where the Fermi function and its slope vanish."""
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("60 GB")
    ng = int(np.prod(N))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    few = torch.randn(2, ng, 16, generator=gen, device="cuda") * 0.3
    eps16 = torch.linspace(-0.2, 0.2, 16, device="cuda", dtype=torch.float64)
    V = torch.randn(1, ng, generator=gen, device="cuda")
    want, mu = _forward([few[0].contiguous(), few[1].contiguous()], eps16, V)
    ns = 32768
    psi = torch.zeros(2, ng, ns, device="cuda")
    eps = torch.full((ns,), 50.0, device="cuda", dtype=torch.float64)
    at = torch.cat([torch.arange(8), torch.arange(ns - 8, ns)]).cuda()
    psi[:, :, at] = few
    eps[at] = eps16
    got, mu2 = _forward([psi[0].contiguous(), psi[1].contiguous()], eps, V)
    # the same FP32 products; sums of 64 and 16 terms in another order
    assert float((got - want).abs().max()) <= 2.0 ** -16 * float(want.abs().max())
    assert float((mu2 - mu).abs().max()) <= 2.0 ** -16 * max(1.0, float(mu.abs().max()))
