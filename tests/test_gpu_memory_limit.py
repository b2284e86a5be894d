"""Contexts near the device's limit: where the buffers that only buy speed (several
row ranges of the projections, blocks of small buffers) do not fit, the context is
made without them and answers the same."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, K = (20, 20, 20), 64


def _make(kind, psi, im, eps):
    from paper_2211_07894_gb300 import Context, KpContext
    ns = psi.shape[1]
    if kind == "kp":
        return KpContext(N, (0.5,) * 3, [psi, im, psi], [im, psi, im], [eps] * 3, [0.25, 0.5, 0.25], 0.9 * ns, 0.05,
                         rho_floor=1e-3, prec="fp32", io_dtype=torch.float32, k_max=K)
    return Context([dict(n=N, h=(0.5,) * 3, psi=[psi], eps=[eps], n_electrons=0.9 * ns, kT=0.05, g=2.0,
                         rho_floor=1e-3, k_max=K)], prec="fp32", io_dtype=torch.float32, k_max=K)


# projections of 64 directions at four ranges: 400 MB for X and for Gbar (a
# point's Gram), 100 MB at one
@pytest.mark.parametrize("kind,ns,left", [("real", 640, 600), ("kp", 320, 700)])
def test_fewer_ranges_where_memory_is_short(kind, ns, left):
    ng = int(np.prod(N))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(12)
    psi = (torch.linalg.qr(torch.randn(ng, ns, generator=gen, device="cuda", dtype=torch.float64))[0]
           / 0.5 ** 1.5).float().contiguous()
    im = (0.5 * psi.flip(1)).contiguous()
    eps = torch.linspace(-1, 1, ns, device="cuda", dtype=torch.float64)
    V = torch.randn((K, ng) if kind == "kp" else (K, 1, ng), generator=gen, device="cuda")
    F = torch.empty_like(V)
    dmu = torch.empty(K, dtype=torch.float64, device="cuda")

    def run():
        ctx = _make(kind, psi, im, eps)
        ctx.gateaux(V if kind == "kp" else [V], out=F if kind == "kp" else [F], dmu=dmu)
        torch.cuda.synchronize()
        ctx.close()

    run()
    want, mu = F.cpu(), dmu.cpu()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    F.fill_(float("nan"))
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (left << 20), dtype=torch.uint8, device="cuda")
    try:
        run()
    finally:
        del filler
        torch.cuda.empty_cache()
    # the same FP32 sums of 8,000 rows over one range in place of four
    assert float((F.cpu() - want).abs().max()) <= 2.0 ** -14 * float(want.abs().max())
    assert float((dmu.cpu() - mu).abs().max()) <= 2.0 ** -14 * float(mu.abs().max())
