"""A forward call replayed from its graph after another forward with other row
ranges (an adaptive-rank step, one direction at a time) ran on the same context:
the adjoint and the projections that follow read X with the replayed call's
ranges, as they do on a context without graphs."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _context(n, ns, K, prec, io, graph):
    from paper_2211_07894_gb300 import Context
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(ns)
    psi = torch.linalg.qr(torch.randn(ng, ns, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    eps = torch.linspace(-1, 1, ns, device="cuda", dtype=torch.float64)
    return Context([dict(n=n, h=(0.5,) * 3, psi=[psi.to(io).contiguous()], eps=[eps], n_electrons=0.9 * ns, kT=0.05,
                         g=2.0, rho_floor=1e-3, k_max=K)], prec=prec, io_dtype=io, k_max=K, use_graph=graph)


# 16^3 / 32, FP64: 38 ranges at K = 4, 63 at K = 1; 24^3 / 200: other tiles and counts
@pytest.mark.parametrize("prec", ["fp64", "fp32", "tf32", "bf16x3"])
@pytest.mark.parametrize("n,ns,K", [((16, 16, 16), 32, 4), ((24, 24, 24), 200, 6)])
def test_replay_after_another_forward(prec, n, ns, K):
    io = torch.float64 if prec == "fp64" else torch.float32
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    V = torch.randn(K, 1, ng, generator=gen, device="cuda", dtype=io)
    R = torch.randn(1, ng, generator=gen, device="cuda", dtype=io)
    fbar = torch.randn(K, 1, ng, generator=gen, device="cuda", dtype=io)
    torch.cuda.synchronize()
    got = []
    for graph in (False, True):
        with torch.cuda.stream(torch.cuda.Stream()):
            ctx = _context(n, ns, K, prec, io, graph)
            F = [torch.empty_like(V)]
            dmu = torch.empty(K, dtype=torch.float64, device="cuda")
            ctx.gateaux([V], out=F, dmu=dmu)                     # captured where graphs are used
            ctx.krylov_step(R, s_tol=0.0, r_max=2)
            F[0].fill_(float("nan"))
            ctx.gateaux([V], out=F, dmu=dmu)                     # replayed
            X = [ctx.projection(k) for k in range(K)]
            vbar, eps_bar, occ_bar = ctx.backward([fbar])
            X2 = ctx.projection(K - 1)
            torch.cuda.current_stream().synchronize()
            got.append([F[0].clone(), dmu.clone(), *X, X2, vbar[0].clone(), eps_bar[0].clone(), occ_bar[0].clone()])
            assert ctx.status() == 0
            ctx.close()
    for a, b in zip(*got):
        assert torch.isfinite(a).all() and torch.equal(a, b)
