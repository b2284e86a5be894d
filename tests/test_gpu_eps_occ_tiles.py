"""eps_bar and occ_bar over the ways k_eps_occ_bar shares out a row: fewer to more
quads of states than threads, one and several row ranges, directions not a
multiple of the groups, against torch in FP64 on the library's own projections
and f_bar's adjoint through the FP64 mode.

The FP32 modes sum G X over K directions (K 2^-24 of the sum of magnitudes) of
X and G within 2^-20 of sum_g |a psi_i psi_j| (FP32 sums of some 10^3 to 10^4 terms);
with magnitudes at most sqrt(N_g) = 106 times the entries' root mean square, that is
3e-4 of the largest entries' products.  A direction, range or column left out or
taken twice is off by 1 / (K nsplit) >= 1e-2 of them."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["fp32", "bf16x3"])
@pytest.mark.parametrize("ns,K", [(2, 1), (5, 8), (64, 3), (130, 7), (256, 8), (512, 5), (513, 2), (1030, 2)])
def test_eps_occ_bar_every_share(prec, ns, K):
    from paper_2211_07894_gb300 import Context
    n = (24, 22, 21)
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(ns)
    psi = torch.linalg.qr(torch.randn(ng, ns, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    eps = torch.linspace(-1, 1, ns, device="cuda", dtype=torch.float64)      # no pair within the tolerance
    V = torch.randn(K, 1, ng, generator=gen, device="cuda")
    fbar = torch.randn(K, 1, ng, generator=gen, device="cuda")
    out = []
    for p in ("fp64", prec):
        dt = torch.float64 if p == "fp64" else torch.float32
        ctx = Context([dict(n=n, h=(0.5,) * 3, psi=[psi.to(dt).contiguous()], eps=[eps],
                            n_electrons=max(1.0, 0.9 * ns), kT=0.5, g=2.0, rho_floor=1e-3, k_max=K)],
                      prec=p, io_dtype=dt, k_max=K)
        ctx.gateaux([V.to(dt)])
        _, e, o = ctx.backward([fbar.to(dt)])
        out.append((e[0].double(), o[0].double()))
        assert ctx.status() == 0
    for x64, x32 in zip(*out):
        assert (x32 - x64).norm() <= 1e-3 * x64.norm()
