"""The pair response multiplies the triangle of X'' alone, in columns of 32: every
remainder of N_s against a j-tile (256) and a stage (32), one to three j-tiles,
against the single-CTA kernel, which multiplies whole blocks.  Each row sums the
same terms in the same order (the left-out ones are zeros), so the results are
equal bit for bit."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
@pytest.mark.parametrize("ns", [2, 31, 33, 64, 97, 128, 129, 161, 200, 225, 255, 256, 257, 289, 350, 385, 449, 500,
                                512, 513, 577, 700])
def test_pair_response_equals_single_cta(prec, ns):
    from paper_2211_07894_gb300 import Context
    n = (13, 11, 10)                                   # 1,430 rows: an odd number of 128-row blocks, a ragged last one
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(ns)
    psi = torch.linalg.qr(torch.randn(ng, ns, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    eps = torch.sort(torch.rand(ns, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1).values
    V = torch.randn(3, 1, ng, generator=gen, device="cuda")
    F = []
    for bn in (512, 256):
        ctx = Context([dict(n=n, h=(0.5,) * 3, psi=[psi.float().contiguous()], eps=[eps],
                            n_electrons=max(1.0, 0.9 * ns), kT=0.02, g=2.0, rho_floor=1e-3, k_max=3)],
                      prec=prec, io_dtype=torch.float32, k_max=3)
        ctx.set_tuning(g2_bn=bn)
        (f,), _ = ctx.gateaux([V])
        assert ctx.status() == 0
        F.append(f)
    assert torch.equal(F[0], F[1])
