"""The pair projection covers the symmetric X_k by items of one row block, two
column blocks and two directions (and 256 x 256 tiles for the last direction of
an odd number): one to ten block rows, every remainder of a group of four, odd and
even numbers of directions, one and two row ranges, against the square single-CTA
tiles, which cover it block by block.

Both round the operands, in blocks below the diagonal with the weights on the
other factor.  Each is within eps sum_g |a psi_i psi_j| of the exact value: BF16x3
drops lo x lo and rounds both lo (3 x 2^-18) and truncates 192 sums a segment
(192 x 2^-24), 2.3e-5; TF32 rounds both factors (2 x 2^-11) and truncates 128 (128
x 2^-24).  For the random data here sum_g |a psi_i psi_j| is at most sqrt(N_g) = 106
times the root mean square of X's entries off the diagonal, so the two differ by
at most 2 x 106 x 2.3e-5 = 5e-3 (0.21 for TF32) of that.  A block left out,
repeated with another direction or stored elsewhere is off by 1 and more."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
@pytest.mark.parametrize("ns,K", [(3, 2), (128, 3), (130, 2), (255, 4), (257, 1), (300, 5), (384, 2), (450, 3), (512, 2),
                                  (513, 3), (700, 2), (800, 4), (897, 2), (1024, 1), (1025, 2), (1153, 3)])
def test_pair_projection_covers_every_block(prec, ns, K):
    from paper_2211_07894_gb300 import Context
    n = (24, 22, 21)                                   # 11,088 rows: 346 or 347 stages, two row ranges where few items
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(ns)
    psi = torch.linalg.qr(torch.randn(ng, ns, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    eps = torch.sort(torch.rand(ns, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1).values
    V = torch.randn(K, 1, ng, generator=gen, device="cuda")
    X = []
    for nb in (512, 128):
        ctx = Context([dict(n=n, h=(0.5,) * 3, psi=[psi.float().contiguous()], eps=[eps],
                            n_electrons=max(1.0, 0.9 * ns), kT=0.02, g=2.0, rho_floor=1e-3, k_max=K)],
                      prec=prec, io_dtype=torch.float32, k_max=K)
        ctx.set_tuning(g1_nb=nb, g1_dpt=1)
        ctx.gateaux([V])
        assert ctx.status() == 0
        X.append(torch.stack([ctx.projection(k).clone() for k in range(K)]))
    off = X[1] - torch.diag_embed(X[1].diagonal(dim1=1, dim2=2))
    rms = (off.pow(2).sum((1, 2)) / (ns * (ns - 1))).sqrt()
    bound = {"bf16x3": 5e-3, "tf32": 0.21}[prec]
    assert ((X[0] - X[1]).abs().amax((1, 2)) <= bound * rms).all()
    assert torch.equal(X[0], X[0].transpose(1, 2))
