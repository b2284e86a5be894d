"""mu' and the occupation gradient of a gapped spectrum: with given occupations
the weights L_ii = -f_i (1 - f_i) / kT of a gap of many kT lie far below the FP32
range, and mu' = sum L_ii X_ii / sum L_ii stays their weighted mean."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, H, KT, K = (16, 15, 14), 0.5, 0.002, 3
NV = 8                                            # states on either side of the gap


def _system(gap, io):
    """Plane-wave-like orthonormal columns, band edges spread over a few kT, Fermi
    occupations of a mid-gap mu, smooth directions."""
    ng, ns = int(np.prod(N)), 2 * NV
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    psi = torch.linalg.qr(torch.randn(ng, ns, generator=gen, device="cuda", dtype=torch.float64))[0] / H ** 1.5
    step = 1.7 * KT * torch.arange(NV, device="cuda", dtype=torch.float64)
    eps = torch.cat([-0.5 * gap * KT - step.flip(0), 0.5 * gap * KT + step])
    occ = 1.0 / (1.0 + torch.exp(eps / KT))
    x = [torch.arange(m, device="cuda", dtype=torch.float64) * (2 * np.pi / m) for m in N]
    V = torch.stack([(torch.cos((k + 1) * x[0])[:, None, None] + torch.sin(x[1])[None, :, None] * (0.5 + k)
                      + torch.cos(x[2] + k)[None, None, :]).reshape(1, -1) for k in range(K)])
    fbar = torch.roll(V, 1, 0) + 0.3 * V
    d = dict(n=N, h=(H,) * 3, psi=[psi.to(io).contiguous()], eps=[eps], occ=[occ], n_electrons=2.0 * NV, kT=KT,
             g=2.0, rho_floor=1e-3, k_max=K)
    return d, V.to(io).contiguous(), fbar.to(io).contiguous()


def _run(prec, gap):
    from paper_2211_07894_gb300 import Context
    io = torch.float64 if prec == "fp64" else torch.float32
    d, V, fbar = _system(gap, io)
    ctx = Context([d], prec=prec, io_dtype=io, k_max=K)
    _, dmu = ctx.gateaux([V])
    X = torch.stack([ctx.projection(k) for k in range(K)])
    _, _, occ_bar = ctx.backward([fbar])
    assert ctx.status() == 0
    return dmu.clone(), X, occ_bar[0].clone()


# X carries the rounding of its operands: 2^-20 (FP32 sums of 3,360 terms), 2^-15
# (BF16x3: three terms of 2^-17 and the sums), 2^-10 (TF32) of the directions'
# range, which X reaches to a factor of 8; occ_bar is a sum of 16 products of two such.
UNIT = {"fp32": 2.0 ** -20, "bf16x3": 2.0 ** -15, "tf32": 2.0 ** -10}


@pytest.mark.parametrize("prec", ["fp32", "tf32", "bf16x3"])
@pytest.mark.parametrize("gap", [60, 190, 260, 1200])
def test_mu_and_occupation_gradient(prec, gap):
    dmu64, X64, ob64 = _run("fp64", gap)
    dmu, X, ob = _run(prec, gap)
    u = UNIT[prec]
    assert float(dmu64.abs().max()) > 0.01 * float(X64.abs().max())
    assert float((X - X64).abs().max()) <= 8 * u * float(X64.abs().max())
    assert float((dmu - dmu64).abs().max()) <= 8 * u * float(X64.abs().max())
    assert float((ob - ob64).abs().max()) <= 128 * u * float(ob64.abs().max())


@pytest.mark.parametrize("prec", ["fp32", "tf32", "bf16x3"])
@pytest.mark.parametrize("gap", [60, 260])
def test_kpoint_mu(prec, gap):
    """Two k-points: mu lies where the first occupations leave 0 or 1."""
    from paper_2211_07894_gb300 import KpContext

    def run(p):
        io = torch.float64 if p == "fp64" else torch.float32
        d, V, _ = _system(gap, io)
        re, eps = d["psi"][0], d["eps"][0]
        im = (0.5 * re.flip(1)).contiguous()
        ctx = KpContext(N, (H,) * 3, [re, im], [im, re], [eps, eps + 0.1 * KT], [0.25, 0.75], 2.0 * NV, KT,
                        rho_floor=1e-3, prec=p, io_dtype=io, k_max=K)
        _, dmu = ctx.gateaux(V[:, 0].contiguous())
        return dmu.clone()

    ref, got = run("fp64"), run(prec)
    # |X_ii| <= (1 + 0.5)^2 max |dV|, dV no more than ten times the directions' range of 4
    assert torch.isfinite(ref).all()
    assert float((got - ref).abs().max()) <= 8 * UNIT[prec] * max(1.0, float(ref.abs().max()))
