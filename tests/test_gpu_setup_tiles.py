"""Set-up kernels at the edges of their tiles.

k_loewner takes 32 x 32 blocks of the upper triangle and mirrors them: permuting
the states of a system leaves every result as it is, so an entry left out, taken
from elsewhere or not mirrored moves to another pair of states and shows.  FP64
sums of at most 10^3 terms, reordered: 10^3 2^-53, 1e-12 with the cancellation of
F = dV - V.

k_copy_tc converts 32 rows x 128 states, with 16-byte loads where the rows allow:
rows at another leading dimension and at an odd address hold the same values, so
the results are equal bit for bit."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = (11, 10, 9)
NG = int(np.prod(N))


def _system(ns, gen):
    psi = torch.linalg.qr(torch.randn(NG, ns, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    eps = torch.sort(torch.rand(ns, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1).values
    return psi, eps


def _forward(psi, eps, V, prec, **kw):
    from paper_2211_07894_gb300 import Context
    d = dict(n=N, h=(0.5,) * 3, psi=[psi], eps=[eps], n_electrons=max(1.0, 0.9 * len(eps)), kT=kw.pop("kT"), g=2.0,
             rho_floor=1e-3, k_max=2)
    if "occ" in kw:
        d["occ"] = [kw.pop("occ")]
    ctx = Context([d], prec=prec, io_dtype=V.dtype, k_max=2, **kw)
    (F,), _ = ctx.gateaux([V])
    assert ctx.status() == 0
    return F


@pytest.mark.parametrize("mode", ["fermi", "log", "occ", "fermi_T"])
@pytest.mark.parametrize("ns", [2, 31, 32, 33, 64, 65, 100])
def test_loewner_follows_the_states(mode, ns):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(ns)
    psi, eps = _system(ns, gen)
    V = torch.randn(2, 1, NG, generator=gen, device="cuda", dtype=torch.float64)
    kw = {"fermi": dict(kT=0.05), "log": dict(kT=1e-3), "occ": dict(kT=0.05), "fermi_T": dict(kT=0.05, fermi_T=8)}[mode]
    p = torch.randperm(ns, generator=gen, device="cuda")
    kw2 = dict(kw)
    if mode == "occ":
        occ = torch.sigmoid(-eps / 0.05)
        kw["occ"], kw2["occ"] = occ, occ[p].contiguous()
    a = _forward(psi.contiguous(), eps, V, "fp64", **kw)
    b = _forward(psi[:, p].contiguous(), eps[p].contiguous(), V, "fp64", **kw2)
    assert (a - b).norm() <= 1e-12 * a.norm()


@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
@pytest.mark.parametrize("ns", [1, 4, 31, 127, 128, 130, 256, 301])
def test_copies_do_not_depend_on_the_layout(prec, ns):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(ns)
    psi, eps = _system(ns, gen)
    V = torch.randn(2, 1, NG, generator=gen, device="cuda")
    psi = psi.float()
    n4 = (ns + 3) // 4 * 4
    results = []
    for ld, off in ((n4, 0), (n4 + 1, 0), (n4 + 4, 1)):      # 16-byte rows; other rows; rows off by 4 bytes
        buf = torch.full((NG * ld + off,), float("nan"), device="cuda")
        view = buf[off:].view(NG, ld)[:, :ns]
        view.copy_(psi)
        results.append(_forward(view, eps, V, prec, kT=0.05))
    assert torch.equal(results[0], results[1]) and torch.equal(results[0], results[2])
    assert torch.isfinite(results[0]).all()
