"""Contexts made one after another, side by side and from several threads on
streams of their own: the transform plans of closed contexts are taken over by
later ones of the same grid, batch and precision, more sizes than are kept go
through, and every context answers as the first of its kind did, bit for bit."""

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [((8, 9, 10), 1, "fp64"), ((8, 9, 10), 2, "fp64"), ((8, 9, 10), 1, "fp32"), ((10, 9, 8), 1, "fp64"),
         ((12, 12, 12), 3, "fp32"), ((5, 7, 11), 2, "fp64")]


def _system(n, K, prec):
    ng, ns = int(np.prod(n)), 6
    gen = torch.Generator(device="cuda")
    gen.manual_seed(ng + K)
    dt = torch.float64 if prec == "fp64" else torch.float32
    psi = torch.linalg.qr(torch.randn(ng, ns, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    eps = torch.linspace(-1, 1, ns, device="cuda", dtype=torch.float64)
    V = torch.randn(K, 1, ng, generator=gen, device="cuda", dtype=dt)
    return dict(n=n, h=(0.5,) * 3, psi=[psi.to(dt).contiguous()], eps=[eps], n_electrons=5.0, kT=0.05, g=2.0,
                rho_floor=1e-3, k_max=K), V, dt


def _run(ctx, V):
    (F,), _ = ctx.gateaux([V])
    torch.cuda.current_stream().synchronize()
    return F.clone()


def test_contexts_share_nothing_but_plans():
    from paper_2211_07894_gb300 import Context
    made = {}
    for c in CASES:
        d, V, dt = _system(*c)
        ctx = Context([d], prec=c[2], io_dtype=dt, k_max=c[1])
        made[c] = (d, V, dt, _run(ctx, V))
        ctx.close()
    torch.cuda.synchronize()
    bad = []

    def work(seed):
        rng = np.random.default_rng(seed)
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(6):
                pair = []
                for i in (0, rng.integers(len(CASES))):      # two alive at a time, often of one kind
                    c = CASES[i]
                    d, V, dt, F = made[c]
                    pair.append((Context([d], prec=c[2], io_dtype=dt, k_max=c[1]), V, F))
                for ctx, V, F in pair:
                    if not torch.equal(_run(ctx, V), F):
                        bad.append(seed)
                for ctx, _, _ in pair:
                    ctx.close()

    threads = [threading.Thread(target=work, args=(s,)) for s in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
