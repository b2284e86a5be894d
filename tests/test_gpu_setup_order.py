"""Set-up of a context on a stream of the caller's that does not wait for the
legacy stream: what set-up reads and zeroes is ordered on that stream, so a call
right after it answers as on an idle device while the legacy stream is busy."""

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, NS, K = (14, 13, 12), 200, 16


def _inputs(prec):
    io = torch.float64 if prec == "fp64" else torch.float32
    ng = int(np.prod(N))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)
    q = torch.linalg.qr(torch.randn(ng, NS, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    q2 = torch.linalg.qr(torch.randn(ng, NS, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    eps = torch.linspace(-1, 1, NS, device="cuda", dtype=torch.float64)
    V = torch.randn(K, 1, ng, generator=gen, device="cuda", dtype=io)
    return io, q.to(io).contiguous(), (q2 * 0.1).to(io).contiguous(), eps, V


def _run(kind, prec, io, psi, psi2, eps, V, stream):
    """One context made and called on `stream`, its eigenvalues written there just before."""
    from paper_2211_07894_gb300 import Context, KpContext
    with torch.cuda.stream(stream):
        e = eps + 0.0
        if kind == "kp":
            ctx = KpContext(N, (0.5,) * 3, [psi], [psi2], [e], [1.0], 0.9 * NS, 0.05, rho_floor=1e-3, prec=prec,
                            io_dtype=io, k_max=K)
            F, dmu = ctx.gateaux(V[:, 0].contiguous())
        else:
            ctx = Context([dict(n=N, h=(0.5,) * 3, psi=[psi], eps=[e], n_electrons=0.9 * NS, kT=0.05, g=2.0,
                                rho_floor=1e-3, k_max=K)], prec=prec, io_dtype=io, k_max=K)
            (F,), dmu = ctx.gateaux([V])
        out = F.clone(), dmu.clone()
        stream.synchronize()
        ctx.close()
    return out


# K N_s^2 words of X, Gbar and X'' are more than 2 MB, allocations of their own
@pytest.mark.parametrize("kind,prec", [("real", "fp64"), ("real", "fp32"), ("real", "bf16x3"), ("kp", "fp64"),
                                       ("kp", "fp32"), ("kp", "tf32")])
def test_busy_legacy_stream(kind, prec):
    args = _inputs(prec)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    ref = _run(kind, prec, *args, side)
    torch.cuda.synchronize()
    A = torch.randn(4096, 4096, device="cuda")
    B = torch.empty_like(A)

    def feed():                                   # some 0.5 s of work on the legacy stream
        for _ in range(200):
            torch.mm(A, A, out=B)

    for _ in range(3):
        t = threading.Thread(target=feed)
        t.start()
        got = _run(kind, prec, *args, side)
        t.join()
        torch.cuda.synchronize()
        for a, b in zip(ref, got):
            assert torch.isfinite(a).all() and torch.equal(a, b)


def test_driver_state_after_create():
    """The accumulated driver's arrays hold what was loaded right after create."""
    from paper_2211_07894_gb300 import binding
    import ctypes
    n, m = 1 << 20, 4
    lib = binding.load()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    U = torch.randn(m, n, generator=gen, device="cuda")
    T = torch.randn(m, n, generator=gen, device="cuda")
    R = torch.randn(n, generator=gen, device="cuda")
    A = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for _ in range(20):
        torch.mm(A, A)
    h = ctypes.c_void_p()
    assert lib.lrdm_lrdma_create(ctypes.byref(h), ctypes.c_longlong(n), binding.DTYPE_F32, ctypes.c_double(1.0), m) == 0
    st = ctypes.c_void_p(side.cuda_stream)
    p = ctypes.c_void_p
    assert lib.lrdm_lrdma_import(h, m, 0, p(U.data_ptr()), p(T.data_ptr()), p(R.data_ptr()), st) == 0
    side.synchronize()
    torch.cuda.synchronize()
    U2, T2, R2 = torch.empty_like(U), torch.empty_like(T), torch.empty_like(R)
    assert lib.lrdm_lrdma_export(h, p(U2.data_ptr()), p(T2.data_ptr()), p(R2.data_ptr()), st) == 0
    side.synchronize()
    lib.lrdm_lrdma_destroy(h)
    assert torch.equal(U, U2) and torch.equal(T, T2) and torch.equal(R, R2)
