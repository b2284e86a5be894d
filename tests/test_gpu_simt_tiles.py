"""The CUDA-core contractions at the edges of their tiles (64 and 128 states in
FP32, 32 states and 2 x 2 micro-tiles in FP64), of the vector loads (N_s a multiple
of 4 or not) and of the row ranges, against the oracle; real subspaces, spin pairs
and the stacked operand of k-point systems."""

import numpy as np
import pytest

import oracle
import workloads
from gates import TOL
from helpers import oracle_system, per_direction_rel_err

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

IO = {"fp64": torch.float64, "fp32": torch.float32}
# FP32: products and sums over N_g <= 720 rows and N_s <= 320 states rounded to
# 2^-24, random signs: sqrt(N_g N_s) 2^-24 = 3e-5 of the largest term at most
GATE = {"fp64": TOL["fp64"], "fp32": 3e-5}


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("ns", [3, 31, 32, 33, 63, 64, 65, 97, 127, 128, 129, 160, 200, 257, 320])
@pytest.mark.parametrize("K", [1, 3])
def test_contractions_at_tile_edges(prec, ns, K):
    from gpu_helpers import directions, make_context
    cfg = workloads.random_system(70 + ns, (10, 9, 8), ns, max(1.0, 0.9 * ns), 0.02, K)
    ctx, _ = make_context([cfg], prec, IO[prec])
    F, dmu = ctx.gateaux([directions(cfg, IO[prec])])
    ref = oracle.gateaux(oracle_system(cfg), cfg["V"])
    assert per_direction_rel_err(F[0].double().cpu().numpy(), ref["F"]) < GATE[prec]
    X = ctx.projection(K - 1).cpu().numpy()
    assert np.array_equal(X, X.T)
    Xr = ref["X"][0][K - 1]
    assert np.linalg.norm(X - Xr) < GATE[prec] * np.linalg.norm(Xr)
    assert ctx.status() == 0


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("ns", [16, 45, 64, 65])
def test_kpoint_stacked_at_tile_edges(prec, ns):
    from paper_2211_07894_gb300 import KpContext
    cfg = workloads.kpoint_system(90 + ns, (9, 8, 10), ns, 2, 0.8 * ns, 0.02, 2)
    dt = IO[prec]
    ctx = KpContext(cfg["n"], cfg["h"], [torch.as_tensor(np.ascontiguousarray(p.real), dtype=dt, device="cuda") for p in cfg["psi"]],
                    [torch.as_tensor(np.ascontiguousarray(p.imag), dtype=dt, device="cuda") for p in cfg["psi"]],
                    [torch.as_tensor(e, dtype=torch.float64, device="cuda") for e in cfg["eps"]], cfg["k_weights"],
                    cfg["n_electrons"], cfg["kT"], g=cfg["g"], rho_floor=cfg["rho_floor"], prec=prec, io_dtype=dt, k_max=2)
    F, dmu = ctx.gateaux(torch.as_tensor(cfg["V"], dtype=dt, device="cuda"))
    ks = oracle.KpointSystem(n=cfg["n"], h=cfg["h"], psi=cfg["psi"], eps=cfg["eps"], k_weights=cfg["k_weights"],
                             rho=np.zeros(int(np.prod(cfg["n"]))), n_electrons=cfg["n_electrons"],
                             kT=cfg["kT"], g=cfg["g"])
    mu = oracle.solve_mu_kpoints(cfg["eps"], cfg["k_weights"], cfg["n_electrons"], cfg["kT"], cfg["g"])
    ks.rho = oracle.density_kpoints(ks, mu, cfg["rho_floor"])
    ref = oracle.gateaux_kpoints(ks, cfg["V"])
    for k in range(2):
        f, r = F[k].double().cpu().numpy(), ref["F"][k]
        assert np.linalg.norm(f - r) < GATE[prec] * np.linalg.norm(r)
