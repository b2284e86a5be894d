"""A tuning cache written against earlier contraction kernels: its shapes are not
taken over, the candidates are timed again."""

import json
import re

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_cache_of_other_kernels_is_not_used(tmp_path, monkeypatch):
    from paper_2211_07894_gb300 import Context
    cache = tmp_path / "tune.jsonl"
    monkeypatch.setenv("LRDM_TUNE_CACHE", str(cache))
    n, ns = (12, 12, 12), 40
    ng = int(np.prod(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    psi = torch.linalg.qr(torch.randn(ng, ns, generator=gen, device="cuda", dtype=torch.float64))[0] / 0.5 ** 1.5
    d = dict(n=n, h=(0.5,) * 3, psi=[psi.float().contiguous()],
             eps=[torch.linspace(-1, 1, ns, device="cuda", dtype=torch.float64)], n_electrons=30.0, kT=0.05, g=2.0,
             rho_floor=1e-3, k_max=4)

    def make():
        ctx = Context([d], prec="bf16x3", io_dtype=torch.float32, k_max=4, autotune=True)
        t = ctx.tuning()
        ctx.close()
        return t

    first = make()
    (line,) = cache.read_text().splitlines()
    assert make() == first and len(cache.read_text().splitlines()) == 1       # its own entry is used
    old = json.loads(line)
    old["key"] = re.sub(r";kernels\d+", "", old["key"])
    cache.write_text(json.dumps(old) + "\n")
    make()
    lines = cache.read_text().splitlines()
    assert len(lines) == 2 and json.loads(lines[1])["key"] != old["key"]
