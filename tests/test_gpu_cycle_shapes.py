"""The band solve with other multigrid cycles than the default: one smoothing sweep a side, more
sweeps on the coarsest level, fewer levels down to plain Jacobi, on bands of each engine.

Every choice is a symmetric preconditioner, so the FP64 solve reaches its tolerance; an FP32 one may
stall above 1e-6 (128x128x64 with one sweep a side and six on the coarsest level does), and then has
to say so.  Of a solution that is returned as one, the residual is formed by the oracle's operator,
with the bounds of the large-band tests (FP64 1e-10; FP32 1e-3, which rounding w to FP32 alone can
leave).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import band as obm  # noqa: E402
from oracle import model as omodel  # noqa: E402
from paper_2606_04347_gb300 import Plan  # noqa: E402
from paper_2606_04347_gb300 import workloads as wl  # noqa: E402
from paper_2606_04347_gb300.abi import EtdError  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,eps", [((32, 32, 32), 0.25),      # a cluster
                                   ((64, 96, 1), 0.25),       # a cluster, 2D
                                   ((128, 128, 64), 0.09),    # hybrid from three levels on, else the grid
                                   ((128, 128, 128), 0.09)])  # the grid
def test_cycle_shapes_reach_the_tolerance(monkeypatch, n, eps, prec):
    dim = 2 if n[2] == 1 else 3
    p = wl.workload("c2", n=16)[0].replace(dim=dim, n=n, model=0, precision=prec, cg_rtol=1e-12 if prec == 0 else 1e-6, cg_maxit=5000)
    dt, tdt = (np.float64, torch.float64) if prec == 0 else (np.float32, torch.float32)
    r = np.sqrt(sum(c ** 2 for c in wl.grid(n, p.half_len, dim)))
    phi = (wl.tanh_profile(1.6 - r, eps) * np.ones(p.shape)).astype(dt).astype(np.float64)
    band, g = obm.band_mask(phi, p.band_mask_hi), omodel.g_loc(phi)
    f = np.where(band, np.random.default_rng(7).uniform(-1.0, 1.0, size=p.shape), 0.0).astype(dt).astype(np.float64)
    b = np.where(band, f - f[band].mean(), 0.0)
    cf = obm.face_coeffs(g, band)
    phid, fd = (torch.tensor(a, dtype=tdt, device="cuda:0") for a in (phi, f))
    iters = {}
    for shape in ("", "NU=1", "CSWEEPS=4", "NU=1,CSWEEPS=6", "LEVELS=3", "LEVELS=3,NU=1", "LEVELS=2", "LEVELS=2,CSWEEPS=4", "LEVELS=1"):
        env = dict(kv.split("=") for kv in shape.split(",") if kv)
        for k, v in env.items():
            monkeypatch.setenv("ETD_MG_" + k, v)
        plan = Plan(p)
        for k in env:
            monkeypatch.delenv("ETD_MG_" + k)
        w = torch.zeros(p.shape, dtype=tdt, device="cuda:0")
        try:
            iters[shape], res = plan.nonlocal_solve(phid, fd, w)
            assert res <= p.cg_rtol and iters[shape] > 0, shape
        except EtdError as e:
            assert e.code == 5 and prec == 1 and shape, shape
            iters[shape] = p.cg_maxit
            continue
        finally:
            plan.close()
        got = w.cpu().numpy().astype(np.float64)
        err = b - obm.apply_neg_lap(got, cf, p.h[:dim])
        assert np.linalg.norm(err) <= (1e-10 if prec == 0 else 1e-3) * np.linalg.norm(b), shape
    assert iters["LEVELS=1"] > iters[""] and iters["NU=1"] >= iters[""]
