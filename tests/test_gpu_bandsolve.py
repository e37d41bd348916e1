"""The band solve's two engines at the sizes where they can go wrong.

Bands that fit one thread-block cluster and bands that do not; levels of the multigrid hierarchy
that every block holds itself and coarsest levels that stay distributed; node counts that are no
multiple of a warp or of the blocks.  The solve is compared with the oracle's Jacobi-CG: with a
relative residual of 1e-13 (FP64) and 1e-6 (FP32) and condition numbers of these bands below
1e3, the solutions agree to 1e-10 and 1e-3 * 1e-6 * 20 = 2e-5 or better (the bounds of the other
band-solve tests).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import band as obm  # noqa: E402
from oracle import model as omodel  # noqa: E402
from paper_2606_04347_gb300 import Plan  # noqa: E402
from paper_2606_04347_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _params(n, prec):
    dim = 2 if n[2] == 1 else 3
    return wl.workload("c2", n=16)[0].replace(dim=dim, n=n, model=0, precision=prec, cg_rtol=1e-13 if prec == 0 else 1e-6)


def _membrane(p, kind, rng):
    if kind == "full":      # every point in the band, g between 0.46 and 1.125
        return rng.uniform(0.2, 0.8, size=p.shape)
    ax = wl.grid(p.n, p.half_len, p.dim)
    if kind == "corner":    # a sphere around the box's corner: the band crosses every boundary
        r = np.sqrt(sum((np.pi - np.abs(c)) ** 2 for c in ax))
        return wl.tanh_profile(1.6 - r, 0.09) * np.ones(p.shape)
    r = np.sqrt(sum(c ** 2 for c in ax))
    eps = {"shell": 0.25, "thin": 0.09}[kind]
    return wl.tanh_profile(1.6 - r, eps) * np.ones(p.shape)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,kind", [
    ((8, 8, 1), "full"), ((16, 8, 1), "full"), ((64, 96, 1), "shell"),      # a few nodes a block; 2D levels
    ((8, 8, 8), "full"), ((32, 32, 32), "shell"), ((64, 64, 32), "thin"),
    ((32, 32, 16), "full"), ((32, 32, 32), "full"),                          # near and past the cluster's capacity
    ((128, 16, 8), "full"), ((256, 16, 8), "full"),                          # coarsest level distributed
])
def test_band_solve_sizes_match_oracle(n, kind, prec):
    p = _params(n, prec)
    rng = np.random.default_rng(11)
    dt = np.float64 if prec == 0 else np.float32
    phi = _membrane(p, kind, rng).astype(dt).astype(np.float64)
    band = obm.band_mask(phi, p.band_mask_hi)
    f = np.where(band, rng.uniform(-1.0, 1.0, size=p.shape), 0.0).astype(dt).astype(np.float64)
    want, _, _ = obm.solve_neg_lap(f, omodel.g_loc(phi), band, p.h[:p.dim], rtol=1e-14)
    plan = Plan(p)
    dev = lambda a: torch.tensor(a, dtype=plan.dtype, device=DEV)  # noqa: E731
    w = torch.zeros(p.shape, dtype=plan.dtype, device=DEV)
    it, res = plan.nonlocal_solve(dev(phi), dev(f), w)
    assert res <= p.cg_rtol and it > 0
    got = w.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - want) / np.linalg.norm(want) < (1e-10 if prec == 0 else 2e-5)
    assert not got[~band].any()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,kind", [((128, 128, 64), "thin"), ((128, 128, 128), "shell"), ((256, 64, 64), "thin"),
                                    ((256, 128, 128), "shell"), ((256, 128, 128), "corner"), ((64, 64, 64), "corner")])
def test_large_band_solve_residual(n, kind, prec):
    """Bands past one cluster, of a size the host does not know (the hybrid or the grid engine; the
    largest with the packed matrix, and across the periodic boundary, where it does not apply):
    the solution's own residual, formed by the oracle's operator, and its mean.  FP32: rounding w
    to FP32 alone leaves a residual of eps32 max(diag) |w| / |b|, below 1e-3 here."""
    p = _params(n, prec)
    rng = np.random.default_rng(2)
    dt = np.float64 if prec == 0 else np.float32
    phi = _membrane(p, kind, rng).astype(dt).astype(np.float64)
    band, g = obm.band_mask(phi, p.band_mask_hi), omodel.g_loc(phi)
    f = np.where(band, rng.uniform(-1.0, 1.0, size=p.shape), 0.0).astype(dt).astype(np.float64)
    plan = Plan(p.replace(cg_rtol=1e-12 if prec == 0 else 1e-6))
    dev = lambda a: torch.tensor(a, dtype=plan.dtype, device=DEV)  # noqa: E731
    w = torch.zeros(p.shape, dtype=plan.dtype, device=DEV)
    it, res = plan.nonlocal_solve(dev(phi), dev(f), w)
    got = w.cpu().numpy().astype(np.float64)
    b = np.where(band, f - f[band].mean(), 0.0)
    r = b - obm.apply_neg_lap(got, obm.face_coeffs(g, band), p.h)
    assert it > 0 and res <= (1e-12 if prec == 0 else 1e-6)
    assert np.linalg.norm(r) <= (1e-10 if prec == 0 else 1e-3) * np.linalg.norm(b)
    assert abs(got[band].mean()) <= (1e-12 if prec == 0 else 1e-5) * np.abs(got).max() and not got[~band].any()


@pytest.mark.parametrize("n,kind,prec,tol", [((64, 64, 64), "shell", 0, 1e-11), ((96, 64, 32), "shell", 0, 1e-11),
                                             ((64, 64, 64), "shell", 1, 3e-5), ((64, 64, 32), "thin", 1, 3e-5)])
def test_frozen_band_step_matches_oracle(n, kind, prec, tol):
    """A frozen band's engine is chosen from its level counts (64^3 shell: the hybrid engine).  The
    bounds are those of the fixed-membrane step tests."""
    from oracle import etd as oetd
    p = _params(n, prec).replace(scheme=1, tau=1e-3, M=100.0)
    rng = np.random.default_rng(4)
    dt = np.float64 if prec == 0 else np.float32
    phi = _membrane(p, kind, rng).astype(dt).astype(np.float64)
    u = rng.uniform(0.3, 0.7, size=p.shape).astype(dt).astype(np.float64)
    want = oetd.FixedStepper(p.replace(cg_rtol=1e-13), phi).run(u.copy(), 1)
    plan = Plan(p)
    dev = lambda a: torch.tensor(a, dtype=plan.dtype, device=DEV)  # noqa: E731
    ud = dev(u)
    plan.step(dev(phi), ud, 1, diag=True)
    assert np.linalg.norm(ud.cpu().numpy() - want) < tol * np.linalg.norm(want)
