"""The energy sums and bound statistics on random fields, against the oracle: 2D and 3D, ragged and
small grids (fewer points than a block), both precisions."""
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
    r = np.sqrt(sum(c ** 2 for c in wl.grid(p.n, p.half_len, p.dim)))
    eps = {"shell": 0.25, "thin": 0.09}[kind]
    return wl.tanh_profile(1.6 - r, eps) * np.ones(p.shape)


@pytest.mark.parametrize("prec,tol", [(0, 1e-11), (1, 3e-6)])
@pytest.mark.parametrize("n,kind", [((8, 8, 1), "full"), ((96, 64, 1), "shell"), ((32, 16, 8), "full"), ((64, 32, 32), "shell")])
def test_energy_sums_match_oracle(n, kind, prec, tol):
    """Every sum of Eq. (2.16) on random fields.  FP32: g, W(u) and f(u) carry a few FP32
    roundings (below 1e-6 relative, all terms positive but the mass, whose square enters), the
    sums themselves none."""
    p = _params(n, prec).replace(gamma=20.0, M=30.0, ubar=0.3)
    rng = np.random.default_rng(5)
    dt = np.float64 if prec == 0 else np.float32
    phi = _membrane(p, kind, rng).astype(dt).astype(np.float64)
    u = rng.uniform(0.2, 0.9, size=p.shape).astype(dt).astype(np.float64)
    band, G = obm.band_mask(phi, p.band_mask_hi), omodel.g_loc(phi)
    want = omodel.energy(u, G, band, p, rtol=1e-13)
    plan = Plan(p)
    dev = lambda a: torch.tensor(a, dtype=plan.dtype, device=DEV)  # noqa: E731
    d = plan.energy(dev(phi), dev(u))
    assert abs(d["energy"] - want["total"]) <= tol * abs(want["total"])
    assert abs(d["mass"] - want["mass"]) <= tol * abs(want["mass"])
    mb, lo, hi = omodel.bound_stats(u, G, p.recover_delta)
    assert d["band_size"] == band.sum() and (d["max_bound"], d["umin"], d["umax"]) == (mb, lo, hi)
    assert abs(d["volume"] - omodel.volume(phi, p)) <= 1e-13 * phi.sum()


def test_step_of_an_unaligned_field():
    """u one element past a 16-byte boundary: the mass sum takes its one-value loads.  Only the
    order of that sum differs, so the FP64 results agree to a few roundings of the mass (its
    relative error is below 1e-14 and the step is Lipschitz in it: 1e-12)."""
    p = _params((64, 64, 1), 0).replace(scheme=1, tau=1e-3, M=100.0, cg_rtol=1e-13)
    rng = np.random.default_rng(8)
    phi = _membrane(p, "shell", rng)
    u = rng.uniform(0.3, 0.7, size=p.shape)
    plan = Plan(p)
    phid, ud = torch.tensor(phi, device=DEV), torch.tensor(u, device=DEV)
    buf = torch.zeros(u.size + 1, dtype=torch.float64, device=DEV)
    buf[1:] = ud.reshape(-1)
    uu = buf[1:].view(u.shape)
    assert uu.data_ptr() % 16 != 0
    a = plan.step(phid, ud, 1, diag=True)
    b = plan.step(phid, uu, 1, diag=True)
    assert abs(a["mass"] - b["mass"]) <= 1e-13 * abs(a["mass"])
    assert float((ud - uu).norm()) <= 1e-12 * float(ud.norm())


@pytest.mark.parametrize("at", ["all", "one"])
def test_energy_sums_past_fp32_range(at):
    """Sums that leave FP32's range come out as the FP64 sums of the FP32 terms: |u| = 2e9, where
    W(u) = 2.88e38 still fits FP32, at every point (the sums do not fit) or at one."""
    p = _params((64, 32, 32), 1).replace(gamma=0.0, M=0.0, ubar=0.3)
    rng = np.random.default_rng(8)
    phi = _membrane(p, "full", rng).astype(np.float32).astype(np.float64)
    u = np.full(p.shape, 2e9) if at == "all" else rng.uniform(0.2, 0.9, size=p.shape)
    if at == "one":
        u[7, 9, 11] = 2.1e9        # W(u) past FP32: infinite, as FP32 has it
    u = u.astype(np.float32).astype(np.float64)
    band, G = obm.band_mask(phi, p.band_mask_hi), omodel.g_loc(phi)
    plan = Plan(p)
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device=DEV)  # noqa: E731
    d = plan.energy(dev(phi), dev(u))
    h3 = float(np.prod(p.h[:3]))
    if at == "all":
        want = h3 * float((G * 18.0 * (u * u - u) ** 2).sum()) / p.eps_u
        assert abs(d["energy"] - want) <= 3e-6 * want
    else:
        assert d["energy"] == np.inf and d["umax"] == u.max()
    mass = h3 * float((G * (3 * u * u - 2 * u ** 3 - p.ubar)).sum())
    assert abs(d["mass"] - mass) <= 3e-6 * abs(mass)
