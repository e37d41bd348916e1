"""Component labels of a frozen band, which are made once for all its steps.

The labels have to be there, or be reported as missing by every step, whatever was reported
before: an earlier solve that did not converge, or a band of more components than the solve takes.
Bounds: those of the fixed-membrane step tests.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import band as obm  # noqa: E402
from oracle import etd as oetd  # noqa: E402
from paper_2606_04347_gb300 import Plan  # noqa: E402
from paper_2606_04347_gb300 import workloads as wl  # noqa: E402
from paper_2606_04347_gb300.abi import EtdError  # noqa: E402

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.tensor(a, dtype=torch.float64, device="cuda:0")


def _params(n, **kw):
    return wl.workload("c2", n=16)[0].replace(dim=3, n=(n, n, n), model=0, precision=0, scheme=1, tau=1e-3, cg_rtol=1e-13, **kw)


def _pairs(n):
    """Pairs of nodes along z in columns that touch diagonally: labelled by the union-find, and
    solved in two or three iterations."""
    z, y, x = np.meshgrid(*[np.arange(n)] * 3, indexing="ij")
    return np.where(((x + y) % 2 == 0) & (z % 4 < 2), 0.5, 0.0)


def _step_matches_oracle(plan, p, phi, u):
    want = oetd.FixedStepper(p, phi).run(u.copy(), 1)
    ud = _dev(u)
    plan.step(None, ud, 1, diag=True)
    assert np.linalg.norm(ud.cpu().numpy() - want) < 1e-11 * np.linalg.norm(want)


def test_band_frozen_after_a_solve_that_did_not_converge():
    p = _params(16, cg_maxit=6)
    rng = np.random.default_rng(1)
    full, pairs = rng.uniform(0.2, 0.8, size=p.shape), _pairs(16)
    u = rng.uniform(0.3, 0.7, size=p.shape)
    assert obm.components(obm.band_mask(pairs, p.band_mask_hi))[1] == 512
    plan = Plan(p)
    plan.step(_dev(full), _dev(u), 1)          # 15 iterations wanted; nothing looks at it yet
    plan.step(_dev(pairs), _dev(u), 0)
    with pytest.raises(EtdError) as ei:
        plan.step(None, _dev(u), 0, diag=True)
    assert ei.value.code == 5
    _step_matches_oracle(plan, p, pairs, u)


def test_too_many_components_are_reported_by_every_step():
    p = _params(32)
    z, y, x = np.meshgrid(*[np.arange(32)] * 3, indexing="ij")
    u = np.random.default_rng(2).uniform(0.3, 0.7, size=p.shape)
    plan, ud = Plan(p), _dev(u)
    phi = _dev(np.where((x + y + z) % 2 == 0, 0.5, 0.0))      # 16384 single nodes
    for k in range(3):
        with pytest.raises(EtdError) as ei:
            plan.step(phi if k == 0 else None, ud, 1, diag=True)
        assert ei.value.code == 1
    pairs = _pairs(32)                                         # 4096 components: the most it takes
    assert obm.components(obm.band_mask(pairs, p.band_mask_hi))[1] == 4096
    plan.step(_dev(pairs), ud, 0, diag=True)
    _step_matches_oracle(plan, p, pairs, u)
