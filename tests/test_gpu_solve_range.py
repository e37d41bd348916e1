"""The band solve over the range of its right-hand sides and guesses.

(b,b) and its like are formed in double-float, which has FP32's exponents.  The solve is linear
and every scaling in it is by a power of two, so a right-hand side times 2^k has the solution times
2^k to the bit as long as nothing of it is denormal.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2606_04347_gb300 import Plan  # noqa: E402
from paper_2606_04347_gb300 import workloads as wl  # noqa: E402
from paper_2606_04347_gb300.abi import EtdError  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(32, 32, 32), (128, 128, 64), (128, 128, 128)])   # cluster, hybrid, grid engine
@pytest.mark.parametrize("blobs", [1, 2])
def test_solution_scales_with_the_right_hand_side(n, blobs):
    p = wl.workload("c2", n=16)[0].replace(dim=3, n=n, model=0, precision=1, cg_rtol=1e-6)
    x, y, z = wl.grid(n, p.half_len, 3)
    if blobs == 1:
        phi = wl.tanh_profile(1.6 - np.sqrt(x * x + y * y + z * z), 0.25)
    else:   # two components: the per-component means, which are summed in FP64
        phi = sum(wl.tanh_profile(0.9 - np.sqrt((x - s) ** 2 + y * y + z * z), 0.2) for s in (-1.6, 1.6))
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda:0")  # noqa: E731
    phid = dev(phi * np.ones(p.shape))
    f = dev(np.random.default_rng(6).uniform(-1.0, 1.0, size=p.shape))
    plan = Plan(p)
    w = torch.zeros_like(f)
    it, res = plan.nonlocal_solve(phid, f, w)
    assert it > 0 and 0 < res <= 1e-6
    for k in (-80, -50, 40, 62, 100):
        wk = torch.zeros_like(f)
        got = plan.nonlocal_solve(phid, f * 2.0 ** k, wk)
        if blobs == 1:
            assert got == (it, res) and torch.equal(wk, w * 2.0 ** k)
        else:   # sums of FP64 atomics, whose order varies: the bound of the residual
            assert got[0] > 0 and 0 < got[1] <= 1e-6
            d = (wk.double() * 2.0 ** -k - w.double()).norm() / w.double().norm()
            assert float(d) < 2e-5
    wk = torch.zeros_like(f)
    assert plan.nonlocal_solve(phid, torch.zeros_like(f), wk)[0] == 0 and not wk.any()


@pytest.mark.parametrize("n", [(32, 32, 32), (128, 128, 64), (128, 128, 128)])
@pytest.mark.parametrize("prec,guess,rhs", [(0, 1e30, 1e-15), (1, 1e20, 1e-5)])
def test_hopeless_guess_is_not_reported_as_converged(n, prec, guess, rhs):
    """A guess whose rounding errors alone are far above the right-hand side cannot be brought to the
    tolerance; its residual leaves FP32's range if the right-hand side sets the scale."""
    p = wl.workload("c2", n=16)[0].replace(dim=3, n=n, model=0, precision=prec, cg_rtol=1e-12 if prec == 0 else 1e-6, cg_maxit=30)
    x, y, z = wl.grid(n, p.half_len, 3)
    phi = wl.tanh_profile(1.6 - np.sqrt(x * x + y * y + z * z), 0.25) * np.ones(p.shape)
    rng = np.random.default_rng(9)
    dev = lambda a: torch.tensor(a, dtype=torch.float64 if prec == 0 else torch.float32, device="cuda:0")  # noqa: E731
    with pytest.raises(EtdError) as ei:
        Plan(p).nonlocal_solve(dev(phi), dev(rhs * rng.uniform(-1, 1, p.shape)), dev(guess * rng.uniform(-1, 1, p.shape)))
    assert ei.value.code == 5
