"""The grid barrier's verdict and what the band solve does when one gives up.

On the CPU: every order of the steps of three blocks over two barriers, with the functions of
csrc/barrier.h themselves deciding, any block free to give up while it waits.  A barrier has to
end the same way in every block: blocks of one thread-block cluster that disagreed about it would
part, and one would read the shared memory of another that has left.

On the GPU: the grid and the hybrid engine (bands past one cluster; the 32^3 band of
test_gpu_timeouts.py runs on the cluster engine) with limits that run out before the solve, in
the middle of it, and not at all.
"""
import ctypes as ct
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2606_04347_gb300.build import CSRC

WAIT, PASS, FAIL = 'wait', 'pass', 'fail'
SHIM = """
#include "barrier.h"
extern "C" {
uint32_t target(uint32_t w, uint32_t nb) { return etd::bar_target(w, nb); }
int decided(uint32_t w, uint32_t t) { return etd::bar_decided(w, t); }
int passed(uint32_t w, uint32_t t, uint32_t nb) { return etd::bar_passed(w, t, nb); }
uint32_t closed(uint32_t t) { return etd::bar_closed(t); }
}
"""


@pytest.fixture(scope="module")
def word(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("barrier")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    lib = ct.CDLL(str(d / "shim.so"))
    u32 = ct.c_uint32
    lib.target.restype, lib.target.argtypes = u32, [u32, u32]
    lib.decided.restype, lib.decided.argtypes = ct.c_int, [u32, u32]
    lib.passed.restype, lib.passed.argtypes = ct.c_int, [u32, u32, u32]
    lib.closed.restype, lib.closed.argtypes = u32, [u32]
    return lib


def _verdict(word, w, target, nb):
    return WAIT if not word.decided(w, target) else PASS if word.passed(w, target, nb) else FAIL


def _endings(word, nb, nbar, start, private):
    """All reachable endings: for each, the verdicts of every barrier over the blocks.  A block is
    ("run", e): about to arrive at barrier e; ("wait", e, t); ("swap", e, t, w): about to close the
    word it saw as w; ("left",).  private: a block that gives up fails by itself, the word open."""
    seen, ends = set(), set()
    todo = [(start, (("run", 0),) * nb, ((),) * nbar)]
    while todo:
        s = todo.pop()
        if s in seen:
            continue
        seen.add(s)
        w, blocks, verd = s
        if all(b[0] == "left" for b in blocks):
            ends.add(verd)
            continue
        for k, b in enumerate(blocks):
            def go(nw, nbk, e=None, v=None):
                nv = verd if e is None else tuple(tuple(sorted(x + (v,))) if i == e else x for i, x in enumerate(verd))
                todo.append((nw, blocks[:k] + (nbk,) + blocks[k + 1:], nv))

            def judged(nw, e, t, v):
                if v == WAIT:
                    go(nw, ("wait", e, t))
                else:
                    go(nw, ("run", e + 1) if v == PASS and e + 1 < nbar else ("left",), e, v)
            if b[0] == "run":
                t = word.target(w, nb)
                judged(w + 1, b[1], t, _verdict(word, w + 1, t, nb))
            elif b[0] == "wait":
                v = _verdict(word, w, b[2], nb)
                if v != WAIT:
                    judged(w, b[1], b[2], v)
                elif private:
                    go(w, ("left",), b[1], FAIL)
                else:
                    go(w, ("swap", b[1], b[2], w))
            elif b[0] == "swap":
                if w == b[3]:
                    judged(word.closed(b[2]), b[1], b[2], FAIL)
                else:
                    go(w, ("wait", b[1], b[2]))
    return ends


@pytest.mark.parametrize("start", [0, 3 * 1000])
def test_every_block_gets_the_same_verdict(word, start):
    ends = _endings(word, 3, 2, start, private=False)
    assert ((PASS,) * 3, (PASS,) * 3) in ends and any(FAIL in v for e in ends for v in e)
    for e in ends:
        for v in e:
            assert len(set(v)) <= 1 and len(v) in (0, 3), ends   # nobody ends a barrier that others never reach


def test_verdicts_taken_alone_differ(word):
    """The rule that the word replaces: a block that gives up fails by itself."""
    assert any(set(v) == {PASS, FAIL} for e in _endings(word, 3, 2, 0, private=True) for v in e)


def test_word_of_late_and_early_blocks(word):
    nb = 152
    v = lambda w, t: _verdict(word, w, t, nb)  # noqa: E731
    w = word.closed(6 * nb)                        # barrier 6 given up with 7 blocks there
    for late in range(nb - 7):
        assert v(w + late + 1, word.target(w + late, nb)) == FAIL and v(w + late + 1, 6 * nb) == FAIL
        assert v(w + late + 1, 5 * nb) == PASS     # still polling barrier 5, which was complete
    assert v(5 * nb + 7, 6 * nb) == WAIT and v(6 * nb, 6 * nb) == PASS and v(7 * nb - 1, 6 * nb) == PASS


# ---- the band solve ------------------------------------------------------------------------

torch = pytest.importorskip("torch")

from oracle import band as obm  # noqa: E402
from oracle import model as omodel  # noqa: E402
from paper_2606_04347_gb300 import Plan  # noqa: E402
from paper_2606_04347_gb300 import workloads as wl  # noqa: E402
from paper_2606_04347_gb300.abi import EtdError  # noqa: E402


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [(128, 128, 64),    # 93 k nodes, the hybrid engine
                               (128, 128, 128)])  # 186 k nodes, the grid engine
def test_solve_that_gives_up_leaves_the_device_usable(monkeypatch, n, prec):
    """Limits from none to more than a whole solve: each call reports ETD_ETIMEOUT or the solution
    (its residual formed by the oracle's operator, with the bound of the large-band tests), and the
    first limit always gives up."""
    p = wl.workload("c2", n=16)[0].replace(dim=3, n=n, model=0, precision=prec, cg_rtol=1e-12 if prec == 0 else 1e-6)
    r = np.sqrt(sum(c ** 2 for c in wl.grid(n, p.half_len, 3)))
    dt = np.float64 if prec == 0 else np.float32
    phi = (wl.tanh_profile(1.6 - r, 0.09) * np.ones(p.shape)).astype(dt).astype(np.float64)
    band, g = obm.band_mask(phi, p.band_mask_hi), omodel.g_loc(phi)
    f = np.where(band, np.random.default_rng(3).uniform(-1.0, 1.0, size=p.shape), 0.0).astype(dt).astype(np.float64)
    b = np.where(band, f - f[band].mean(), 0.0)
    cf = obm.face_coeffs(g, band)
    tdt = torch.float64 if prec == 0 else torch.float32
    phid, fd = (torch.tensor(a, dtype=tdt, device="cuda:0") for a in (phi, f))
    w = torch.zeros(p.shape, dtype=tdt, device="cuda:0")
    gave_up = []
    for budget in (-1, 0, 500, 1500, 2000, 2500, 3000, 4000, 6000, 10000, 30000, None):
        if budget is not None:
            monkeypatch.setenv("ETD_WAIT_BUDGET", str(budget))
        plan = Plan(p)
        monkeypatch.delenv("ETD_WAIT_BUDGET", raising=False)
        for _ in range(4):
            w.zero_()
            try:
                plan.nonlocal_solve(phid, fd, w)
            except EtdError as e:
                assert e.code == 6
                gave_up.append(budget)
                continue
            res = b - obm.apply_neg_lap(w.cpu().numpy().astype(np.float64), cf, p.h)
            assert np.linalg.norm(res) <= (1e-10 if prec == 0 else 1e-3) * np.linalg.norm(b)
        plan.close()
    assert gave_up.count(-1) == 4 and None not in gave_up


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(32, 32, 32), (128, 128, 64), (128, 128, 128)])   # cluster, hybrid, grid engine
def test_solves_after_a_failure_keep_its_report(n):
    """A solve that does not converge sets the status word; the solves after it return at once, the
    report is the first failure's, and the plan works on."""
    p = wl.workload("c2", n=16)[0].replace(dim=3, n=n, model=0, precision=1, scheme=1, cg_rtol=1e-6, cg_maxit=2)
    r = np.sqrt(sum(c ** 2 for c in wl.grid(n, p.half_len, 3)))
    phi = torch.tensor(wl.tanh_profile(1.6 - r, 0.09) * np.ones(p.shape), dtype=torch.float32, device="cuda:0")
    u = torch.tensor(np.random.default_rng(5).uniform(0.3, 0.7, size=p.shape), dtype=torch.float32, device="cuda:0")
    plan = Plan(p)
    for _ in range(2):
        plan.step(phi, u, 3)
        with pytest.raises(EtdError) as ei:
            plan.step(None, u, 0, diag=True)
        assert ei.value.code == 5
        assert plan.step(None, u, 0, diag=True)["cg_iters_last"] == 2
