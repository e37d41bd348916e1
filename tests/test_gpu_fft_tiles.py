"""Transforms at the sizes where the tile rules change, and R1 where its wide loads cannot run.

Pass A with fewer row pairs than teams (small extents, 2D, FP64's two-plane tiles), pass B with
one and with several pencil blocks per CTA and a ragged last one.  Against numpy's FP64 FFT of
the same input: an FFT of N points keeps a relative L2 error of about eps log2 N (1e-13 and 2e-6
are the bounds of the other transform tests).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2606_04347_gb300 import Plan  # noqa: E402
from paper_2606_04347_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("prec,tol", [(0, 1e-13), (1, 2e-6)])
@pytest.mark.parametrize("n", [(8, 8, 8), (16, 64, 128), (64, 64, 64), (128, 128, 64), (256, 32, 16), (32, 256, 32),
                               (64, 128, 96), (96, 16, 64), (8, 256, 1), (256, 8, 1), (96, 128, 1)])
def test_transforms_match_numpy(n, prec, tol):
    dim = 2 if n[2] == 1 else 3
    p = wl.workload("c2", n=16)[0].replace(dim=dim, n=n, model=0, precision=prec)
    plan = Plan(p)
    f = torch.tensor(wl.random_fields(p.shape, 3, -1.0, 1.0), dtype=plan.dtype, device=DEV)
    half = torch.zeros(p.shape[:-1] + (n[0] // 2 + 1,), dtype=plan.cdtype, device=DEV)
    back = torch.zeros_like(f)
    plan.fft_forward(f, half)
    plan.fft_inverse(half, back)
    want = np.fft.rfftn(f.cpu().numpy().astype(np.float64))
    assert np.linalg.norm(half.cpu().numpy() - want) < tol * np.linalg.norm(want)
    assert float((back.double() - f.double()).norm()) < tol * float(f.double().norm())


@pytest.mark.parametrize("prec,tol", [(0, 1e-11), (1, 2e-5)])
def test_r1_of_an_unaligned_field_matches_oracle(prec, tol):
    """u one element past a 16-byte boundary takes the one-point loads (the bounds of the aligned
    R1 test; not bit for bit, the volume in R1 being a sum of atomics)."""
    from oracle import model as omodel
    p, phi, u, _ = wl.workload("c3", n=32, precision=prec)
    p = p.replace(A0=omodel.volume(phi, p) - 0.05)
    plan = Plan(p)
    dt = plan.dtype
    phid = torch.tensor(phi, dtype=dt, device=DEV)
    buf = torch.zeros(u.size + 1, dtype=dt, device=DEV)
    buf[1:] = torch.tensor(u, dtype=dt, device=DEV).reshape(-1)
    uu = buf[1:].view(u.shape)
    assert uu.data_ptr() % 16 != 0
    out = torch.zeros_like(phid)
    plan.remainder(1, phid, None, uu, out)
    want = omodel.R1(phi, u, p, p.A0)
    assert np.linalg.norm(out.cpu().numpy() - want) < tol * np.linalg.norm(want)


@pytest.mark.parametrize("n", [(256, 256, 256), (128, 256, 256), (256, 128, 128), (256, 256, 64), (96, 256, 64)])
def test_large_standard_layout_transforms_match_numpy(n):
    """FP32 pass B with several kx a CTA on its way to and from the standard layout, with whole
    and ragged last groups (the bound of the transforms above; the arrays end exactly at the grid)."""
    p = wl.workload("c2", n=16)[0].replace(dim=3, n=n, model=0, precision=1)
    plan = Plan(p)
    f = torch.tensor(wl.random_fields(p.shape, 5, -1.0, 1.0), dtype=plan.dtype, device=DEV)
    half = torch.zeros(p.shape[:-1] + (n[0] // 2 + 1,), dtype=plan.cdtype, device=DEV)
    back = torch.zeros_like(f)
    plan.fft_forward(f, half)
    plan.fft_inverse(half, back)
    want = np.fft.rfftn(f.cpu().numpy().astype(np.float64))
    assert np.linalg.norm(half.cpu().numpy() - want) < 2e-6 * np.linalg.norm(want)
    assert float((back.double() - f.double()).norm()) < 2e-6 * float(f.double().norm())
