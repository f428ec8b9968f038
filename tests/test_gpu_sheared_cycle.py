"""Packing and residual kernels of the sheared wavefront at the edges of their
tiles (columns of 70, 130 and 32 points in tiles of 64 and 32, two and three
strips, planes beyond the strip): a two-level V-cycle, which residuals and packs
straight into the sweeps' order, equals the same cycle put together from single
level operations in natural order.  Both form the same sums in the same order
from the same stored values, so what may differ is a last-bit rounding of each
of the six operations, not amplified: the smoothers contract (rows of 77/128)."""
import numpy as np
import pytest

from paper_2506_21932_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = {0: 2.3e-16, 1: 1.2e-7, 2: 1.2e-7}


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_21932_gb300 import build, smg
    build.build()
    return smg


@pytest.mark.parametrize("smoother", ["ILU0", "SGS"])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("mask", [7, 19, 27])
@pytest.mark.parametrize("d", [(34, 10, 70), (8, 12, 130), (70, 8, 32)])
def test_cycle_equals_its_level_operations(S, d, mask, prec, smoother):
    off = {7: I.OFF7, 19: I.OFF19, 27: I.OFF27}[mask]
    rng = np.random.default_rng(3)
    i, j, k = np.meshgrid(*(np.arange(t) for t in d), indexing="ij")
    A = np.zeros((*d, len(off)))
    for e, o in enumerate(off):
        ok = np.ones(d, dtype=bool)
        for x, t, n in zip((i, j, k), o, d):
            ok &= (x + t >= 0) & (x + t < n)
        A[..., e] = np.where(ok, -rng.integers(1, 4, size=d), 0.0)
    A[..., off.index((0, 0, 0))] = 128.0
    n, nc = int(np.prod(d)), int(np.prod(d)) // 8
    h = S.SMG(d, off, torch.from_numpy(A.reshape(n, -1)).cuda(), smoother=getattr(S, smoother), precision=prec,
              krylov=S.PCG if prec == 0 else S.FPCG, max_levels=2)
    dt = torch.float64 if prec == 0 else torch.float32
    new = lambda m: torch.zeros(m, dtype=dt, device="cuda")
    r = torch.from_numpy(rng.normal(size=n)).cuda()
    z = torch.zeros_like(r)
    h.vcycle(r, z)
    f, u, t, c = r.to(dt), new(n), new(n), new(nc)
    if smoother == "ILU0":
        h.level_apply(0, S.OP_ILU_APPLY, b=f, y=u)
    else:
        h.level_apply(0, S.OP_GS_ZERO, x=u, b=f)
        h.level_apply(0, S.OP_GS_BACKWARD, x=u, b=f)
    h.level_apply(0, S.OP_RESIDUAL, x=u, b=f, y=t)
    h.level_apply(0, S.OP_RESTRICT, x=t, y=c)
    uc = torch.zeros(nc, dtype=torch.float64, device="cuda")
    h.level_apply(1, S.OP_COARSE_SOLVE, b=c.double(), y=uc)
    h.level_apply(0, S.OP_PROLONG_ADD, x=uc.to(dt), y=u)
    if smoother == "ILU0":
        e = new(n)
        h.level_apply(0, S.OP_RESIDUAL, x=u, b=f, y=t)
        h.level_apply(0, S.OP_ILU_APPLY, b=t, y=e)
        u += e
    else:
        h.level_apply(0, S.OP_GS_FORWARD, x=u, b=f)
        h.level_apply(0, S.OP_GS_BACKWARD, x=u, b=f)
    # six operations of at most 28 rounded terms each
    assert torch.linalg.norm(z - u.double()) <= 6 * 28 * EPS[prec] * torch.linalg.norm(z)
    h.close()
