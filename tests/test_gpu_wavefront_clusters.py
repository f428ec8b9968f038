"""Tile shapes of the sheared wavefront that only wide grids reach: four planes
(FP64) and eight planes (FP32) per tile, clusters of two, four and eight tiles,
units that end early, and more tiles than clusters are resident at once.
Sequential sweeps and factors of the oracle in FP64; the matrices are small
integers over powers of two, so reduced precision only rounds values and sums
(27 terms and a diagonal, contracting by 78/128 a row: 27 * eps / (1 - 78/128),
with the larger of that and the repository's bounds)."""
import numpy as np
import pytest

from paper_2506_21932_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 2e-5}
# planes per tile, tiles per cluster
# planes per tile, tiles per cluster
CASES = [((200, 200, 2), 27, 0),   # 4, 4
         ((416, 240, 2), 27, 0),   # 4, 2
         ((336, 328, 2), 27, 1),   # 8, 4
         ((152, 280, 3), 7, 1),    # 4, 4
         ((96, 88, 4), 19, 1),     # 4, 8
         ((72, 64, 3), 27, 0)]     # 2, 8


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_21932_gb300 import build, smg
    build.build()
    return smg


@pytest.fixture(scope="module")
def orc():
    from oracle import oracle
    oracle.build()
    return oracle


@pytest.mark.parametrize("d,mask,prec", CASES)
def test_wide_grids_equal_the_sequential_sweeps(S, orc, d, mask, prec):
    off = {7: I.OFF7, 19: I.OFF19, 27: I.OFF27}[mask]
    rng = np.random.default_rng(11)
    i, j, k = np.meshgrid(*(np.arange(t) for t in d), indexing="ij")
    A = np.zeros((*d, len(off)))
    for e, o in enumerate(off):
        ok = np.ones(d, dtype=bool)
        for x, t, n in zip((i, j, k), o, d):
            ok &= (x + t >= 0) & (x + t < n)
        A[..., e] = np.where(ok, -rng.integers(1, 4, size=d), 0.0)
    A[..., off.index((0, 0, 0))] = 128.0
    A = A.reshape(-1, len(off))
    n = A.shape[0]
    dt = torch.float64 if prec == 0 else torch.float32
    dev = lambda v: torch.from_numpy(v).to(dt).cuda()
    b, u0 = rng.normal(size=(2, n))
    Dinv = orc.diag_inverse(d, off, A)
    err = lambda got, ref: np.linalg.norm(got.double().cpu().numpy() - ref) / np.linalg.norm(ref)
    kry = S.PCG if prec == 0 else S.FPCG
    h = S.SMG(d, off, torch.from_numpy(A).cuda(), smoother=S.SGS, precision=prec, krylov=kry,
              transfer=S.C16XY)
    x = dev(u0)
    h.level_apply(0, S.OP_GS_FORWARD, x=x, b=dev(b))
    fwd = orc.gs_forward(d, off, A, Dinv, b, u0)
    assert err(x, fwd) <= TOL[prec]
    x = dev(u0)
    h.level_apply(0, S.OP_GS_BACKWARD, x=x, b=dev(b))
    assert err(x, orc.gs_backward(d, off, A, Dinv, b, u0)) <= TOL[prec]
    h.close()
