"""Tile shapes of the sheared wavefront that only wide grids reach: four planes
(FP64) and eight planes (FP32) per tile, clusters of two, four and eight tiles,
units that end early, and more tiles than clusters are resident at once.
Single sweeps against the oracle's sequential ones in FP64; the matrices are
small integers over powers of two, so reduced precision only rounds values and
sums (27 terms and a diagonal, contracting by 78/128 a row: 27 * eps /
(1 - 78/128), with the larger of that and the repository's bounds).  Cycles, whose
solves write to the mirrored stream, in place, with sums handed on and with a
weight, against the same cycle put together from single level operations."""
import numpy as np
import pytest

from paper_2506_21932_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 2e-5}
EPS = {0: 2.3e-16, 1: 1.2e-7, 2: 1.2e-7}
# planes per tile, tiles per cluster
CASES = [((200, 200, 2), 27, 0),   # 4, 4
         ((416, 240, 2), 27, 0),   # 4, 2
         ((336, 328, 2), 27, 1),   # 8, 4
         ((152, 280, 3), 7, 1),    # 4, 4
         ((96, 88, 4), 19, 1),     # 4, 8
         ((72, 64, 3), 27, 0),     # 2, 8
         ((24, 400, 3), 27, 0)]    # 2, 8; its level operations run in natural order


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


def matrix(d, off, rng):
    i, j, k = np.meshgrid(*(np.arange(t) for t in d), indexing="ij")
    A = np.zeros((*d, len(off)))
    for e, o in enumerate(off):
        ok = np.ones(d, dtype=bool)
        for x, t, n in zip((i, j, k), o, d):
            ok &= (x + t >= 0) & (x + t < n)
        A[..., e] = np.where(ok, -rng.integers(1, 4, size=d), 0.0)
    A[..., off.index((0, 0, 0))] = 128.0
    return A.reshape(-1, len(off))


@pytest.mark.parametrize("d,mask,prec", CASES)
def test_wide_grids_equal_the_sequential_sweeps(S, orc, d, mask, prec):
    off = {7: I.OFF7, 19: I.OFF19, 27: I.OFF27}[mask]
    rng = np.random.default_rng(11)
    A = matrix(d, off, rng)
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


@pytest.mark.parametrize("smoother,w", [("ILU0", 1.0), ("SGS", 1.0), ("SGS", 0.8)])
@pytest.mark.parametrize("d,mask,prec", CASES + [((200, 200, 2), 27, 2), ((264, 104, 3), 19, 2)])  # BF16: 4, 4 and 4, 8
def test_wide_cycles_equal_their_level_operations(S, d, mask, prec, smoother, w):
    off = {7: I.OFF7, 19: I.OFF19, 27: I.OFF27}[mask]
    rng = np.random.default_rng(13)
    h = S.SMG(d, off, torch.from_numpy(matrix(d, off, rng)).cuda(), smoother=getattr(S, smoother), precision=prec,
              krylov=S.PCG if prec == 0 else S.FPCG, transfer=S.C16XY, relax_w=w)
    nl = h.stats()["levels"]
    size = [int(np.prod(h.level_info(l)[0])) for l in range(nl)]
    dt = torch.float64 if prec == 0 else torch.float32
    new = lambda m: torch.zeros(m, dtype=dt, device="cuda")

    def cycle(l, f):
        n, u = size[l], new(size[l])
        if l == nl - 1:
            u = u.double()
            h.level_apply(l, S.OP_COARSE_SOLVE, b=f.double(), y=u)
            return u.to(dt)
        t, c = new(n), new(size[l + 1])
        if smoother == "ILU0":
            h.level_apply(l, S.OP_ILU_APPLY, b=f, y=u)
        else:
            h.level_apply(l, S.OP_GS_ZERO, x=u, b=f)
            h.level_apply(l, S.OP_GS_BACKWARD, x=u, b=f)
        h.level_apply(l, S.OP_RESIDUAL, x=u, b=f, y=t)
        h.level_apply(l, S.OP_RESTRICT, x=t, y=c)
        h.level_apply(l, S.OP_PROLONG_ADD, x=cycle(l + 1, c), y=u)
        if smoother == "ILU0":
            e = new(n)
            h.level_apply(l, S.OP_RESIDUAL, x=u, b=f, y=t)
            h.level_apply(l, S.OP_ILU_APPLY, b=t, y=e)
            u += e
        else:
            h.level_apply(l, S.OP_GS_FORWARD, x=u, b=f)
            h.level_apply(l, S.OP_GS_BACKWARD, x=u, b=f)
        return u

    r = torch.from_numpy(rng.normal(size=size[0])).cuda()
    z = torch.zeros_like(r)
    h.vcycle(r, z)
    u = cycle(0, r.to(dt)).double()
    # per level six operations of at most 28 rounded terms each, of stored values
    # that are the same in both; none amplifies (rows of 77/128)
    assert torch.linalg.norm(z - u) <= 6 * 28 * EPS[prec] * nl * torch.linalg.norm(z)
    h.close()
