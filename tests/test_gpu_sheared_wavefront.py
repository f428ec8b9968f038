"""Edges of the sheared wavefront solves: strips of 32 x-points (31, 32, 33,
65 and 1 points), fewer y-points than planes in a tile, columns of one and two
points, every mask and precision, weights other than one.  The solves of one
level are compared with dense triangular solves of the same matrix in FP64;
the bounds are those of the repository's parity tests (27 terms and a diagonal
in FP64, FP32 rounding of the stored values otherwise)."""
import numpy as np
import pytest

from paper_2506_21932_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = [(33, 3, 5), (31, 4, 2), (32, 2, 9), (65, 2, 1), (1, 1, 7), (2, 41, 3), (40, 1, 6), (5, 19, 4)]
MASKS = {7: I.OFF7, 19: I.OFF19, 27: I.OFF27}
TOL = {0: 1e-12, 1: 2e-5, 2: 2e-5}


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


def matrix(d, off, seed):
    """Nonsymmetric diagonally dominant stencil matrix with powers of two and
    small integers, exact in FP32 and (divided by its row scale) in BF16."""
    rng = np.random.default_rng(seed)
    i, j, k = np.meshgrid(*(np.arange(t) for t in d), indexing="ij")
    A = np.zeros((*d, len(off)))
    for e, o in enumerate(off):
        ok = np.ones(d, dtype=bool)
        for x, t, n in zip((i, j, k), o, d):
            ok &= (x + t >= 0) & (x + t < n)
        A[..., e] = np.where(ok, -rng.integers(1, 4, size=d), 0.0)
    A[..., off.index((0, 0, 0))] = 128.0
    return A.reshape(-1, len(off))


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("mask", [7, 19, 27])
@pytest.mark.parametrize("d", DIMS)
def test_gauss_seidel_and_ilu_solves_equal_dense_ones(S, orc, d, mask, prec):
    off = MASKS[mask]
    A = matrix(d, off, 3)
    n = A.shape[0]
    full = orc.assemble_dense(d, off, A)
    lo, up, D = np.tril(full, -1), np.triu(full, 1), np.diag(np.diag(full))
    rng = np.random.default_rng(5)
    b, u0 = rng.normal(size=n), rng.normal(size=n)
    dt = torch.float64 if prec == 0 else torch.float32
    dev = lambda v: torch.from_numpy(v).to(dt).cuda()
    host = lambda t: t.double().cpu().numpy()
    close = lambda got, ref: np.linalg.norm(host(got) - ref) <= TOL[prec] * np.linalg.norm(ref)
    kry = S.PCG if prec == 0 else S.FPCG
    for w in (1.0, 0.75):
        h = S.SMG(d, off, torch.from_numpy(A).cuda(), smoother=S.SGS, precision=prec, krylov=kry, relax_w=w,
                  max_levels=1)
        for op, low, high in ((S.OP_GS_FORWARD, lo, up), (S.OP_GS_BACKWARD, up, lo)):
            # one unknown at a time: u_p <- (1 - w) u_p + w (b_p - ...) / a_pp
            x = dev(u0)
            h.level_apply(0, op, x=x, b=dev(b))
            ref = np.linalg.solve(D / w + low, b - high @ u0 + (1.0 / w - 1.0) * (D @ u0))
            assert close(x, ref), (op, w)
        x = dev(u0)
        h.level_apply(0, S.OP_GS_ZERO, x=x, b=dev(b))
        assert close(x, np.linalg.solve(D / w + lo, b)), ("zero", w)
        h.close()
    h = S.SMG(d, off, torch.from_numpy(A).cuda(), smoother=S.ILU0, precision=prec, krylov=kry, max_levels=1)
    if prec == 0:  # the reduced factors are rounded: parity with the oracle's cycle covers them
        LU = orc.assemble_dense(d, off, orc.ilu0_factor(d, off, A))
        y, z = dev(b), torch.empty(n, dtype=dt, device="cuda")
        h.level_apply(0, S.OP_ILU_LOWER, b=y, y=y)
        ref = np.linalg.solve(np.tril(LU, -1) + np.eye(n), b)
        assert close(y, ref)
        h.level_apply(0, S.OP_ILU_UPPER, b=y, y=z)
        assert close(z, np.linalg.solve(np.triu(LU), ref))
        h.level_apply(0, S.OP_ILU_APPLY, b=dev(b), y=y)
        assert torch.equal(y, z)
    h.close()
