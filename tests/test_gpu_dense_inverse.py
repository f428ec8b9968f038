"""The coarsest level's dense inverse at the edges of its blocks (16 columns,
8 CTAs of rows): direct solves of matrices whose pivots need row exchanges,
within and across blocks, against numpy.  The bound on the solution's error is
the first-order one of elimination with partial pivoting, n^2 eps times the
condition number."""
import numpy as np
import pytest

from paper_2506_21932_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_21932_gb300 import build, smg
    build.build()
    return smg


@pytest.mark.parametrize("d", [(1, 1, 1), (1, 1, 2), (3, 5, 1), (1, 4, 4), (1, 1, 17), (1, 31, 1), (3, 11, 1),
                               (5, 5, 5), (1, 129, 1), (5, 3, 17), (9, 8, 7), (3, 9, 33)])
def test_direct_solve_with_row_exchanges(S, d):
    rng = np.random.default_rng(int(np.prod(d)))
    n = int(np.prod(d))
    off = I.OFF27
    A = np.zeros((*d, 27))
    i, j, k = np.meshgrid(*(np.arange(t) for t in d), indexing="ij")
    full = np.zeros((n, n))
    idx = np.arange(n).reshape(d)
    for e, o in enumerate(off):
        ok = np.ones(d, dtype=bool)
        for x, t, m in zip((i, j, k), o, d):
            ok &= (x + t >= 0) & (x + t < m)
        # a small diagonal: most columns take their pivot from another row
        v = rng.uniform(-1, 1, size=d) * (0.05 if o == (0, 0, 0) else 1.0) + (0.01 if o == (0, 0, 0) else 0.0)
        A[..., e] = np.where(ok, v, 0.0)
        p = idx[ok]
        q = p + (o[0] * d[1] + o[1]) * d[2] + o[2]
        full[p, q] = A[..., e][ok]
    h = S.SMG(d, off, torch.from_numpy(A.reshape(n, 27)).cuda(), smoother=S.SGS, max_levels=1)
    b = rng.normal(size=n)
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    h.level_apply(0, S.OP_COARSE_SOLVE, b=torch.from_numpy(b).cuda(), y=y)
    ref = np.linalg.solve(full, b)
    bound = n * n * 2.0 ** -53 * np.linalg.cond(full) + 1e-15
    assert np.linalg.norm(y.cpu().numpy() - ref) <= bound * np.linalg.norm(ref)


def test_singular_matrix_is_a_breakdown(S):
    d = (2, 3, 4)
    A = np.zeros((24, 7))
    A[:, 3] = 1.0
    A[20, 3] = 0.0  # a zero column past the first block
    with pytest.raises(S.SmgError) as e:
        S.SMG(d, I.OFF7, torch.from_numpy(A).cuda(), smoother=S.SGS, max_levels=1)
    assert e.value.status == S.EBREAKDOWN
