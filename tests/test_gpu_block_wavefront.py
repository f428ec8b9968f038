"""Edges of the point-block wavefront solves (three unknowns per point, 7-point
mask): strips of 32 x-points (31, 32, 33, 65 and 1 points), fewer y-points than
planes in a tile, columns of one and two points, both precisions, weights other
than one.  The sweeps and one V(1,1)-cycle of a single level are compared with
dense block solves in FP64.

Bounds: a solve is a chain of products with D^-1 A, whose rows sum to less than
1/2, so errors of single steps add up to twice one step's error: 12 products
with blocks that carry the error of D^-1 (condition below 4): 2 * 12 * 4 * eps,
eps = 1.1e-16 or 6e-8, with a factor of 4 for the norm of the difference."""
import numpy as np
import pytest

from paper_2506_21932_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = [(33, 3, 5), (31, 4, 2), (32, 2, 9), (65, 2, 1), (1, 1, 7), (2, 41, 3), (40, 5, 6), (5, 19, 4)]
TOL = {0: 4 * 96 * 1.2e-16, 1: 4 * 96 * 6e-8}


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_21932_gb300 import build, smg
    build.build()
    return smg


def blocks(d, seed):
    """Nonsymmetric blocks, the diagonal ones dominant by a factor above 2."""
    rng = np.random.default_rng(seed)
    A = rng.uniform(-1, 1, size=(int(np.prod(d)), 7, 3, 3))
    A[:, 3] += 40.0 * np.eye(3)
    for p, ijk in enumerate(np.ndindex(*d)):
        for e, o in enumerate(I.OFF7):
            if not all(0 <= a + t < m for a, t, m in zip(ijk, o, d)):
                A[p, e] = 0.0
    return A


def dense(d, A):
    n = A.shape[0]
    full = np.zeros((n, 3, n, 3))
    for p, ijk in enumerate(np.ndindex(*d)):
        for e, o in enumerate(I.OFF7):
            q = tuple(a + t for a, t in zip(ijk, o))
            if all(0 <= a < m for a, m in zip(q, d)):
                full[p, :, np.ravel_multi_index(q, d), :] = A[p, e]
    return full.reshape(3 * n, 3 * n)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("d", DIMS)
def test_block_sweeps_and_smoothing_equal_dense_solves(S, d, prec):
    A = blocks(d, 3)
    if prec:
        A = A.astype(np.float32).astype(np.float64)
    full = dense(d, A)
    n = full.shape[0]
    blk = np.arange(n) // 3
    lo, up = full * (blk[:, None] > blk[None, :]), full * (blk[:, None] < blk[None, :])
    D = full - lo - up
    rng = np.random.default_rng(5)
    b, u0 = rng.normal(size=n), rng.normal(size=n)
    dt = torch.float64 if prec == 0 else torch.float32
    dev = lambda v: torch.from_numpy(v).to(dt).cuda()
    if prec:
        b, u0 = b.astype(np.float32).astype(np.float64), u0.astype(np.float32).astype(np.float64)
    err = lambda got, ref: np.linalg.norm(got.double().cpu().numpy() - ref) / np.linalg.norm(ref)
    for w in (1.0, 0.75):
        h = S.SMG(d, I.OFF7, torch.from_numpy(A).cuda(), block=3, smoother=S.SGS, precision=prec, krylov=S.FGMRES,
                  relax_w=w, max_levels=1)

        def half(low, high, u):
            return np.linalg.solve(D / w + low, b - high @ u + (1.0 / w - 1.0) * (D @ u))

        for op, low, high in ((S.OP_GS_FORWARD, lo, up), (S.OP_GS_BACKWARD, up, lo)):
            x = dev(u0)
            h.level_apply(0, op, x=x, b=dev(b))
            assert err(x, half(low, high, u0)) <= TOL[prec], (op, w)
        x = dev(u0)
        h.level_apply(0, S.OP_GS_ZERO, x=x, b=dev(b))
        assert err(x, np.linalg.solve(D / w + lo, b)) <= TOL[prec], ("zero", w)
        h.close()


@pytest.mark.parametrize("w", [1.0, 0.75])
@pytest.mark.parametrize("prec", [0, 1])
def test_block_cycle_equals_its_sweeps(S, prec, w):
    """The V-cycle hands one sweep's sums to the next; composed of single
    level operations it has to give the same."""
    d = (36, 12, 20)
    A = blocks(d, 7)
    h = S.SMG(d, I.OFF7, torch.from_numpy(A).cuda(), block=3, transfer=S.PC8C, smoother=S.SGS, precision=prec,
              krylov=S.FGMRES, relax_w=w, max_levels=2)
    n = int(np.prod(d)) * 3
    dt = torch.float64 if prec == 0 else torch.float32
    r = torch.from_numpy(np.random.default_rng(1).normal(size=n)).cuda()
    z = torch.zeros_like(r)
    h.vcycle(r, z)
    f, u, t = r.to(dt), torch.zeros(n, dtype=dt, device="cuda"), torch.zeros(n, dtype=dt, device="cuda")
    h.level_apply(0, S.OP_GS_ZERO, x=u, b=f)
    h.level_apply(0, S.OP_GS_BACKWARD, x=u, b=f)
    h.level_apply(0, S.OP_RESIDUAL, x=u, b=f, y=t)
    fc = torch.zeros(n // 8, dtype=dt, device="cuda")
    h.level_apply(0, S.OP_RESTRICT, x=t, y=fc)
    fc64, uc = fc.double(), torch.zeros(n // 8, dtype=torch.float64, device="cuda")
    h.level_apply(1, S.OP_COARSE_SOLVE, b=fc64, y=uc)
    h.level_apply(0, S.OP_PROLONG_ADD, x=uc.to(dt), y=u)
    h.level_apply(0, S.OP_GS_FORWARD, x=u, b=f)
    h.level_apply(0, S.OP_GS_BACKWARD, x=u, b=f)
    # four sweeps, a residual and the coarse solve, each within TOL; residuals of
    # values of the size of u amplify by the row sums, below 2
    assert torch.linalg.norm(z - u.double()) <= 8 * TOL[prec] * torch.linalg.norm(u.double())
    h.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_block_zero_wait_budget_aborts_and_context_survives(S, prec):
    """With a zero wait budget the block solves give up at their first unsatisfied
    wait and every CTA drains, those of one cluster with each other's mailboxes
    half written; with the budget restored the same context runs the cycle of a
    context that never gave up, to the bit."""
    d = (40, 40, 12)  # 36 and 24 FP64 tiles, in clusters of eight
    A = torch.from_numpy(blocks(d, 7)).cuda()
    new = lambda: S.SMG(d, I.OFF7, A, block=3, transfer=S.PC8C, smoother=S.SGS, precision=prec, krylov=S.FGMRES,
                        max_levels=2)
    r = torch.from_numpy(np.random.default_rng(1).normal(size=int(np.prod(d)) * 3)).cuda()
    want, z = torch.zeros_like(r), torch.zeros_like(r)
    fresh, h = new(), new()
    fresh.vcycle(r, want)
    fresh.close()
    for _ in range(2):
        h.set_wait_budget_ns(0)
        status = S.OK
        try:
            h.vcycle(r, z)
        except S.SmgError as e:
            status = e.status
        assert status in (S.OK, S.ETIMEOUT)
        h.set_wait_budget_ns(10 ** 9)
        h.vcycle(r, z)
        assert torch.equal(z, want)
    h.close()
