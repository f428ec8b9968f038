"""The line sweep's wait for a column's records is bounded by the wait budget
also where no other wait is: one x-plane has no earlier plane to wait for, so a
copy in flight is all its helper warps wait for."""
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


@pytest.fixture(scope="module")
def orc():
    from oracle import oracle
    oracle.build()
    return oracle


# columns too long for more than one in shared memory: each one's copy is issued
# when the one before is solved, and waited for
@pytest.mark.parametrize("d", [(1, 7, 600), (1, 4, 1024)])
def test_a_copy_in_flight_counts_against_the_budget(S, orc, d):
    off, n = I.OFF27, int(np.prod(d))
    A = I.q1_aniso27(d, 2).numpy()
    h = S.SMG(d, off, torch.from_numpy(A).cuda(), smoother=S.LGS, max_levels=1)
    b = torch.from_numpy(I.rhs(n, 5).numpy()).cuda()
    h.set_wait_budget_ns(0)
    with pytest.raises(S.SmgError) as e:
        h.level_apply(0, S.OP_LGS_FORWARD, x=torch.zeros_like(b), b=b)
    assert e.value.status == S.ETIMEOUT
    h.set_wait_budget_ns(10 ** 9)
    ref = orc.lgs_forward(d, off, A, b.cpu().numpy(), np.zeros(n))
    for _ in range(2):
        x = torch.zeros_like(b)
        h.level_apply(0, S.OP_LGS_FORWARD, x=x, b=b)
        assert np.abs(x.cpu().numpy() - ref).max() < 1e-12 * np.abs(ref).max()
    h.close()
