"""Device memory of the point smoothers' streams on flat and narrow boxes: one
slot per point, so a hierarchy of a flat box takes what one of a compact box with
as many points and the same x-y coarsening takes (the strips of 32 x-points and
groups of 2 to 8 y-points are full in all of these; the tenth is for allocations
rounded up on the small levels)."""
import numpy as np
import pytest

from paper_2506_21932_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COMPACT = (128, 128, 128)
FLAT = [(512, 512, 8), (1024, 1024, 2), (2048, 1024, 1), (128, 1024, 16)]


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_21932_gb300 import build, smg
    build.build()
    return smg


def matrix(d, off):
    """-1 for every neighbour on the grid, 40 on the diagonal."""
    A = torch.full((*d, len(off)), -1.0, dtype=torch.float64, device="cuda")
    for e, o in enumerate(off):
        for ax in range(3):
            if o[ax]:
                A[..., e].select(ax, d[ax] - 1 if o[ax] > 0 else 0).zero_()
    A[..., off.index((0, 0, 0))] = 40.0
    return A.reshape(-1, len(off))


def hierarchy_bytes(S, d, off, smoother, prec, block):
    A = matrix(d, off)
    if block == 3:
        A = A[:, :, None, None] * torch.eye(3, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    h = S.SMG(d, off, A, smoother=smoother, precision=prec, krylov=S.FPCG, block=block,
              transfer=S.C16XY)
    used = free - torch.cuda.mem_get_info()[0]
    h.close()
    return used


@pytest.mark.parametrize("smoother,mask,prec,block", [("ILU0", 27, 0, 1), ("ILU0", 27, 1, 1), ("ILU0", 27, 2, 1),
                                                      ("SGS", 7, 0, 1), ("SGS", 7, 0, 3)])
def test_flat_boxes_take_no_more_memory_than_compact_ones(S, smoother, mask, prec, block):
    off = I.OFF27 if mask == 27 else I.OFF7
    compact = hierarchy_bytes(S, COMPACT, off, getattr(S, smoother), prec, block)
    for d in FLAT:
        assert np.prod(d) == np.prod(COMPACT)
        assert hierarchy_bytes(S, d, off, getattr(S, smoother), prec, block) <= 1.1 * compact, d
