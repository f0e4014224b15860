"""The warp-pair DP's sweep at the sizes where its trips, slots and links can go
wrong (odd sub-chunk counts, one sub-chunk, strips of one row, several tickets
of a cluster), one and two strips per CTA, one to four cost warps per strip: every
form must return the one-row-per-lane kernel's path and total, bit for bit (every
cell is the same FP32 arithmetic, so no tolerance)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(2, 2), (8, 9), (17, 24), (93, 120), (94, 101), (187, 186), (188, 97), (500, 263),
         (743, 800), (1490, 1337), (1489, 2971)]


@pytest.fixture(scope="module")
def aligner():
    from paper_2607_15478_gb300 import build, pardtw
    build.build()
    a = pardtw.Aligner(0)
    yield a
    a.close()


def pair(La, Lb, D):
    g = torch.Generator(device="cuda")
    g.manual_seed(La * 10007 + Lb * 31 + D)
    return (torch.rand((La, D), device="cuda", generator=g),
            torch.rand((Lb, D), device="cuda", generator=g))


def same(aligner, A, B, ref, **opts):
    path, total = aligner.align(A, B, wait_limit_us=500000, **opts)
    assert total == ref[1] and torch.equal(path, ref[0]), opts


@pytest.mark.parametrize("D", [3, 8, 12, 16, 20, 64, 100])
@pytest.mark.parametrize("La,Lb", SIZES)
def test_sweeps_equal_one_row_per_lane(aligner, La, Lb, D):
    A, B = pair(La, Lb, D)
    ref = aligner.align(A, B, rows_per_lane=1)
    for transpose in (1, 2):
        for clusters in (0, 1):
            same(aligner, A, B, ref, transpose=transpose, clusters=clusters)
    if D <= 16:
        same(aligner, A, B, ref, strips_per_cta=4)
        same(aligner, A, B, ref, rows_per_lane=2)


@pytest.mark.parametrize("La,Lb", SIZES)
def test_bf16_sweeps_agree(aligner, La, Lb):
    A, B = pair(La, Lb, 100)
    ref = aligner.align(A, B, cost_precision=1, clusters=1, transpose=1)
    for transpose in (1, 2):
        same(aligner, A, B, ref, cost_precision=1, transpose=transpose)


@pytest.mark.parametrize("La,Lb,D", [(16001, 14003, 12), (16001, 14003, 20), (16001, 14003, 100),
                                     (33001, 35003, 12)])
def test_several_tickets_per_cluster(aligner, La, Lb, D):
    A, B = pair(La, Lb, D)
    ref = aligner.align(A, B, clusters=1, transpose=1)
    for transpose in (1, 2):
        same(aligner, A, B, ref, transpose=transpose)
