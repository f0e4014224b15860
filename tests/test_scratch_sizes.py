"""The backtrace's scratch holds what the backtrace lays out in it, for every band height
that a call may take for a pair (CPU): the one chosen for its rows, and 128 rows in
a call of more than 1e9 cells, where bands longer than a short pair still have whole
pieces of the path."""
import ctypes

import pytest

from paper_2607_15478_gb300 import build as pbuild


@pytest.fixture(scope="module")
def scratch_bytes():
    pbuild.build()
    f = ctypes.CDLL(pbuild.LIB)["_ZN6pardtw21bandmap_scratch_bytesEii"]
    f.restype = ctypes.c_size_t
    return lambda La, Lb: f(La, Lb)


def laid_out(La, Lb, band):
    n = (La + band - 1) // band
    twos = (n - 2) // 2 if n >= 4 else 0
    fours = (n - 6) // 4 + 1 if n >= 6 else 0
    cells = (n + twos + fours) * Lb + n + n * band  # (row, column) pairs: maps, crossings, pieces
    return 8 * cells + 4 * (n + 1)  # and the pieces' lengths, the end cell's entry


def heights(La):
    return (32 if La <= 1536 else (64 if La <= 6144 else 128), 128)


def test_scratch_holds_every_band_height(scratch_bytes):
    lens = list(range(1, 200)) + [511, 512, 1535, 1536, 1537, 6143, 6144, 6145, 20000, 126231]
    for La in lens:
        for Lb in {(La + 1) // 2, La, 2 * La}:
            for band in heights(La):
                assert scratch_bytes(La, Lb) >= laid_out(La, Lb, band), (La, Lb, band)


@pytest.mark.gpu
def test_short_pairs_in_a_large_call():
    torch = pytest.importorskip("torch")
    from paper_2607_15478_gb300 import pardtw
    pbuild.build()
    sizes = [(1, 1), (30000, 34000), (2, 3), (20, 37), (33, 64), (65, 60)]
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    for D in (3, 12):
        A = [torch.rand((a, D), device="cuda", generator=g) for a, _ in sizes]
        B = [torch.rand((b, D), device="cuda", generator=g) for _, b in sizes]
        with pardtw.Aligner(0) as aligner:
            paths, cost, status = aligner.align_many(A, B)
            for k, path in enumerate(paths):
                ref, total = aligner.align(A[k], B[k], rows_per_lane=1)
                assert status[k] == 0 and float(cost[k]) == total and torch.equal(path, ref), k


def test_growing_pairs_allocate_seldom():
    """A handle fed pairs whose needs grow by 1% a call allocates once per eighth, and a
    first small allocation has no spare room."""
    pbuild.build()
    grown = ctypes.CDLL(pbuild.LIB)["_ZN6pardtw11grown_bytesEmm"]
    grown.restype = ctypes.c_size_t
    grown.argtypes = [ctypes.c_size_t, ctypes.c_size_t]
    assert grown(1 << 20, 0) == 1 << 20
    for start in (100 << 10, 1 << 20, 3 << 20, 64 << 20):
        need, cap, allocations = float(start), 0, 0
        while need < 4 * start:
            if need > cap:
                cap = grown(int(need) + 1, cap)
                allocations += 1
            need *= 1.01
        assert allocations <= 14  # ln 4 / ln 1.125 = 11.8, the first, one of rounding
