"""The exact DP sweeps, per strip of rows, only the columns that the strip's
rows can reach on a path (strip_range in csrc/dp_split.cuh).  This restates the
strip-wise sweep (whole 16-column words, borders from the strip above only for
the columns both sweep) and compares it with the full matrix, cell by cell on
the cells that a path can cross."""
import numpy as np
import pytest

INF = np.inf


def path_lo(i, La, Lb):
    return max((i + 1) // 2, Lb - 1 - 2 * (La - 1 - i))


def path_hi(i, La, Lb):
    return min(2 * i, Lb - 1 - (La - i) // 2)


def strip_range(s, rps, La, Lb):
    """Sub-chunks [x, y) of 8 columns."""
    nsub = (Lb + 7) // 8
    r0, r1 = s * rps, min((s + 1) * rps, La) - 1
    x = (max(path_lo(r0, La, Lb) - 2, 0) // 8) & ~1
    y = min(max(path_hi(r1, La, Lb), 0) // 8 + 1, nsub)
    return x, max(y, x + 1)


def full(C):
    La, Lb = C.shape
    D = np.full((La + 2, Lb + 2), INF)
    F = np.zeros((La, Lb), dtype=np.int8)
    for i in range(La):
        for j in range(Lb):
            c = (D[i + 1, j + 1] + 2 * C[i, j], D[i + 1, j] + 3 * C[i, j], D[i, j + 1] + 3 * C[i, j])
            F[i, j] = int(np.argmin(c))
            D[i + 2, j + 2] = C[0, 0] if i == j == 0 else c[F[i, j]]
    return D[2:, 2:], F


def swept(C, rps):
    """The strip-wise sweep; NaN where no strip computed a cell."""
    La, Lb = C.shape
    D = np.full((La, Lb), np.nan)
    F = np.full((La, Lb), -1, dtype=np.int8)
    ranges = [strip_range(s, rps, La, Lb) for s in range((La + rps - 1) // rps)]
    for s, (x, y) in enumerate(ranges):
        c0, c1 = 8 * x, min(8 * y, Lb)
        a0, a1 = (8 * ranges[s - 1][0], min(8 * ranges[s - 1][1], Lb)) if s else (0, 0)
        for i in range(s * rps, min((s + 1) * rps, La)):
            for j in range(c0, c1):
                def e(r, q):
                    if r < 0 or q < c0:  # nothing of the columns before the first one is kept
                        return INF
                    if r < s * rps and not (a0 <= q < a1):
                        return INF
                    return D[r, q]
                c = (e(i - 1, j - 1) + 2 * C[i, j], e(i - 1, j - 2) + 3 * C[i, j],
                     e(i - 2, j - 1) + 3 * C[i, j])
                F[i, j] = int(np.argmin(c))
                D[i, j] = C[0, 0] if i == j == 0 else c[F[i, j]]
    return D, F, ranges


@pytest.mark.parametrize("La,Lb", [(1, 1), (2, 3), (9, 17), (17, 9), (40, 79), (79, 40), (60, 60),
                                   (97, 130), (130, 97), (188, 96), (95, 189), (64, 127)])
@pytest.mark.parametrize("rps", [30, 62, 93])
def test_sweep_of_the_path_region_is_exact(La, Lb, rps):
    C = np.random.default_rng(La * 1000 + Lb).random((La, Lb))
    Df, Ff = full(C)
    D, F, ranges = swept(C, rps)
    for i in range(La):
        for j in range(max(path_lo(i, La, Lb), 0), path_hi(i, La, Lb) + 1):
            assert D[i, j] == Df[i, j], (i, j)
            if np.isfinite(Df[i, j]) and (i, j) != (0, 0):
                assert F[i, j] == Ff[i, j], (i, j)
    assert np.isfinite(D[-1, -1])
    assert ranges[0][0] == 0 and ranges[-1][1] == (Lb + 7) // 8
    for a, b in zip(ranges, ranges[1:]):  # a staircase without gaps
        assert a[0] <= b[0] <= a[1] <= b[1] and a[0] < a[1]
