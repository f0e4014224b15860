"""Frames of B that are NaN: a segment's match is never attained there, and the other
columns are as without it, in each form of the segment-level DP (one cluster up to
131072 columns, one grid above): the recurrence in numpy on the device's own C_seg, NaN
read as +inf, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lb", [3000, 131072, 131073])
def test_a_nan_frame_is_never_an_end(Lb):
    from paper_2607_15478_gb300 import build, pardtw
    build.build()
    La, N = 60, 3
    g = torch.Generator(device="cuda")
    g.manual_seed(Lb)
    A = torch.rand((La, 12), device="cuda", generator=g)
    B = torch.rand((Lb, 12), device="cuda", generator=g)
    B[::1024] = float("nan")  # the first column of every tile of the grid's scan
    nan = (Lb + 1023) // 1024
    with pardtw.Aligner(0) as aligner:
        _, ends, total = aligner.wsdtw(A, B, N)
        cseg = aligner.wsdtw_cseg(N, Lb).cpu().numpy()
    assert np.isnan(cseg).sum() == nan * N
    cseg = np.where(np.isnan(cseg), np.float32(np.inf), cseg)
    args, D, d = [], None, La // N // 2
    for k in range(N):
        m = cseg[k].copy()
        if k:
            m = np.full(Lb, np.inf, np.float32)
            m[d:] = D[:Lb - d] + cseg[k][d:]
        D = np.minimum.accumulate(m)
        first = np.concatenate([[True], m[1:] < D[:-1]])
        args.append(np.maximum.accumulate(np.where(first, np.arange(Lb), 0)))
    e, want = Lb - 1, []
    for k in range(N - 1, -1, -1):
        e = int(args[k][e])
        want.append(e)
        e -= d
    assert np.float32(total) == D[-1]
    np.testing.assert_array_equal(ends.cpu().numpy(), np.array(want[::-1], np.int32))
