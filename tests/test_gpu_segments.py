"""The segment-level DP of WSDTW against its recurrence, run in numpy on the
device's own C_seg: the same FP32 additions and comparisons, so the end frames
and the total are equal bit for bit.  Sizes at the edges of its forms: one
cluster with 4, 8 or 16 columns a thread (up to 32768, 65536, 131072 columns),
the grid of one launch above, one CTA and several, half fragments longer than the
columns of a CTA, one fragment and more fragments than warps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [(60, 47, 3), (64, 4096, 64), (90, 4097, 5), (60, 8193, 1), (200, 32768, 7),
         (200, 32769, 7), (80, 65536, 4), (80, 65537, 4), (60, 131072, 3), (60, 131073, 3),
         (24001, 21011, 2), (30000, 50021, 3)]


@pytest.mark.parametrize("La,Lb,N", CASES)
def test_ends_and_total_follow_from_cseg(La, Lb, N):
    from paper_2607_15478_gb300 import build, pardtw
    build.build()
    aligner = pardtw.Aligner(0)
    try:
        g = torch.Generator(device="cuda")
        g.manual_seed(La + Lb + N)
        B = torch.rand((Lb, 12), device="cuda", generator=g)
        at = torch.arange(La, device="cuda") * max(Lb // La, 1) % Lb
        A = (B[at] + 0.05 * torch.rand((La, 12), device="cuda", generator=g)).contiguous()
        _, ends, total = aligner.wsdtw(A, B, N)
        cseg = aligner.wsdtw_cseg(N, Lb).cpu().numpy()
    finally:
        aligner.close()
    args, D = [], None
    rows = [(k + 1) * La // N - k * La // N for k in range(N)]
    for k in range(N):
        m = cseg[k].copy()
        if k:
            d = rows[k] // 2
            m = np.full(Lb, np.inf, np.float32)
            m[d:] = D[:Lb - d] + cseg[k][d:]
        D = np.minimum.accumulate(m)
        first = np.concatenate([[True], m[1:] < D[:-1]])
        args.append(np.maximum.accumulate(np.where(first, np.arange(Lb), 0)))
    e = Lb - 1
    want = []
    for k in range(N - 1, -1, -1):
        e = int(args[k][e])
        want.append(e)
        e -= rows[k] // 2
    assert np.float32(total) == D[-1]
    np.testing.assert_array_equal(ends.cpu().numpy(), np.array(want[::-1], np.int32))
