"""Calls queued one behind the other on one handle, with no synchronisation in
between: their kernels share the workspace and are placed before the kernel in
front has finished, so every result must still be the one of a call made alone.
Sizes with one band of the backtrace, without and with each of its map
compositions, and with more bands than an SM count; every cell is the same FP32
arithmetic, so no tolerance."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(2, 2), (31, 40), (97, 110), (129, 130), (200, 333), (1536, 1537), (6145, 5001), (9001, 12007)]


@pytest.mark.parametrize("D,opts", [(12, {}), (20, {}), (100, {}), (100, {"cost_precision": 1}),
                                    (12, {"clusters": 1})])
def test_calls_in_a_row_equal_single_calls(D, opts):
    from paper_2607_15478_gb300 import build, pardtw
    build.build()
    aligner = pardtw.Aligner(0)
    try:
        g = torch.Generator(device="cuda")
        g.manual_seed(D)
        pairs = [(torch.rand((La, D), device="cuda", generator=g),
                  torch.rand((Lb, D), device="cuda", generator=g)) for La, Lb in SIZES + SIZES[::-1]]
        alone = []
        for A, B in pairs:
            alone.append([x.cpu() if torch.is_tensor(x) else x for x in aligner.align(A, B, **opts)])
            torch.cuda.synchronize()
        rows = [aligner.align(A, B, **opts) for _ in range(3) for A, B in pairs]
        torch.cuda.synchronize()
        for k, (path, total) in enumerate(rows):
            ref = alone[k % len(pairs)]
            assert torch.equal(path.cpu(), ref[0]) and float(total) == float(ref[1]), k
    finally:
        aligner.close()
