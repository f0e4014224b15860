"""Calls queued without a synchronisation, every result against the kernel with one
row per lane (BF16 cost: against the kernel without clusters), bit for bit: the
warps of the warp-pair DP hand slots, borders and releases to one another, and a
load that does not wait for what it reads shows as a wrong path in one call of many.
Both orientations of the sweep, each form of the kernel (strips and cost warps a
CTA, clusters and none, FP32 and BF16 cost, batch), pairs of one strip, of a few,
and of more strip groups than are resident in clusters."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(9001, 12007), (31, 40), (1537, 1536), (12007, 9001), (200, 333), (6145, 5001)]
ROUNDS = 200
NEVER, ALWAYS = {"transpose": 1}, {"transpose": 2}


def outputs(A, B):
    n = min(A.shape[0], B.shape[0])
    return (torch.zeros((n, 2), dtype=torch.int32, device="cuda"),
            torch.zeros(1, dtype=torch.int32, device="cuda"),
            torch.zeros(1, dtype=torch.float32, device="cuda"))


def same(x, y):
    return all(torch.equal(a, b) for a, b in zip(x, y))


def draw(D):
    g = torch.Generator(device="cuda")
    g.manual_seed(D)
    return [(torch.rand((La, D), device="cuda", generator=g),
             torch.rand((Lb, D), device="cuda", generator=g)) for La, Lb in SIZES]


@pytest.mark.parametrize("D,opts", [
    (4, {}), (8, {}), (12, {}), (16, {}), (20, {}), (32, {}), (64, {}), (100, {}), (128, {}),
    (64, {"cost_precision": 1}), (128, {"cost_precision": 1}),
    (12, {"clusters": 1}), (32, {"clusters": 1}), (100, {"clusters": 1}),
    (100, {"cost_precision": 1, "clusters": 1}), (12, {"strips_per_cta": 4})])
def test_queued_pairs(D, opts):
    from paper_2607_15478_gb300 import build, pardtw
    build.build()
    plain = {"rows_per_lane": 1}
    if "cost_precision" in opts:
        plain = {"cost_precision": 1, "clusters": 1, "transpose": 1}
    aligner = pardtw.Aligner(0)
    try:
        pairs = draw(D)
        want = []
        for A, B in pairs:
            want.append(outputs(A, B))
            aligner.align_into(A, B, *want[-1], **plain)
        calls = [(k, o) for o in (NEVER, ALWAYS) for k in range(len(pairs))]
        got = [outputs(*pairs[k]) for k, _ in calls]
        wrong = []
        for _ in range(ROUNDS):
            for (k, o), out in zip(calls, got):
                out[0].zero_()
                aligner.align_into(*pairs[k], *out, **opts, **o)
            torch.cuda.synchronize()
            wrong += [(SIZES[k], o) for (k, o), out in zip(calls, got) if not same(out, want[k])]
        assert not wrong, (len(wrong), sorted(set(map(str, wrong))))
    finally:
        aligner.close()


@pytest.mark.parametrize("D,opts", [(8, {}), (12, {}), (12, {"strips_per_cta": 2}), (20, {}),
                                    (24, {}), (25, {}), (28, {}), (29, {}),
                                    (12, {"rows_per_lane": 2})])
def test_repeated_batches(D, opts):
    from paper_2607_15478_gb300 import build, pardtw
    build.build()
    aligner = pardtw.Aligner(0)
    try:
        pairs = draw(D) * 3
        want = []
        for A, B in pairs[:len(SIZES)]:
            p, total = aligner.align(A, B, rows_per_lane=1)
            want.append((p, total))
        for _ in range(ROUNDS // 2):
            paths, cost, status = aligner.align_many([a for a, _ in pairs], [b for _, b in pairs],
                                                     **opts)
            for k, p in enumerate(paths):
                ref = want[k % len(SIZES)]
                assert status[k] == 0 and torch.equal(p, ref[0]) and float(cost[k]) == ref[1], k
    finally:
        aligner.close()
