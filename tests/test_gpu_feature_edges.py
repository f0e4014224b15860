"""Feature dimensions at the edges of the groups that the cost warps take: they leave
out groups of features in which both frames hold only padding, which changes no
bit of a cost, so every form returns the one-row-per-lane kernel's path and total
(which sums all padded features)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [17, 19, 20, 21, 24, 32, 33, 47, 48, 49, 64, 65, 80, 81, 96, 97, 112,
                               113, 127, 128])
def test_padding_is_left_out_of_costs_only(D):
    from paper_2607_15478_gb300 import build, pardtw
    build.build()
    aligner = pardtw.Aligner(0)
    try:
        g = torch.Generator(device="cuda")
        g.manual_seed(D)
        pairs = [(torch.randn((La, D), device="cuda", generator=g),
                  torch.randn((Lb, D), device="cuda", generator=g))
                 for La, Lb in ((300, 350), (411, 400), (94, 93))]
        refs = [aligner.align(A, B, rows_per_lane=1) for A, B in pairs]
        for opts in ({}, {"clusters": 1}, {"transpose": 1}):
            for (A, B), ref in zip(pairs, refs):
                path, total = aligner.align(A, B, **opts)
                assert float(total) == float(ref[1]) and torch.equal(path, ref[0]), opts
        many = aligner.align_many([p[0] for p in pairs], [p[1] for p in pairs])
        for k, ref in enumerate(refs):
            path, total = many[0][k], many[1][k]
            assert float(total) == float(ref[1]) and torch.equal(path, ref[0])
    finally:
        aligner.close()
