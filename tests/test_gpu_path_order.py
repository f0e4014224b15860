"""The embedding gradient does not depend on the order of the path's pairs: the targets
are means over a coarse row's pairs, wherever they stand.  Loss and gradients are sums
of the same FP32 terms in any order (atomics): at most Lac = 188 of them, a relative
error of 188 x 2^-24 = 1.2e-5 of the largest partial sums; the gradients' bound is
that of their comparison with autograd."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["descending", "shuffled"])
def test_gradient_takes_pairs_in_any_order(order):
    from paper_2607_15478_gb300 import band_train, build, pardtw, synth
    build.build()
    wp = synth.warped_pair(synth.rng_for(70, 1500), 1500, 1300, 12, knots=8, tmin=0.6, tmax=1.6)
    A, B = torch.from_numpy(wp.A).cuda(), torch.from_numpy(wp.B).cuda()
    P = torch.from_numpy(band_train.init_params(12, seed=3)).cuda()
    with pardtw.Aligner(0) as aligner:
        path, _ = aligner.align(A, B)
        n = path.shape[0]
        perm = np.arange(n)[::-1] if order == "descending" else np.random.default_rng(5).permutation(n)
        got = []
        for p in (path, path[torch.from_numpy(perm.copy()).cuda()]):
            G, loss = torch.zeros_like(P), torch.zeros(1, device="cuda")
            plen = torch.tensor([n], dtype=torch.int32, device="cuda")
            pardtw.dtw_encoder_grad(aligner.h, P, A, B, p.contiguous(), plen, 0, G, loss)
            torch.cuda.synchronize()
            got.append((G.cpu().numpy(), float(loss)))
    (g0, l0), (g1, l1) = got
    assert abs(l1 - l0) <= 1.2e-5 * abs(l0)
    np.testing.assert_allclose(g1, g0, atol=2e-4 * np.abs(g0).max(), rtol=0)
