"""Encoder kernels at their tiles' edges (64 coarse rows a convolution tile, 128 a
weight-gradient block, 32 and 16 in the heads) and at input widths beside the
trained one (16 or 32 lanes per pooled frame, one or two features a lane), against
the FP64 PyTorch reference and the tolerances of test_gpu_encoder."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_15478_gb300 import band_train  # noqa: E402
from tests.test_gpu_encoder import (aligner, blocks, dev, params_t, ref_forward,  # noqa: E402,F401
                                    ref_loss_emb, targets)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1, 16, 17, 33, 64])
@pytest.mark.parametrize("L", [8 * 63 + 1, 8 * 64, 8 * 64 + 1])
@pytest.mark.parametrize("bf16", [False, True])
def test_encode_widths(aligner, D, L, bf16):  # noqa: F811
    X = np.random.default_rng(L + D).random((L, D)).astype(np.float32) + 0.1
    p = band_train.init_params(D, seed=D)
    e_ref, _, hw_ref, _ = ref_forward(X, params_t(p, D), 8, bf16)
    emb, hw = aligner.encode(dev(X), dev(p), downsample=8, bf16=bf16)
    tol = 2e-3 if bf16 else 2e-5
    np.testing.assert_allclose(emb.cpu().numpy(), e_ref.numpy(), atol=tol, rtol=0)
    np.testing.assert_allclose(hw.cpu().numpy(), hw_ref.detach().numpy(), rtol=tol * 10)


@pytest.mark.parametrize("La,Lb,D", [(8 * 128, 8 * 127 + 1, 12), (8 * 65, 8 * 63, 20),
                                     (8 * 129 + 3, 8 * 140, 64), (8 * 17, 8 * 16, 3)])
def test_gradient_tiles(aligner, La, Lb, D):  # noqa: F811
    from paper_2607_15478_gb300 import pardtw
    rng = np.random.default_rng(La + D)
    A = rng.random((La, D)).astype(np.float32) + 0.1
    B = rng.random((Lb, D)).astype(np.float32) + 0.1
    path, _ = aligner.align(dev(A), dev(B))
    plen = torch.tensor([path.shape[0]], dtype=torch.int32, device="cuda")
    p = band_train.init_params(D, seed=4)
    P = dev(p)
    G, loss = torch.zeros_like(P), torch.zeros(1, device="cuda")
    pardtw.dtw_encoder_grad(aligner.h, P, dev(A), dev(B), path.contiguous(), plen, 0, G, loss)
    prm = params_t(p, D, grad=True)
    L = ref_loss_emb(A, B, prm, 8, targets(path.cpu().numpy(), La, Lb, 8))
    L.backward()
    assert abs(float(loss.item()) - float(L.detach())) <= 1e-4 * abs(float(L.detach())) + 1e-6
    g = blocks(G.cpu().numpy(), D)
    for k, t in prm.items():
        if k not in ("W5", "b5"):
            ref = t.grad.numpy()
            np.testing.assert_allclose(g[k], ref, atol=2e-4 * (np.abs(ref).max() + 1e-12), rtol=0,
                                       err_msg=k)
