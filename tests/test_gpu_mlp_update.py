"""The fused update of the warm-start network (Adam and the BF16 copies of the updated weights in one pass
over 64 x 64 tiles): odd and even row lengths, partial tiles, batches of one row and of the full tile.
The parameters follow from the step's own gradient by Adam in FP64 within FP32 rounding (a handful of
roundings of w and of the update: 4e-7 of |w| plus 1e-5 of the step size), and the forward pass afterwards
uses the updated weights (against the FP64 oracle of the network with the same BF16 rounding points, with
the tolerance of the other forward tests)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_06650_gb300.build import build
    build()
    from paper_2310_06650_gb300 import qg as mod
    return mod


@pytest.mark.parametrize("n_in,n_h,n_out,B", [(64, 64, 64, 64), (65, 33, 127, 1), (190, 130, 66, 63), (501, 96, 1031, 17)])
def test_update_and_next_forward(qg, n_in, n_h, n_out, B):
    from oracle import mlp
    lr, b1, b2 = 1e-3, 0.9, 0.999
    m = qg.qg_mlp_create(n_in, n_h, n_out, 64, seed=11)
    npar = qg.qg_mlp_num_params(m)
    gen = torch.Generator().manual_seed(4)
    w = torch.zeros(npar, device="cuda")
    g = torch.zeros(npar, device="cuda")
    y = torch.zeros(B, n_out, device="cuda")
    mom, var = np.zeros(npar), np.zeros(npar)
    qg.qg_mlp_get_params(m, w)
    for step in (1, 2):
        x = torch.randn(B, n_in, generator=gen).cuda()
        t = torch.randn(B, n_out, generator=gen).cuda()
        w0 = w.cpu().numpy().astype(np.float64)
        qg.qg_mlp_train_step(m, x, t, B, lr, b1, b2)
        qg.qg_mlp_get_grads(m, g)
        qg.qg_mlp_get_params(m, w)
        torch.cuda.synchronize()
        gr = g.cpu().numpy().astype(np.float64)
        mom = b1 * mom + (1 - b1) * gr
        var = b2 * var + (1 - b2) * gr * gr
        ref = w0 - lr * (mom / (1 - b1 ** step)) / (np.sqrt(var / (1 - b2 ** step)) + 1e-8)
        wn = w.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(wn - ref) <= 4e-7 * np.abs(ref) + 1e-5 * lr)
        assert not np.array_equal(wn, w0)
        qg.qg_mlp_forward(m, x, B, y)
        torch.cuda.synchronize()
        X = x.cpu().numpy().astype(np.float64)
        Y = mlp.forward_backward(wn, X, np.zeros((B, n_out)), n_in, n_h, n_out)[0]
        assert np.linalg.norm(y.cpu().numpy() - Y) <= 2e-3 * np.linalg.norm(Y)
    qg.qg_mlp_check(m)
    qg.qg_mlp_destroy(m)
