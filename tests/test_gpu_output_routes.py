"""Outputs that take a copy instead of the kernels' own stores (arrays that overlap an input or each other,
arrays not aligned to their elements) hold the same bits as separate aligned ones."""
import numpy as np
import pytest

import oracle
import synth

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


class At:
    """A device address inside a byte tensor, with the value there as a tensor of n elements."""

    def __init__(self, buf, off, n, dtype):
        self.buf, self.off, self.n, self.dtype = buf, off, n, dtype

    def data_ptr(self):
        return self.buf.data_ptr() + self.off

    def value(self):
        size = torch.empty(0, dtype=self.dtype).element_size()
        return self.buf[self.off:self.off + self.n * size].clone().view(self.dtype)


@pytest.mark.parametrize("precision", [0, 1])
def test_eval_grad_into_any_array(qg, precision):
    c = synth.mid()
    s = qg.Solver(c, precision=precision)
    w, n = s.g.element_size(), s.n_x
    x0 = np.clip(synth.random_point(c, 2), *oracle.box(c))
    x = torch.tensor(x0, dtype=s.dtype, device="cuda")
    obj, g = (t.clone() for t in s.eval_grad(x))
    raw = x.view(torch.uint8)

    def call(px, po, pg):
        qg.qg_eval_grad(s.h, px, po, pg)
        torch.cuda.synchronize()

    for off in (0, w, 8 * w):  # g on x, from the start or later
        buf = torch.zeros(n * w + 8 * w, dtype=torch.uint8, device="cuda")
        buf[:n * w] = raw
        out, o = At(buf, off, n, s.dtype), torch.zeros(1, dtype=torch.float64, device="cuda")
        call(At(buf, 0, n, s.dtype), o, out)
        assert torch.equal(out.value(), g) and torch.equal(o, obj), off
    for off in (1, 2, w // 2):  # not a multiple of the element
        buf = torch.zeros(n * w + 16, dtype=torch.uint8, device="cuda")
        ob = torch.zeros(16, dtype=torch.uint8, device="cuda")
        out, o = At(buf, off, n, s.dtype), At(ob, off, 1, torch.float64)
        call(x, o, out)
        assert torch.equal(out.value(), g) and torch.equal(o.value(), obj), off
    # obj on the last 8 bytes of g: written first, then g over it
    buf = torch.zeros((n + 2) * 8, dtype=torch.uint8, device="cuda")
    out = At(buf, 0, n, s.dtype)
    call(x, At(buf, (n * w - 8) // 8 * 8, 1, torch.float64), out)
    assert torch.equal(out.value(), g)
    # either one alone
    o = torch.zeros(1, dtype=torch.float64, device="cuda")
    call(x, o, None)
    out = At(torch.zeros(n * w, dtype=torch.uint8, device="cuda"), 0, n, s.dtype)
    call(x, None, out)
    assert torch.equal(o, obj) and torch.equal(out.value(), g)
    s.close()


@pytest.mark.parametrize("B", [1, 64])
def test_mlp_forward_into_any_array(qg, B):
    m = qg.qg_mlp_create(190, 130, 601, 64, seed=3)
    x = torch.randn(B, 190, generator=torch.Generator().manual_seed(1)).cuda()
    y = torch.zeros(B * 601, device="cuda")
    qg.qg_mlp_forward(m, x, B, y)
    for off in (1, 2, 3):
        out = At(torch.zeros(4 * B * 601 + 16, dtype=torch.uint8, device="cuda"), off, B * 601, torch.float32)
        qg.qg_mlp_forward(m, x, B, out)
        torch.cuda.synchronize()
        assert torch.equal(out.value(), y)
    qg.qg_mlp_check(m)
    qg.qg_mlp_destroy(m)
