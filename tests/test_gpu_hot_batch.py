"""Hot rows of stage 2 (see test_gpu_hot_rows.py) where their buffers are laid out for more than one user: a
batch of two uneven instances, before and after qg_autotune has given the plan another block shape, and the
static work array of qg_eval_grad_noalloc, whose second half holds them.  Tolerances as in the other parity
tests (1e-10 FP64 path, 1e-4 mixed path); the no-allocation entry is bitwise qg_eval_grad."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from gradcheck import check_prec

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


def grid(n, M, K, T, scale):
    c = synth.make_case("hot", n, M, max(5, n // 10), T=T, K=K, seed=n + K)
    return dataclasses.replace(c, s_max_ctg=scale * c.s_max_ctg)


def point(c):
    return np.clip(synth.random_point(c, 3, 0.2), *oracle.box(c)).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("precision,sizes", [(0, [(90, 140, 3, 480), (700, 1100, 998, 5)]),
                                             (1, [(1350, 2100, 1999, 1), (1350, 2100, 2001, 3)])])
def test_uneven_batch_before_and_after_autotune(qg, precision, sizes):
    cases = [grid(*s, 0.3) for s in sizes]
    xs = [point(c) for c in cases]
    refs = [oracle.evaluate(c, x) for c, x in zip(cases, xs)]
    s = qg.Solver(cases, precision=precision)
    x = torch.tensor(np.concatenate(xs), dtype=s.dtype, device="cuda")
    tol = 1e-10 if precision == 0 else 1e-4
    for stage in ("created", "tuned"):
        obj, g = s.eval_grad(x)
        torch.cuda.synchronize()
        g, o = g.double().cpu().numpy(), 0
        terms = s.breakdown()
        for b, (c, r) in enumerate(zip(cases, refs)):
            assert abs(obj[b].item() - r.obj) <= tol * abs(r.obj), (stage, b)
            assert r.terms["zctg"] > 0 and abs(terms[b, 7] - r.terms["zctg"]) <= tol * abs(r.terms["zctg"]), (stage, b)
            check_prec(g[o:o + c.n_x], r.grad, c, precision, f"{stage}, instance {b}")
            o += c.n_x
        if stage == "created":
            qg.qg_autotune(s.h, x, 3)
    s.close()


@pytest.mark.parametrize("scale", [0.2, 1e-3])
def test_noalloc_with_hot_rows(qg, scale):
    """A plan with hot rows that fits the array, some rows hot or every row, twice in a row after another handle."""
    other = qg.Solver(synth.rt617(), precision=0)
    xo = torch.tensor(synth.rt617().flat_start(), dtype=torch.float64, device="cuda")
    c = grid(90, 140, 3, 480, scale)
    s = qg.Solver(c, precision=0)
    x = torch.tensor(point(c), dtype=torch.float64, device="cuda")
    ref = tuple(t.clone() for t in s.eval_grad(x))
    for first, xf in ((other, xo), (s, x), (s, x)):
        for h, xx in ((first, xf), (s, x)):
            obj = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
            g = torch.full((h.n_x,), float("nan"), dtype=torch.float64, device="cuda")
            qg.qg_eval_grad_noalloc(h.h, xx, obj, g)
            torch.cuda.synchronize()
        assert torch.equal(obj, ref[0]) and torch.equal(g, ref[1])
    s.close()
    other.close()
