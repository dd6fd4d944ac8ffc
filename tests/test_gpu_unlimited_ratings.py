"""Branches without a post-contingency limit, given as a huge finite rating whose square is beyond FP32
(1e20, 1e30), among branches with overloads.  They are never over their limit, and stage 2 still has to
write their row partials wherever another row of their 64-row tile has one: the static work array of
qg_eval_grad_noalloc holds whatever its last user left.  Handles take turns on that array, and each call is
bitwise its handle's qg_eval_grad and agrees with the FP64 oracle (1e-10 FP64 path, 1e-4 mixed path); one
plan has hot rows, for which the limited branches are over their limit before any outage."""
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


def unlimited(c, scale, rating):
    s = scale * c.s_max_ctg
    s[::3] = rating
    return dataclasses.replace(c, s_max_ctg=s)


@pytest.mark.parametrize("precision", [0, 1])
def test_unlimited_rows_among_overloads(qg, precision):
    dirty = synth.rt617()  # its contents are what the others find in the array
    hot = synth.make_case("hot", 90, 140, 9, T=480, K=3, seed=93)  # FP64 path: hot rows
    cases = [dataclasses.replace(dirty, s_max_ctg=1e-2 * dirty.s_max_ctg), unlimited(synth.mid(), 0.3, 1e20),
             unlimited(synth.mid(), 0.3, 1e30), unlimited(hot, 0.2, 1e20)]
    xs = [np.clip(synth.random_point(c, 3, 0.2), *oracle.box(c)).astype(np.float32).astype(np.float64) for c in cases]
    solvers = [qg.Solver(c, precision=precision) for c in cases]
    xd = [torch.tensor(x, dtype=s.dtype, device="cuda") for x, s in zip(xs, solvers)]
    refs = [tuple(t.clone() for t in s.eval_grad(x)) for s, x in zip(solvers, xd)]
    for k in (1, 2, 3):
        ref = oracle.evaluate(cases[k], xs[k])
        assert ref.terms["zctg"] > 0
        for _ in range(2):
            for j in (0, k):
                s = solvers[j]
                obj = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
                g = torch.full((s.n_x,), float("nan"), dtype=s.dtype, device="cuda")
                qg.qg_eval_grad_noalloc(s.h, xd[j], obj, g)
                torch.cuda.synchronize()
            assert torch.equal(obj, refs[k][0]) and torch.equal(g, refs[k][1]), k
        tol = 1e-10 if precision == 0 else 1e-4
        assert abs(obj.item() - ref.obj) <= tol * abs(ref.obj)
        check_prec(g.cpu().numpy(), ref.grad, cases[k], precision, f"unlimited rows, case {k}")
    for s in solvers:
        s.close()
