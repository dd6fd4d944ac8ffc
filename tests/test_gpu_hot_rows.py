"""Stage 2's hot rows (branches over their post-contingency limit in the base case, evaluated over every
outage by blocks of their own) against the FP64 oracle: outage counts around the 1,024 columns of a block
and not multiples of a thread's four, no row, some rows and every row hot (more than the 32 staged at a
time), several row groups, many periods, and plans of both paths large enough to
take them (FP64: more than 65,536 branch-periods; mixed: 2^22 (branch, outage) pairs per period).

Tolerances as in the other parity tests: 1e-10 (FP64 path), 1e-4 (mixed path, the oracle at the same
FP32-rounded point)."""
import dataclasses
import functools

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


@functools.lru_cache(maxsize=None)
def grid(n, M, K, T):
    return synth.make_case("hot", n, M, max(5, n // 10), T=T, K=K, seed=n + K)


@pytest.mark.parametrize("precision,n,M,K,T,scale", [
    (0, 90, 140, 3, 480, 1.0), (0, 700, 1100, 1023, 60, 1.0), (0, 700, 1100, 1025, 60, 1e-3),
    (0, 700, 1100, 1024, 61, 1e3), (0, 700, 1100, 998, 64, 0.5), (1, 1350, 2100, 2001, 2, 0.5), (1, 1350, 2100, 2001, 1, 1e-3)])
def test_hot_rows_match_the_oracle(qg, precision, n, M, K, T, scale):
    c = grid(n, M, K, T)
    c = dataclasses.replace(c, s_max_ctg=scale * c.s_max_ctg)
    x = np.clip(synth.random_point(c, 3, 0.2), *oracle.box(c))
    if precision == 1:
        x = x.astype(np.float32).astype(np.float64)
    s = qg.Solver(c, precision=precision)
    obj, g = s.eval_grad(torch.tensor(x, dtype=s.dtype, device="cuda"))
    torch.cuda.synchronize()
    ref = oracle.evaluate(c, x)
    tol = 1e-10 if precision == 0 else 1e-4
    assert abs(obj.item() - ref.obj) <= tol * abs(ref.obj)
    assert abs(s.breakdown()[0, 7] - ref.terms["zctg"]) <= tol * abs(ref.terms["zctg"])
    check_prec(g.cpu().numpy(), ref.grad, c, precision, "hot rows")
    s.close()


def test_hot_rows_screening_scores(qg):
    """A screening handle: the scores of the selected outages hold the hot rows' share."""
    c = grid(700, 1100, 998, 64)
    c = dataclasses.replace(c, s_max_ctg=0.5 * c.s_max_ctg)
    x = np.clip(synth.random_point(c, 3, 0.2), *oracle.box(c))
    s = qg.Solver(c, precision=0, ctg_frac=0.5)
    Ks = int(np.ceil(0.5 * c.K))
    sel = np.sort(np.random.default_rng(1).choice(c.K, Ks, replace=False)).astype(np.int32)
    qg.qg_ctg_select(s.h, 0, sel)
    obj, g = s.eval_grad(torch.tensor(x, dtype=s.dtype, device="cuda"))
    z = qg.qg_ctg_scores(s.h, c.T * Ks).reshape(c.T, Ks)
    sub = dataclasses.replace(c, ctg=c.ctg[sel])
    ref = oracle.evaluate(sub, x)
    floor = c.dt[:, None] * c.c_s * c.beta * c.eps * (c.n_branch - 1)
    assert abs(obj.item() - ref.obj) <= 1e-10 * abs(ref.obj)
    assert np.max(np.abs(z - (ref.z_ctg - floor))) <= 1e-10 * np.abs(ref.z_ctg).max()
    check_prec(g.cpu().numpy(), ref.grad, c, 0, "hot rows, screening")
    s.close()
