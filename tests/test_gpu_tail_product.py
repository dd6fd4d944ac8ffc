"""The dense-tail product of the sparse DC solver (error-free splitting into 8-bit digits on the tensor
cores) where its tiling can go wrong: one period, 16 and 17 (one and two column tiles), two passes over the
periods, tails below and above one 128-row tile and of many 64-column blocks; against the dense solver, which
shares nothing of it.  Digits carry 54 bits of a row's largest entry on the mixed path and 62 on the FP64
path, so the two solvers agree to the tolerances of the parity tests (1e-10, 1e-4); a product that were
not exact in FP32 accumulation would miss the first by orders of magnitude.  A NaN in the dispatch
reaches the objective."""
import numpy as np
import pytest

import oracle
import synth
from gradcheck import check_at

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


def evaluate(qg, c, x, precision, solver):
    s = qg.Solver(c, precision=precision, dc_solver=solver)
    obj, g = s.eval_grad(torch.tensor(x, dtype=s.dtype, device="cuda"))
    torch.cuda.synchronize()
    f = qg.qg_dc_flows(s.h, c.T * c.n_branch)
    out = obj.item(), g.cpu().numpy().astype(np.float64), f.astype(np.float64)
    s.close()
    return out


@pytest.mark.parametrize("n,T", [(617, 1), (1200, 16), (1576, 17), (2400, 49), (3300, 33)])
@pytest.mark.parametrize("precision", [0, 1])
def test_sparse_against_dense(qg, n, T, precision):
    c = synth.make_case("tail", n, int(1.5 * n), n // 7, T=T, K=20, seed=n + T)
    x = np.clip(synth.random_point(c, 5, 0.2), *oracle.box(c))
    od, gd, fd = evaluate(qg, c, x, precision, qg.QG_DC_DENSE)
    os_, gs, fs = evaluate(qg, c, x, precision, qg.QG_DC_SPARSE)
    tol = 1e-10 if precision == 0 else 1e-4
    assert abs(os_ - od) <= tol * abs(od)
    check_at(gs, gd, c, tol, "sparse against dense")
    # FP32 values of flows that agree to far below one FP32 rounding: at most one unit in the last place apart
    assert np.all(np.abs(fs - fd) <= 2.0 ** -23 * np.abs(fd) + 1e-9 * np.abs(fd).max())


def test_nan_reaches_the_objective(qg):
    c = synth.make_case("tail", 1200, 1800, 170, T=3, K=20, seed=9)
    x = np.clip(synth.random_point(c, 5, 0.2), *oracle.box(c))
    x[2 * c.T * c.n_bus + c.n_gen] = np.nan  # a dispatch of period 1
    for precision in (0, 1):
        obj, _, f = evaluate(qg, c, x, precision, qg.QG_DC_SPARSE)
        assert np.isnan(obj)
        f = f.reshape(c.T, c.n_branch)
        assert np.isnan(f[1]).any() and np.isfinite(f[[0, 2]]).all()
