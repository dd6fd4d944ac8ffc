"""The dense-tail product of the sparse DC solver at injections of any size and of very different sizes, against
the dense solver, which shares nothing of it.  Its operands are integers relative to the power of two above
the largest entry of a row of the matrix and of a period's right-hand side, so what it owes is
    |error| <= K (S + 1) 2^(4 - 8 S) max|a| max|z|     (K columns, S = 8 digits on the FP64 path, 7 on the mixed path)
per output: with K = 160 and angles to flows costing at most 1e3 of max|z|, 2e-12 of the largest flow of the
period on the FP64 path and 2e-9 on the mixed path (the dense solver's own rounding is below that), besides
one FP32 unit of the flow itself, as which it is read."""
import dataclasses

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
    f = qg.qg_dc_flows(s.h, c.T * c.n_branch).reshape(c.T, c.n_branch).astype(np.float64)
    out = obj.item(), s.breakdown()[0, 7], g.cpu().numpy().astype(np.float64), f
    s.close()
    return out


def both(qg, c, precision):
    x = np.clip(synth.random_point(c, 5, 0.2), *oracle.box(c)).astype(np.float32).astype(np.float64)
    return evaluate(qg, c, x, precision, qg.QG_DC_DENSE), evaluate(qg, c, x, precision, qg.QG_DC_SPARSE)


def grid():
    return synth.make_case("tail", 1200, 1800, 170, T=3, K=20, seed=9)


def close_flows(fs, fd, precision):
    tol = 2e-12 if precision == 0 else 2e-9
    for t in range(len(fd)):
        ok = np.isfinite(fd[t])  # FP32 copies of FP64 flows beyond FP32: infinite in both
        assert np.array_equal(fs[t][~ok], fd[t][~ok]), t
        assert np.all(np.abs(fs[t][ok] - fd[t][ok]) <= 2.0 ** -23 * np.abs(fd[t][ok]) + tol * np.abs(fd[t][ok]).max()), t


@pytest.mark.parametrize("precision,size", [(0, 1e30), (0, 3e38), (0, 1e39), (0, 1e42), (1, 1e30), (1, 3e38)])
def test_injections_up_to_the_end_of_the_range(qg, precision, size):
    """One period with two opposite injections of that size at the buses of highest degree, which the
    elimination leaves to the tail; the others as usual."""
    c = grid()
    deg = np.bincount(np.concatenate([c.br_from, c.br_to]), minlength=c.n_bus)
    a, b = [k for k in np.argsort(-deg, kind="stable") if k != c.ref_bus][:2]
    load = c.load_p.copy()
    load[1, a], load[1, b] = size, -size
    c = dataclasses.replace(c, load_p=load)
    (od, zd, gd, fd), (os_, zs, gs, fs) = both(qg, c, precision)
    close_flows(fs, fd, precision)
    if precision == 0:  # (the mixed path's objective is beyond FP32)
        assert np.isfinite(od) and np.isfinite(os_) and np.all(np.isfinite(gs))
    if precision == 0 and size <= 3e38:  # beyond it the FP32 screen sees infinities
        # (no gradients: at a bus with two branches, the outage of one leaves the other an own injection of about 1
        # as the difference of flows of 1e30, and the sign of what rounding leaves of it is the adjoint)
        assert zd > 0
        assert abs(os_ - od) <= 1e-10 * abs(od) and abs(zs - zd) <= 1e-10 * abs(zd)


@pytest.mark.parametrize("precision", [0, 1])
def test_injections_across_twelve_decades(qg, precision):
    c = grid()
    rng = np.random.default_rng(4)
    load = c.load_p.copy()
    load[1] = rng.choice([-1.0, 1.0], c.n_bus) * 10.0 ** rng.uniform(-6, 6, c.n_bus)
    load[2, rng.permutation(c.n_bus)[:3]] = [1e6, -1e6, 1e-6]
    c = dataclasses.replace(c, load_p=load)
    (od, zd, gd, fd), (os_, zs, gs, fs) = both(qg, c, precision)
    close_flows(fs, fd, precision)
    tol = 1e-10 if precision == 0 else 1e-4
    assert abs(os_ - od) <= tol * abs(od) and abs(zs - zd) <= tol * abs(zd)
    check_at(gs, gd, c, tol, "sparse against dense")
