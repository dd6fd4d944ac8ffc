"""The index-checked build on the kernels that only larger plans take: hot rows of stage 2 on both paths (with
screening scores too), the adjoint DC products of large dense plans, the on-demand contingency path, and the
tail product of the sparse DC solver (whose tiles the copy engine fetches within its tensor maps; the rest of
its accesses is checked).  Results are those of the oracle (1e-9 FP64 path, 1e-4 mixed path, in the norm) and no
checked access misses."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import dataclasses, json, sys
sys.path.insert(0, ROOT)
import numpy as np, torch
import oracle, synth
from paper_2310_06650_gb300 import qg

def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-300))

res = {}
def run(name, c, prec, path, **kw):
    x0 = np.clip(synth.random_point(c, 3, 0.2), *oracle.box(c)).astype(np.float32).astype(np.float64)
    s = qg.Solver(c, precision=prec, **kw)
    x = torch.tensor(x0, dtype=s.dtype, device="cuda")
    obj, g = (t.clone() for t in s.eval_grad(x))
    torch.cuda.synchronize()
    ref = oracle.evaluate(c, x0)
    got = (rel(obj.item(), ref.obj), rel(g.double().cpu().numpy(), ref.grad), 1e-9 if prec == qg.QG_FP64 else 1e-4)
    shapes = qg.qg_launches_per_eval(s.h), qg.qg_ctg_path(s.h)
    qg.qg_solve(s.h, x, 2, 1e-3, 0.9, 0.999)
    torch.cuda.synchronize()
    s.close()
    assert shapes[1] == path, (name, shapes)
    res[name] = got

def grid(n, M, K, T, scale):
    c = synth.make_case("hot", n, M, max(5, n // 10), T=T, K=K, seed=n + K)
    return dataclasses.replace(c, s_max_ctg=scale * c.s_max_ctg)

F64, MIXED = qg.QG_FP64, qg.QG_MIXED
run("hot rows, adjoint products, FP64", grid(90, 140, 3, 480, 0.2), F64, 0)
run("adjoint products, mixed", grid(90, 140, 3, 480, 0.2), MIXED, 0)
run("hot rows of two column blocks, FP64", grid(700, 1100, 1025, 60, 0.5), F64, 0)
run("hot rows, on-demand path, mixed", grid(1350, 2100, 2001, 2, 0.5), MIXED, 2)
run("hot rows, compact block, mixed", grid(1350, 2100, 2001, 2, 0.5), MIXED, 2, lodf_dtype=qg.QG_LODF_BF16X2)
run("hot rows, scores, FP64", grid(700, 1100, 998, 64, 0.5), F64, 0, ctg_frac=1.0 - 1e-9)
for prec in (F64, MIXED):
    run(f"on-demand path {prec}", synth.mid(), prec, 2, ctg_bound=qg.QG_CTG_BOUND_LAZY)
    run(f"eager bound test {prec}", synth.mid(), prec, 1, ctg_bound=qg.QG_CTG_BOUND_EAGER)
    run(f"tail, two passes {prec}", synth.make_case("tail", 1200, 1800, 170, T=50, K=20, seed=9), prec, 0,
        dc_solver=qg.QG_DC_SPARSE)
print(json.dumps({"cases": res, "report": qg.qg_bounds_report()}))
"""


def test_checked_build_sees_no_bad_index_on_larger_plans():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_06650_gb300.build import build
    lib = build(check_bounds=True)
    env = dict(os.environ, QG_LIBRARY=lib)
    out = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + CHILD], env=env, capture_output=True,
                         text=True, timeout=1200)
    assert out.returncode == 0, out.stderr[-3000:]
    res = json.loads(out.stdout.strip().splitlines()[-1])
    assert res["report"] is None, f"a checked access missed: line {res['report'][0]}"
    for name, (ro, rg, tol) in res["cases"].items():
        assert ro <= tol and rg <= tol, (name, ro, rg)
