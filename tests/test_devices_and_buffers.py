"""The host side of the entry points on a process with two GPUs, without a GPU: the library's objects linked
with a fake CUDA runtime (fake_cudart.cpp, where "device" memory is host memory with a device ordinal and
kernels do not run) in a child process.

Limits: shared memory above 48 KB has to be granted on each GPU.  Outputs: a kernel may write the caller's array only if it is aligned memory of the handle's own GPU apart
from the inputs; every other array takes a copy after the kernels, as it did when all of them did."""
import json
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = r"""
import ctypes as C, json, sys
sys.path.insert(0, ROOT)
import numpy as np
import synth
from paper_2310_06650_gb300 import qg

fake = C.CDLL(LIB)
fake.fake_alloc.restype = C.c_void_p
fake.fake_alloc.argtypes = [C.c_size_t, C.c_int, C.c_int]
fake.fake_watch.argtypes = [C.c_void_p]
fake.fake_copies_to.argtypes = [C.c_void_p]
fake.fake_hits.restype = fake.fake_copies_to.restype = C.c_longlong
HOST, DEVICE, MANAGED = 1, 2, 3

class Buf:
    def __init__(self, n, dev=0, kind=DEVICE):
        self.p = fake.fake_alloc(n, dev, kind)
    def at(self, off):
        b = Buf.__new__(Buf)
        b.p = self.p + off
        return b
    def data_ptr(self):
        return self.p

def routed(out, call):
    # (launches that were handed `out`, copies into it after the last launch)
    fake.fake_watch(out.p)
    call()
    return int(fake.fake_hits()), int(fake.fake_copies_to(out.p))

def handle(case, precision, **kw):
    return qg.qg_create(case, qg.case_options(case, precision=precision, **kw))

res = {}
"""


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    from paper_2310_06650_gb300 import build as b
    gxx, nvcc = shutil.which("g++"), b._nvcc()
    if gxx is None:
        pytest.skip("no host C++ compiler")
    objs = [os.path.join(b.OUT, os.path.splitext(s)[0] + ".o") for s in b.SOURCES]
    b.build(force=not all(os.path.exists(o) for o in objs))
    lib = str(tmp_path_factory.mktemp("fake") / "libqg_fake.so")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run([gxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-I", include, "-I", b.CSRC,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", lib, "-Wl,-Bsymbolic", "-ldl", "-lpthread"],
                   check=True, capture_output=True, text=True)

    def run(code):
        env = dict(os.environ, QG_LIBRARY=lib)
        out = subprocess.run([sys.executable, "-c", f"ROOT, LIB = {ROOT!r}, {lib!r}\n" + PRELUDE + code +
                              "\nprint(json.dumps(res))"], env=env, capture_output=True, text=True, timeout=600)
        assert out.returncode == 0, out.stderr[-3000:]
        return json.loads(out.stdout.strip().splitlines()[-1])

    return run


def test_eval_grad_writes_only_arrays_of_its_own_gpu(child):
    """On both paths and for handles on either GPU.  qg_eval_grad_noalloc asks for such arrays and has no
    copies."""
    r = child(r"""
c = synth.tiny()
for prec, w in ((qg.QG_FP64, 8), (qg.QG_MIXED, 4)):
    h = handle(c, prec)
    n = qg.qg_num_vars(h)
    x, obj, g = Buf(w * n + 64), Buf(8), Buf(w * n + 64)
    ev = lambda o, gg: (lambda: qg.qg_eval_grad(h, x, o, gg))
    far_g, far_o = Buf(w * n, 1), Buf(8, 1)
    man = Buf(w * n, 0, MANAGED)
    both = Buf(w * n + 8)
    res[f"own g {prec}"] = routed(g, ev(obj, g))
    res[f"own obj {prec}"] = routed(obj, ev(obj, g))
    res[f"other gpu g {prec}"] = routed(far_g, ev(obj, far_g))
    res[f"other gpu obj {prec}"] = routed(far_o, ev(far_o, g))
    res[f"managed g {prec}"] = routed(man, ev(obj, man))
    res[f"g on x {prec}"] = routed(x.at(w * 8), ev(obj, x.at(w * 8)))
    res[f"g is x {prec}"] = routed(x, ev(obj, x))
    res[f"misaligned g {prec}"] = routed(g.at(2), ev(obj, g.at(2)))
    res[f"g over obj {prec}"] = routed(both, ev(both.at(w * n - 8), both))
    res[f"obj in g {prec}"] = routed(both.at(w * n - 8), ev(both.at(w * n - 8), both))
    res[f"no obj {prec}"] = routed(g, ev(None, g))
    res[f"no g {prec}"] = routed(obj, ev(obj, None))
    qg.qg_destroy(h)
    fake.fake_set_device(1)
    h = handle(c, prec)
    x1, obj1, g1 = Buf(w * n, 1), Buf(8, 1), Buf(w * n, 1)
    res[f"own g on 1 {prec}"] = routed(g1, lambda: qg.qg_eval_grad(h, x1, obj1, g1))
    res[f"other gpu g on 0 {prec}"] = routed(g, lambda: qg.qg_eval_grad(h, x1, obj1, g))
    qg.qg_destroy(h)
    fake.fake_set_device(0)
""")
    for name, (hits, copies) in r.items():
        kernel = name.split(" ")[0] in ("own", "no")
        assert (hits > 0, copies) == ((True, 0) if kernel else (False, 1)), (name, hits, copies)


def test_mlp_forward_writes_only_arrays_of_its_own_gpu(child):
    r = child(r"""
m = qg.qg_mlp_create(65, 33, 127, 7)
for B in (7, 1):
    x, y, far, man = Buf(4 * 65 * 7), Buf(4 * 127 * 7 + 64), Buf(4 * 127 * 7, 1), Buf(4 * 127 * 7, 0, MANAGED)
    for name, out in (("own", y), ("other gpu", far), ("managed", man), ("misaligned", y.at(2))):
        res[f"{name} {B}"] = routed(out, lambda: qg.qg_mlp_forward(m, x, B, out))
qg.qg_mlp_destroy(m)
""")
    for name, (hits, copies) in r.items():
        assert (hits, copies) == ((1, 0) if name.startswith("own") else (0, 1)), (name, hits, copies)


def test_sparse_handles_evaluate_on_every_gpu(child):
    """The tail product's shared-memory limit is an attribute of its kernel on one GPU."""
    r = child(r"""
c = synth.make_case("tail", 617, 925, 88, T=3, K=20, seed=1)
for dev in (0, 1):
    fake.fake_set_device(dev)
    for prec, w in ((qg.QG_FP64, 8), (qg.QG_MIXED, 4)):
        h = handle(c, prec, dc_solver=qg.QG_DC_SPARSE)
        x, obj, g = Buf(w * qg.qg_num_vars(h), dev), Buf(8, dev), Buf(w * qg.qg_num_vars(h), dev)
        for _ in range(2):
            qg.qg_eval_grad(h, x, obj, g)
        qg.qg_destroy(h)
        res[f"{dev} {prec}"] = True
""")
    assert len(r) == 4


def test_contingency_blocks_evaluate_on_every_gpu(child):
    """A contingency block of many periods (above 48 KB on both paths), then a smaller one, on the first GPU
    and then on the second."""
    r = child(r"""
big, small = synth.make_case("big", 90, 140, 9, T=48, K=20, seed=1), synth.mid()
for dev in (0, 1):
    fake.fake_set_device(dev)
    for prec, w in ((qg.QG_FP64, 8), (qg.QG_MIXED, 4)):
        hs = [handle(c, prec, ctg_bound=qg.QG_CTG_BOUND_LAZY) for c in (big, small)]
        for h in hs:
            n = qg.qg_num_vars(h)
            qg.qg_eval_grad(h, Buf(w * n, dev), Buf(8, dev), Buf(w * n, dev))
        for h in hs:
            qg.qg_destroy(h)
        res[f"{dev} {prec}"] = True
""")
    assert len(r) == 4


def test_networks_run_on_every_gpu(child):
    r = child(r"""
for dev in (0, 1):
    fake.fake_set_device(dev)
    m = qg.qg_mlp_create(65, 33, 127, 7)
    x, t, y = Buf(4 * 65 * 7, dev), Buf(4 * 127 * 7, dev), Buf(4 * 127 * 7, dev)
    qg.qg_mlp_forward(m, x, 7, y)
    qg.qg_mlp_train_step(m, x, t, 7, 1e-3)
    qg.qg_mlp_destroy(m)
    res[str(dev)] = True
""")
    assert len(r) == 2
