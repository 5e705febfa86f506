"""The library's launches against a CUDA runtime without a GPU (fake_cudart.c, preloaded
into a child process): nothing runs, so every device pointer may be any aligned address."""
import os
import subprocess
import sys

import pytest

from paper_2609_38169_gb300 import build_ext

HERE = os.path.dirname(os.path.abspath(__file__))

# The calls by name, each a function of no arguments that returns the status.
CALLS = """
import ctypes as C
import numpy as np
from paper_2609_38169_gb300 import api as A, _lib
fake = C.CDLL(None)
L, p, B = _lib.lib(), C.c_void_p(1 << 20), 4
assert fake.fake_launches() == 0
def plan_of(gate):
    cfg = A.Config(2, 1, 2, gate)
    n, rng = A.stepq_num_units(cfg), np.random.default_rng(0)
    omega, ell = rng.lognormal(size=(2, 2, 128)).astype(np.float32), np.log(rng.uniform(0.85, 0.99, n))
    dist = rng.uniform(size=(n, 4)) * 4.0 ** -np.arange(4)
    return cfg, A.stepq_fit_scales(cfg, omega, ell, dist)
cfg, plan = {}, {}
for kind, gate in (("heads", A.GATE_SCALAR), ("rows", A.GATE_CHANNEL)):
    cfg[kind], plan[kind] = plan_of(gate)
c = {k: v.c() for k, v in cfg.items()}
calls = {"fp32": lambda: L.stepq_fp32_decode_step(c["heads"], 0, p, B, p, B, p, p, p, p, p, p, None),
         "int8": lambda: L.stepq_intb_decode_step(c["heads"], 8, 0, p, B, p, B, p, p, p, p, p, p, None),
         "prefill": lambda: L.stepq_prefill_fp32(c["heads"], B, 40, p, p, p, p, p, p, p, None),
         "observe": lambda: L.stepq_calib_observe(c["heads"], 0, p, p, p, p, B, p, p, None)}
for k in ("heads", "rows"):
    h = plan[k].handle
    calls.update({
        k + " decode": lambda h=h: L.stepq_decode_step(h, 0, p, B, p, B, p, p, p, p, p, p, None),
        k + " readout": lambda h=h: L.stepq_decode_readout(h, 0, p, B, p, B, p, p, p, p, p, p, p, None),
        k + " writeback": lambda h=h: L.stepq_decode_writeback(h, 0, p, B, p, B, p, p, p, p, None),
        k + " pack": lambda h=h: L.stepq_quantize_pool(h, -1, p, p, B, p, B, None),
        k + " unpack": lambda h=h: L.stepq_dequantize_pool(h, -1, p, B, p, B, p, None)})
"""
LAUNCH, SET_ATTRIBUTE, GET_ATTRIBUTES = range(3)
STEPQ_ERR_CUDA = 5


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    build_ext.build()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build_ext.nvcc())))
    fake = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-Wall", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "fake_cudart.c"), "-o", fake], check=True)

    def child(code):
        r = subprocess.run([sys.executable, "-c", CALLS + code], cwd=os.path.dirname(HERE), capture_output=True,
                           text=True, env={**os.environ, "LD_PRELOAD": fake}, timeout=120)
        assert r.returncode == 0, r.stderr
        return r.stdout
    return child


@pytest.mark.parametrize("kind", [LAUNCH, SET_ATTRIBUTE])
def test_a_refused_launch_leaves_no_error(run, kind):
    """A call whose launch (or shared-memory opt-in) the runtime refuses returns
    STEPQ_ERR_CUDA and leaves nothing behind: the next call is not failed by it."""
    run(f"""
for name, call in calls.items():
    fake.fake_refuse({kind}, 1)
    before, status = fake.fake_launches(), call()
    fake.fake_refuse({kind}, 0)
    assert status == (0 if fake.fake_launches() > before else {STEPQ_ERR_CUDA}), (name, status)
    assert fake.fake_pending_error() == 0, name
    assert calls["observe"]() == 0, name           # a plain launch, checked by the last error
    assert call() == 0, name
""")


def test_prefill_after_a_failed_attribute_query(run):
    """A failed query of prefill's register count fails that call alone."""
    run(f"""
fake.fake_refuse({GET_ATTRIBUTES}, 1)
assert calls["prefill"]() == {STEPQ_ERR_CUDA}
assert fake.fake_pending_error() == 0 and fake.fake_launches() == 0
assert calls["observe"]() == 0 and calls["prefill"]() == 0
""")
