"""The network's host code on a CUDA runtime without a GPU (fake_cudart.c): what it launches, in which order, and what it
does when a launch fails."""
import os
import subprocess
import sys

import pytest

from paper_2312_07440_gb300 import rwgt

HERE = os.path.dirname(os.path.abspath(__file__))
PRELUDE = """
import ctypes, re
import numpy as np
from paper_2312_07440_gb300 import rwgt
lib, fake = rwgt.load(), ctypes.CDLL(None)
fake.fake_log.restype = ctypes.c_char_p
B = 2100  # rows: enough for the tensor-core backward pass
x, y, out = np.zeros((B, 40), np.float32), np.zeros(B, np.float32), np.zeros((B, 2), np.float32)

def kernels():
    return re.findall(r"k_[a-z0-9_]+?(?=E|I[Li])", fake.fake_log().decode())

def model(device):
    m = ctypes.c_void_p()
    assert lib.rw_mlp_create(ctypes.byref(m), device, None, 40, 256, 4, B, 7) == 0
    return m

def train(m, steps):
    return lib.rw_mlp_train(m, x.ctypes.data, y.ctypes.data, B, B, steps, 1e-3, 0.3, 0.1, 5)

def forward(m):
    return lib.rw_mlp_forward(m, x.ctypes.data, B, out.ctypes.data)
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "fake_cudart.c")], check=True)
    if not os.path.exists(rwgt.LIB_PATH):
        pytest.skip("the CUDA library is not built")

    def go(body):
        r = subprocess.run([sys.executable, "-c", PRELUDE + body], capture_output=True, text=True, timeout=300,
                           cwd=os.path.join(HERE, ".."), env={**os.environ, "LD_PRELOAD": so})
        assert r.returncode == 0, r.stdout + r.stderr
    return go


def test_a_model_on_a_second_device(run):
    """The limit on dynamic shared memory belongs to a function on one device: each model raises it on its own."""
    run("""
for device in (0, 1):
    m = model(device)
    for gemm in (0, 2):
        assert lib.rw_mlp_set_gemm(m, gemm) == 0
        assert train(m, 2) == 0 and forward(m) == 0, (device, gemm, lib.rw_mlp_last_error(m))
    lib.rw_mlp_destroy(m)
""")


def test_packed_weights_follow_the_parameters_after_a_failed_step(run):
    """Whichever launch of a training run fails, the inference that follows packs or has packed the weights after the last
    update of the parameters, and so have the transposes been made."""
    run("""
m = model(0)
fake.fake_clear()
assert train(m, 1) == 0
step = kernels()
assert step.count("k_adam") == 1 and step[-2:] == ["k_transpose_bf16", "k_pack_infer"], step
for n in range(1, 3 * len(step)):
    fake.fake_clear()
    fake.fake_fail_launch(n)
    rc = train(m, 3)
    fake.fake_fail_launch(0)
    assert rc == (-5 if n <= 3 * len(step) - 2 else 0), (n, rc)  # all but the last step leave the packing out
    assert forward(m) == 0
    log = kernels()
    assert log[-1] == "k_mlp_infer", log
    if "k_adam" in log:
        after = log[len(log) - 1 - log[::-1].index("k_adam"):]
        assert "k_transpose_bf16" in after and "k_pack_infer" in after, (n, after)
""")
