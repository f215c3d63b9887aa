"""Reads and checkpoints of a batch while another device is current (CPU only,
two pretended GPUs): they were always plain copies for the caller, which take any
current device, and must not ask for the batch's now that kernels gather for them."""
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = """
import ctypes
from paper_2403_04714_gb300 import netgen, sim

fake = ctypes.CDLL(None)
def current():
    d = ctypes.c_int()
    fake.cudaGetDevice(ctypes.byref(d))
    return d.value

text = netgen.gen_flat(5, n_ops=900, n_regs=60, depth=12, n_inputs=4, rams=((3, 64),)).to_text()
for n_inst in (1, 33):
    fake.cudaSetDevice(0)
    b = sim.Batch(sim.Netlist(text), n_inst)
    b.step(3)
    for device in (0, 1):
        fake.cudaSetDevice(device)
        b.regs(n_inst - 1)
        b.mem_all(n_inst - 1, 0)
        b.restore(b.save())
        b.peek_reg(0, 1)
        assert current() == device
    b.close()
print("done")
"""


def test_reads_and_checkpoints_take_any_current_device(tmp_path):
    if not shutil.which("g++") or not os.path.exists(f"{CUDA}/include/cuda_runtime_api.h"):
        pytest.skip("needs g++ and the CUDA headers")
    so = str(tmp_path / "fake_cuda_runtime.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", f"-I{CUDA}/include", "-o", so, os.path.join(HERE, "fake_cuda_runtime.cpp")],
                   check=True)
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=os.path.dirname(HERE), capture_output=True, text=True, timeout=120,
                       env={**os.environ, "LD_PRELOAD": so})
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr
