"""Host calls (CPU only, behind a stand-in for the CUDA runtime with two pretended
GPUs).  Reads and checkpoints while another device than the batch's is current,
and without pinned memory: for the caller they are plain copies, which need
neither.  Launch plans of several instances with lane = operation, and of
generated code."""
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


NO_PINNED = """
from paper_2403_04714_gb300 import netgen, sim

text = netgen.gen_flat(5, n_ops=900, n_regs=60, depth=12, n_inputs=4, rams=((3, 64),)).to_text()
nl = sim.Netlist(text)
init = [int(l.split()[2]) for l in text.splitlines() if l.startswith("reg ")]
width = [int(l.split()[1]) for l in text.splitlines() if l.startswith("reg ")]
assert any(init) and {1, 32, 64} <= set(width)
for n_inst in (1, 70):
    b = sim.Batch(nl, n_inst)
    b.step(2)                                   # pretended kernels change nothing
    for i in {0, n_inst // 2, n_inst - 1}:
        assert list(b.regs(i)) == init
        want = [hash((i, r)) % 2 ** w for r, w in enumerate(width)]
        for r, v in enumerate(want):
            b.poke_reg(i, r, v)
        words = [hash((i, a)) % 2 ** 64 for a in range(8)]
        for a, v in enumerate(words):
            b.poke_mem(i, 0, a, v)
        assert list(b.regs(i)) == want and list(b.mem_all(i, 0)) == words
print("done")
"""

PLANS = """
from paper_2403_04714_gb300 import netgen, sim

def plan(nl, n_inst):
    b = sim.Batch(nl, n_inst)
    i = b.launch_info()
    b.close()
    return i["ctas"] * i["warps_per_cta"], i["tasks_per_cycle"]

# few large processes: a warp for every task, not one for several instances in turn
text = open(netgen.cached_netlist("mid")).read()
few = sim.Netlist(text, mode="lane_op", target_processes=30)
for n in (8, 16, 31, 64):
    warps, tasks = plan(few, n)
    assert tasks == 30 * n and warps >= tasks, (n, warps, tasks)
warps, tasks = plan(few, 200)
assert warps >= 1216, warps
# resident programs where they are the better ones
assert plan(few, 5)[0] == 150
some = sim.Netlist(text, mode="lane_op", target_processes=152)
assert plan(some, 16)[0] == 1216
assert plan(sim.Netlist(open(netgen.cached_netlist("tiny")).read(), mode="lane_op"), 8)[0] == 560
print("done")
"""

GENERATED = """
from paper_2403_04714_gb300 import netgen, sim

text = open(netgen.cached_netlist("tiny")).read()
for warps in (1, 2, 3, 4, 6, 8):
    nl = sim.Netlist(text, mode="lane_inst", lowering="generated", warps_per_cta=warps)
    for n in (1, 700, 2500, 4096, 9999):
        b = sim.Batch(nl, n)
        i = b.launch_info()
        assert i["warps_per_cta"] == warps
        need = -(-i["tasks_per_cycle"] // warps)
        most = 32 // warps * 152
        rounds = -(-need // most)
        assert i["ctas"] == (-(-need // rounds) if warps <= 4 else min(need, most)), (warps, n, i)
        b.close()

# launches of one cycle: few tasks are spread over the SMs unless they are brief
def warps(text, **cfg):
    b = sim.Batch(sim.Netlist(text, mode="lane_inst", lowering="generated", **cfg), 32)
    return b.launch_info()["warps_per_cta"]

longer = netgen.gen_flat(21, 5000, 400, 20, 9).to_text()
assert warps(text) == 2 and warps(longer) == 2
assert warps(text, kernel="graph") == 8 and warps(text, kernel="per_cycle") == 8
assert warps(longer, kernel="graph") == 2 and warps(text, kernel="persistent_graph") == 2
print("done")
"""


def run(program, tmp_path, **env):
    if not shutil.which("g++") or not os.path.exists(f"{CUDA}/include/cuda_runtime_api.h"):
        pytest.skip("needs g++ and the CUDA headers")
    so = str(tmp_path / "fake_cuda_runtime.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", f"-I{CUDA}/include", "-o", so, os.path.join(HERE, "fake_cuda_runtime.cpp")],
                   check=True)
    r = subprocess.run([sys.executable, "-c", program], cwd=os.path.dirname(HERE), capture_output=True, text=True, timeout=120,
                       env={**os.environ, "LD_PRELOAD": so, **env})
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr


def test_reads_and_checkpoints_take_any_current_device(tmp_path):
    run(PROGRAM, tmp_path)


def test_reads_without_pinned_memory(tmp_path):
    run(NO_PINNED, tmp_path, FAKE_CUDA_NO_PINNED="1")


def test_plans_of_several_instances(tmp_path):
    run(PLANS, tmp_path)


def test_plans_of_generated_code(tmp_path):
    run(GENERATED, tmp_path)
