"""Lane = instance bytecode with areas packed by process: warps per CTA given
or chosen, one round and several, in bands, launches of one cycle; every
instruction kind; against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2403_04714_gb300 import netgen, sim
from test_gpu_step_ops import ops_netlist

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["persistent", "per_cycle", "graph"])
@pytest.mark.parametrize("n_inst,warps,procs", [(1, 0, 0), (33, 0, 0), (100, 1, 3), (100, 6, 40), (900, 0, 40), (2100, 32, 9)])
def test_packed_areas(kernel, n_inst, warps, procs):
    text = ops_netlist(9, n_chains=90)
    b = sim.Batch(sim.Netlist(text, mode="lane_inst", kernel=kernel, warps_per_cta=warps, target_processes=procs), n_inst, seed=2)
    b.hold_input(0, 3, 0x7FFFFFFF)
    b.step(70)
    net = oracle.Net(text=text)
    got = b.state_digests()
    for i in {0, n_inst // 2, n_inst - 1}:
        ref = oracle.Sim(net, seed=2, inst=i)
        if i == 0:
            ref.hold_input(3, 0x7FFFFFFF)
        ref.run(70)
        assert got[i] == ref.digest(), i
        assert np.array_equal(b.regs(i), ref.regs()), i


def test_bands_with_memories():
    # many instances of a netlist whose processes differ in size: several rounds
    text = netgen.gen_flat(21, n_ops=20_000, n_regs=900, depth=30, n_inputs=9, rams=((5, 64), (3, 17))).to_text()
    b = sim.Batch(sim.Netlist(text, mode="lane_inst"), 1500, seed=6)
    b.step(30)
    net = oracle.Net(text=text)
    got = b.state_digests()
    for i in (0, 31, 32, 777, 1499):
        ref = oracle.Sim(net, seed=6, inst=i)
        ref.run(30)
        assert got[i] == ref.digest(), i


def test_configured_warps_that_do_not_fit():
    # 32 warps' slots of the 200k-op netlist exceed an SM: fewer run
    b = sim.Batch(sim.Netlist(open(netgen.cached_netlist("mid")).read(), mode="lane_inst", warps_per_cta=32), 33, seed=1)
    assert 1 <= b.launch_info()["warps_per_cta"] < 32
    b.step(5)
    ref = oracle.Sim(oracle.Net(text=open(netgen.cached_netlist("mid")).read()), seed=1, inst=32)
    ref.run(5)
    assert b.state_digests()[32] == ref.digest()
