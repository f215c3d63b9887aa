"""Persistent launches of more CTAs than the grid barrier polls quickly for: states
against the oracle, and its wait running out."""
import pytest

import oracle
from paper_2403_04714_gb300 import netgen, sim

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tiny_text():
    return open(netgen.cached_netlist("tiny")).read()


@pytest.mark.parametrize("warps", [1, 2, 6])
def test_states_and_time_out(tiny_text, warps):
    nl = sim.Netlist(tiny_text, mode="lane_inst", lowering="generated", warps_per_cta=warps)
    b = sim.Batch(nl, 2500, seed=4)
    assert b.launch_info()["ctas"] > 608
    b.step(50)
    b.step(1)
    got = b.state_digests()
    net = oracle.Net(text=tiny_text)
    for i in (0, 1000, 2499):
        ref = oracle.Sim(net, seed=4, inst=i)
        ref.run(51)
        assert got[i] == ref.digest(), i
    b.debug_skip_arrival(20)
    b.step(3)
    with pytest.raises(sim.SimError) as e:
        b.sync()
    assert e.value.name == "SIM_ERR_TIMEOUT"
