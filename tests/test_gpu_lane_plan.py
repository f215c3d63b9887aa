"""Launch plans of lane = instance batches on the GPU."""
import pytest

import oracle
from paper_2403_04714_gb300 import netgen, sim

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tiny_text():
    return open(netgen.cached_netlist("tiny")).read()


@pytest.mark.parametrize("lowering", ["bytecode", "generated"])
def test_a_pool_plans_again_only_when_its_groups_or_share_change(tiny_text, lowering):
    nl = sim.Netlist(tiny_text, mode="lane_inst", lowering=lowering)
    s = sim.Server(pool_slots=256, chunk_cycles=1)
    try:
        job = s.submit(nl, 40, 3, 60)
        s.wait(job)
        before = sim.debug_count(sim.SIM_COUNT_PLANS)
        job = s.submit(nl, 40, 3, 60)           # sixty steps of one cycle
        s.wait(job)
        assert sim.debug_count(sim.SIM_COUNT_PLANS) - before <= 1
        got = s.digests(job, 40)
    finally:
        s.close()
    net = oracle.Net(text=tiny_text)
    for i in (0, 39):
        ref = oracle.Sim(net, seed=3, inst=i)
        ref.run(60)
        assert got[i] == ref.digest(), i
