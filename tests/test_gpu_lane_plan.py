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


@pytest.fixture(scope="module")
def mid_text():
    return open(netgen.cached_netlist("mid")).read()


@pytest.fixture(scope="module")
def mid_net(mid_text):
    return oracle.Net(text=mid_text)


@pytest.mark.parametrize("procs,n_inst,kernel", [(0, 1000, "persistent"), (256, 1500, "persistent_graph"), (256, 500, "persistent")])
def test_bands(mid_text, mid_net, procs, n_inst, kernel):
    nl = sim.Netlist(mid_text, mode="lane_inst", target_processes=procs, kernel=kernel)
    plan = nl.debug_lane_plan((n_inst + 31) // 32)
    assert plan["banded"] and plan["rounds"] > 1
    b = sim.Batch(nl, n_inst, seed=6)
    info = b.launch_info()
    assert (info["ctas"], info["warps_per_cta"]) == (plan["ctas"], plan["warps_per_cta"])
    b.step(7)
    got = b.state_digests()
    for i in (0, 33, n_inst // 2, n_inst - 1):
        ref = oracle.Sim(mid_net, seed=6, inst=i)
        ref.run(7)
        assert got[i] == ref.digest(), i


def test_pools_in_bands_as_jobs_come_and_go(mid_text, mid_net, tiny_text):
    # two pools, so that the groups in use and the share change between steps
    nl = sim.Netlist(mid_text, mode="lane_inst", target_processes=256)
    assert nl.debug_lane_plan(16, 1)["banded"] and nl.debug_lane_plan(16, 2)["banded"] and nl.debug_lane_plan(32, 2)["banded"]
    assert not nl.debug_lane_plan(1, 2)["banded"]
    tiny = sim.Netlist(tiny_text, mode="lane_inst")
    s = sim.Server(pool_slots=1024, chunk_cycles=3)
    try:
        jobs = [(s.submit(n, size, seed, cycles), n, size, seed, cycles)
                for n, size, seed, cycles in [(nl, 32, 1, 20), (nl, 500, 2, 14), (tiny, 100, 3, 40), (nl, 450, 4, 5), (tiny, 64, 5, 11),
                                              (nl, 400, 6, 9)]]
        for job, *_ in jobs:
            s.wait(job)
        digests = {job: s.digests(job, size) for job, _, size, _, _ in jobs}
    finally:
        s.close()
    nets = {nl: mid_net, tiny: oracle.Net(text=tiny_text)}
    for job, n, size, seed, cycles in jobs:
        for i in (0, size // 2, size - 1):
            ref = oracle.Sim(nets[n], seed=seed, inst=i)
            ref.run(cycles)
            assert digests[job][i] == ref.digest(), (size, i)
