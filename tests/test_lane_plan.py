"""Launch plans of the lane = instance bytecode (CPU only): a pool on 1 / share
of the GPU takes at most that share of the CTAs that fit, also with a configured
CTA size whose value slots leave room for fewer CTAs per SM than its warps
would.  Launches of one cycle get small CTAs unless larger ones let more warps
share an SM."""
import pytest

from paper_2403_04714_gb300 import netgen, sim


@pytest.fixture(scope="module")
def mid_text():
    return open(netgen.cached_netlist("mid")).read()


@pytest.mark.parametrize("warps", [0, 4, 8, 16, 22, 32])
def test_a_pool_keeps_to_its_share(mid_text, warps):
    nl = sim.Netlist(mid_text, mode="lane_inst", warps_per_cta=warps)
    tasks = nl.info()["n_processes"]
    for groups in (1, 3, 32, 128):
        for share in (1, 2, 3, 5, 200):
            for per_cycle in (False, True):
                p = nl.debug_lane_plan(groups, share, per_cycle)
                assert 1 <= p["ctas"] <= max(1, p["max_ctas"] // share), (groups, share, p)
                assert p["rounds"] * p["ctas"] * p["warps_per_cta"] >= tasks * groups
                assert p["smem"] <= 227 * 1024 - 32
                assert not (per_cycle and p["banded"])


def test_a_configured_cta_size_is_kept_where_it_fits(mid_text):
    for warps in (1, 4, 8):
        nl = sim.Netlist(mid_text, mode="lane_inst", warps_per_cta=warps)
        assert nl.debug_lane_plan(128)["warps_per_cta"] == warps


def test_launches_of_one_cycle(mid_text):
    tiny = sim.Netlist(open(netgen.cached_netlist("tiny")).read(), mode="lane_inst")
    for groups in (22, 79, 128):
        assert tiny.debug_lane_plan(groups, per_cycle=True)["warps_per_cta"] == 4
    assert tiny.debug_lane_plan(4, per_cycle=True)["warps_per_cta"] == 2       # 280 tasks on 152 SMs
    assert tiny.debug_lane_plan(1, per_cycle=True)["warps_per_cta"] == 1
    mid = sim.Netlist(mid_text, mode="lane_inst")
    p = mid.debug_lane_plan(79, per_cycle=True)      # 69 slots and fewer: three CTAs of four warps
    assert p["max_ctas"] * p["warps_per_cta"] >= 152 * 16
