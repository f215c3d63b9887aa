"""What admission counts for a pool (CPU only): its state and the programs that
are uploaded for it, which are the lane = instance ones whatever else the netlist
was lowered to."""
import pytest

from paper_2403_04714_gb300 import netgen, sim


@pytest.fixture(scope="module")
def text():
    return netgen.gen_flat(7, n_ops=3000, n_regs=200, depth=15, n_inputs=6, rams=((4, 64), (3, 16))).to_text()


def test_programs_a_pool_does_not_have_are_not_counted(text):
    base = sim.Netlist(text, target_processes=16)
    pairs = sim.Netlist(text, target_processes=16, chain=2)
    cluster = sim.Netlist(text, target_processes=16, mode="lane_op", cluster_size=2, warps_per_cta=8)
    assert len(pairs.table("c_words")) != len(base.table("c_words"))
    for other in (pairs, cluster):
        assert len(other.table("b_ins")) == len(base.table("b_ins"))
        assert sim.Server.footprint(other, 64) == sim.Server.footprint(base, 64)


def test_the_program_is_counted_as_uploaded(text):
    a, b = (sim.Netlist(text, target_processes=n) for n in (4, 40))
    tables = [nl.table("b_ins").nbytes + 4 * nl.table("b_off").nbytes for nl in (a, b)]
    assert tables[0] != tables[1]
    assert sim.Server.footprint(b, 64) - sim.Server.footprint(a, 64) == tables[1] - tables[0]
