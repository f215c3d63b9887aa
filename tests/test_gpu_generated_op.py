"""Generated code with lane = operation, whose kernels take more registers than
those of lane = instance: configured CTA sizes up to ones that do not fit."""
import numpy as np
import pytest

import oracle
from paper_2403_04714_gb300 import netgen, sim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warps", [0, 1, 24, 25, 32])
@pytest.mark.parametrize("n_inst", [1, 9])
def test_cta_sizes(warps, n_inst):
    text = open(netgen.cached_netlist("tiny")).read()
    b = sim.Batch(sim.Netlist(text, mode="lane_op", lowering="generated", warps_per_cta=warps), n_inst, seed=3)
    got = b.launch_info()["warps_per_cta"]
    assert got == warps if warps in (1, 24) else 2 <= got <= 24
    b.step(40)
    ref = oracle.Sim(oracle.Net(text=text), seed=3, inst=n_inst - 1)
    ref.run(40)
    assert np.array_equal(b.regs(n_inst - 1), ref.regs())
