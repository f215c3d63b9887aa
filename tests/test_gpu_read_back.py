"""Read-back of registers and memories through pinned buffers."""
import threading

import numpy as np
import pytest

import oracle
from paper_2403_04714_gb300 import netgen, sim

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def text():
    return netgen.gen_flat(5, n_ops=900, n_regs=60, depth=12, n_inputs=4, rams=((3, 64), (8, 17))).to_text()


def check(b, ref, inst):
    assert np.array_equal(b.regs(inst), ref.regs())
    for m, depth in enumerate((8, 256)):
        assert np.array_equal(b.mem_all(inst, m), [ref.mem(m, a) for a in range(depth)])


def test_batches_one_after_another_share_the_pinned_buffer(text):
    nl = sim.Netlist(text)
    net = oracle.Net(text=text)
    before = sim.debug_count(sim.SIM_COUNT_PINNED)
    for seed in range(5):
        b = sim.Batch(nl, 1, seed=seed)
        b.step(9)
        ref = oracle.Sim(net, seed=seed, inst=0)
        ref.run(9)
        check(b, ref, 0)
        b.close()
    assert sim.debug_count(sim.SIM_COUNT_PINNED) - before == 1


def test_read_backs_on_several_threads(text):
    nl = sim.Netlist(text)
    net = oracle.Net(text=text)
    errors = []

    def work(seed):
        try:
            b = sim.Batch(nl, 33, seed=seed)
            ref = oracle.Sim(net, seed=seed, inst=32)
            for _ in range(10):
                b.step(3)
                ref.run(3)
                check(b, ref, 32)
        except Exception as e:      # reported on the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in range(7)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
