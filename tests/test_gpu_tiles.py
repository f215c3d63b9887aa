"""Lane = instance state in group tiles: a checkpoint stays in [register]
[instance] order, read back register by register, and moves between batches."""
import numpy as np
import pytest

import oracle
from paper_2403_04714_gb300 import netgen, sim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lowering", ["bytecode", "generated"])
@pytest.mark.parametrize("n_inst", [1, 33, 100])
def test_checkpoint_order(lowering, n_inst):
    text = netgen.gen_flat(11, n_ops=1500, n_regs=90, depth=14, n_inputs=5, rams=((4, 64),)).to_text()
    nl = sim.Netlist(text, mode="lane_inst", lowering=lowering)
    b = sim.Batch(nl, n_inst, seed=3)
    b.step(37)
    r = 7
    b.poke_reg(n_inst - 1, r, 0x5A5A5A5A5A5A5A5A)
    blob = b.save()
    I = -(-n_inst // 32) * 32
    cls, idx = nl.table("reg_cls"), nl.table("reg_idx")
    n1, n32, n64 = (int((cls == c).sum()) for c in range(3))
    raw = np.frombuffer(blob, dtype=np.uint8)[64:]
    bits = raw[:n1 * I // 8].view(np.uint32).reshape(n1, I // 32)
    w32 = raw[n1 * I // 8:][:n32 * I * 4].view(np.uint32).reshape(n32, I)
    w64 = raw[n1 * I // 8 + n32 * I * 4:][:n64 * I * 8].view(np.uint64).reshape(n64, I)
    for i in {0, n_inst // 2, n_inst - 1}:
        regs = b.regs(i)
        want = [int(w64[x, i]) if c == 2 else int(w32[x, i]) if c == 1 else int(bits[x, i // 32]) >> (i % 32) & 1
                for c, x in zip(cls, idx)]
        assert regs.tolist() == want, i
        assert b.peek_reg(i, r) == want[r]
    other = sim.Batch(nl, n_inst, seed=3)
    other.step(3)
    other.restore(blob)
    assert other.save() == blob
    b.step(20)
    other.step(20)
    assert np.array_equal(b.state_digests(), other.state_digests())
    ref = oracle.Sim(oracle.Net(text=text), seed=3, inst=0)
    ref.run(37)
    if n_inst == 1:
        ref.set_reg(r, 0x5A5A5A5A5A5A5A5A)
    ref.run(20)
    assert b.state_digests()[0] == ref.digest()


@pytest.mark.parametrize("n_inst", [32, 64, 96, 250, 600])
def test_spread_small_batches(n_inst):
    # few tasks run in smaller CTAs: every size matches the oracle
    text = netgen.gen_flat(12, n_ops=6000, n_regs=400, depth=16, n_inputs=6).to_text()
    b = sim.Batch(sim.Netlist(text, mode="lane_inst", lowering="generated"), n_inst, seed=4)
    b.step(50)
    net = oracle.Net(text=text)
    got = b.state_digests()
    for i in {0, n_inst // 2, n_inst - 1}:
        ref = oracle.Sim(net, seed=4, inst=i)
        ref.run(50)
        assert got[i] == ref.digest(), i
