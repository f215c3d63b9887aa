"""The step interpreter's one-formula operators at the edges of its encoding:
every operator over widths 1..64, shift amounts of 0, 63, 64 and more and of
more than 32 bits, muxes selected by wide values, pairs whose second operator
takes the first result in every position (also in two at once), and several
instances spread over warps; per-cycle digests against the oracle."""
import random

import numpy as np
import pytest

import oracle
from paper_2403_04714_gb300 import netgen, sim

pytestmark = pytest.mark.gpu

OPS = ("add", "sub", "mul", "and", "or", "xor", "shl", "shr", "eq", "lt", "mux", "slice", "concat")


def ops_netlist(seed, n_chains=60, length=9):
    rng = random.Random(seed)
    nl = netgen.Netlist()
    widths = (1, 2, 6, 7, 31, 32, 33, 63, 64)
    leaves = [nl.node("input", w, nl.add_input(w)) for w in widths]
    regs = [nl.add_reg(rng.choice(widths), 1) for _ in range(n_chains)]
    leaves += [nl.node("reg", nl.regs[r][0], r) for r in regs]
    for v in (0, 1, 31, 32, 63, 64, 65, (1 << 40) + 3, (1 << 64) - 1):
        leaves.append(nl.node("const", max(1, v.bit_length()), v))
    for r in regs:
        x = rng.choice(leaves)
        for _ in range(length):
            # the previous result in one operand or in several
            def arg():
                return x if rng.random() < 0.5 else rng.choice(leaves)
            op = rng.choice(OPS)
            w = rng.choice(widths)
            if op in ("eq", "lt"):
                y = nl.node(op, 1, arg(), arg())
            elif op == "mux":
                y = nl.node(op, w, arg(), arg(), arg())
            elif op == "slice":
                a = arg()
                lo = rng.choice((0, nl.width(a) - 1, rng.randrange(nl.width(a))))
                y = nl.node(op, rng.randint(1, nl.width(a) - lo), a, lo)
            elif op == "concat":
                a, b = arg(), arg()
                if nl.width(a) + nl.width(b) > 64:
                    a, b = (nl.node("slice", min(20, nl.width(v)), v, 0) for v in (a, b))
                y = nl.node(op, nl.width(a) + nl.width(b), a, b)
            else:
                y = nl.node(op, w, arg(), arg())
            x = y
        nl.set_next(r, x)
    return nl.to_text()


@pytest.mark.parametrize("cfg", [dict(), dict(chain=2), dict(chain=2, cluster_size=2, warps_per_cta=3, target_processes=11),
                                 dict(cluster_size=2, warps_per_cta=3, target_processes=11), dict(chain=2, target_processes=3)])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_operator_edges(cfg, seed):
    text = ops_netlist(seed)
    n = 120
    b = sim.Batch(sim.Netlist(text, mode="lane_op", digest_capacity=n + 1, **cfg), 1, seed=seed)
    b.step(n)
    ref = oracle.Sim(oracle.Net(text=text), seed=seed, inst=0)
    want = np.concatenate([np.array([ref.digest()], dtype=np.uint64), ref.run(n, digests=True)])
    got = b.digests(0, 0, n + 1)
    assert np.array_equal(got, want), int(np.nonzero(got != want)[0][0])
    assert np.array_equal(b.regs(0), ref.regs())


@pytest.mark.parametrize("chain", [0, 2])
@pytest.mark.parametrize("n_inst", [2, 7, 31, 64])
@pytest.mark.parametrize("procs", [0, 3, 200])
def test_instances_over_warps(chain, n_inst, procs):
    text = ops_netlist(5)
    n = 40
    track = sorted({0, n_inst // 2, n_inst - 1})
    b = sim.Batch(sim.Netlist(text, mode="lane_op", digest_capacity=n + 1, chain=chain, target_processes=procs), n_inst, seed=8,
                  track=track)
    b.hold_input(n_inst - 1, 4, 0x1234567)
    b.step(n)
    net = oracle.Net(text=text)
    for i in track:
        ref = oracle.Sim(net, seed=8, inst=i)
        if i == n_inst - 1:
            ref.hold_input(4, 0x1234567)
        assert np.array_equal(b.digests(i, 1, n), ref.run(n, digests=True)), i
        assert np.array_equal(b.regs(i), ref.regs()), i
