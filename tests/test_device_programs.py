"""The per-operation programs as the GPU runs them (CPU only)."""
import numpy as np
import pytest

from paper_2403_04714_gb300 import sim

D_CONST, D_MEMRD, D_ADD, D_MUX, D_STR, D_STX = 3, 4, 5, 15, 18, 22
GENERIC, LEAF, CHAIN, STORE = 1 << 31, 1 << 30, 1 << 29, 1 << 28


def program(steps):
    """Words of a compact program: steps of (flags, instructions)."""
    words, ins = [len(steps)], []
    for flags, step in steps:
        words.append(len(ins) | len(step) << 16 | flags)
        ins += step
    words += [0] * (-len(words) % 4)
    return np.concatenate([np.array(words, dtype=np.uint32), np.array(ins, dtype=sim.DINS).view(np.uint32)])


def ins(op, dst=0, a=0, b=0, c=0, imm=0, w=0, x=0):
    return (op, w, dst, a, b, c, x, imm)


CONSTS = (GENERIC | LEAF, [ins(D_CONST, k, imm=k) for k in range(3)])
SUM = [ins(D_ADD, 3, 0, 1)]
STORES = (GENERIC, [ins(D_STR, a=3)])


@pytest.mark.parametrize("why,steps", [
    ("operators in its last step", [CONSTS, (0, SUM)]),
    ("operators in its last step", [CONSTS, (GENERIC | CHAIN | 2 << 24, SUM * 2)]),
    ("an empty step", [CONSTS, (0, []), STORES]),
    ("an empty step", [CONSTS, (GENERIC | CHAIN | 2 << 24, []), STORES]),
    ("an empty step", [CONSTS, (0, SUM), (GENERIC, [])]),
    ("a step too wide", [CONSTS, (0, SUM * 33), STORES]),
    ("a step too wide", [CONSTS, (GENERIC | CHAIN | 2 << 24, SUM * 3), STORES]),
    ("a step too wide", [CONSTS, (GENERIC | CHAIN | 2 << 24, SUM * 66), STORES]),
    ("a step too wide", [CONSTS, (0, SUM), (GENERIC | STORE, STORES[1] * 129)]),
])
def test_programs_the_interpreter_could_not_end_are_refused(why, steps):
    with pytest.raises(sim.SimError) as e:
        sim.debug_encode(program(steps))
    assert e.value.name == "SIM_ERR_STATE" and why in str(e.value)


def test_malformed_step_tables_are_refused():
    good = program([CONSTS, (0, SUM), STORES])
    sim.debug_encode(good)
    for cut in (0, 1, 4, len(good) - 4):
        with pytest.raises(sim.SimError):
            sim.debug_encode(good[:cut])
    gap = good.copy()
    gap[2] += 1                      # the second step starts one instruction late
    with pytest.raises(sim.SimError) as e:
        sim.debug_encode(gap)
    assert "out of order" in str(e.value)


def test_the_widest_steps_are_taken():
    sim.debug_encode(program([(GENERIC | LEAF, CONSTS[1] * 42), (0, SUM * 32), (GENERIC | CHAIN | 2 << 24, SUM * 64),
                              (GENERIC | STORE, STORES[1] * 128)]))
