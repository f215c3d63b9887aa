"""The programs as the GPU runs them (CPU only): operators as instances of one
formula over a constant table, a step's pairs side by side, merged store steps,
kinds above the opcodes.  Checked by static rules, by running them in an emulator
of that form against the oracle, and operator by operator at the edges of their
widths and operands."""
import random

import numpy as np
import pytest

import oracle
from bytecode_emu import Emu, mask
from paper_2403_04714_gb300 import netgen, sim
from test_oracle_bruteforce import random_tiny_circuit

M64 = (1 << 64) - 1
D_NOP, D_CONST, D_MEMRD, D_ADD, D_SUB, D_MUL, D_AND, D_OR, D_XOR, D_SHL, D_SHR, D_EQ, D_LT = 0, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14
D_MUX, D_SLICE, D_CONCAT, D_STR, D_STX = 15, 16, 17, 18, 22
OPS = range(D_ADD, D_CONCAT + 1)
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


# The device form, written from the layout's description (kOpMark and the
# constants beside it), not from the kernel.
MARK, SLOT0 = 1 << 7, 1024
TABLE = [0, M64] + [1 << k for k in range(64)] + [v for v in range(3, 64) if v & (v - 1)]


def sign_bits(word, byte):
    return M64 if word >> (8 * byte + 7) & 1 else 0


def shift(v, n, left):
    return 0 if n >= 64 else (v << n) & M64 if left else v >> n


def run_op(o, value, first=None):
    """Result of one encoded operator (four words); value(offset) reads an
    operand, `first` is the lane's first result (second rows only)."""
    w0, bits = int(o[0]), int(o[3])
    assert first is not None or not bits & 0x3C, "chain bits in a first row"
    # (a chained operand's slot is loaded too, but what it holds is not used)
    a = first if bits & 1 << 2 else value(int(o[1]) & 0xFFFF)
    m = value(int(o[1]) >> 16)
    x = first if bits & 1 << 3 else value(int(o[2]) & 0xFFFF)
    d = first if bits & 1 << 4 else value(int(o[2]) >> 16)
    c = x if (d != 0) != bool(bits & 1 << 5) else m
    k_and, k_orc = sign_bits(bits, 1), sign_bits(bits, 2)
    f = (a & c if k_and else a ^ c) | c & k_orc
    n = d & 0xFFFFFFFF
    s = shift(a, n | bits & 1 << 6, False) | shift(a, n | bits & 1 << 7, True)
    compare = (bits & 1 if f == 0 else 0) | (w0 & 1 if a < x else 0)
    return ((a * m + f) & M64 | s) & shift(M64, bits >> 25, False) | compare


def device_program(nl, p):
    """Steps of process p: (flags and count word, instruction words [n, 4])."""
    off, size = int(nl.table("c_off")[p]), int(nl.table("c_size")[p])
    return split_program(nl.table("e_words")[off:off + size], int(nl.table("e_tab")[p]))


def split_program(prog, tab=None):
    ne, units = int(prog[0]) & 0xFFFF, int(prog[0]) >> 16
    assert tab is None or units == tab
    ins = prog[units * 4:].reshape(-1, 4)
    steps, at = [], 0
    for b, e in enumerate(int(v) for v in prog[1:1 + ne]):
        assert e & 0xFFFF == at, "instructions left out between steps"
        cnt = e >> 16 & 0xFF
        if e & CHAIN or not e & GENERIC:
            assert cnt <= 31
            cnt = (cnt + 1) * (2 if e & CHAIN else 1)
        else:
            assert 1 <= cnt <= (128 if e & (LEAF | STORE) else 32)
        steps.append((e, ins[at:at + cnt]))
        at += cnt
    assert at == len(ins) and not prog[1 + ne:units * 4].any()
    return steps


class DeviceEmu(Emu):
    """The emulator on the device form: registers, memories and mirrors as Emu has them."""

    def __init__(self, text, netlist, mode):
        super().__init__(text, netlist, mode)
        self.progs = [device_program(netlist, p) for p in range(len(netlist.table("c_off")))]

    def step(self, order):
        nxt, recs = [None] * len(self.regs), {}
        if self.cluster:
            self.cluster["nxt"] = [[None] * len(v) for v in self.cluster["cur"]]
        for p in order:
            self.proc = p
            slots = [None] * int(self.nslots[p])
            read = set()

            def value(off):
                assert off % 8 == 0
                if off < SLOT0:
                    return TABLE[off // 8]
                read.add(off)
                return slots[off // 8 - SLOT0 // 8]
            for e, ins in self.progs[p]:
                outs = []
                read.clear()
                if e & CHAIN:
                    for o1, o2 in zip(ins[::2], ins[1::2]):
                        assert o1[0] & MARK and o2[0] & MARK
                        r = run_op(o1, value)
                        outs += [(int(o1[0]) >> 16, r), (int(o2[0]) >> 16, run_op(o2, value, r))]
                elif not e & GENERIC:
                    assert all(o[0] & MARK for o in ins)
                    outs = [(int(o[0]) >> 16, run_op(o, value)) for o in ins]
                else:
                    for d in ins.copy().view(sim.DINS).reshape(-1):
                        assert int(d["op"]) < 32 and not (e & STORE and d["op"] not in (D_STR, D_STX))
                        v = self._exec(d, slots, nxt, recs)
                        if v is not None:
                            outs.append((SLOT0 + int(d["dst"]) * 8, v))
                written = [off for off, _ in outs if off]     # 0: the spare slot
                assert len(written) == len(set(written)) and not read & set(written)
                for off, v in outs:
                    if off:
                        assert off >= SLOT0 and off % 8 == 0
                        slots[off // 8 - SLOT0 // 8] = v
        assert all(v is not None for v in nxt)
        if self.cluster:
            assert all(x is not None for v in self.cluster["nxt"] for x in v)
            self.cluster["cur"] = self.cluster["nxt"]
        self.regs, self.pending = nxt, recs
        self.cycle += 1


def run_compare(text, cycles, cluster=None, **cfg):
    if cluster:
        cfg.update(cluster_size=cluster[0], warps_per_cta=cluster[1])
    emu = DeviceEmu(text, sim.Netlist(text, mode="lane_op", **cfg), "lane_op_cluster" if cluster else "lane_op_compact")
    ref = oracle.Sim(oracle.Net(text=text), seed=42, inst=0)
    rng = random.Random(1)
    order = list(range(len(emu.progs)))
    for t in range(cycles):
        rng.shuffle(order)
        emu.step(order)
        ref.run(1)
        assert emu.regs == [int(v) for v in ref.regs()], t
    emu.finish()
    for m in range(len(emu.mems)):
        assert emu.mems[m] == [ref.mem(m, a) for a in range(len(emu.mems[m]))]


@pytest.mark.parametrize("chain", [0, 2])
@pytest.mark.parametrize("seed", range(6))
def test_random_circuits(seed, chain):
    text = random_tiny_circuit(seed).to_text()
    for target in (1, 2, 4):
        run_compare(text, 20, target_processes=target, chain=chain)
    for C, W, target in ((2, 1, 2), (4, 1, 4), (2, 2, 3)):
        run_compare(text, 15, cluster=(C, W), target_processes=target, chain=chain)


@pytest.mark.parametrize("chain", [0, 2])
def test_workload_and_memories(chain):
    run_compare(open(netgen.cached_netlist("tiny")).read(), 10, chain=chain)
    run_compare(open(netgen.cached_netlist("tiny")).read(), 10, cluster=(4, 2), target_processes=16, chain=chain)
    text = netgen.gen_flat(7, n_ops=3000, n_regs=200, depth=15, n_inputs=6, rams=((4, 64), (3, 16))).to_text()
    run_compare(text, 10, target_processes=16, chain=chain)
    run_compare(text, 10, cluster=(4, 2), target_processes=16, chain=chain)


def plain(op, w, a, b, c, x):
    v = {D_ADD: a + b, D_SUB: a - b, D_MUL: a * b, D_AND: a & b, D_OR: a | b, D_XOR: a ^ b, D_SHL: shift(a, b, True),
         D_SHR: shift(a, b, False), D_EQ: int(a == b), D_LT: int(a < b), D_MUX: b if a else c, D_SLICE: shift(a, x, False),
         D_CONCAT: (a << x) | b}[op]
    return v & mask(w)


def encode(steps):
    """Encoded operators of the steps between constants and a store."""
    full = [CONSTS, *steps, STORES]
    return [ins for _, ins in split_program(sim.debug_encode(program(full)))[1:-1]]


VALUES = (0, 1, 2, 31, 32, 63, 64, 65, (1 << 31) - 1, 1 << 31, (1 << 32) - 1, 1 << 32, (1 << 63) + 5, M64 - 1, M64)


@pytest.mark.parametrize("op", OPS)
def test_operators_at_their_edges(op):
    rng = random.Random(op)
    for w in (1, 2, 31, 32, 33, 63, 64) if op not in (D_EQ, D_LT) else (1,):
        for x in (range(64) if w == 64 and op in (D_SLICE, D_CONCAT) else (0, 7, 63)):
            (o,) = encode([(0, [ins(op, 9, 4, 5, 6, w=w, x=x if op in (D_SLICE, D_CONCAT) else 0)])])[0]
            assert int(o[0]) >> 16 == SLOT0 + 9 * 8
            for a in VALUES:
                for b in VALUES:
                    if op in (D_SHL, D_SHR) and b >> 32:
                        continue                # amounts of more than 32 bits run in generic steps
                    if op == D_CONCAT:
                        b &= mask(x)            # the lower part's width is the shift
                    c = rng.choice(VALUES)
                    vals = {SLOT0 + 32: a, SLOT0 + 40: b, SLOT0 + 48: c}
                    got = run_op(o, lambda f: TABLE[f // 8] if f < SLOT0 else vals[f])
                    assert got == plain(op, w, a, b, c, x if op in (D_SLICE, D_CONCAT) else 0), (w, x, a, b, c)


@pytest.mark.parametrize("op", OPS)
def test_pairs_in_every_position(op):
    # which of the operands a, b, c are the first result, as pair_fits admits them
    masks = [0, 1] if op == D_SLICE else [0, 1, 2] if op == D_MUL else [0, 1, 2, 4, 3, 5] if op == D_MUX else [0, 1, 2, 3]
    w = 1 if op in (D_EQ, D_LT) else 37
    x = 5 if op in (D_SLICE, D_CONCAT) else 0
    for flags in masks:
        # three lanes: this operator second, nothing second, a second operator alone
        rows = [ins(D_ADD, 9, 4, 5, w=32)] * 3 + [ins(op, 10, 9 if flags & 1 else 6, 9 if flags & 2 else 7, 9 if flags & 4 else 8,
                                                     imm=flags, w=w, x=x), ins(D_NOP, w=64), ins(D_XOR, 11, 6, 7, w=64)]
        got = encode([(GENERIC | CHAIN | 2 << 24, rows)])[0]
        assert len(got) == 6 and int(got[3][0]) >> 16 == 0, "an empty second row writes the spare slot"
        for va, vb, vc in ((0, 0, 0), (5, 40, 9), (M64, 31, M64), (1 << 33, 1 << 20, 0)):
            if op == D_CONCAT and not flags & 2:
                vb &= 31
            for first in (0, 1, 31, 32, (1 << 32) - 1):
                if op == D_CONCAT and flags & 2:
                    first &= 31
                vals = {SLOT0 + 48: va, SLOT0 + 56: vb, SLOT0 + 64: vc}      # not the first result's slot
                value = lambda f: TABLE[f // 8] if f < SLOT0 else vals[f]
                a, b, c = (first if flags >> k & 1 else v for k, v in enumerate((va, vb, vc)))
                assert run_op(got[1], value, first) == plain(op, w, a, b, c, x), (flags, a, b, c)
                assert run_op(got[5], value, first) == va ^ vb


@pytest.mark.parametrize("chain", [0, 2])
def test_kinds_of_the_instructions(chain):
    text = netgen.gen_flat(7, n_ops=3000, n_regs=200, depth=15, n_inputs=6, rams=((4, 64), (3, 16))).to_text()
    nl = sim.Netlist(text, target_processes=16, chain=chain)
    k, b = nl.table("k_ins"), nl.table("b_ins")
    kinds = {1: 1, D_CONST: 2, D_STR: 3, D_ADD: 4, D_SUB: 4, D_MUL: 4, D_EQ: 5, D_LT: 5, D_MUX: 5, D_SHL: 6, D_SHR: 6, D_SLICE: 6,
             D_CONCAT: 6, D_AND: 7, D_OR: 7, D_XOR: 7}
    assert [int(v) for v in k["op"]] == [int(v) | kinds.get(int(v), 0) << 5 for v in b["op"]]
    for field in ("w", "dst", "a", "b", "c", "x", "imm"):
        assert np.array_equal(k[field], b[field])
    assert {int(v) for v in b["op"]} >= set(OPS), "every operator occurs"


@pytest.mark.parametrize("sizes,merged", [((32, 32, 32, 32, 32), (128, 32)), ((100, 29), (100, 29)), ((100, 28, 1), (128, 1)),
                                          ((1, 1, 1), (3,))])
def test_store_steps_are_merged_up_to_their_width(sizes, merged):
    steps = [CONSTS, (0, SUM)] + [(GENERIC | (STORE if n > 32 else 0), [ins(D_STX if k else D_STR, a=3, imm=k)] * n)
                                  for k, n in enumerate(sizes)]
    got = split_program(sim.debug_encode(program(steps)))[2:]
    assert tuple(len(i) for _, i in got) == merged and all(e & STORE and e & GENERIC for e, _ in got)
    assert [int(d["imm"]) for _, i in got for d in i.copy().view(sim.DINS).reshape(-1)] == [k for k, n in enumerate(sizes) for _ in range(n)]
