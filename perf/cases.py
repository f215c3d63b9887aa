"""The performance cases of the simulator: what its users have it do.

A program loads a design once (`sim.Netlist`), creates batches of instances
with their own stimulus seeds (`sim.Batch`) or a job server (`sim.Server`),
and then steps them and reads results.  A case is a design, a load
configuration, an instance count and the cycles of one pass; its inputs are
the stimulus seeds and, for some, held input values.

Every output is a whole number and has to be equal: registers, memory words
and state digests (a digest is the sum of a hash of every register and memory
word of an instance, so it differs if any of them does).  One-instance cases
return all their registers and memories, the checkpoint cases the whole saved
state; the 4,096-instance batch (360 MB of state) returns what `sim_step_host`
gives its callers, the digest of every instance.
"""
from __future__ import annotations

import functools
import math

import numpy as np

from paper_2403_04714_gb300 import netgen, sim

# Load configurations, as the benchmark and the autotuner use them.
CONFIGS = {
    # what sim.Netlist(text) gives: one instance on the grid barrier, or lane = instance bytecode from 32 on
    "default": dict(),
    "pairs": dict(mode="lane_op", chain=2),
    # one thread-block cluster, for designs of a few thousand operators
    "one_cluster": dict(mode="lane_op", chain=2, cluster_size=8, warps_per_cta=8, target_processes=64),
    # the autotuner's pick for one instance of the 200k-operator design
    "tuned": dict(mode="lane_op", chain=2, cluster_size=2, warps_per_cta=4, partitioner="hypergraph"),
    "clusters_of_4": dict(mode="lane_op", chain=2, cluster_size=4, warps_per_cta=4),
    "hypergraph": dict(partitioner="hypergraph"),
    "generated": dict(mode="lane_inst", lowering="generated"),
    # the autotuner's pick for the 4,096-instance batch, as the benchmark runs it
    "generated_graph": dict(mode="lane_inst", lowering="generated", warps_per_cta=6,
                            task_order="process_major", kernel="persistent_graph"),
    # every cycle its own kernel, replayed from a CUDA graph
    "graph": dict(kernel="graph"),
}


def listed():
    return [
        # a testbench that looks at the design every few cycles: launch and read-back latency
        dict(name="tiny_short_step", design="tiny", config="default", n_inst=1, cycles=8, reads="regs"),
        # a small design simulated for long, in its best configuration
        dict(name="tiny_one_cluster", design="tiny", config="one_cluster", n_inst=1, cycles=4000, reads="regs"),
        # a trace: the digest of every cycle, to find where two runs part
        dict(name="tiny_cycle_digests", design="tiny", config="default", n_inst=1, cycles=2000, reads="trace"),
        # a few instances with inputs from the host, too few for lane = instance
        dict(name="tiny_x8_held", design="tiny", config="default", n_inst=8, cycles=1000, reads="host"),
        # one instance of the 200k-operator design: as loaded by default, and tuned (the headline)
        dict(name="mid_default", design="mid", config="default", n_inst=1, cycles=1000, reads="regs"),
        dict(name="mid_tuned", design="mid", config="tuned", n_inst=1, cycles=2000, reads="regs"),
        # a 500k-operator mesh of cores with register files and RAMs, eight processes per SM
        dict(name="mesh_4x4", design="mesh_4x4", config="default", n_inst=1, cycles=1000, reads="regs"),
        # many instances without run-time compilation
        dict(name="mid_x100_bytecode", design="mid", config="default", n_inst=100, cycles=40, reads="digests"),
        # a regression of a small design: many seeds, an odd number of them, then a checkpoint
        dict(name="tiny_x1000_save", design="tiny", config="generated", n_inst=1000, cycles=1000, reads="save"),
        # the same of a larger one
        dict(name="mid_x250_save", design="mid", config="generated", n_inst=250, cycles=200, reads="save"),
        # the batched workload at full size
        dict(name="mid_x4096", design="mid", config="generated_graph", n_inst=4096, cycles=100, reads="host_free"),
        # a server's jobs of several designs and sizes at once
        dict(name="served", design="served", config="generated", n_inst=256, cycles=10000, jobs=10, trace=7),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    if u < 0.08:
        return dict(design="served", config="generated", n_inst=_log(rng, 32, 256), cycles=_log(rng, 2000, 10000),
                    jobs=rng.randint(3, 10), trace=rng.randrange(1000))
    if u < 0.55:    # one instance, or a few
        config = rng.choice(["default", "default", "pairs", "tuned", "clusters_of_4", "hypergraph", "graph"])
        n_inst = 1 if config in ("tuned", "clusters_of_4") else rng.choice([1, 1, 1, _log(rng, 2, 31)])
        design = rng.choice(["flat", "flat", "tiny", "mid", "mesh_small"])
        case = dict(design=design, config=config, n_inst=n_inst, cycles=_log(rng, 4, 2000) if n_inst == 1 else _log(rng, 4, 200),
                    reads=rng.choice(["regs", "host", "trace"]) if design != "mid" else "regs")
        if design == "flat":
            case.update(n_ops=_log(rng, 2000, 200_000), depth=rng.randint(16, 60))
        return case
    config = rng.choice(["default", "generated", "generated", "generated_graph"])
    design = rng.choice(["tiny", "mid", "mesh_small", "flat"])
    n_inst = _log(rng, 32, 4096)
    case = dict(design=design, config=config, n_inst=n_inst, reads="digests" if n_inst > 512 else rng.choice(["digests", "host", "save"]))
    ops = {"tiny": 2080, "mid": 207_743, "mesh_small": 124_654}.get(design)
    if design == "flat":
        case.update(n_ops=_log(rng, 2000, 20_000), depth=rng.randint(16, 60))
        ops = case["n_ops"]
    # at most the work of the 4,096-instance batch (the bytecode takes some twenty times longer for it)
    most = (3e9 if config == "default" else 8e10) / (ops * (n_inst + 256))
    case["cycles"] = max(2, min(_log(rng, 10, 1000), int(most)))
    return case


@functools.lru_cache(maxsize=None)
def _text(design, n_ops, depth):
    if design == "tiny":
        return netgen.gen_tiny().to_text()
    if design == "mid":
        return netgen.gen_mid().to_text()
    if design == "mesh_small":
        return netgen.gen_mesh_small().to_text()
    if design == "mesh_4x4":
        return netgen.gen_mesh(mesh=4, ops_per_block=30_000, regs_per_block=2_000).to_text()
    return netgen.gen_flat(n_ops, n_ops, max(48, n_ops // 12), depth, 8 + n_ops // 4000,
                           rams=((8, 32),) if n_ops >= 8000 else ()).to_text()


# A loaded design is kept for the life of a program; batches come and go.
@functools.lru_cache(maxsize=None)
def _netlist(design, config, n_ops, depth, ring):
    nl = sim.Netlist(_text(design, n_ops, depth), digest_capacity=ring, **CONFIGS[config])
    if CONFIGS[config].get("lowering") == "generated" and not ring:
        nl.compile_generated("lane_inst")
    return nl


def _design(case):
    ring = case["cycles"] + 1 if case.get("reads") == "trace" else 0
    return _netlist(case["design"], case["config"], case.get("n_ops", 0), case.get("depth", 0), ring)


def _jobs(case):
    """(design, instances, cycles) of each job of a server case."""
    trace = netgen.served_trace(n_jobs=case["jobs"], seed=case["trace"], inst_max=case["n_inst"],
                                cycles_lo=max(1, case["cycles"] // 10), cycles_hi=case["cycles"])
    return [(shape, n_inst, cyc) for _, shape, _, n_inst, cyc, _ in trace]


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["design"] == "served":
        jobs = [(_netlist(shape, case["config"], 0, 0, 0), n_inst, int(rng.integers(1 << 62)), cyc)
                for shape, n_inst, cyc in _jobs(case)]
        return dict(case=case, server=sim.Server(pool_slots=1024, chunk_cycles=1000), jobs=jobs)
    nl = _design(case)
    state = dict(case=case, batch=sim.Batch(nl, case["n_inst"], seed=int(rng.integers(1 << 62))))
    if case["reads"] == "host":
        state["held"] = rng.integers(0, 1 << 64, size=(case["n_inst"], nl.info()["n_inputs"]), dtype=np.uint64)
    if case["reads"] in ("host", "host_free"):
        state["digests"] = np.zeros(case["n_inst"], dtype=np.uint64)
    return state


def _memories(batch):
    return [batch.mem_all(0, m).view(np.int64) for m in range(batch.info["n_mems"])]


def run(state):
    case = state["case"]
    if "server" in state:
        server = state["server"]
        ids = [(server.submit(nl, n_inst, seed, cyc), n_inst) for nl, n_inst, seed, cyc in state["jobs"]]
        for job, _ in ids:
            server.wait(job)
        return [server.digests(job, n_inst).view(np.int64) for job, n_inst in ids]
    batch, n, reads = state["batch"], case["cycles"], case["reads"]
    if reads in ("host", "host_free"):      # inputs from the host, digests to the host, in one call
        return batch.step_host(n, state.get("held"), state["digests"]).view(np.int64).copy()
    batch.step(n)
    if reads == "save":
        return [np.frombuffer(batch.save(), dtype=np.uint8), batch.state_digests().view(np.int64)]
    if reads == "trace":
        at = batch.cycle
        return [batch.digests(0, at - n + 1, n).view(np.int64), batch.regs(0).view(np.int64)]
    if reads == "digests":
        return [batch.state_digests().view(np.int64), batch.regs(case["n_inst"] - 1).view(np.int64)]
    return [batch.regs(0).view(np.int64)] + _memories(batch)


def work(case):
    """Word operations of every simulated cycle; the state read and written once in each."""
    if case["design"] == "served":
        parts = [(_netlist(shape, case["config"], 0, 0, 0), n_inst * cyc) for shape, n_inst, cyc in _jobs(case)]
    else:
        parts = [(_design(case), case["n_inst"] * case["cycles"])]
    out = {"bytes": 0.0, "flops": 0.0}
    for nl, inst_cycles in parts:
        per_class = np.bincount(nl.table("reg_cls"), minlength=3)
        out["bytes"] += 2.0 * (per_class[0] / 8 + per_class[1] * 4 + per_class[2] * 8) * inst_cycles
        out["flops"] += float(nl.info()["n_ops"]) * inst_cycles
    return out


def exact(case, seed):
    """No output is a computed real number: all are compared for equality."""
    return None
