"""Performance cases of the mapping search: what its users have it do, through the public entry points.

A case names the entry point, the problem (dimensions of the chain C = A(I x K) B(K x L), E = C D(L x J), the
accelerator, the search options) and nothing else.  The seed stands for the accelerator a user happens to have: it
moves the energy of every access, the DRAM rate and the share of the buffer that the mapping may use a little around
the named accelerator's, so that two seeds are two different searches of the same size.

  search       a planned search (mmee_create in advance) into device records: mmee_search
  solve        the one-shot call with host records, planning included: mmee_solve_host
  shapes       one energy-delay search per logical array shape: mmee_search_shapes
  front        the energy-latency Pareto front of a mapping space: mmee_pareto_front
  front_bs_da  the buffer-size / DRAM-traffic Pareto front: mmee_pareto_front_bs_da
"""
import math
import random

import numpy as np
import torch

import mmee_inputs as mi
import paper_2604_03446_b200 as mm

ARCHS = {"tiny": mi.arch_tiny, "edge": mi.arch_edge, "cloud": mi.arch_cloud, "accel1": mi.arch_accel1}
FRONT_CAPACITY = 4096


def _case(name, call, arch, seq_q, seq_kv, d_qk, d_v, groups=1, objective=mi.OBJ_ENERGY, topk=1,
          tiling_set=mi.TILE_ALL_DIVISORS, order_set=mi.ORD_ALL6, fuse_mask=mi.FUSE_ALL, row_pruning=0, rf_tiling=0,
          shapes=0, buffer_kb=0):
    case = dict(call=call, arch=arch, seq_q=seq_q, seq_kv=seq_kv, d_qk=d_qk, d_v=d_v, groups=groups,
                objective=objective, topk=topk, tiling_set=tiling_set, order_set=order_set, fuse_mask=fuse_mask,
                row_pruning=row_pruning, rf_tiling=rf_tiling, shapes=shapes, buffer_kb=buffer_kb)
    return dict(case, name=name) if name else case


def listed():
    return [
        # A design-space loop around very small kernels: ragged dimensions, one host call per point, where the
        # launches and the host's own work are what counts.
        _case("tiny_ragged_solve_edp", "solve", "tiny", 24, 20, 8, 6, objective=mi.OBJ_EDP, topk=3),
        # The smallest benchmark configuration: power-of-two tilings, two loop orders, fused or fully unfused.
        _case("tiny_s64_d64_energy", "search", "tiny", 64, 64, 64, 64, tiling_set=mi.TILE_POW2,
              order_set=mi.ORD_NORECOMP2, fuse_mask=mi.FUSE_FUSED | mi.FUSE_SEPARATE),
        # BERT-base attention on the edge accelerator: the ordinary search, on a plan that is kept.
        _case("bert_base_s512_energy", "search", "edge", 512, 512, 64, 64),
        # The same chain with the third tiling level (register files), latency-driven.
        _case("bert_base_s512_latency_rf", "search", "edge", 512, 512, 64, 64, objective=mi.OBJ_LATENCY, rf_tiling=1),
        # Llama-style prefill on the cloud accelerator: the sixteen best mappings, one-shot with host records.
        _case("llama_prefill_s4096_latency_top16", "solve", "cloud", 4096, 4096, 128, 128, objective=mi.OBJ_LATENCY,
              topk=16),
        # Grouped-query attention (four query heads stacked on a K/V head): the default benchmark's two searches, the
        # first on a kept plan, the second as one call.
        _case("gqa_s8192_latency", "search", "cloud", 8192, 8192, 128, 128, groups=4, objective=mi.OBJ_LATENCY),
        _case("gqa_s8192_edp_solve", "solve", "cloud", 8192, 8192, 128, 128, groups=4, objective=mi.OBJ_EDP),
        # Longest sequence of the sweep, with the offline row pruning that long sweeps use.
        _case("sweep_s65536_energy_pruned", "search", "edge", 65536, 65536, 128, 128, row_pruning=1),
        # A convolution chain beyond attention: ragged divisor lists, the most tilings of all, sixteen best mappings.
        _case("conv_chain_cc1_energy_top16", "search", "accel1", 12544, 192, 576, 128, topk=16,
              fuse_mask=mi.FUSE_FUSED),
        # A reconfigurable array: every power-of-two shape with 1024 PEs, energy-delay product.
        _case("reconfig_11_shapes_edp", "shapes", "accel1", 512, 512, 64, 64, objective=mi.OBJ_EDP,
              fuse_mask=mi.FUSE_FUSED, shapes=11),
        # The energy-latency trade-off of a 4096-token head on the edge accelerator.
        _case("front_s4096_d128", "front", "edge", 4096, 4096, 128, 128),
        # The DRAM-traffic-against-buffer-size study of a large feed-forward block.
        _case("ffn_dram_front", "front_bs_da", "accel1", 32768, 16384, 4096, 4096, fuse_mask=mi.FUSE_FUSED,
              buffer_kb=1024),
    ]


def _divisors(n, pow2):
    ds = [d for d in range(1, math.isqrt(n) + 1) if n % d == 0]
    ds = sorted(set(ds + [n // d for d in ds]))
    return sum(1 for d in ds if not pow2 or d & (d - 1) == 0)


def _rows(case):
    """Tilings times rows (fusion mode, loop order, buffering levels; nine mappings each) of the case's space, and the
    longest divisor list."""
    pow2 = case["tiling_set"] == mi.TILE_POW2
    n = [_divisors(d, pow2) for d in (case["groups"] * case["seq_q"], case["d_qk"], case["seq_kv"], case["d_v"])]
    orders = 2 if case["order_set"] == mi.ORD_NORECOMP2 else 6
    unfused = bin(case["fuse_mask"] >> 1).count("1")
    return math.prod(n) * orders * ((case["fuse_mask"] & 1) * 3125 + unfused * 625), max(n)


def _length(rng, lo, hi):
    """A length between lo and hi, even over the logarithm: a power of two, a multiple of 8 or 96, or any number."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    kind = rng.randrange(4)
    if kind == 0:
        return min(hi, max(lo, 1 << round(math.log2(n))))
    step = (8, 96, 1)[kind - 1]
    return min(hi, max(lo, round(n / step) * step))


def draw(rng):
    """One more case of the same ranges; spaces larger than the listed cases of the same call are drawn again."""
    most = {"search": 1.2e9, "solve": 4e8, "shapes": 1e8, "front": 4e7, "front_bs_da": 3e8}
    while True:
        call = rng.choice(("search", "search", "search", "solve", "solve", "shapes", "front", "front_bs_da"))
        arch = rng.choice(("tiny", "edge", "edge", "cloud", "cloud", "accel1"))
        groups = rng.choice((1, 1, 1, 2, 4, 8))
        seq_q = _length(rng, 16, 65536 // groups)
        seq_kv = seq_q if rng.random() < 0.6 else _length(rng, 16, 65536)
        d_qk = rng.choice((8, 24, 32, 40, 64, 64, 72, 80, 96, 128, 128, 192, 256))
        d_v = d_qk if rng.random() < 0.7 else rng.choice((6, 16, 32, 64, 80, 96, 128))
        objective = rng.choice((mi.OBJ_ENERGY, mi.OBJ_LATENCY, mi.OBJ_EDP))
        topk = rng.choice((1, 1, 3, 16))
        case = _case("", call, arch, seq_q, seq_kv, d_qk, d_v, groups, objective, topk,
                     tiling_set=rng.choice((mi.TILE_ALL_DIVISORS,) * 3 + (mi.TILE_POW2,)),
                     order_set=rng.choice((mi.ORD_ALL6,) * 3 + (mi.ORD_NORECOMP2,)),
                     fuse_mask=rng.choice((mi.FUSE_ALL, mi.FUSE_ALL, mi.FUSE_FUSED, mi.FUSE_FUSED | mi.FUSE_SEPARATE)),
                     row_pruning=int(call == "search" and topk == 1 and rng.random() < 0.3),
                     rf_tiling=int(call in ("search", "solve") and objective != mi.OBJ_EDP and arch != "tiny"
                                   and rng.random() < 0.2),
                     buffer_kb=rng.choice((0, 0, 64, 192, 1024)))
        if call == "shapes":
            case.update(objective=rng.choice((mi.OBJ_ENERGY, mi.OBJ_EDP)), topk=1, shapes=rng.randrange(1, 12))
        if call in ("front", "front_bs_da"):
            case.update(objective=mi.OBJ_ENERGY, topk=1)
        rows, longest = _rows(case)
        if 1e5 <= rows <= most[call] and longest <= 64 and groups * seq_q * seq_kv <= 1 << 32:
            return case


def _inputs(case, seed):
    """(workload, accelerator, search options) of one seed."""
    rng = random.Random(seed)
    arch = ARCHS[case["arch"]]()
    q = arch["energy_quantum_pj"]
    for name in ("e_dram_pj", "e_gb_pj", "e_rf_pj", "e_mac_pj"):
        if arch[name]:
            arch[name] = q * max(1, round(arch[name] / q * rng.uniform(0.8, 1.25)))
    arch["dram_words_per_cycle"] = max(1, round(arch["dram_words_per_cycle"] * rng.uniform(0.8, 1.2)))
    if case["buffer_kb"]:
        arch["gb_bytes"] = case["buffer_kb"] * mi.KiB
    arch["gb_bytes"] = arch["gb_bytes"] * rng.randrange(960, 1025) // 1024 // 2 * 2
    work = mi.workload(1, case["groups"], 1, case["seq_q"], case["seq_kv"], case["d_qk"], case["d_v"])
    opts = mi.objective(case["objective"], case["topk"], case["tiling_set"], case["order_set"], case["fuse_mask"],
                        row_pruning=case["row_pruning"], rf_tiling=case["rf_tiling"])
    return work, arch, opts


class _Plan:
    """A planned search with its device records; the plan is released with the object."""

    def __init__(self, inputs):
        self.handle = mm.mmee_create(*inputs)
        self.best = mm.result_buffer(1)
        self.topk = mm.result_buffer(inputs[2]["topk"])

    def __del__(self):
        mm.mmee_destroy(self.handle)


def prepare(case, seed):
    inputs = _inputs(case, seed)
    state = {"call": case["call"], "inputs": inputs}
    if case["call"] == "search":
        state["plan"] = _Plan(inputs)
    elif case["call"] == "shapes":
        # shapes with the same number of PEs, the squarest first
        a = inputs[1]
        pes = a["pe_rows"] * a["pe_cols"]
        every = [(1 << i, pes >> i) for i in range(pes.bit_length())]
        every.sort(key=lambda rc: (abs(math.log2(rc[0]) - math.log2(rc[1])), rc))
        state["shapes"] = every[:case["shapes"]]
    return state


def _raw(records):
    """Result records as bytes in one array."""
    return np.frombuffer(b"".join(bytes(r) for r in records), dtype=np.uint8)


def run(state):
    call = state["call"]
    if call == "search":
        plan = state["plan"]
        mm.mmee_search(plan.handle, plan.best, plan.topk)
        return {"best": plan.best, "topk": plan.topk}
    work, arch, opts = state["inputs"]
    if call == "solve":
        best, topk, _, _ = mm.mmee_solve_host(work, arch, opts)
        return {"best": _raw([best]), "topk": _raw(topk)}
    if call == "shapes":
        per_shape, best = mm.mmee_search_shapes(work, arch, opts, state["shapes"])
        return {"per_shape": _raw(per_shape), "best": -1 if best is None else best}
    if call == "front":
        return {"points": _raw(mm.mmee_pareto_front(work, arch, opts, FRONT_CAPACITY))}
    return {"points": _raw(mm.mmee_pareto_front_bs_da(work, arch, opts, FRONT_CAPACITY))}


def work(case):
    """A search has to decide every row of its space (the two buffer needs against the capacity, the DRAM words against
    the best so far: five operations with the sums) and to write its records; a front is at least one such pass, a set
    of shapes one pass each."""
    rows, _ = _rows(case)
    passes = max(1, case["shapes"])
    records = case["topk"] + 1 if case["call"] in ("search", "solve") else passes
    return {"bytes": 336 * records, "flops": 5 * rows * passes}


def tolerance(case):
    """Counts, indices and keys are whole numbers, and the floating-point fields are single correctly rounded products
    of them: records are compared byte for byte."""
    return "exact"
