"""The kernels' arithmetic that the host can run as well, compiled for the CPU and checked there: no GPU is used."""
import ctypes as C
import multiprocessing
import os
import subprocess

import numpy as np
import pytest

import mmee_inputs as mi
import oracle
import paper_2604_03446_b200.binding as mm
from paper_2604_03446_b200 import build as lib_build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="session")
def host(tmp_path_factory):
    """host_math.cu and the planner as a shared object."""
    out = str(tmp_path_factory.mktemp("host_math") / "host_math.so")
    flags = [f for f in lib_build.NVCC_FLAGS if f not in ("-lineinfo", "-O3")]
    subprocess.check_call([lib_build._nvcc()] + flags + ["-O1", "-o", out, os.path.join(HERE, "host_math.cu")] +
                          [os.path.join(lib_build.CSRC, f) for f in ("mmee_plan.cu", "mmee_prune.cu")])
    lib = C.CDLL(out)
    lib.path = out
    return lib


def tile_terms(lib, dims, pe, tile, op, sm, objective=mi.OBJ_ENERGY, rf_words=0):
    """(words, cycles, block) of one tile with extents (i, k, l, j)."""
    w = mm._fill(mm.Workload(), mi.workload(1, 1, 1, dims[0], dims[2], dims[1], dims[3], 2))
    a = mm._fill(mm.Arch(), dict(mi.arch(pe[0], pe[1], 1, 1 << 20, 2 * rf_words, 1, 1.0, 1.0, 1.0, 1.0)))
    o = mm._fill(mm.Objective(), mi.objective(objective, 1, rf_tiling=1 if rf_words else 0))
    b = (C.c_uint32 * 8)(*([d // t for d, t in zip(dims, tile)] + list(tile)))
    out, blk = (C.c_int64 * 2)(), (C.c_uint32 * 3)()
    assert lib.host_tile_terms(C.byref(w), C.byref(a), C.byref(o), b, op, sm, out, blk) == mm.OK
    return out[0], out[1], list(blk)


def _tile_terms_at(path, *args):
    return tile_terms(C.CDLL(path), *args)


def ceil_div(a, b):
    return -(-a // b)


def divisors(n):
    ds = [d for d in range(1, int(n ** 0.5) + 2) if n % d == 0 and d * d <= n]
    return sorted(set(ds + [n // d for d in ds]))


def expected_terms(pe, tile, op, sm, objective, rf_words):
    """The definition, in Python integers: the stationary operand's extents cut into parts of the array (or, with a
    register file, of the best admissible block), operands and partial sums moved once per part."""
    m, r, n = (tile[0], tile[1], tile[2]) if op == 0 else (tile[0], tile[2], tile[3])
    ea, eb = {0: (r, n), 1: (m, r), 2: (m, n)}[sm]

    def terms(qa, qb, held):
        words = {0: r * n + m * r * qb + m * n * (2 * qa - 1), 1: m * r + r * n * qa + m * n * (2 * qb - 1),
                 2: m * r * qb + r * n * qa + m * n}[sm]
        return words, {0: m, 1: n, 2: r}[sm] * qa * qb * held

    if not rf_words:
        return terms(ceil_div(ea, pe[0]), ceil_div(eb, pe[1]), 1) + ([0, 0, 0],)
    best = None
    for a in divisors(ea):
        for b in divisors(eb):
            held = ceil_div(a, pe[0]) * ceil_div(b, pe[1])
            if held + 2 > rf_words:
                continue
            w, c = terms(ea // a, eb // b, held)
            key = (w, c) if objective == mi.OBJ_ENERGY else (c, w)
            if best is None or key < best[0]:
                best = (key, w, c, [1, a, b] if sm == 0 else ([a, b, 1] if sm == 1 else [a, 1, b]))
    return best[1:]


HUGE = 2 ** 32 - 1


@pytest.mark.parametrize("dims,pe,rf_words", [
    ((2, 4294967294, 3, 4), (4, 7), 0),              # extents within one fold of 2^32
    ((4294967294, 2, 3, 4), (2147483648, 5), 0),
    ((48, 30, 20, 6), (HUGE, HUGE - 7), 0),          # arrays that hold any tile
    ((2, 4294967294, 3, 4), (4, 7), 12),
    ((4294967294, 2, 3, 4), (65536, 65536), 70000),
    ((48, 30, 20, 6), (HUGE, HUGE - 7), 6),
], ids=["k", "i", "array", "k_rf", "i_rf", "array_rf"])
def test_folds_near_the_32_bit_limit(host, dims, pe, rf_words):
    """ceil(extent / rows) where extent + rows - 1 exceeds 32 bits."""
    for op in (0, 1):
        for sm in (0, 1, 2):
            for objective in (mi.OBJ_ENERGY, mi.OBJ_LATENCY):
                want = expected_terms(pe, dims, op, sm, objective, rf_words)
                assert tile_terms(host, dims, pe, dims, op, sm, objective, rf_words) == want, (op, sm, objective)


@pytest.mark.parametrize("dims,pe,rf_words", [
    ((HUGE, 3, 5, 1), (65536, 65536), 2 ** 31 - 1),      # every divisor of 2^32 - 1 is admissible
    ((3, HUGE, 1, 1), (2, 3), 2 ** 32 - 1),
    ((HUGE, 1, 3, 2), (HUGE, 1), 7),
])
def test_register_file_walk_ends_at_an_extent_of_all_ones(host, dims, pe, rf_words):
    """The walk over the two divisor lists, with an extent equal to its mark for "no divisor left"; in a process of its own
    with a time limit, since a walk that mistakes one for the other does not end."""
    pool = multiprocessing.get_context("spawn").Pool(1)
    try:
        for op in (0, 1):
            for sm in (0, 1, 2):
                for objective in (mi.OBJ_ENERGY, mi.OBJ_LATENCY):
                    args = (dims, pe, dims, op, sm, objective, rf_words)
                    got = pool.apply_async(_tile_terms_at, (host.path,) + args).get(timeout=60)
                    assert got == expected_terms(pe, dims, op, sm, objective, rf_words), args
    finally:
        pool.terminate()


NO_ROW = 2 ** 62


@pytest.mark.parametrize("dims", [(12, 4, 20, 6), (30, 12, 8, 18), (7, 5, 1, 3), (16, 16, 16, 16)])
@pytest.mark.parametrize("order_set", [mi.ORD_ALL6, mi.ORD_NORECOMP2])
def test_classes_of_levels_against_the_rows_of_the_oracle(host, dims, order_set):
    """The search's closed forms -- how many rows of a block fit, the least DRAM words of one that does, the least buffer
    need at those words, with and without row pruning -- against every row of the block as the oracle evaluates it, for
    tilings all over the space and capacities from one at which nothing fits to one at which everything does."""
    w = mi.workload(1, 1, 1, dims[0], dims[2], dims[1], dims[3], 1)
    base = mi.objective(mi.OBJ_ENERGY, 1, order_set=order_set, fuse_mask=mi.FUSE_FUSED | mi.FUSE_SOFTMAX_IN_OP1, row_pruning=1)
    arch = mi.arch(2, 3, 1, 1 << 20, 0, 1, 1.0, 0.0, 0.0, 0.0)
    p = oracle.make_problem(w, arch, base)
    keep = np.array(mm.mmee_row_pruning_keep(base), dtype=bool)
    rng = np.random.default_rng(sum(dims))
    n_orders = p.n_orders
    for t in sorted({0, p.T - 1} | set(int(v) for v in rng.integers(0, p.T, size=6))):
        raw = np.frombuffer(oracle.evaluate_range(p, t * p.R * 9, p.R * 9), dtype=np.dtype(oracle.Record))[::9]
        words, need, lc, da1, da2 = (np.ascontiguousarray(v, dtype=np.int64) for v in
                                     (raw["n"][:, 0], raw["bs"], raw["beta"][:, 2] - 3, raw["da1"], raw["da2"]))
        split = n_orders * 3125
        caps = np.unique(np.concatenate([[need.min() - 1, need.max()], rng.choice(need, size=4)]))
        for cap in (int(v) for v in caps if v > 0):
            fits = need <= cap
            for slot in range(n_orders):
                out = ((C.c_int64 * 8) * 4)()
                args = [C.byref(mm._fill(s(), d)) for s, d in ((mm.Workload, w), (mm.Arch, dict(arch, gb_bytes=cap)), (mm.Objective, base))]
                assert host.host_classes(*args, C.c_uint32(t), slot, out) == mm.OK
                for c in range(3):
                    first, width, rows, x, least_need, rows2, x2, kept = out[c]
                    here = np.zeros(p.R, dtype=bool)
                    here[slot * 3125:(slot + 1) * 3125] = True
                    here &= fits & (lc >= first) & (lc < first + width)
                    assert rows == rows2 == here.sum() and kept == (here & keep).sum()
                    want = words[here].min() if here.any() else NO_ROW
                    assert x == x2 == want
                    if here.any():
                        assert least_need == need[here & (words == want)].min()
                _, _, rows, x1, least_need, rows2, x2, kept = out[3]
                here = np.zeros(p.R, dtype=bool)
                here[split + slot * 625:split + (slot + 1) * 625] = True
                here &= fits
                assert rows == rows2 == here.sum() and kept == (here & keep).sum()
                if here.any():
                    assert (x1, x2) == (da1[here].min(), da2[here].min())
                    assert least_need == need[here & (da1 == x1) & (da2 == x2)].min()
                else:
                    assert x1 == NO_ROW
