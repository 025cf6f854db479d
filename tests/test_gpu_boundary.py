"""GPU tests of the C-ABI boundary's helpers: decoding one index, launch counters, device checks."""
import ctypes as C
import os

import numpy as np
import pytest
import torch

import mmee_inputs as mi
import oracle
import paper_2604_03446_b200.binding as mm
from test_gpu_parity import Handle, assert_same_record

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [1, 4, 9])
def test_decode_returns_the_mapping_and_its_evaluation(seed):
    """mmee_decode against the oracle's evaluation of the same index: sampled indices of the whole space,
    its first and its last index; an index outside the space is an argument error."""
    cfg = mi.random_tiny_problem(seed)
    obj = cfg["searches"][0]
    p = oracle.make_problem(cfg["workload"], cfg["arch"], obj)
    rng = np.random.default_rng(seed)
    picks = [0, p.N - 1] + [int(i) for i in rng.integers(0, p.N, size=40)]
    with Handle(cfg, obj) as h:
        assert mm.mmee_num_candidates(h) == p.N
        for idx in picks:
            got = mm.mmee_decode(h, idx)
            want = oracle.evaluate(p, idx)
            assert_same_record(got, want, "idx %d" % idx)
            assert got.status == mm.OK
        assert mm.library().mmee_decode(h, p.N, C.byref(mm.Result())) == mm.ERR_ARG
        assert mm.library().mmee_decode(h, 0, None) == mm.ERR_ARG


def test_decode_at_full_size():
    cfg = mi.config4()
    obj = cfg["searches"][1]
    p = oracle.make_problem(cfg["workload"], cfg["arch"], obj)
    with Handle(cfg, obj) as h:
        for idx in (0, p.N // 3 + 7, p.N - 1):
            assert_same_record(mm.mmee_decode(h, idx), oracle.evaluate(p, idx), "idx %d" % idx)


def test_search_with_host_records_equals_the_device_path():
    cfg = mi.random_tiny_problem(3)
    obj = dict(cfg["searches"][0], topk=5)
    want = oracle.search(oracle.make_problem(cfg["workload"], cfg["arch"], obj))
    with Handle(cfg, obj) as h:
        for _ in range(2):
            best, topk = mm.mmee_search_host(h, True, 5)
            assert [r.idx for r in topk if r.idx != mm.NO_INDEX] == [r.idx for r in want.topk]
            assert best.n_feasible == want.n_feasible and best.n_total == want.n_total
            if want.topk:
                assert_same_record(best, want.topk[0])
        best_only, none = mm.mmee_search_host(h)
        assert none is None and bytes(best_only) == bytes(best)


def test_launch_counters_of_a_search():
    """Create time, launches, persistent CTAs and the number of groups that went to the exact path are reported;
    a search cannot find an optimum without at least one visit of the exact path."""
    cfg = mi.config1()
    obj = cfg["searches"][0]
    best = mm.result_buffer(1)
    with Handle(cfg, obj) as h:
        assert mm.mmee_last_search_stats(h).exact_path_visits == 0
        mm.mmee_search(h, best)
        torch.cuda.synchronize()
        st = mm.mmee_last_search_stats(h)
        assert st.kernels_launched == 1 and st.grid >= 1 and st.block == 256
        assert st.create_ms > 0.0
        assert 1 <= st.exact_path_visits <= st.tasks * 25
        first = st.exact_path_visits
        mm.mmee_search(h, best)
        torch.cuda.synchronize()
        assert mm.mmee_last_search_stats(h).exact_path_visits > 0
        assert first > 0
    assert mm.read_results(best, 1)[0].status == mm.OK


def test_a_handle_is_refused_on_another_device():
    """A handle lives on the device that was current at mmee_create; calls with another device current are
    argument errors and launch nothing."""
    if torch.cuda.device_count() < 2:
        pytest.skip("needs two devices")
    cfg = mi.config1()
    obj = dict(cfg["searches"][0], t_begin=0, t_end=50)
    with torch.cuda.device(0):
        h = mm.mmee_create(cfg["workload"], cfg["arch"], obj)
    try:
        with torch.cuda.device(1):
            best = mm.result_buffer(1, device="cuda:1")
            lib = mm.library()
            assert lib.mmee_search(h, None, C.c_void_p(best.data_ptr()), None) == mm.ERR_ARG
            assert lib.mmee_decode(h, 0, C.byref(mm.Result())) == mm.ERR_ARG
            assert lib.mmee_eval(h, None, 0, 1, C.c_void_p(best.data_ptr())) == mm.ERR_ARG
    finally:
        with torch.cuda.device(0):
            mm.mmee_destroy(h)


def _bs_da_of_every_candidate(cfg, obj, limit):
    """(buffer words, DRAM words, idx) of every candidate of the range-limited problem, from the oracle's records."""
    p = oracle.make_problem(cfg["workload"], cfg["arch"], obj)
    if p.N > limit:
        obj = dict(obj, t_begin=0, t_end=max(1, limit // (p.R * 9)))
        p = oracle.make_problem(cfg["workload"], cfg["arch"], obj)
    begin, count = p.t_begin * p.R * 9, (p.t_end - p.t_begin) * p.R * 9
    recs = oracle.evaluate_range(p, begin, count)
    raw = np.frombuffer(recs, dtype=np.uint8).reshape(count, C.sizeof(oracle.Record))
    field = lambda off: raw[:, off:off + 8].copy().view(np.int64).ravel()
    bs = field(oracle.Record.bs.offset)
    da = field(oracle.Record.n.offset)
    return obj, p, bs, da, np.arange(begin, begin + count, dtype=np.int64)


@pytest.mark.parametrize("seed", [2, 3, 6, 8, 11])
def test_buffer_size_dram_traffic_pareto_front(seed):
    """The buffer-size / DRAM-traffic front (Section VI-A, Section VII-C) by device searches under a shrinking buffer,
    against a brute-force front over the oracle's (BS, N_DRAM) pair of every candidate: by increasing traffic,
    each point the least buffer that reaches that traffic, with the lowest index that attains the pair."""
    cfg = mi.random_tiny_problem(seed)
    obj, p, bs, da, idx = _bs_da_of_every_candidate(cfg, dict(cfg["searches"][0], objective=mi.OBJ_ENERGY, topk=1), 250_000)
    fits = bs <= p.cap_words
    want, best_bs = [], None
    for d in np.unique(da[fits]):
        sel = fits & (da == d)
        b = int(bs[sel].min())
        if best_bs is None or b < best_bs:
            want.append((b, int(d), int(idx[sel & (bs == b)].min())))
            best_bs = b
    got = mm.mmee_pareto_front_bs_da(cfg["workload"], cfg["arch"], obj)
    assert [(r.bs, r.n[0], r.idx) for r in got] == want
    assert len(want) >= 2
    for r in got:
        assert r.e_key == r.n[0]                # the search's key was the DRAM word count


@pytest.mark.parametrize("seed", [1, 4, 5, 7, 9, 10, 13, 21])
def test_chained_front_equals_one_search_after_the_other(seed):
    """The buffer-size / DRAM-traffic front takes its searches' bounds from the device, block by block; its records are
    those of plain searches, each allowed one word of buffer less than the mapping before it needs, byte for byte (the
    count of fitting mappings included, which depends on the bound a point was found under)."""
    cfg = mi.random_tiny_problem(seed)
    obj = shrink_to(cfg, dict(cfg["searches"][0], objective=mi.OBJ_ENERGY, topk=1), 1_000_000)
    wb = cfg["workload"]["word_bytes"]
    arch = dict(cfg["arch"], e_dram_pj=1.0, e_gb_pj=0.0, e_rf_pj=0.0, e_mac_pj=0.0, c_softmax=0.0, energy_quantum_pj=1.0)
    want, held, cap = [], None, arch["gb_bytes"] // wb
    while cap > 0:
        r = mm.mmee_solve_host(cfg["workload"], dict(arch, gb_bytes=cap * wb), obj)[0]
        if held is not None and (r.idx == mm.NO_INDEX or r.e_key != held.e_key):
            want.append(bytes(held))
        if r.idx == mm.NO_INDEX:
            break
        held, cap = r, r.bs - 1
    got = mm.mmee_pareto_front_bs_da(cfg["workload"], cfg["arch"], obj)
    assert [bytes(r) for r in got] == want and len(want) >= 2


@pytest.mark.parametrize("shape,gb_bytes,tilings,least_searches", [
    ((12544, 576, 192, 128), 1 << 20, None, 2),     # 63 504 tilings: several passes of tables in every search
    ((5040, 360, 1680, 96), 8 << 20, 42000, 33),    # more searches than one chain has
    ((64, 64, 64, 64), 1 << 18, 3, 2),              # one block of threads
], ids=["passes", "chains", "few"])
def test_chains_of_searches_equal_plain_searches(shape, gb_bytes, tilings, least_searches):
    """The searches of a front as steps of one kernel, at the edges of its shapes: tables that do not stay between steps,
    a front that needs a second chain, a handful of tilings; byte for byte the records of plain searches."""
    w, arch = mi.two_gemm(*shape), mi.arch_dram_only(gb_bytes)
    obj = mi.objective(mi.OBJ_ENERGY, 1, t_end=tilings or 0)
    want, held, cap, searches = [], None, gb_bytes // 2, 0
    while True:
        r = mm.mmee_solve_host(w, dict(arch, gb_bytes=cap * 2), obj)[0]
        searches += 1
        if held is not None and (r.idx == mm.NO_INDEX or r.e_key != held.e_key):
            want.append(bytes(held))
        if r.idx == mm.NO_INDEX:
            break
        held, cap = r, r.bs - 1
    assert [bytes(r) for r in mm.mmee_pareto_front_bs_da(w, arch, obj)] == want
    assert min(searches, len(want) + 1) >= least_searches


def test_buffer_size_dram_traffic_front_of_the_ffn_task():
    """On the fused feed-forward GEMMs of the paper's buffer-size study the front is a staircase: strictly less
    buffer and strictly more traffic from point to point, no point above the buffer, the last one at the
    smallest buffer any mapping needs; a plain search at a point's buffer size finds that point's traffic."""
    cfg = [c for c in mi.ffn_dram_sweep_configs() if c["name"] == "ffn_gpt3_dram_1024KB"][0]
    obj = dict(cfg["searches"][0], t_begin=0, t_end=4000)
    got = mm.mmee_pareto_front_bs_da(cfg["workload"], cfg["arch"], obj)
    cap = cfg["arch"]["gb_bytes"] // cfg["workload"]["word_bytes"]
    assert len(got) >= 3 and got[0].bs <= cap
    for a, b in zip(got, got[1:]):
        assert b.bs < a.bs and b.n[0] > a.n[0]
    mid = got[len(got) // 2]
    arch = dict(cfg["arch"], gb_bytes=mid.bs * cfg["workload"]["word_bytes"])
    best = mm.mmee_solve_host(cfg["workload"], arch, obj)[0]
    assert (best.n[0], best.bs, best.idx) == (mid.n[0], mid.bs, mid.idx)
    below = dict(cfg["arch"], gb_bytes=(got[-1].bs - 1) * cfg["workload"]["word_bytes"])
    assert mm.mmee_solve_host(cfg["workload"], below, obj)[0].idx == mm.NO_INDEX


def _group_minima(cfg, obj):
    """Least key of the feasible mappings of every group of 45 consecutive candidates (INT64_MAX: none), from the
    oracle's keys."""
    p = oracle.make_problem(cfg["workload"], cfg["arch"], obj)
    begin, count = p.t_begin * p.R * 9, (p.t_end - p.t_begin) * p.R * 9
    keys, feas = oracle.keys_range(p, begin, count)
    masked = np.where(feas.astype(bool), keys, np.iinfo(np.int64).max)
    return masked.reshape(-1, 45).min(axis=1), keys[feas.astype(bool)]


def _filter_flags(cfg, obj, thr, n_groups):
    flags = torch.empty(n_groups, dtype=torch.uint8, device="cuda")
    with Handle(cfg, obj) as h:
        mm.mmee_filter_flags(h, int(thr), flags)
        torch.cuda.synchronize()
    return flags.cpu().numpy().astype(bool)


@pytest.mark.parametrize("objective", [mi.OBJ_ENERGY, mi.OBJ_LATENCY, mi.OBJ_EDP])
@pytest.mark.parametrize("seed", [1, 2, 5, 7, 10, 12])
def test_the_filter_flags_every_group_that_holds_a_passing_mapping(seed, objective):
    """The search kernel's filter against fixed thresholds (the 1st, 50th and 99th percentile of the oracle's feasible
    keys, just above the optimum, the optimum itself and the largest key): every group of five rows that holds a
    feasible mapping with a key below the threshold is flagged.  In these small problems the energy and latency
    filters work in units of one quantum / one word, where they are exact: nothing else is flagged either; the
    energy-delay filter also flags groups whose least key equals the threshold or lies within its rounding margin."""
    cfg = mi.random_tiny_problem(seed)
    obj = shrink_to(cfg, dict(cfg["searches"][0], objective=objective, topk=1), 1_200_000)
    gmin, fkeys = _group_minima(cfg, obj)
    if fkeys.size == 0:
        pytest.skip("nothing fits")
    ranked = np.sort(fkeys)
    thresholds = [ranked[(ranked.size - 1) * q // 100] for q in (1, 50, 99)] + [ranked[0] + 1, ranked[0], ranked[-1] + 1]
    for thr in thresholds:
        flags = _filter_flags(cfg, obj, thr, gmin.size)
        must = gmin < int(thr)
        assert not (must & ~flags).any(), "a group with a passing mapping was not flagged (threshold %d)" % thr
        extra = flags & ~must
        if objective == mi.OBJ_EDP:
            # (keys are bit patterns of positive doubles; the filter compares products rounded in floating point
            # with "<=" against the threshold widened by 1e-14: a group is flagged beyond need only if its least key
            # is within that margin of the threshold)
            as_double = lambda a: np.asarray(a, dtype=np.int64).view(np.float64)
            assert (as_double(gmin[extra]) <= as_double([int(thr)])[0] * (1.0 + 1e-13)).all()
        else:
            assert not extra.any()


@pytest.mark.parametrize("log2_quantum", [-12, -24])
@pytest.mark.parametrize("seed", [3, 4, 8])
def test_the_filter_in_coarse_units_never_misses(seed, log2_quantum):
    """The same with a tiny energy quantum: keys are then large, the 32-bit filter works in units of many quanta with
    every term rounded down (and the largest ones capped), so it may flag more groups than pass, never fewer."""
    cfg = mi.random_tiny_problem(seed)
    arch = dict(cfg["arch"], energy_quantum_pj=cfg["arch"]["energy_quantum_pj"] * 2.0 ** log2_quantum)
    cfg = dict(cfg, arch=arch)
    obj = shrink_to(cfg, dict(cfg["searches"][0], objective=mi.OBJ_ENERGY, topk=1), 1_200_000)
    gmin, fkeys = _group_minima(cfg, obj)
    if fkeys.size == 0:
        pytest.skip("nothing fits")
    ranked = np.sort(fkeys)
    for q in (1, 50, 99):
        thr = ranked[(ranked.size - 1) * q // 100]
        flags = _filter_flags(cfg, obj, thr, gmin.size)
        must = gmin < int(thr)
        assert not (must & ~flags).any()
        assert (flags & ~must).sum() <= max(16, gmin.size // 4)


def shrink_to(cfg, obj, limit):
    p = oracle.make_problem(cfg["workload"], cfg["arch"], obj)
    if p.N <= limit:
        return dict(obj)
    return dict(obj, t_begin=0, t_end=max(1, limit // (p.R * 9)))


# ---- register-file-level tiling ------------------------------------------------------------------------------------

def _with_register_file_tiling(cfg, objective, rf_words, topk=1):
    arch = dict(cfg["arch"], rf_bytes=rf_words * cfg["workload"]["word_bytes"])
    if arch["e_rf_pj"] == 0:
        arch["e_rf_pj"] = arch["energy_quantum_pj"]
    obj = dict(cfg["searches"][0], objective=objective, topk=topk, rf_tiling=1, row_pruning=0)
    return dict(cfg, arch=arch), obj


@pytest.mark.parametrize("objective", [mi.OBJ_ENERGY, mi.OBJ_LATENCY])
@pytest.mark.parametrize("seed,rf_words", [(1, 6), (2, 7), (4, 8), (6, 16), (9, 64)])
def test_register_file_tiling_keys_records_and_search(seed, rf_words, objective):
    """The third tiling level on small problems: every candidate's key, sampled full records (with the register-file
    block of each operator) and the top-5 of the search equal the oracle's, from a register file that holds a single
    stationary element per PE to one that holds whole tiles."""
    cfg, obj = _with_register_file_tiling(mi.random_tiny_problem(seed), objective, rf_words, topk=5)
    obj = shrink_to(cfg, obj, 600_000)
    p = oracle.make_problem(cfg["workload"], cfg["arch"], obj)
    begin, count = p.t_begin * p.R * 9, (p.t_end - p.t_begin) * p.R * 9
    want_keys, want_feas = oracle.keys_range(p, begin, count)
    want_keys = np.where(want_feas.astype(bool), want_keys, np.iinfo(np.int64).max)
    keys = torch.empty(count, dtype=torch.int64, device="cuda")
    with Handle(cfg, obj) as h:
        mm.mmee_dump_keys(h, keys)
        torch.cuda.synchronize()
        rng = np.random.default_rng(seed)
        for idx in [begin, begin + count - 1] + [int(i) for i in rng.integers(begin, begin + count, size=60)]:
            assert_same_record(mm.mmee_decode(h, idx), oracle.evaluate(p, idx), "idx %d" % idx)
        best, topk = mm.mmee_search_host(h, True, 5)
    assert np.array_equal(keys.cpu().numpy(), want_keys)
    want = oracle.search(p)
    assert [r.idx for r in topk if r.idx != mm.NO_INDEX] == [r.idx for r in want.topk]
    assert best.n_feasible == want.n_feasible
    for g, o in zip(topk, want.topk):
        assert_same_record(g, o)
        assert any(g.rf_block)


def test_register_file_tiling_at_full_size_sampled():
    """BERT-base on the edge accelerator with the third tiling level: sampled candidates against the oracle, and the
    search's optimum is a mapping whose record the oracle reproduces and whose key no sampled candidate beats; a
    larger register file never makes the optimum worse."""
    cfg = mi.config2()
    rng = np.random.default_rng(17)
    best_keys = []
    for rf_words in (8, 512):
        cfgr, obj = _with_register_file_tiling(cfg, mi.OBJ_ENERGY, rf_words)
        p = oracle.make_problem(cfgr["workload"], cfgr["arch"], obj)
        with Handle(cfgr, obj) as h:
            best, _ = mm.mmee_search_host(h)
            assert best.status == mm.OK
            assert_same_record(best, oracle.evaluate(p, best.idx), "optimum")
            for idx in rng.integers(0, p.N, size=300):
                o = oracle.evaluate(p, int(idx))
                assert_same_record(mm.mmee_decode(h, int(idx)), o, "idx %d" % idx)
                assert not o.feasible or (o.e_key, o.idx) >= (best.e_key, best.idx)
        best_keys.append(best.e_key)
    assert best_keys[1] <= best_keys[0]
    plain, _, _ = __import__("test_gpu_parity").gpu_search(cfg, cfg["searches"][0])
    assert plain.rf_block[0] == 0


def test_fronts_and_flags_on_a_problem_in_which_nothing_fits():
    """A buffer smaller than any tile set: both Pareto fronts are empty, no group is flagged, and the plain search
    reports that nothing fits."""
    cfg = mi.random_tiny_problem(3)
    arch = dict(cfg["arch"], gb_bytes=2 * cfg["workload"]["word_bytes"])
    obj = dict(cfg["searches"][0], objective=mi.OBJ_ENERGY, topk=1)
    assert mm.mmee_pareto_front_bs_da(cfg["workload"], arch, obj) == []
    assert mm.mmee_pareto_front(cfg["workload"], arch, obj) == []
    small = dict(cfg, arch=arch)
    obj = shrink_to(small, obj, 400_000)
    p = oracle.make_problem(small["workload"], small["arch"], obj)
    n_groups = (p.t_end - p.t_begin) * p.R // 5
    assert not _filter_flags(small, obj, 2 ** 62, n_groups).any()
    with Handle(small, obj) as h:
        best, _ = mm.mmee_search_host(h)
    assert best.idx == mm.NO_INDEX and best.status == mm.ERR_NO_FEASIBLE and best.n_feasible == 0


def test_workspaces_are_not_shared_between_live_handles_threads_or_streams():
    """Released workspaces serve the next handle: one-shot calls from several threads, handles released while their
    search is still in flight on a side stream, and more live handles than workspaces are kept, each with the oracle's
    optimum; after mmee_trim everything works as before."""
    import threading
    cfgs = [mi.random_tiny_problem(s) for s in (2, 3, 5, 7)]
    jobs = [(c, shrink_to(c, dict(c["searches"][0], topk=2), 2_000_000)) for c in cfgs]
    want = [[r.idx for r in oracle.search(oracle.make_problem(c["workload"], c["arch"], o)).topk] for c, o in jobs]
    found = lambda topk: [r.idx for r in topk if r.idx != mm.NO_INDEX]

    errors = []

    def worker(i):
        try:
            torch.cuda.set_device(0)
            for n in range(40):
                c, o = jobs[(i + n) % len(jobs)]
                assert found(mm.mmee_solve_host(c["workload"], c["arch"], o)[1]) == want[(i + n) % len(jobs)]
        except Exception as e:                       # noqa: BLE001 (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=worker, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]

    streams = [torch.cuda.Stream() for _ in range(3)]
    pending = []
    for n in range(60):                              # released while in flight, the next handle at once
        c, o = jobs[n % len(jobs)]
        st = streams[n % len(streams)]
        top = mm.result_buffer(2)
        st.wait_stream(torch.cuda.current_stream())
        h = mm.mmee_create(c["workload"], c["arch"], o)
        mm.mmee_search(h, mm.result_buffer(1), top, stream=st)
        mm.mmee_destroy(h)
        pending.append((top, n % len(jobs)))
    torch.cuda.synchronize()
    for top, j in pending:
        assert found(mm.read_results(top, 2)) == want[j]

    handles = [mm.mmee_create(c["workload"], c["arch"], o) for c, o in jobs * 4]     # more than are kept
    tops = [mm.result_buffer(2) for _ in handles]
    best = [mm.result_buffer(1) for _ in handles]
    for h, b, t in zip(handles, best, tops):
        mm.mmee_search(h, b, t)
    for h in handles:
        mm.mmee_destroy(h)
    mm.mmee_trim()
    for i, t in enumerate(tops):
        assert found(mm.read_results(t, 2)) == want[i % len(jobs)]
    c, o = jobs[0]
    assert found(mm.mmee_solve_host(c["workload"], c["arch"], o)[1]) == want[0]


def test_searches_that_follow_one_another_on_a_stream():
    """A search starts while the kernel before it on the stream ends: alternating searches of different problems and
    list lengths into the same buffers, each followed by copies of its records on the same stream, without any wait
    between; an empty tiling range among them; then the same from a captured graph."""
    cfgs = [mi.random_tiny_problem(s) for s in (3, 5, 9)]
    jobs = [(c, shrink_to(c, dict(c["searches"][0], topk=k), 2_000_000)) for c, k in zip(cfgs, (1, 16, 3))]
    want = [[(r.idx, r.e_key) for r in oracle.search(oracle.make_problem(c["workload"], c["arch"], o)).topk] for c, o in jobs]
    empty = (cfgs[1], dict(jobs[1][1], t_begin=3, t_end=3))
    want.append([])
    handles = [mm.mmee_create(c["workload"], c["arch"], o) for c, o in jobs + [empty]]
    ks = [1, 16, 3, 16]
    best, top = mm.result_buffer(1), mm.result_buffer(16)

    def one_round():
        out = []
        for h, k in zip(handles, ks):
            mm.mmee_search(h, best, top)
            out.append((best.clone(), top.clone()))
        return out

    def check(rounds):
        for b, (j, k) in zip(rounds, [(j, ks[j]) for j in range(4)] * (len(rounds) // 4)):
            got = [(r.idx, r.e_key) for r in mm.read_results(b[1], k) if r.idx != mm.NO_INDEX]
            assert got == want[j] and mm.read_results(b[0], 1)[0].idx == (want[j][0][0] if want[j] else mm.NO_INDEX)

    try:
        rounds = []
        for _ in range(50):
            rounds += one_round()
        for _ in range(30):                      # no copies between: the last search's records stay
            for h in handles[:3]:
                mm.mmee_search(h, best, top)
        rounds_end = (best.clone(), top.clone())
        torch.cuda.synchronize()
        check(rounds)
        assert [(r.idx, r.e_key) for r in mm.read_results(rounds_end[1], 3) if r.idx != mm.NO_INDEX] == want[2]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            captured = one_round()
        for _ in range(5):
            graph.replay()
        torch.cuda.synchronize()
        check(captured)
    finally:
        for h in handles:
            mm.mmee_destroy(h)


@pytest.mark.parametrize("objective", [mi.OBJ_ENERGY, mi.OBJ_LATENCY])
@pytest.mark.parametrize("pe,rf_words", [((7, 3), 6), ((8, 8), 5), ((1, 16), 40), ((4, 6), 3)])
def test_register_file_blocks_with_many_divisors(pe, rf_words, objective):
    """The block search walks one divisor list down and the other up instead of trying every pair: extents with many
    divisors, arrays that do not divide them, register files from the smallest on; sampled candidates (block, words and
    cycles among their fields) against the oracle, which tries every block."""
    cfg = dict(name="rf_ragged", workload=mi.workload(1, 1, 1, 360, 120, 48, 30, 1),
               arch=mi.arch(pe[0], pe[1], 1, 40000, 64, 4, 120.0, 4.0, 1.0, 0.5, c_softmax=3.0, energy_quantum_pj=0.5))
    cfg["arch"]["rf_bytes"] = max(6, rf_words)
    obj = mi.objective(objective, 1, rf_tiling=1)
    p = oracle.make_problem(cfg["workload"], cfg["arch"], obj)
    rng = np.random.default_rng(rf_words)
    buf = mm.result_buffer(9)
    with Handle(cfg, obj) as h:
        for start in rng.integers(0, p.N // 9, size=250):
            mm.mmee_eval(h, int(start) * 9, 9, buf)          # one row: the nine stationary pairs
            for g, o in zip(mm.read_results(buf, 9), oracle.evaluate_range(p, int(start) * 9, 9)):
                assert_same_record(g, o, "idx %d" % o.idx)


RESET_SCRIPT = """
import ctypes, glob, os, sys
import mmee_inputs as mi
import paper_2604_03446_b200.binding as mm
cfg = mi.random_tiny_problem(3)
obj = dict(cfg["searches"][0], topk=2)
args = (cfg["workload"], cfg["arch"], obj)
solve = lambda: [bytes(r) for r in mm.mmee_solve_host(*args)[1]]
front = lambda: [bytes(r) for r in mm.mmee_pareto_front_bs_da(cfg["workload"], cfg["arch"], obj)]
runtime = ctypes.CDLL(glob.glob(sys.argv[1])[0])
want = solve(), front()
held = mm.mmee_create(*args)
for _ in range(2):
    assert runtime.cudaDeviceReset() == 0
    assert (solve(), front()) == want
    mm.mmee_destroy(held)                       # its workspace went with the first context
    held = mm.mmee_create(*args)
    assert bytes(mm.mmee_search_host(held, True, 2)[1][0]) == want[0][0]
assert runtime.cudaDeviceReset() == 0
mm.mmee_trim()
assert (solve(), front()) == want
print("same records")
"""


def test_one_shot_calls_after_a_device_reset():
    """cudaDeviceReset (between calls, nothing in flight) takes the kept workspaces with it: what follows gets memory of its
    own.  In a process of its own, since a reset ends torch's context as well."""
    import glob
    import subprocess
    import sys
    libs = [p for d in sys.path for p in glob.glob(os.path.join(d, "nvidia", "cuda_runtime", "lib", "libcudart.so.*"))]
    libs += glob.glob("/usr/local/cuda/lib64/libcudart.so.1*")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RESET_SCRIPT, libs[0]], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "same records" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("buffer_dram", [0, 1])
def test_fronts_whose_waits_run_out(buffer_dram):
    """The searches of a front wait for one another on the device, a limited number of looks: with a limit that is too low
    the call ends with a status of its own and leaves nothing behind that a later call would see.  (A limit in between may
    suffice or not; what is returned then is the whole front.)"""
    cfg = mi.random_tiny_problem(9)
    obj = shrink_to(cfg, dict(cfg["searches"][0], objective=mi.OBJ_ENERGY, topk=1), 1_000_000)
    args = [C.byref(mm._fill(s(), d)) for s, d in ((mm.Workload, cfg["workload"]), (mm.Arch, cfg["arch"]), (mm.Objective, obj))]
    public = (mm.mmee_pareto_front, mm.mmee_pareto_front_bs_da)[buffer_dram]
    want = [bytes(r) for r in public(cfg["workload"], cfg["arch"], obj)]
    assert want

    def limited(polls):
        pts, n = (mm.Result * 256)(), C.c_uint32()
        status = mm.library().mmee_front_with_polls(buffer_dram, *args, C.c_uint32(polls), pts, 256, C.byref(n))
        return status, [bytes(r) for r in pts[:n.value]]

    assert limited(1 << 22) == (mm.OK, want)
    for polls in (0, 0, 1, 10, 30, 100, 300, 1000):
        status, got = limited(polls)
        assert status == mm.ERR_TIMEOUT if polls == 0 else (status == mm.ERR_TIMEOUT or (status, got) == (mm.OK, want))
        if polls in (0, 100):
            assert [bytes(r) for r in public(cfg["workload"], cfg["arch"], obj)] == want
    assert limited(1 << 22) == (mm.OK, want)


PART_SCRIPT = """
import ctypes as C
import mmee_inputs as mi
import paper_2604_03446_b200.binding as mm
w, a, o = mi.workload(1, 1, 1, 4096, 4096, 128, 128), mi.arch_edge(), mi.objective(mi.OBJ_ENERGY, 1)
fronts = lambda: [[bytes(r) for r in f(w, a, o)] for f in (mm.mmee_pareto_front, mm.mmee_pareto_front_bs_da)]
want = fronts()
driver = C.CDLL("libcuda.so.1")
def call(name, *args):
    status = getattr(driver, name)(*args)
    assert status == 0, (name, status)
dev, whole, rest, part = C.c_int(), (C.c_ubyte * 256)(), (C.c_ubyte * 256)(), (C.c_ubyte * 256)()
call("cuDeviceGet", C.byref(dev), 0)
call("cuDeviceGetDevResource", dev, whole, 1)
n, desc, green, context = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
call("cuDevSmResourceSplitByCount", part, C.byref(n), whole, rest, 0, 32)
call("cuDevResourceGenerateDesc", C.byref(desc), part, 1)
call("cuGreenCtxCreate", C.byref(green), desc, dev, 1)
call("cuCtxFromGreenCtx", C.byref(context), green)
call("cuCtxSetCurrent", context)
assert fronts() == want
print("same records")
"""


def test_fronts_in_a_context_with_a_part_of_the_sms():
    """In a context that owns 32 SMs the steps of a front cannot have as many CTAs as the device holds: the fronts' points are
    those found with all SMs.  In a process of its own, which ends with that context."""
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PART_SCRIPT], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "same records" in r.stdout, r.stdout + r.stderr


def _raw(buf):
    return buf.cpu().numpy().tobytes()


def _problems_that_follow():
    """Searches of one CTA and of all, with lists of one and of sixteen, each with its records found by a search of its own, the small
    one's checked against the oracle (the large one's answers are the stored ones of test_gpu_parity)."""
    out = []
    small, large = mi.random_tiny_problem(3), mi.config4()
    for cfg, k in ((small, 1), (small, 16), (large, 1), (large, 16)):
        obj = dict(cfg["searches"][0], topk=k)
        if cfg is small:
            obj = shrink_to(cfg, obj, 2_000_000)
        best, top = mm.result_buffer(1), mm.result_buffer(k)
        with Handle(cfg, obj) as h:
            mm.mmee_search(h, best, top)
            torch.cuda.synchronize()
        if cfg is small:
            want = oracle.search(oracle.make_problem(cfg["workload"], cfg["arch"], obj))
            assert [r.idx for r in mm.read_results(top, k) if r.idx != mm.NO_INDEX] == [r.idx for r in want.topk]
        out.append((cfg, obj, (_raw(best), _raw(top))))
    return out


def test_many_searches_in_a_row_into_buffers_of_their_own():
    """More searches one after the other than a handle has scratches, with nothing between them, on one handle and on two in
    alternation: every one's records."""
    jobs = _problems_that_follow()
    for pair in [[j] for j in jobs] + [[jobs[0], jobs[2]], [jobs[1], jobs[3]], [jobs[1], jobs[2]], [jobs[0], jobs[0]]]:
        handles = [mm.mmee_create(c["workload"], c["arch"], o) for c, o, _ in pair]
        runs = [(i % len(pair), mm.result_buffer(1), mm.result_buffer(pair[i % len(pair)][1]["topk"])) for i in range(24)]
        torch.cuda.synchronize()
        for _ in range(10):
            for i, b, t in runs:
                b.zero_()
                t.zero_()
            for i, b, t in runs:
                mm.mmee_search(handles[i], b, t)
            torch.cuda.synchronize()
            for n, (i, b, t) in enumerate(runs):
                assert (_raw(b), _raw(t)) == pair[i][2], n
        for h in handles:
            mm.mmee_destroy(h)


def test_captured_searches_among_launched_ones():
    """Searches of one handle on a stream, behind other work, while another stream's capture records searches of the same handle in
    between: the launched ones' records, then those of the captured graph, launched several times."""
    eager, side = torch.cuda.Stream(), torch.cuda.Stream()
    for cfg, obj, want in _problems_that_follow()[:3]:
        h = mm.mmee_create(cfg["workload"], cfg["arch"], obj)
        outs = [[(mm.result_buffer(1), mm.result_buffer(obj["topk"])) for _ in range(24)] for _ in range(2)]
        launched, captured = [], []
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(eager):
            torch.cuda._sleep(2_000_000)                # about a millisecond
        with torch.cuda.stream(side):
            graph.capture_begin(capture_error_mode="relaxed")
        for turn, n in enumerate((2, 1, 3, 2, 1, 1, 4, 3, 2, 5, 6, 6)):
            for _ in range(n):
                done, stream, left = (captured, side, outs[1]) if turn % 2 else (launched, eager, outs[0])
                b, t = left[len(done)]
                mm.mmee_search(h, b, t, stream=stream)
                done.append((b, t))
        with torch.cuda.stream(side):
            graph.capture_end()
        torch.cuda.synchronize()
        assert all((_raw(b), _raw(t)) == want for b, t in launched)
        for _ in range(3):
            for b, t in captured:
                b.zero_()
                t.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert all((_raw(b), _raw(t)) == want for b, t in captured)
        for b, t in launched:
            b.zero_()
            t.zero_()
        graph.replay()
        for b, t in launched:
            mm.mmee_search(h, b, t)
        torch.cuda.synchronize()
        assert all((_raw(b), _raw(t)) == want for b, t in launched + captured)
        del graph
        mm.mmee_destroy(h)


def test_handles_that_take_over_the_workspace_of_a_call_with_host_records():
    """A call with host records returns before its kernel has ended, and its handle may be released: the next handle takes the same
    workspace and searches on another stream at once."""
    jobs = _problems_that_follow()[:3]
    stream = torch.cuda.Stream()
    outs = [(mm.result_buffer(1), mm.result_buffer(jobs[n % 3][1]["topk"])) for n in range(60)]
    torch.cuda.synchronize()
    for n, (b, t) in enumerate(outs):
        cfg, obj, want = jobs[n % 3]
        mm.mmee_solve_host(*[(jobs[(n + 1) % 3][0][key]) for key in ("workload", "arch")], jobs[(n + 1) % 3][1])
        h = mm.mmee_create(cfg["workload"], cfg["arch"], obj)
        best, top = mm.mmee_search_host(h, want_topk=True, topk=obj["topk"])
        assert (bytes(best), b"".join(bytes(r) for r in top)) == want
        mm.mmee_destroy(h)
        h = mm.mmee_create(cfg["workload"], cfg["arch"], obj)
        for _ in range(5):
            mm.mmee_search(h, b, t, stream=stream)
        stream.synchronize()
        mm.mmee_destroy(h)
        assert (_raw(b), _raw(t)) == want
