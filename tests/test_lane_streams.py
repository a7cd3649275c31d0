"""The lane kernel where its rings can go wrong: records in flight around what a lane keeps in shared memory and in
its spill ring, replica counts around the two sizes of the batch ring, trace lengths around a turn and around a tile
of the packed trace, and more candidates than the device holds at once."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def same(w, oracle, ring=0):
    import torch
    import paper_1812_01776_b200 as il
    exp = oracle.estimate_workload(w)
    with il.Estimator.from_workload(w) as est:
        if ring:
            est.set_test_knob(1, ring)
        est.set_test_knob(3, 2)
        a, b = est.estimate_device(torch.from_numpy(w.configs).cuda(), w.slo_us)
        st = est.stats()
        assert np.array_equal(a.cpu().numpy(), exp[0]) and np.array_equal(b.cpu().numpy(), exp[1])
        assert np.array_equal(est.feasible(w.configs, w.slo_us), exp[0] <= w.slo_us)
    return st


@pytest.mark.parametrize("ring", [0, 7, 9])
@pytest.mark.parametrize("burst", [30, 47, 65, 130, 260, 1100])
def test_records_in_flight(oracle, burst, ring):
    """Bursts of arrivals at one instant, on as many replicas as take them all: that many records wait at once."""
    w = workloads.random_small(burst, S=3, H=2, Bmax=64, n=4000, C=48, max_replicas=32, lat_lo=500, lat_hi=900000)
    w.arrival_us = (np.arange(4000) // burst * 400_000).astype(np.int64)
    w.configs[::2, :, 2] = 32
    st = same(w, oracle, ring)
    assert ring or st["fallback_candidates"] == 0


@pytest.mark.parametrize("replicas", [1, 2, 14, 15, 16, 17, 31, 32])
def test_replicas_around_the_ring_sizes(oracle, replicas):
    w = workloads.random_small(replicas, S=4, H=2, Bmax=4, n=1500, C=40, max_replicas=replicas, qps=900.0, cv=4.0,
                               lat_lo=1, lat_hi=60000, equal_stamp_every=2)
    w.configs[::3, :, 2] = replicas
    same(w, oracle)


@pytest.mark.parametrize("n", [1, 2, 3, 15, 16, 17, 32, 33, 510, 511, 512, 513, 1024])
def test_trace_lengths(oracle, n):
    w = workloads.random_small(n, S=5, H=2, Bmax=8, n=n, C=33, max_replicas=3, tree=n % 2 == 1)
    same(w, oracle)


@pytest.mark.parametrize("S", [1, 4, 9])
@pytest.mark.parametrize("n", [63, 64, 65, 66, 96, 97, 127, 128, 129])
def test_trace_lengths_around_a_root_s_stretch(oracle, n, S):
    """Record 64 of the trace is copied to where record 0 was, in the turn in which that one opens its batch; by another
    lane where the candidate has several."""
    w = workloads.random_small(n + S, S=S, H=2, Bmax=8, n=n, C=700, max_replicas=3, qps=5000.0, lat_lo=1, lat_hi=3000)
    same(w, oracle)


@pytest.mark.parametrize("bits_too", [False, True], ids=["query-index", "query-index-and-bits"])
@pytest.mark.parametrize("over", [0, 1], ids=["just-below", "at-the-limit"])
@pytest.mark.parametrize("shape", ["chain", "tree", "fan_out", "diamond", "two_joins"])
def test_times_at_the_limit_of_a_record(oracle, shape, over, bits_too):
    """Records are compared as doubles, so their words stay below 0x7fe0 << 48: traces whose last possible time is just below
    what the query index (and the branch bits) leave room for, and traces one microsecond beyond."""
    import torch
    import paper_1812_01776_b200 as il
    n = 1000
    if shape in ("chain", "tree"):
        w = workloads.random_small(3, S=5, H=2, Bmax=8, n=n, C=40, max_replicas=4, tree=shape == "tree", qps=900.0, cv=3.0,
                                   equal_stamp_every=3)
    elif shape == "fan_out":
        w = workloads.fan_out_small(11, n=n, C=40, max_replicas=4, Bmax=8)
    else:
        w = workloads.join_small(4, n=n, C=40, max_replicas=4, Bmax=8, shape=shape)
    guards = [w.cond_bit] + ([w.join[1]] if w.join is not None else [])
    bits = max(int(g.max()) for g in guards) + 1
    q = 10 + (bits if bits_too else 0)                                    # 1,000 queries: 10 bits
    worst = n * int(w.latency_us.max(axis=(1, 2)).astype(np.int64).sum())
    exp = oracle.estimate_workload(w)
    _, _, lat = oracle.estimate_one(w.parent, w.cond_bit, w.cond_val, w.latency_us, w.arrival_us, w.branch_bits, w.configs[0],
                                    w.slo_us, want_latency=True, join=w.join)
    w.arrival_us = w.arrival_us + ((0x7fe0 << 48 >> q) - 1 + over - worst - int(w.arrival_us[-1]))
    with il.Estimator.from_workload(w) as est:
        if w.join is None and (not over or bits_too and bits):
            assert est.kernel_name() == "des_lane_kernel"
        elif shape in ("chain", "tree"):
            assert est.kernel_name() == "des_packed_kernel"
        a, b = est.estimate_device(torch.from_numpy(w.configs).cuda(), w.slo_us)
        assert np.array_equal(a.cpu().numpy(), exp[0]) and np.array_equal(b.cpu().numpy(), exp[1])
        for slo in (w.slo_us, int(np.median(exp[0])), 1 << 62):
            assert np.array_equal(est.feasible(w.configs, slo), exp[0] <= slo)
        assert np.array_equal(est.latencies(w.configs[0]), lat)


def rare_branch(rows, n=20_000, C=590):
    """A stage that only the queries in `rows` visit, one behind it, and the other way with a stage behind it."""
    w = workloads.random_small(5, S=5, H=2, Bmax=8, n=n, C=C, max_replicas=4, tree=True, qps=300.0, lat_lo=500, lat_hi=9000)
    w.parent = np.array([-1, 0, 0, 1, 2], np.int32)
    w.cond_bit, w.cond_val = np.array([-1, 0, 0, -1, -1], np.int8), np.array([0, 0, 1, 0, 0], np.uint8)
    w.branch_bits = np.zeros(n, np.uint8)
    w.branch_bits[rows] = 1
    return w


@pytest.mark.parametrize("rows", [[], [0], [1999], [0, 1999], [1900, 1930], list(range(40)), list(range(1000, 2000, 400))])
def test_rarely_taken_branches(oracle, rows):
    same(rare_branch(rows, n=2000, C=40), oracle)


def test_a_branch_taken_late_costs_no_short_turns():
    """The time of a batch does not depend on where in the trace a branch is taken for the first time (while a stage waits
    for its first record, or has seen its last one, there is nothing to look at every few iterations)."""
    import torch
    import paper_1812_01776_b200 as il
    ms = {}
    for name, rows in (("late", slice(19_980, None)), ("even", slice(0, None, 1000))):
        w = rare_branch(rows)
        cfg = torch.from_numpy(w.configs).cuda()
        with il.Estimator.from_workload(w) as est:
            ms[name] = min((est.estimate_device(cfg, w.slo_us), est.stats()["sim_ms"])[1] for _ in range(7))
    assert ms["late"] < 1.12 * ms["even"], ms


@pytest.mark.parametrize("skip", [16, 1024, 3072, 4080, 8192])
@pytest.mark.parametrize("replicas", [3, 32])
def test_shared_memory_that_starts_elsewhere(oracle, replicas, skip):
    """The batch keys are aligned wherever shared memory starts; what that takes comes out of the words of examined records,
    down to 32 a lane (here with more than that in flight, on a tree and with a join)."""
    import paper_1812_01776_b200 as il
    w = workloads.random_small(skip + replicas, S=6, H=3, Bmax=33, n=2500, C=48, max_replicas=replicas, tree=True, qps=3000.0,
                               cv=4.0, lat_lo=500, lat_hi=90000)
    j = workloads.join_small(replicas, n=1500, C=48, max_replicas=replicas, Bmax=8, shape="two_joins")
    for x in (w, j):
        exp = oracle.estimate_workload(x)
        many = np.arange(20_000) % x.n_candidates                  # every resident CTA, and as few words as there can be
        with il.Estimator.from_workload(x) as est:
            est.set_test_knob(3, 2)
            est.set_test_knob(6, skip)
            a, b = est.estimate(x.configs[many], x.slo_us)
            assert np.array_equal(a, exp[0][many]) and np.array_equal(b, exp[1][many])
            assert np.array_equal(est.feasible(x.configs[many], x.slo_us), exp[0][many] <= x.slo_us)
            with pytest.raises(Exception):
                est.set_test_knob(6, 8)


@pytest.mark.parametrize("S", [1, 3])
def test_more_candidates_than_resident_groups(oracle, S):
    w = workloads.random_small(S, S=S, H=2, Bmax=4, n=60, C=90_001, max_replicas=3)
    w.configs = np.ascontiguousarray(w.configs[np.arange(90_001) % 5_000])
    exp = oracle.estimate_workload(workloads.Workload(w.name, w.parent, w.cond_bit, w.cond_val, w.latency_us, w.arrival_us,
                                                      w.branch_bits, w.configs[:5_000].copy(), w.slo_us))
    import torch
    import paper_1812_01776_b200 as il
    with il.Estimator.from_workload(w) as est:
        est.set_test_knob(3, 2)
        a, _ = est.estimate_device(torch.from_numpy(w.configs).cuda(), w.slo_us)
    assert np.array_equal(a.cpu().numpy(), exp[0][np.arange(w.n_candidates) % 5_000])


@pytest.mark.parametrize("slow", [1, 2])
@pytest.mark.parametrize("shape", ["diamond", "guarded", "two_joins", "skip"])
def test_joins_with_one_slow_input(oracle, shape, slow):
    """One of two branches falls behind the other by hundreds to thousands of queries: more than a join keeps in
    shared memory of its incoming streams, and of its queries' bits."""
    import torch
    import paper_1812_01776_b200 as il
    w = workloads.join_small(slow, n=6000, C=40, max_replicas=4, Bmax=8, shape=shape)
    if shape == "skip" and slow == 2:
        slow = 1                                  # (the other input there comes straight from stage 0)
    w.configs[:20, slow] = (0, 1, 1, 0)
    w.latency_us[slow, 0, 0] = 9000               # 110 a second of 300
    exp = oracle.estimate_workload(w)
    with il.Estimator.from_workload(w) as est:
        a, b = est.estimate_device(torch.from_numpy(w.configs).cuda(), w.slo_us)
        assert np.array_equal(a.cpu().numpy(), exp[0]) and np.array_equal(b.cpu().numpy(), exp[1])
