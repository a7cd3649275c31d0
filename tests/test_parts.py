"""Pipelines cut at their branch points (the lane kernel's parts): shapes of the tree that make every kind of stream between
two parts, trace lengths around a pair of records, a group's stretch and the publishing of a count, and as many candidates
as one warp, several warps and several rounds of groups hold.  Exact against the oracle."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

# parent, guard bit and value per stage
SHAPES = {
    "root_leaves": ([-1, 0, 1, 1], [-1, 0, 1, 1], [0, 1, 0, 1]),                    # some queries leave at the root
    "cascades": ([-1, 0, 1, 2, 3], [-1, -1, 0, -1, 1], [0, 0, 1, 0, 0]),            # one guarded way on, twice
    "late_branch": ([-1, 0, 1, 2, 2, 3], [-1, -1, -1, 0, 0, -1], [0, 0, 0, 0, 1, 0]),
    "three_levels": ([-1, 0, 0, 1, 1, 3, 3], [-1, 0, 0, 1, 1, 2, 2], [0, 0, 1, 0, 1, 0, 1]),
    "side_leaves": ([-1, 0, 0, 1, 2], [-1, 0, 0, 1, 3], [0, 1, 0, 1, 0]),           # both sides lose queries
    "fan_out": ([-1, 0, 0, 1, 2, 2], [-1, -1, -1, -1, 0, -1], [0, 0, 0, 0, 1, 0]),
    "fan_out_some": ([-1, 0, 0, 1, 1], [-1, 0, 1, -1, 2], [0, 1, 0, 0, 1]),         # none, one or both ways
}


def small(shape, seed, n, C, **more):
    parent, bit, val = SHAPES[shape]
    w = workloads.random_small(seed, S=len(parent), H=2, Bmax=8, n=n, C=C, max_replicas=more.pop("replicas", 6), qps=700.0,
                               cv=4.0, lat_lo=1, lat_hi=9000, equal_stamp_every=more.pop("stamps", 0))
    w.parent, w.cond_bit, w.cond_val = np.array(parent, np.int32), np.array(bit, np.int8), np.array(val, np.uint8)
    w.branch_bits = np.random.default_rng(seed).integers(0, 256, size=n).astype(np.uint8)
    return w


def same(w, oracle, at=slice(None), knobs=()):
    import torch
    import paper_1812_01776_b200 as il
    exp = oracle.estimate_workload(w)
    p99, miss, cfg = exp[0][at], exp[1][at], np.ascontiguousarray(w.configs[at])
    with il.Estimator.from_workload(w) as est:
        est.set_test_knob(3, 2)
        for k, v in knobs:
            est.set_test_knob(k, v)
        a, b = est.estimate_device(torch.from_numpy(cfg).cuda(), w.slo_us)
        assert np.array_equal(a.cpu().numpy(), p99) and np.array_equal(b.cpu().numpy(), miss)
        for slo in (w.slo_us, int(np.median(p99)), 0):
            assert np.array_equal(est.feasible(cfg, slo), p99 <= slo), slo
        a, b = est.estimate(cfg, w.slo_us)
        assert np.array_equal(a, p99) and np.array_equal(b, miss)


@pytest.mark.parametrize("n", [1, 2, 3, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 257, 700])
@pytest.mark.parametrize("shape", SHAPES)
def test_trace_lengths(oracle, shape, n):
    same(small(shape, n, n, 12, stamps=3 if n % 2 else 0), oracle)


@pytest.mark.parametrize("C", [1, 2, 31, 33, 700, 9000])
@pytest.mark.parametrize("shape", ["root_leaves", "late_branch", "three_levels", "fan_out"])
def test_candidates_of_one_warp_and_of_several_rounds(oracle, shape, C):
    same(small(shape, C, 333, 64, replicas=20), oracle, at=np.arange(C) % 64)


@pytest.mark.parametrize("knobs", [((5, 0),), ((1, 6),), ((6, 4080),)], ids=["bits_looked_up", "short_rings", "shared_memory_elsewhere"])
@pytest.mark.parametrize("shape", SHAPES)
def test_other_forms(oracle, shape, knobs):
    """Branch bits looked up; parts that give a candidate (or a root node that several share) up, so that whoever reads
    their streams gives up too; fewer words of examined records."""
    same(small(shape, 5, 900, 40, replicas=32), oracle, knobs=knobs)


@pytest.mark.parametrize("shape", SHAPES)
def test_latencies(oracle, shape):
    import paper_1812_01776_b200 as il
    w = small(shape, 9, 801, 3)
    with il.Estimator.from_workload(w) as est:
        for c in range(3):
            _, _, exp = oracle.estimate_one(w.parent, w.cond_bit, w.cond_val, w.latency_us, w.arrival_us, w.branch_bits,
                                            w.configs[c], w.slo_us, want_latency=True)
            assert np.array_equal(est.latencies(w.configs[c]), exp)


@pytest.mark.parametrize("shape", ["root_leaves", "three_levels", "side_leaves", "fan_out"])
def test_small_workspace_and_bad_candidates(oracle, shape):
    import torch
    import paper_1812_01776_b200 as il
    from paper_1812_01776_b200 import estimator as E
    w = small(shape, 3, 2000, 60)
    exp = oracle.estimate_workload(w)
    d = torch.from_numpy(w.configs).cuda()
    with il.Estimator.from_workload(w) as est:
        est.set_test_knob(3, 2)
        est.reserve_workspace(60, max_bytes=il.il_workspace_min_bytes(est._h) + 30 * 2016 * 8)
        a, _ = est.estimate_device(d, w.slo_us)
        assert est.stats()["chunks"] > 1 and np.array_equal(a.cpu().numpy(), exp[0])
        assert np.array_equal(est.feasible_device(d, w.slo_us).cpu().numpy().astype(bool), exp[0] <= w.slo_us)
        bad = w.configs.copy()
        bad[7, -1, 2] = 0
        for call in (est.estimate_device, est.feasible_device):
            with pytest.raises(E.ILError) as ei:
                call(torch.from_numpy(bad).cuda(), w.slo_us)
            assert ei.value.code == E.IL_ERR_BAD_CONFIG
        a, _ = est.estimate_device(d, w.slo_us)
        assert np.array_equal(a.cpu().numpy(), exp[0])


@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 65, 129, 1025, 2100])
@pytest.mark.parametrize("C", [1, 40, 20_000])
@pytest.mark.parametrize("shape", ["diamond", "guarded", "two_joins", "skip"])
def test_merges(oracle, shape, C, n):
    """Lengths around a merge's windows and around what it keeps of the queries' bits (1,024 at the least); one, a few and
    several rounds of candidates per lane; one input slow, so that it falls far behind."""
    import paper_1812_01776_b200 as il
    w = workloads.join_small(n, n=n, C=24, max_replicas=3, Bmax=8, shape=shape)
    w.configs[:8, 1] = (0, 1, 1, 0)
    w.latency_us[1, 0, 0] = 9000
    at = np.arange(C) % 24
    exp = oracle.estimate_workload(w)
    with il.Estimator.from_workload(w) as est:
        a, b = est.estimate(w.configs[at], w.slo_us)
        assert np.array_equal(a, exp[0][at]) and np.array_equal(b, exp[1][at])


@pytest.mark.parametrize("shape", ["late_branch", "fan_out"])
def test_iteration_bound(shape):
    import paper_1812_01776_b200 as il
    from paper_1812_01776_b200 import estimator as E
    w = small(shape, 4, 3000, 20)
    with il.Estimator.from_workload(w) as est:
        est.set_test_knob(2, 64)
        with pytest.raises(E.ILError) as ei:
            est.estimate(w.configs, w.slo_us)
        assert ei.value.code == E.IL_ERR_ITER_LIMIT
        est.set_test_knob(2, 0)
        assert (est.estimate(w.configs, w.slo_us)[0] > 0).all()


@pytest.mark.parametrize("C,sms", [(300, 1), (4096, 1), (4096, 2), (4096, 40)])
def test_ctas_that_come_to_few_sms_still_work(oracle, C, sms):
    """The first CTA on an SM may take it for root nodes, and others that come there leave.  Where the rest of the device is
    taken by somebody else's kernel all CTAs come to the same few SMs; all but the planned ones must work all the same,
    or the first few do everything (which takes some forty times as long)."""
    import torch
    import paper_1812_01776_b200 as il
    w = workloads.make(3, n_queries=3000, n_candidates=400)
    exp = oracle.estimate_workload(w)
    at = np.arange(C) % 400
    d = torch.from_numpy(np.ascontiguousarray(w.configs[at])).cuda()
    ms = {}
    with il.Estimator.from_workload(w) as est:
        for seen in (0, sms):
            est.set_test_knob(7, seen)
            for _ in range(4):
                p99, miss = est.estimate_device(d, w.slo_us)
                assert np.array_equal(p99.cpu().numpy(), exp[0][at]) and np.array_equal(miss.cpu().numpy(), exp[1][at])
                ms[seen] = min(ms.get(seen, 1e9), est.stats()["sim_ms"])
            assert np.array_equal(est.feasible(w.configs[at], w.slo_us), exp[0][at] <= w.slo_us)
    print(f"{C} candidates, {sms} SMs: {ms[0]:.2f} / {ms[sms]:.2f} ms")
    assert ms[sms] < 4.0 * ms[0] + 0.5, ms
