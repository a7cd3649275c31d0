"""P99 and misses of rows long enough for the percentile kernel's one-pass form: latencies known by construction, in the
order of the row, so that its sample (the first four of every 64 records) can be made to tell the truth or to deceive."""
import numpy as np
import pytest

from select_cases import grouped_workload

pytestmark = pytest.mark.gpu


def blocks(n, block):
    """Group sizes that add up to n, from a function of the number of a block of 64."""
    sizes, j = [], 0
    while sum(sizes) < n:
        sizes += block(j)
        j += 1
    while sum(sizes) > n:
        sizes.pop()
    return sizes + [1] * (n - sum(sizes))


def honest(j):
    return [1 + (j * 7 + k) % 5 for k in range(12)] + [30] if j % 9 else [16, 16, 32]


def hidden(j):         # late queries only where the sample does not look
    return [1, 1, 1, 1, 60] if j % 40 == 0 else [1] * 64


def shown(j):          # hardly any late queries, all of them where it looks
    return [4] + [1] * 60 if j % 50 == 0 else [1] * 64


LAT = {b: 900 + 17 * b * b for b in range(1, 65)}
FAR = {**{b: 40 + b for b in range(1, 65)}, 60: 3 * 2 ** 32}
CASES = {
    "honest": (honest, LAT, 1), "hidden": (hidden, LAT, 1), "shown": (shown, LAT, 1), "far": (hidden, FAR, 7),
    "all_equal": (lambda j: [64], {64: 1_000_003}, 1), "two_values": (lambda j: [1] * 64 if j % 90 else [32, 32], {1: 10, 32: 11}, 1),
}


@pytest.mark.parametrize("n", [16_383, 16_384, 16_387, 20_000, 50_021])
@pytest.mark.parametrize("case", CASES)
def test_percentile_of_long_rows(case, n):
    import paper_1812_01776_b200 as il
    block, lat, S = CASES[case]
    w, want = grouped_workload(blocks(n, block), {b: v for b, v in lat.items()} | {b: 7 for b in range(1, 65) if b not in lat}, S)
    k = (99 * n + 99) // 100
    p99 = int(np.sort(want)[k - 1])
    with il.Estimator.from_workload(w) as est:
        for slo in (int(np.median(want)), p99, 0):
            a, b = est.estimate(w.configs, slo)
            assert a[0] == p99 and b[0] == int((want > slo).sum()), (slo, a, b, p99)


@pytest.mark.parametrize("n", [4095, 4096, 4099, 12_000])
@pytest.mark.parametrize("case", ["ordinary", "one_value", "few_late"])
@pytest.mark.parametrize("tree", [False, True])
def test_largest_latencies_of_shared_nodes(oracle, tree, case, n):
    """The same for the lists of the largest latencies per node that a shared batch is put together from: ordinary rows, rows
    of one value (everything reaches what the sample says) and rows whose late queries the sample does not see."""
    import workloads
    import paper_1812_01776_b200 as il
    w = workloads.random_small(n, S=4 if tree else 2, H=2, Bmax=4, n=n, C=40, max_replicas=6, tree=False, qps=300.0, cv=3.0, lat_lo=1,
                               lat_hi=9000)
    if tree:
        w.parent, w.cond_bit = np.array([-1, 0, 0, 2], np.int32), np.array([-1, 0, 0, 1], np.int8)
        w.cond_val = np.array([0, 0, 1, 0], np.uint8)
        w.branch_bits = np.random.default_rng(n).integers(0, 4, n).astype(np.uint8)
    if case != "ordinary":
        w.latency_us[:] = 100
        w.arrival_us = np.arange(n, dtype=np.int64) * 1000
        w.configs[:, :, 2] = 1
        if case == "few_late":
            late = np.nonzero((np.arange(n) % 64 == 40) & (np.arange(n) // 64 % 2 == 0))[0]
            w.arrival_us[late] = w.arrival_us[late - 1]
            w.configs[:, :, 1] = 1
    exp = oracle.estimate_workload(w)
    with il.Estimator.from_workload(w) as est:
        est.set_test_knob(3, 1)
        a, b = est.estimate(w.configs, w.slo_us)
        assert np.array_equal(a, exp[0]) and np.array_equal(b, exp[1])
