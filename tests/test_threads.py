"""Handles used from different threads at the same time, each on a stream of its own (the header allows it): every call
succeeds and gives the oracle's integers, whatever the other handles launch meanwhile."""
import threading

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _tables(w, H, Bmax):
    """The same workload with tables of another size (other entries are not used), so that its launches take another
    amount of shared memory."""
    lat = np.full((w.latency_us.shape[0], H, Bmax), 77, np.int32)
    h, b = w.latency_us.shape[1:]
    lat[:, :h, :b] = w.latency_us
    w.latency_us = lat
    return w


def _make(kind, k):
    H, Bmax = [(2, 8), (8, 64), (3, 33)][k]
    if kind == "chain":
        w = workloads.random_small(k, S=4, H=2, Bmax=8, n=40 + 20 * k, C=[6, 60, 20][k], max_replicas=[3, 20, 9][k])
    elif kind == "fan_out":
        w = workloads.random_small(k, S=4, H=2, Bmax=8, n=40 + 20 * k, C=[6, 60, 20][k], max_replicas=[3, 20, 9][k])
        w.parent, w.cond_bit, w.cond_val = np.array([-1, 0, 0, 1], np.int32), np.full(4, -1, np.int8), np.zeros(4, np.uint8)
    else:                   # "tree", and "shared": its prefixes
        w = workloads.make(5, n_queries=60 + [0, 20_000, 4_000][k] * (kind == "shared"), n_candidates=[6, 250, 90][k])
        H, Bmax = [(4, 64), (8, 64), (6, 64)][k]
    return _tables(w, H, Bmax)


@pytest.mark.parametrize("kind", ["chain", "tree", "fan_out", "shared"])
def test_handles_on_threads_of_their_own(oracle, kind):
    import torch
    import paper_1812_01776_b200 as il
    ws = [_make(kind, k) for k in range(3)]
    want = [oracle.estimate_workload(w) for w in ws]
    ests = [il.Estimator.from_workload(w) for w in ws]
    streams = [torch.cuda.Stream() for _ in ws]
    failures = []
    start = threading.Barrier(3)

    def calls(k):
        try:
            est, w = ests[k], ws[k]
            il.il_set_stream(est._h, streams[k].cuda_stream)
            start.wait()
            for i in range(1500 if kind != "shared" else 200):
                m = len(w.configs) if i % 3 else 1 + i % len(w.configs)
                p99, miss = est.estimate(w.configs[:m], w.slo_us)
                assert np.array_equal(p99, want[k][0][:m]) and np.array_equal(miss, want[k][1][:m]), (k, i, m)
                if i % 4 == 0:
                    assert np.array_equal(est.feasible(w.configs[:m], w.slo_us), want[k][0][:m] <= w.slo_us), (k, i, m)
        except Exception as e:       # (an assertion of a thread would be lost)
            failures.append((k, repr(e)))

    for est in ests:
        est.set_test_knob(3, 1 if kind == "shared" else 2)
    threads = [threading.Thread(target=calls, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for est in ests:
        est.close()
    assert not failures, failures
