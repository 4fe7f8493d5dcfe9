"""Calls from several threads and on shared streams, against the oracle,
bit-exact: threads at once on streams of their own, calls one after another on
one stream with no synchronisation between, and a thread that ends while
another thread's stream is under capture."""
from __future__ import annotations

import os
import threading
import time
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def words(edges):
    import paper_2207_00514_gb300 as pkg
    return pkg.edges_numpy(edges).view(np.uint32).reshape(-1, 3)


def want(pts):
    return oracle.emst(pts).view(np.uint32).reshape(-1, 3)


def test_threads_at_once():
    import paper_2207_00514_gb300 as pkg
    sets = [synth.blobs(n, 3, n) for n in (700, 40_000, 60_000, 90_001, 33_000, 150_000)]
    wanted = [want(p) for p in sets]
    pkg.load_library()

    def work(k):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            t = torch.from_numpy(sets[k]).cuda()
            got = [pkg.emst_compute(t) for _ in range(6)]
            link, _ = pkg.emst_dendrogram(got[-1])
        stream.synchronize()
        for e in got:
            assert np.array_equal(words(e), wanted[k]), k
        assert int(link[-1, 3]) == len(sets[k])

    with ThreadPoolExecutor(max_workers=len(sets)) as pool:
        list(pool.map(work, range(len(sets))))


def test_calls_on_one_stream():
    # (a call returns when its result is complete, the stream may still report
    # work; the next call's first kernels follow it)
    import paper_2207_00514_gb300 as pkg
    sets = [synth.uniform(n, 2, n) for n in (50_000, 33_000, 200_000, 5_000, 80_000)]
    ts = [torch.from_numpy(p).cuda() for p in sets]
    got = [pkg.emst_compute(t) for t in ts for _ in range(3)]
    torch.cuda.synchronize()
    for k, e in enumerate(got):
        assert np.array_equal(words(e), want(sets[k // 3]))


def test_a_thread_ends_during_a_capture():
    import paper_2207_00514_gb300 as pkg
    pts = synth.uniform(50_000, 3, 5)
    called, leave = threading.Event(), threading.Event()
    tid = []

    def work():
        tid.append(threading.get_native_id())
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            pkg.emst_compute(torch.from_numpy(pts).cuda())
        stream.synchronize()
        called.set()
        leave.wait()

    thread = threading.Thread(target=work)
    thread.start()
    called.wait()

    x = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        x += 1
        leave.set()
        thread.join()
        for _ in range(1000):  # (its thread-local objects go after the Python part has ended)
            if not os.path.exists(f"/proc/self/task/{tid[0]}"):
                break
            time.sleep(0.005)
        assert not os.path.exists(f"/proc/self/task/{tid[0]}")
        x += 1
    graph.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2.0] * 4
