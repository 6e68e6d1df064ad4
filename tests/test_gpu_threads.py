"""Calls of several host threads at once, each with its own objects and stream: launches of one kernel
with different amounts of shared memory do not disturb each other."""
import threading

import numpy as np
import pytest

from afc_inputs import Workload, ws_edges
from tests.test_gpu_sweep_forms import _counts

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
afc = pytest.importorskip("paper_2605_14743_gb300")


def _together(jobs, rounds):
    """Runs every job `rounds` times, each in a thread with a stream of its own."""
    errors, start = [], threading.Barrier(len(jobs))

    def work(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(rounds):
                    job()
        except Exception as e:   # reported by the test
            errors.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not errors, errors[0]


def test_sweeps_of_chains_of_different_size():
    from tests.test_gpu_chain import Chain
    jobs = []
    for c in (163, 200, 300, 420):
        ch = Chain(_counts(440, c, [2, 5], 6000, c, False), 6000, 0.15)
        ref = ch.sweep(0, 1, 0.05, 0.05, 19)[4]

        def job(ch=ch, ref=ref):
            assert (ch.sweep(0, 1, 0.05, 0.05, 19)[4] == ref).all()
        jobs.append(job)
    torch.cuda.synchronize()
    _together(jobs, 400)


def test_counts_of_graphs_of_different_size():
    """Asynchronous calls one after another: the threads' launches follow each other closely."""
    jobs, done = [], []
    for n in (300, 500, 700, 900):
        eu, ev = ws_edges(n, 4, 0.1, n)
        q = afc.Query(Workload("threads", n, eu, ev, 0.9, 1, 9, 1, seed=3), block_threads=512,
                      memory_path=afc.AFC_PATH_SHARED)
        q.run_counts()
        torch.cuda.synchronize()
        done.append((q, q.counts.clone()))
        jobs.append(lambda q=q: q.run_counts())
    _together(jobs, 1500)
    torch.cuda.synchronize()
    for q, ref in done:
        assert bool((q.counts == ref).all())
