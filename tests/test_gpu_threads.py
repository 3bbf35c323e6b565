"""Calls from several host threads, each with its own buffers and stream: the calls whose
kernels take more shared memory the larger their K or their number of noise vectors are
made at once with different ones, and every call must be launched and give its own result."""
import ctypes
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CALLS = 400


@pytest.fixture(scope="module")
def copes():
    from paper_2608_02391_gb300 import copes as c
    c.load()
    return c


def at_once(jobs):
    """Runs each job CALLS times in a thread of its own; the first error of each."""
    start, errors = threading.Barrier(len(jobs)), []

    def loop(job):
        start.wait()
        for i in range(CALLS):
            message = job()
            if message:
                errors.append("call %d: %s" % (i, message))
                return

    threads = [threading.Thread(target=loop, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    return errors


def test_partitions_of_several_sizes(copes):
    L, layout, seed = copes.load(), copes.Layout([40_000, 333]), 1088
    desc, jobs, results = ctypes.byref(layout.desc), [], []
    for K in (64, 16, 48, 32):
        want = [s.tensor for s in copes.hash_partition(layout, K, seed)]
        nbytes = L.copes_hash_workspace_bytes(desc, K)
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        counts, stream = np.zeros(K, np.uint64), torch.cuda.Stream()
        torch.cuda.synchronize()
        rc = L.copes_hash_count(desc, K, seed, ws.data_ptr(), nbytes, counts.ctypes.data, stream.cuda_stream)
        assert rc == 0, copes.last_error()
        lists = [torch.zeros_like(t) for t in want]
        ptrs = (ctypes.c_void_p * K)(*[t.data_ptr() for t in lists])
        torch.cuda.synchronize()

        def fill(K=K, ws=ws, nbytes=nbytes, ptrs=ptrs, stream=stream):
            rc = L.copes_hash_fill(desc, K, seed, ws.data_ptr(), nbytes, ptrs, stream.cuda_stream)
            return copes.last_error() if rc else None

        jobs.append(fill)
        results.append((lists, want))
    assert at_once(jobs) == []
    for lists, want in results:
        assert all(torch.equal(x, y) for x, y in zip(lists, want))


@pytest.mark.parametrize("kind", ["list", "replay"])
def test_updates_of_several_populations(copes, kind):
    n, K = 20_000, 16
    layout, jobs, results = copes.Layout([n]), [], []
    sub = (copes.hash_partition if kind == "list" else copes.hash_replay_partition)(layout, K, 77)[3]
    theta = torch.randn(n, device="cuda")
    for P in (256, 150, 200, 170):
        nid, sign, _ = copes.member_table(P, copes.ONE_SIDED)
        fitness, seeds = torch.linspace(-1, 1, P, device="cuda"), copes.member_seeds(33, 0, 3, P)
        a, b = (copes.Arena(torch.zeros(n, dtype=torch.bfloat16, device="cuda"), theta.clone()) for _ in range(2))
        stream = torch.cuda.Stream()
        for _ in range(CALLS):
            copes.update(b, sub, nid, sign, fitness, seeds, 1e-4)

        def update(a=a, nid=nid, sign=sign, fitness=fitness, seeds=seeds, stream=stream):
            try:
                copes.update(a, sub, nid, sign, fitness, seeds, 1e-4, stream=stream)
            except copes.CopesError as e:
                return str(e)

        jobs.append(update)
        results.append((a, b))
    torch.cuda.synchronize()
    assert at_once(jobs) == []
    for a, b in results:
        assert torch.equal(a.master, b.master) and torch.equal(a.w, b.w)
    copes.check()
