"""Calls on a caller's stream, from several threads beside calls on the
library's own, with memory from the shared pool; a call whose memory is more
than the pool keeps; and the pool's memory handed back on request."""
import threading

import numpy as np
import pytest

import paper_1507_00315_gb300 as sk

pytestmark = pytest.mark.gpu


def test_callers_streams_beside_the_librarys():
    import torch
    primes = sk.default_primes()[:3]
    beta = np.linspace(0.0, 4.0, 12)
    streams = [torch.cuda.Stream().cuda_stream for _ in range(3)] + [None]
    jobs = [lambda s: sk.count_ex(0, 13, stream=s)[1]["residues"],
            lambda s: sk.count_ex(1, 11, stream=s)[1]["residues"],
            lambda s: sk.count_inclusion_exclusion(2, 9, stream=s)[1]["residues"],
            lambda s: sk.pt_estimate(0, 9, 300, beta=beta, ladders=48, seed=5, stream=s)[0],
            lambda s: sk.item_residues_noalloc(0, 12, 9, 3, 64, primes, stream=s)]
    want = [j(None) for j in jobs]
    wrong = []

    def work(k):
        for i in range(16):
            # the static scratch of the last job is not for calls side by side
            j = (k + 3 * i) % (len(jobs) - 1)
            if jobs[j](streams[(k + i) % len(streams)]) != want[j]:
                wrong.append((k, i, j))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(10)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    for s in streams:
        for j in range(len(jobs)):
            assert jobs[j](s) == want[j], (s, j)


def test_more_memory_than_the_pool_keeps():
    # 2^20 items of 4 residues: 32 MiB and the launch record
    primes = sk.default_primes()
    rows = sk.item_residues(0, 14, 6, 0, 1 << 20, primes)
    for lo in (0, 1 << 18, (1 << 20) - 40):
        assert sk.item_residues(0, 14, 6, lo, 40, primes) == rows[lo:lo + 40]


def test_idle_memory_is_handed_back():
    import torch
    sk.item_residues(0, 14, 6, 0, 1 << 19, sk.default_primes())     # 16 MiB stay idle
    before = torch.cuda.mem_get_info()[0]
    sk.release_memory()
    assert torch.cuda.mem_get_info()[0] - before >= 16 << 20
    assert sk.count(0, 8) == 504 // 2
