"""Calls of several threads, with and without a caller's stream, share the
library's pool of streams and memory: every result is the one of a call made
alone, also when the calls need different amounts of memory."""
import threading

import numpy as np
import pytest

import paper_1507_00315_gb300 as sk

pytestmark = pytest.mark.gpu


def test_concurrent_calls_agree_with_single_ones():
    beta = np.linspace(0.0, 4.0, 12)
    primes = sk.default_primes()[:3]
    jobs = [lambda: sk.count_ex(0, 12)[1]["residues"],
            lambda: sk.count_ex(1, 14)[1]["residues"],
            lambda: sk.item_residues(2, 12, 9, 5, 3000, primes),
            lambda: sk.item_residues(0, 16, 8, 0, 200000, primes)[-1],   # beyond what the pool keeps
            lambda: sk.pt_run(0, 9, beta, 40, 300, 30, 3, want_final=True)["final_slots"].tolist(),
            lambda: sk.count_inclusion_exclusion(1, 9)[1]["residues"]]
    want = [j() for j in jobs]
    wrong = []

    def work(k):
        for i in range(12):
            j = (k + 5 * i) % len(jobs)
            if jobs[j]() != want[j]:
                wrong.append((k, i, j))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(12)]   # more than the pool's sets
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
