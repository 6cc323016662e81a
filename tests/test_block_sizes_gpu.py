"""A caller's block size neither changes a count nor makes the zero-skipping
walk (n >= 13) slow: its warps share tables of 54 KB a CTA, so blocks of the
size asked for would leave most of an SM idle (a count at 32 threads took 3.2
times the default's time, a batch 3.6 times).  Kernel times, medians of five,
with half as much again allowed for their spread."""
import statistics

import pytest

import paper_1507_00315_gb300 as sk

pytestmark = pytest.mark.gpu


def _median(call):
    call()
    return statistics.median(call() for _ in range(5))


@pytest.mark.parametrize("symmetry", [sk.SYMMETRY_NEGATION, sk.SYMMETRY_REVERSAL])
def test_counts(symmetry):
    want = sk.count_ex(1, 16, symmetry=symmetry)[0]
    usual = _median(lambda: sk.count_ex(1, 16, symmetry=symmetry)[1]["kernel_ms"])
    for threads in (32, 64, 224, 256):
        kw = dict(symmetry=symmetry, block_threads=threads)
        assert sk.count_ex(1, 16, **kw)[0] == want
        assert _median(lambda: sk.count_ex(1, 16, **kw)[1]["kernel_ms"]) <= 1.5 * usual, threads


@pytest.mark.parametrize("mode", [sk.BATCH_PERSISTENT, sk.BATCH_PER_JOB])
def test_batches(mode):
    jobs = [(0, 16), (1, 16), (2, 15), (0, 9)]
    want = sk.count_batch(jobs, mode=mode)[0]
    usual = _median(lambda: sk.count_batch(jobs, mode=mode)[2]["kernel_ms"])
    for threads in (32, 64, 128):
        kw = dict(mode=mode, block_threads=threads)
        assert sk.count_batch(jobs, **kw)[0] == want
        assert _median(lambda: sk.count_batch(jobs, **kw)[2]["kernel_ms"]) <= 1.5 * usual, threads
