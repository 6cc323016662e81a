"""The autotuner times the kernel that a batch of the order runs: from n = 13
on the zero-skipping walk, whose rate is 2.4 times the dense walk's at n = 18
(which it timed before, 0.42 of a count's rate), and whose walk width is the
planner's; a batch it tuned keeps the counts and is no slower than the
default one (a tenth is allowed for the spread, the configurations being the
same)."""
import statistics

import pytest

import paper_1507_00315_gb300 as sk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,n", [(0, 18), (1, 17), (2, 16)])
def test_rate_is_the_batch_kernels(variant, n):
    r = sk.autotune(variant, n)
    rep = min((sk.count_ex(variant, n)[1] for _ in range(3)), key=lambda x: x["kernel_ms"])
    assert r["terms_per_s"] >= 0.6 * rep["terms"] / (rep["kernel_ms"] * 1e-3)
    assert r["candidates"] == 2 and r["walk_bits"] == sk.count_plan(variant, n)["walk_bits"]


@pytest.mark.parametrize("n", [12, 13, 31])
def test_ends_of_the_ranges(n):
    r = sk.autotune(1, n)
    assert r["terms_per_s"] > 0 and r["block_threads"] in (128, 256)
    assert (r["candidates"] == 2) == (n >= 13)


@pytest.mark.parametrize("mode", [sk.BATCH_PERSISTENT, sk.BATCH_PER_JOB])
def test_tuned_batch_is_no_slower(mode):
    jobs = [(0, 17), (1, 17), (2, 14), (0, 13)]
    want = sk.count_batch(jobs, mode=mode)[0]
    ms = {}
    for tuned in (False, True):
        assert sk.count_batch(jobs, mode=mode, autotune=tuned)[0] == want
        ms[tuned] = statistics.median(
            sk.count_batch(jobs, mode=mode, autotune=tuned)[2]["kernel_ms"] for _ in range(7))
    assert ms[True] <= 1.1 * ms[False], ms
