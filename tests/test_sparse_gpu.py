"""The zero-skipping walk and split work items on the GPU: whole counts
(tiles) against the same counts in ragged parts (the dense walk), aligned
chunks of large orders against the dense walk's item residues, and items that
a launch splits over several lanes against the oracle's block sums."""
import pytest

import oracle
import paper_1507_00315_gb300 as sk

pytestmark = pytest.mark.gpu
SK, LA, HO = 0, 1, 2


@pytest.mark.parametrize("variant", [SK, LA, HO])
@pytest.mark.parametrize("n", [13, 14, 15])
def test_whole_count_equals_ragged_parts(variant, n, tmp_path):
    primes = sk.default_primes()
    whole = sk.count_ex(variant, n, primes=primes, nprimes=4)[1]["residues"]
    path = str(tmp_path / "parts.txt")
    items = sk.count_plan(variant, n)["items"]
    # an odd number of items a launch: never an aligned power-of-two block
    parts = sk.count_ex(variant, n, primes=primes, nprimes=4, checkpoint=path,
                        chunk_items=items // 3 - 1)[1]
    assert parts["chunks_total"] == 4 and parts["residues"] == whole
    assert sk.count_ex(variant, n, primes=primes, nprimes=4,
                       symmetry=sk.SYMMETRY_NEGATION_EVEN)[1]["residues"] in (whole, [0] * 4)
    for kw in ({"block_threads": 32}, {"block_threads": 160, "grid": 3}, {"grid": 1}):
        assert sk.count_ex(variant, n, primes=primes, nprimes=4, **kw)[1]["residues"] == whole, kw


@pytest.mark.parametrize("variant,n,m,lg", [(SK, 20, 14, 17), (LA, 21, 14, 18), (HO, 22, 15, 18),
                                            (SK, 24, 17, 17), (LA, 25, 17, 19)])
def test_aligned_chunk_equals_the_items(variant, n, m, lg, tmp_path):
    # the first chunk of a checkpointed run (2^(m + lg) terms, tiles) and the
    # residues of its work items (dense walk) added up
    primes = sk.default_primes()[:3]
    path = str(tmp_path / "chunk.txt")
    sk.count_ex(variant, n, primes=primes, checkpoint=path, walk_bits=m, chunk_items=1 << lg,
                max_chunks=1)
    chunk = [int(v) for v in open(path).read().splitlines()[1].split()[2:5]]
    items = sk.item_residues(variant, n, m, 0, 1 << lg, primes)
    assert chunk == [sum(r[i] for r in items) % p for i, p in enumerate(primes)]


@pytest.mark.parametrize("m", [9, 10, 12, 13])
@pytest.mark.parametrize("count", [1, 3, 33])
def test_split_items_equal_the_oracle(m, count):
    n = 12
    primes = sk.default_primes()[:3]
    q = (1 << (2 * n - 1 - m)) - count - 2
    want = [[oracle.partial_sum_mod(SK, n, m, q + i, p) for p in primes] for i in range(count)]
    assert sk.item_residues(SK, n, m, q, count, primes) == want
    assert sk.item_residues(SK, n, m, q, count, primes, arith=sk.ARITH_MONTGOMERY) == want
    assert sk.item_residues_noalloc(SK, n, m, q, count, primes) == want
    ie = [[oracle.ie_partial_sum_mod(LA, n, m, q + i, p) for p in primes] for i in range(count)]
    assert sk.ie_item_residues(LA, n, m, q, count, primes) == ie
