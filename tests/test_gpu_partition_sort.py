"""The hash partition's lists at the edges of its counting sort: tensors around one and two
hash tiles of 16,384 elements, stretches of 64 elements a thread, shifts (K a power of two)
and multiplies, and tables of many tensors (the owner search)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 3, 32, 33, 63, 64])
@pytest.mark.parametrize("numel", [[16_383], [16_384, 1], [16_385, 63, 64, 65], [32_768 + 5, 0, 4_097]])
def test_lists_match_the_oracle(K, numel):
    from paper_2608_02391_gb300 import copes
    layout = copes.Layout(numel)
    subs = copes.hash_partition(layout, K, 1088)
    for k in range(K):
        want = oracle.hash_list(numel, range(len(numel)), K, 1088, k)
        assert np.array_equal(subs[k].tensor.cpu().numpy(), want), k
    copes.check()


@pytest.mark.parametrize("n_tensors", [31, 32, 33, 1025, 2000])
def test_many_tensors(n_tensors):
    from paper_2608_02391_gb300 import copes
    numel = [1 + (37 * t) % 90 for t in range(n_tensors)]
    subs = copes.hash_partition(copes.Layout(numel), 4, 7)
    for k in range(4):
        want = oracle.hash_list(numel, range(n_tensors), 4, 7, k)
        assert np.array_equal(subs[k].tensor.cpu().numpy(), want), k
    copes.check()


@pytest.mark.parametrize("n_tensors,K", [(4096, 3), (4097, 3), (8 * 4096, 16), (8 * 4096 + 1, 16), (24 * 4096, 3),
                                         (12_289, 64), (20_481, 64), (1025 * 1024 + 5, 3)])
def test_many_hash_tiles(n_tensors, K):
    """A tensor takes a hash tile at least: one chunk of the scan over the tiles, several, on both
    sides of where chunks are summed first, and more than their scan takes in a step."""
    from paper_2608_02391_gb300 import copes
    numel = np.ones(n_tensors, np.int64)
    subs = copes.hash_partition(copes.Layout(numel), K, 7)
    for k in range(K):
        want = oracle.hash_list(numel, range(n_tensors), K, 7, k)
        assert np.array_equal(subs[k].tensor.cpu().numpy(), want), k
    copes.check()
