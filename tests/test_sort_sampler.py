"""The sampler of the sample sort on the host: a bucket that outgrows shared memory is ranked entry by entry, which is
only right where it hardly ever happens."""
import numpy as np
import pytest

from sorthelpers import bucket_sizes, samples


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("share", [0.002, 0.05, 0.42, 0.76, 0.9, 1.0])
def test_buckets_of_the_longest_lists_fit_shared_memory(form, share):
    n = int(samples(1000)[3 + form] * share)
    room = samples(n)[2]
    for seed in range(4):
        rng = np.random.default_rng(seed)
        for keys in (rng.permutation(n), rng.integers(0, max(2, n // 50), n), (rng.standard_exponential(n) * 1e15).astype(np.int64),
                     np.arange(n)[::-1], np.tile(np.arange(-(-n // 8)), 8)[:n]):
            assert bucket_sizes(keys).max() <= room, (n, seed)


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 511, 512, 513, 5_000, 131_072, 131_073])
def test_samples_are_distinct_positions_of_the_list_in_ascending_order(n):
    at, per = samples(n)[:2]
    assert len(at) == (0 if n <= 256 else per * min(1024, 2 ** int(np.ceil(np.log2(n / 256)))))
    assert len(at) == 0 or (at[0] >= 0 and at[-1] < n and (np.diff(at) > 0).all())
