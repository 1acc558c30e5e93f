"""Canonical order of hashed results at the sizes and key ranges where the sample sort and the radix sort take another
path: one tile, one more, the most pieces, every number of digit passes, equal keys, lists in order already, buckets
beyond shared memory and bins of bunched keys."""
import numpy as np
import pytest
import torch

import paper_2607_07632_b200 as sjq
from sorthelpers import bucket_sizes, samples

pytestmark = pytest.mark.gpu


def _check(keys, capacity):
    n = len(keys)
    rng = np.random.default_rng(n)
    allk = np.full(capacity, 5, dtype=np.int64)
    allk[:n] = keys
    sums, counts = rng.integers(-2**62, 2**62, capacity), rng.integers(0, 2**40, capacity)
    res = sjq.Result("HASHED", torch.from_numpy(sums).cuda(), torch.from_numpy(counts).cuda(),
                     torch.from_numpy(allk.copy()).cuda(), torch.tensor([n], dtype=torch.int64, device="cuda"),
                     torch.zeros(1, dtype=torch.int32, device="cuda"), None)
    res.sort()
    order = np.concatenate([np.argsort(keys, kind="stable"), np.arange(n, capacity)])
    for got, want in ((res.keys, allk), (res.sums, sums), (res.counts, counts)):
        assert np.array_equal(got.cpu().numpy(), want[order])


@pytest.mark.parametrize("n", [2, 31, 255, 256, 257, 512, 513, 2047, 2048, 2049, 4095, 4096, 4097, 148 * 2048 - 1, 148 * 2048 + 1,
                               148 * 4096 + 33, 2**20 - 7, 2**20 - 6, 2_000_003])
def test_list_lengths_around_pieces_and_tiles(n):
    keys = np.random.default_rng(n).permutation(n).astype(np.int64) * 0x9E3779B97F4A7 - 2**40
    _check(keys, n + 7)


@pytest.mark.parametrize("bits", [1, 8, 9, 16, 24, 33, 40, 48, 56, 63])
@pytest.mark.parametrize("capacity", [32_768, 2**20, 2**20 + 1])  # sample sort in one and in either kernel; radix sort
def test_every_number_of_passes_with_equal_keys(bits, capacity):
    n = 20_011
    rng = np.random.default_rng(bits)
    lo = -(2**(bits - 1)) + 12_345
    keys = rng.integers(0, 2**bits - 1, n, endpoint=True, dtype=np.int64) + np.int64(lo)
    keys[:2] = lo, lo + 2**bits - 1  # the whole range, so that the pass count is the intended one
    keys[100:5_000] = keys[7]
    _check(keys, capacity)


@pytest.mark.parametrize("capacity", [300_000, 700_000, 2**20 + 5])
def test_clustered_keys_and_a_lone_outlier(capacity):
    rng = np.random.default_rng(4)
    keys = np.concatenate([rng.permutation(100_000), rng.permutation(100_000) + 2**50, [-2**63, 2**63 - 1],
                           np.full(3_000, 77), 2**62 + 2**40 * rng.integers(0, 50, 5_000)]).astype(np.int64)
    _check(rng.permutation(keys), capacity)
    _check(np.sort(keys)[::-1].copy(), capacity)


def test_buckets_larger_than_shared_memory_are_ranked():
    # the sampled positions hold small keys only: all other entries fall into one bucket
    n = 40_000
    keys = np.random.default_rng(1).permutation(n).astype(np.int64) + 10**6
    at = samples(n)[0]
    keys[at] = np.arange(len(at))
    assert bucket_sizes(keys).max() > 10 * samples(n)[2]
    _check(keys, n)


def test_list_in_order_and_list_of_equal_keys_stay_as_they_are():
    _check(np.arange(100_000, dtype=np.int64) * 3 - 150_000, 131_072)
    _check(np.full(10_000, -9, dtype=np.int64), 10_000)
    swapped = np.arange(60_000, dtype=np.int64)
    swapped[[2047, 2048]] = swapped[[2048, 2047]]  # out of order only across a piece's edge
    _check(swapped, 60_000)


@pytest.mark.parametrize("last", [200, 256, 257, 496, 512, 513, 1500, 2048, 2049])
@pytest.mark.parametrize("bunch", [1, 64, 65, 66])
def test_one_bucket_of_spread_and_of_bunched_keys(last, bunch):
    # the sampled positions hold the smallest keys, so all others share the last bucket with the samples behind the last
    # splitter: `last` entries in all; `bunch` neighbours lie in one bin of the bucket's range
    n = next(n for n in range(last, 2 * last) if n - len(samples(n)[0]) + (samples(n)[1] if n > 256 else 0) == last)
    rng = np.random.default_rng(n + bunch)
    keys = (rng.permutation(n).astype(np.int64) + 10**6) << 40
    bunched = rng.choice(n, bunch, replace=False)
    keys[bunched] = (np.int64(2**62)) + rng.permutation(bunch)
    keys[bunched[: bunch // 8]] = 2**62 + 3  # equal ones keep their order
    at = samples(n)[0]
    keys[at] = np.arange(len(at))
    assert bucket_sizes(keys)[-1] == last
    _check(keys, n + 1)


@pytest.mark.parametrize("last", [200, 1024, 1025, 2048, 2049, 4096, 4097, 8192, 8193])
@pytest.mark.parametrize("bunch", [1, 64, 65, 66, 180])
def test_one_bucket_of_a_long_list(last, bunch):
    # 430,000 entries, whose buckets the larger blocks sort: samples at equal distances, `last` entries beyond the last
    # splitter, `bunch` of them neighbours, all others below it
    n, rng = 430_000, np.random.default_rng(last + bunch)
    at, per = samples(n)[:2]
    assert n > samples(n)[3]
    top, inside = (len(at) - per) << 40, last - per
    rest = rng.permutation(np.setdiff1d(np.arange(n), at))
    keys = np.empty(n, np.int64)
    keys[at] = np.arange(len(at)) << 40
    keys[rest[inside:]] = rng.integers(0, top, n - len(at) - inside)
    keys[rest[:inside]] = top + 1 + rng.permutation(inside) * (2**42 // inside)
    keys[rest[:bunch]] = top + 2**41 + rng.permutation(bunch)
    keys[rest[: bunch // 8]] = top + 2**41 + 3  # equal ones keep their order
    assert bucket_sizes(keys)[-1] == last
    _check(keys, n + 1)


@pytest.mark.parametrize("form", [3, 4])
@pytest.mark.parametrize("beyond", [-7, -6, 200_000])
def test_unordered_lists_on_both_sides_of_the_longest_of_either_form(form, beyond):
    n = samples(1000)[form] + beyond
    keys = np.random.default_rng(n).permutation(n).astype(np.int64) * 0x9E3779B97F4A7 - 2**40
    _check(keys, n + 7)


@pytest.mark.parametrize("n", [1, 2, 300, 5_000, 418_816, 418_817])
def test_lists_shorter_than_their_capacity(n):
    rng = np.random.default_rng(n)
    for capacity in (500_000, 2**20):
        _check(rng.permutation(n).astype(np.int64) * 0x9E3779B97F4A7 - 2**40, capacity)
        _check(np.arange(n, dtype=np.int64), capacity)
        _check(rng.integers(0, 9, n), capacity)
        _check((np.arange(n) // 200 * 2**33 + rng.integers(0, 100, n))[rng.permutation(n)], capacity)  # bunched
