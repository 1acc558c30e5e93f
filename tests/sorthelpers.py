"""The sampler of the sample sort, as the library's own host code gives it, and the buckets it makes of a list."""
import ctypes

import numpy as np

import paper_2607_07632_b200.sjq as b


def samples(n):
    """Of a list of n entries: sampled positions; samples per bucket; entries of a bucket that shared memory holds; the
    longest lists of the two forms of the sample sort."""
    f = b.lib().sjq_result_sort_samples
    f.argtypes = [ctypes.c_int64, ctypes.c_void_p, ctypes.POINTER(ctypes.c_int32), ctypes.POINTER(ctypes.c_int32),
                  ctypes.POINTER(ctypes.c_int64), ctypes.POINTER(ctypes.c_int64)]
    per, room, little, most = ctypes.c_int32(0), ctypes.c_int32(0), ctypes.c_int64(0), ctypes.c_int64(0)
    refs = [ctypes.byref(v) for v in (per, room, little, most)]
    at = np.zeros(f(n, None, *refs), np.int64)
    assert f(n, at.ctypes.data, *refs) == len(at)
    return at, per.value, room.value, little.value, most.value


def bucket_sizes(keys):
    """Entries per bucket: splitters are every per-th of the sorted sample, by key and then by position."""
    n = len(keys)
    at, per = samples(n)[:2]
    if not len(at):
        return np.array([n])
    order = np.argsort(keys, kind="stable")
    rank = np.empty(n, np.int64)
    rank[order] = np.arange(n)  # equal keys by position
    splitters = np.sort(rank[at])[per::per]
    return np.bincount(np.searchsorted(splitters, rank, side="right"), minlength=len(splitters) + 1)
