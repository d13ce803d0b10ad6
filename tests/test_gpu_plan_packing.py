"""Whole series are packed into bins of warps, larger first, each into the first
bin with room: as many bins as the plain search over all bins makes, in time that
does not grow with their number squared."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def first_fit(need, warps):
    room = []
    for w in sorted(need, reverse=True):
        k = next((i for i, r in enumerate(room) if r >= w), None)
        if k is None:
            room.append(warps)
            k = len(room) - 1
        room[k] -= w
    return len(room)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,lo,hi", [(2, 1, 1), (50, 100, 900), (700, 10, 3000), (3000, 1, 640)])
def test_bins_of_the_first_fit(prec, n, lo, hi):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    T = np.random.default_rng(n).integers(lo, hi + 1, n)
    off = np.concatenate([[0], np.cumsum(T)])
    i = rsv.Plan(ctx, off, 10, prec=prec).info()
    whole = T[T <= i["threads"] * i["sites_per_thread"]]
    split = T[T > i["threads"] * i["sites_per_thread"]]
    tile = i["threads"] * i["sites_per_thread"] - 2 * 11 - 3
    bins = first_fit(-(-whole // (32 * i["sites_per_thread"])), i["threads"] // 32) + int((-(-split // tile)).sum())
    assert i["bins"] == bins and i["split_series"] == len(split)
    ctx.close()


def test_many_bins_are_packed_quickly():
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    off = np.concatenate([[0], np.cumsum(np.random.default_rng(0).integers(300, 641, 100000))])
    rsv.Plan(ctx, off[:3], 10)
    t = time.perf_counter()
    rsv.Plan(ctx, off, 10).close()      # 25 000 bins: 3e8 steps by the search over all of them
    assert time.perf_counter() - t < 0.3
    ctx.close()
