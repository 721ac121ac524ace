"""CPU model of the chunk-to-request mapping (csrc/pk_device.cuh, lane_request_guess): every lane of every warp against
searchsorted, on layouts that reach each of its ways out (the guess, the window from the first item's request, the
binary search past it)."""
import numpy as np
import pytest


def window(key_off, R, w0, g0):
    at = w0 + np.arange(32)
    d = np.where(at <= R, key_off[np.minimum(at, R)] - g0, np.iinfo(np.int64).max)
    return np.clip(d, 0, 32)


def warp(key_off, R, g0, total):
    lane = np.arange(32)
    l = np.minimum(g0 + lane, total - 1) - g0
    last = min(total - g0, 32) - 1
    rg = min(int(np.float32(np.float32(g0) / np.float32(total)) * np.float32(R)), R - 1)
    w0 = rg - 8 if rg > 8 else 0
    p = window(key_off, R, w0, g0)
    among = (p >= 1) & (p <= 31)
    places = np.unique(p[among])
    if p[0] == 0 and (p > last).any() and places.size == among.sum():
        return "guess", w0 + (p == 0).sum() - 1 + (places[None, :] <= l[:, None]).sum(1)
    r0, span = 0, R
    while span > 1:
        step = (span + 31) // 32
        c = r0 + (lane + 1) * step
        ok = (c < R) & (key_off[np.minimum(c, R)] <= g0)
        assert not (np.diff(ok.astype(int)) > 0).any()  # a prefix of the lanes
        r0 += step * int(ok.sum())
        span = step
    p = window(key_off, R, r0 + 1, g0)
    lo, hi = np.zeros(32, int), np.full(32, 32)
    for _ in range(6):
        mid = (lo + hi) >> 1
        pm = p[np.minimum(mid, 31)]
        up = (lo < hi) & (pm <= l)
        hi = np.where((lo < hi) & ~up, mid, hi)
        lo = np.where(up, mid + 1, lo)
    if (lo < 32).all():
        return "window", r0 + lo
    r, n = np.full(32, r0), R - r0
    while n > 1:
        h = n >> 1
        r = np.where(key_off[r + h] <= g0 + l, r + h, r)
        n -= h
    return "search", r


def layouts():
    rng = np.random.default_rng(0)
    yield "equal", np.full(500, 32)
    yield "one request", np.array([1000])
    yield "one chunk each", np.ones(4000, int)
    yield "three each", np.full(1000, 3)
    yield "uneven", rng.integers(1, 200, 700)
    yield "some empty", rng.integers(0, 4, 3000)
    yield "mostly empty", (rng.random(5000) < 0.02) * rng.integers(1, 5, 5000)
    yield "runs of empty", np.concatenate([np.zeros(70, int), [5], np.zeros(40, int), [1], np.zeros(33, int), [40], np.zeros(100, int), [2, 1]])
    yield "few long, many short", np.concatenate([rng.integers(1, 3, 900), [5000], rng.integers(1, 3, 900)])
    yield "long first", np.concatenate([[30000], np.ones(1000, int), np.zeros(50, int)])


def test_every_lane_of_every_warp():
    seen = set()
    for name, n in layouts():
        key_off = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
        R, total = n.size, int(key_off[-1])
        for g0 in range(0, total, 32):
            way, r = warp(key_off, R, g0, total)
            seen.add(way)
            g = np.minimum(g0 + np.arange(32), total - 1)
            want = np.searchsorted(key_off, g, side="right") - 1
            assert np.array_equal(r, want), (name, g0, way)
    assert seen == {"guess", "window", "search"}


@pytest.mark.parametrize("R", [1, 2, 31, 32, 33, 1023, 1024, 1025, 4097])
def test_searches_of_every_size(R):
    rng = np.random.default_rng(R)
    key_off = np.concatenate([[0], np.cumsum(rng.integers(0, 3, R))]).astype(np.int64)
    key_off[-1] = max(key_off[-1], 1)
    total = int(key_off[-1])
    for g0 in range(0, total, 32):
        r = warp(key_off, R, g0, total)[1]
        g = np.minimum(g0 + np.arange(32), total - 1)
        assert np.array_equal(r, np.searchsorted(key_off, g, side="right") - 1)
