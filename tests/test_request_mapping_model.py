"""Every lane's request by the chunk-digest warps' mapping (csrc/pk_device.cuh, lane_request_guess), in the model of
test_request_mapping_uniform_model.py: a warp's 32 consecutive chunks g0 .. g0+31 need each lane's request r with
key_off[r] <= g < key_off[r+1].  Layouts of equal, ragged, skewed and mostly empty requests."""
import numpy as np
import pytest
from test_request_mapping_uniform_model import warp


def ref(ko, g):
    return int(np.searchsorted(ko, g, side="right") - 1)


def layouts():
    rng = np.random.default_rng(7)
    yield "equal", np.full(3000, 128)
    yield "equal, few", np.full(5, 40)
    yield "one request", np.array([1000])
    n = rng.integers(0, 9, 4000)
    n[rng.integers(0, 4000, 1500)] = 0
    yield "ragged with empties", n
    n = rng.integers(0, 3, 3000)
    n[rng.integers(0, 3000, 12)] = rng.integers(200, 400, 12)
    yield "skewed", n
    n = np.zeros(6000, np.int64)
    i = 0
    while i < n.size:
        n[i] = rng.integers(1, 6)
        i += 1 + (int(rng.integers(40, 200)) if rng.random() < 0.3 else 0)
    yield "runs of empty requests", n
    n = np.zeros(300, np.int64)
    n[-1] = 50
    yield "empties then one", n


@pytest.mark.parametrize("name,n", list(layouts()), ids=[name for name, _ in layouts()])
def test_every_lane_maps_to_its_request(name, n):
    n = np.asarray(n, np.int64)
    R = n.size
    ko = np.zeros(R + 1, np.int64)
    np.cumsum(n, out=ko[1:])
    total = int(ko[-1])
    paths = set()
    for g0 in range(0, total, 32):
        path, requests = warp(ko, R, g0, total)
        paths.add(path)
        for lane in range(min(32, total - g0)):
            g, r = g0 + lane, int(requests[lane])
            assert r == ref(ko, g), (name, g0, lane, path)
            assert ko[r] <= g < ko[r + 1]
    assert paths, name


def test_all_three_paths_are_reached():
    reached = set()
    for name, n in layouts():
        n = np.asarray(n, np.int64)
        ko = np.zeros(n.size + 1, np.int64)
        np.cumsum(n, out=ko[1:])
        for g0 in range(0, int(ko[-1]), 32):
            reached.add(warp(ko, n.size, g0, int(ko[-1]))[0])
    assert reached == {"guess", "window", "search"}
