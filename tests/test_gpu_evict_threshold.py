"""Where an eviction's threshold falls: at the end of a call's entries (read off the age histogram), one entry before
or after it (the call's stamps split by key index), in calls older than the histogram's last bin, and among entries
without a stamp; each against the oracle's BudgetTable."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


def fill(log2, calls, per_call, unstamped, seed):
    rng = np.random.default_rng(seed)
    keys = rng.integers(0, 256, (unstamped + calls * per_call, 32), dtype=np.uint8)
    keys[:, 0] |= 1
    kt, bt = KeyTable(16, log2), O.BudgetTable(1 << log2)
    slots = np.arange(keys.shape[0], dtype=np.uint32)

    def store(a, b):
        kt.store(torch.from_numpy(keys[a:b]).cuda(), slots[a:b])
        bt.store(keys[a:b], slots[a:b])

    if unstamped:
        store(0, unstamped)
        bt.stamps.clear()
    kt.attach_stamps()
    for c in range(calls):
        store(unstamped + c * per_call, unstamped + (c + 1) * per_call)
    return kt, bt, keys


@pytest.mark.parametrize("calls,per_call,unstamped", [(1, 1500, 0), (5, 400, 0), (4, 300, 100), (300, 7, 0), (520, 4, 50)])
@pytest.mark.parametrize("gone", ["boundary", "before", "after", "inside", "one", "all but one"])
def test_threshold_places(calls, per_call, unstamped, gone):
    kt, bt, keys = fill(12, calls, per_call, unstamped, calls)
    n = keys.shape[0]
    edge = unstamped + max(1, calls // 3) * per_call  # entries up to the end of a call
    k = {"boundary": edge, "before": edge - 1, "after": edge + 1, "inside": unstamped + per_call // 2 + 1, "one": 1,
         "all but one": n - 1}[gone]
    k = min(k, n - 1)
    ev, n_ev = kt.evict(n - k, n - k)
    want = bt.evict(n - k, n - k)
    torch.cuda.synchronize()
    kt.check("evict")
    got = np.sort(ev[: int(n_ev.item())].cpu().numpy().view(np.uint32))
    assert np.array_equal(got, want)
    off = torch.arange(0, n + 1, dtype=torch.int64, device="cuda")
    _, slots = kt.lookup(torch.from_numpy(keys).cuda(), off)
    assert np.array_equal(slots.cpu().numpy().view(np.uint32), bt.table.get(keys))
    kt.close()
