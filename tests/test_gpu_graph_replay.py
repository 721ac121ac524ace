"""Calls captured in a CUDA graph and replayed between live calls.  A captured call carries the number of the store
call it was captured as: replayed, it stands for that call again, however many calls came after it."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300 import pk
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


def random_keys(rng, n):
    k = rng.integers(0, 256, (n, 32), dtype=np.uint8)
    k[:, 0] |= 1
    return k


def new(n):
    return torch.zeros(n, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("R,per", [(40, 5), (3, 150)])  # a warp per request, a warp per 32 keys
@pytest.mark.parametrize("mode", ["list", "range", "lookup_store"])
@pytest.mark.parametrize("log2", [12, 7])  # the call fits; it does not
def test_store_again(log2, mode, R, per):
    """Every replay gives the first one's outputs (its keys count as inserted by the call), and the oracle's."""
    n = R * per
    rng = np.random.default_rng(n + log2)
    keys = random_keys(rng, n)
    keys[per:2 * per] = keys[:per]  # duplicates within the call
    before = keys[2 * per:2 * per + 10]
    kt, table = KeyTable(16, log2), O.DictTable(1 << log2)
    new_slots = np.arange(n, dtype=np.uint32) + 1000
    kt.store(before, np.arange(10, dtype=np.uint32))
    table.store(before, np.arange(10, dtype=np.uint32))
    key_off = np.arange(R + 1, dtype=np.int64) * per
    if mode == "list":
        want = table.store(keys, new_slots)
    elif mode == "range":
        want = O.store_misses(table, keys, key_off, np.zeros(R, np.int32), new_slots)
    else:
        hit_w, slots_w = O.lookup(table, keys, key_off)
        want = (hit_w, slots_w, *O.store_misses(table, keys, key_off, hit_w, new_slots))
    kd, sd, od = torch.from_numpy(keys).cuda(), torch.from_numpy(new_slots.view(np.int32)).cuda(), torch.from_numpy(key_off).cuda()
    hit, slots, result, slot_out = new(R), new(n), new(n), new(n)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        if mode == "lookup_store":
            pk.pk_lookup_store(kt.ctx, kd, sd, od, hit, slots, result, slot_out, kt.status)
        else:
            pk.pk_store(kt.ctx, kd, sd, result, slot_out, kt.status, *(() if mode == "list" else (od, hit)))
    for live in range(3):
        if log2 == 12 and live:
            kt.store(random_keys(rng, 20), np.arange(20, dtype=np.uint32) + 100 * live)
        result.fill_(-99)
        slot_out.fill_(-99)
        g.replay()
        torch.cuda.synchronize()
        got = ((hit.cpu().numpy(), slots.cpu().numpy().view(np.uint32)) if mode == "lookup_store" else ()) + (
            result.cpu().numpy(), slot_out.cpu().numpy().view(np.uint32))
        for a, b in zip(got, want):
            assert np.array_equal(a, b), live
        assert kt.entries() == len(table) + (20 * live if log2 == 12 else 0)
    status = kt.take_status()
    assert status == (pk.PK_OK if log2 == 12 else pk.PK_ERR_TABLE_FULL)
    kt.close()


@pytest.mark.parametrize("calls", [4, 300])  # calls before the capture, 25 keys each
@pytest.mark.parametrize("keep", [1, 24, 40, 50, 60, 99, 100, 120, 149])
def test_evict_after_later_calls(keep, calls):
    """An eviction captured before the last stores: the calls after it are the newest."""
    rng = np.random.default_rng(keep)
    n = 25 * (calls + 2)
    keys, slots = random_keys(rng, n), np.arange(n, dtype=np.uint32)
    kt, bt = KeyTable(16, 14), O.BudgetTable(1 << 14)
    kt.attach_stamps()

    def store(a, b):
        kt.store(keys[a:b], slots[a:b])
        bt.store(keys[a:b], slots[a:b])

    for c in range(calls):
        store(25 * c, 25 * c + 25)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ev, n_ev = kt.evict(keep, keep)
    for c in (calls, calls + 1):
        store(25 * c, 25 * c + 25)
    for again in range(2):
        g.replay()
        want = bt.evict(keep, keep)
        torch.cuda.synchronize()
        kt.check("evict")
        assert np.array_equal(np.sort(ev[: int(n_ev.item())].cpu().numpy().view(np.uint32)), want)
        _, got = kt.lookup(torch.from_numpy(keys).cuda(), torch.arange(n + 1, dtype=torch.int64, device="cuda"))
        assert np.array_equal(got.cpu().numpy().view(np.uint32), bt.table.get(keys))
        store(0, 25)
    kt.close()
