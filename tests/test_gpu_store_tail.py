"""Entries past a batch's last key ([key_off[R], key_capacity)) whose buffers hold the bits of an internal state: they
are no keys of the call, so the finalize kernel must take neither their result nor their slot_out at face value and
marks them SKIPPED.  Both forms of it (one and four entries per thread), every mode with request ranges, calls that
insert keys and calls that find them all."""
import numpy as np
import pytest
import torch

from paper_2609_38706_gb300 import pk
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu

PENDING = 0x40000000  # the internal state of a claimed key; also the bits of 2.0f


# a warp per request and a warp per 32 keys, each with one entry per thread in the finalize kernel and with four
@pytest.mark.parametrize("R,per,capacity", [(40, 5, 700), (2000, 3, 400_000), (3, 150, 700), (3, 150, 400_000)])
@pytest.mark.parametrize("mode", ["lookup_store", "store"])
def test_tail_is_skipped(mode, R, per, capacity):
    rng = np.random.default_rng(R)
    total = R * per
    kt = KeyTable(16, 20)
    keys = torch.zeros((capacity, 32), dtype=torch.uint8, device="cuda")
    keys[:total] = torch.from_numpy(rng.integers(0, 256, (total, 32), dtype=np.uint8)).cuda()
    key_off = torch.arange(R + 1, dtype=torch.int64, device="cuda") * per
    new_slots = torch.arange(capacity, dtype=torch.int32, device="cuda")
    hit, slots = (torch.zeros(k, dtype=torch.int32, device="cuda") for k in (R, capacity))
    for expect in (pk.PK_STORE_INSERTED, None):  # inserts every key; finds every key
        result = torch.full((capacity,), PENDING, dtype=torch.int32, device="cuda")
        slot_out = torch.arange(capacity, dtype=torch.int32, device="cuda")  # (positions inside the table)
        if mode == "store":
            hit.zero_()
            pk.pk_store(kt.ctx, keys, new_slots, result, slot_out, kt.status, key_off, hit)
        else:
            pk.pk_lookup_store(kt.ctx, keys, new_slots, key_off, hit, slots, result, slot_out, kt.status)
        kt.check(mode)
        res, out = result.cpu().numpy(), slot_out.cpu().numpy().view(np.uint32)
        if expect is None:
            expect = pk.PK_STORE_PRESENT if mode == "store" else pk.PK_STORE_SKIPPED
        assert (res[:total] == expect).all()
        assert (res[total:] == pk.PK_STORE_SKIPPED).all() and (out[total:] == pk.PK_NO_SLOT).all()
    assert kt.entries() == total
    kt.close()
