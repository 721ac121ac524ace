"""Key derivation into buffers sized for a far larger batch: the keys bit-exact, nothing written past them, and the time
that of the batch, whose forms and grids follow its tokens and not the buffers."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300 import pk
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


def batch(lens, C, D=3):
    rng = np.random.default_rng(len(lens) + C)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    tokens = rng.integers(0, 1 << 31, int(off[-1]), dtype=np.int64).astype(np.int32)
    idx = rng.integers(0, D, len(lens)).astype(np.int32)
    digests = rng.integers(0, 256, (D, 32), dtype=np.uint8)
    return tokens, off, idx, digests


@pytest.mark.parametrize("capacity", [1 << 12, 1 << 18])
@pytest.mark.parametrize("lens,C", [([5, 0, 3], 8), ([64] * 20, 16), ([0, 0], 4), ([], 4), ([300] * 40, 17), ([70000] * 3, 16)])
def test_keys(lens, C, capacity):
    tokens, off, idx, digests = batch(lens, C)
    capacity += tokens.size // C
    kt = KeyTable(C, 4)
    key_off = torch.full((len(lens) + 1,), -1, dtype=torch.int64, device="cuda")
    keys = torch.full((capacity, 32), 0xA5, dtype=torch.uint8, device="cuda")
    pk.pk_derive_keys(kt.ctx, torch.from_numpy(tokens).cuda(), torch.from_numpy(off).cuda(), torch.from_numpy(idx).cuda(),
                      torch.from_numpy(digests).cuda(), key_off, keys, kt.status)
    kt.check()
    rko, rkeys = O.derive_keys(tokens, off, C, idx.view(np.uint32), digests)
    n, got = int(rko[-1]), keys.cpu().numpy()
    assert np.array_equal(key_off.cpu().numpy(), rko)
    assert np.array_equal(got[:n], rkeys[:n]) and (got[n:] == 0xA5).all()
    kt.close()


def test_time_is_the_batch_s():
    """64 prompts of 512 tokens, into buffers of exactly their keys and of 2^24: at most half as long again (with a
    grid for the buffers, three times as long)."""
    C = 16
    tokens, off, idx, digests = (torch.from_numpy(x).cuda() for x in batch([512] * 64, C))
    kt = KeyTable(C, 4)
    us = []
    for capacity in (64 * 32, 1 << 24):
        key_off = torch.zeros(65, dtype=torch.int64, device="cuda")
        keys = torch.zeros((capacity, 32), dtype=torch.uint8, device="cuda")
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                pk.pk_derive_keys(kt.ctx, tokens, off, idx, digests, key_off, keys, kt.status)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 50)
        us.append(best)
    kt.check()
    kt.close()
    print("us:", us)
    assert us[1] < 1.5 * us[0], us
