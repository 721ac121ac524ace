"""Compaction with several threads per bitmap word, one thread per word, and more words than threads: tables of 64 to
2^23 entries, at loads that give clusters within a part, across parts and across words, with evictions spread over the
table.  Every key's slot against the oracle's BudgetTable."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


def check(log2, n, seed):
    rng = np.random.default_rng(seed)
    keys = rng.integers(0, 256, (n, 32), dtype=np.uint8)
    keys[:, 0] |= 1
    slots = np.arange(n, dtype=np.uint32)
    kt, bt = KeyTable(16, log2), O.BudgetTable(1 << log2)
    kt.attach_stamps()
    for part in np.array_split(np.arange(n), 3):
        kt.store(torch.from_numpy(keys[part]).cuda(), slots[part])
        bt.store(keys[part], slots[part])
    keep = n - max(1, n // 4)
    ev, n_ev = kt.evict(keep, keep)
    want = bt.evict(keep, keep)
    torch.cuda.synchronize()
    kt.check("evict")
    assert np.array_equal(np.sort(ev[: int(n_ev.item())].cpu().numpy().view(np.uint32)), want)
    off = torch.arange(0, n + 1, dtype=torch.int64, device="cuda")
    _, got = kt.lookup(torch.from_numpy(keys).cuda(), off)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), bt.table.get(keys))
    kt.close()


@pytest.mark.parametrize("load", [0.3, 0.6, 0.85])
@pytest.mark.parametrize("log2", [6, 9, 13, 16, 19, 20, 21])
def test_table_sizes(log2, load):
    check(log2, min(int(load * (1 << log2)), 700000), log2 * 100 + int(load * 100))


def test_more_words_than_threads():
    threads = torch.cuda.get_device_properties(0).multi_processor_count * 2 * 512
    log2 = 23
    while (1 << log2) // 32 <= threads:
        log2 += 1
    check(log2, 400000, log2)
