"""The chain's layouts (two lanes per request with one, three or four pairs of warps per CTA, one lane per request) at the
edges of their ranges: requests per pair (16), pairs per SM (2, 3, 4), uneven and empty requests."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


def check(R, C, max_chunks, seed):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, max_chunks * C + C, R)
    lens[rng.integers(0, R)] = max_chunks * C  # at least one request of the largest size
    off = np.zeros(R + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    tokens = rng.integers(0, 1 << 31, int(off[-1]), dtype=np.int64).astype(np.int32)
    D = 5
    idx = rng.integers(0, D, R).astype(np.uint32)
    digests = rng.integers(0, 256, (D, 32), dtype=np.uint8)
    kt = KeyTable(C, 4)
    ko, keys = kt.derive(tokens, off, idx, torch.from_numpy(digests).cuda())
    kt.check()
    rko, rkeys = O.derive_keys(tokens, off, C, idx, digests)
    assert np.array_equal(ko.cpu().numpy(), rko)
    assert np.array_equal(keys.cpu().numpy()[: int(rko[-1])], rkeys)
    kt.close()


@pytest.mark.parametrize("R", [1, 2, 15, 16, 17, 31, 33])
@pytest.mark.parametrize("max_chunks", [1, 2, 3, 9])
def test_few_requests(R, max_chunks):
    check(R, 4, max_chunks, 100 * R + max_chunks)


@pytest.mark.parametrize("pairs_per_sm", [1, 2, 3, 4])
@pytest.mark.parametrize("past", [-1, 0, 1])
def test_layout_boundaries(pairs_per_sm, past):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    check(16 * sms * pairs_per_sm + past, 2, 3, 7 * pairs_per_sm + past)
