"""The chains' order of a CTA's requests, longest first: every layout that sorts (three and four pairs of two lanes per
request, four pairs of one lane), full and partly filled CTAs, for lengths that are equal, rising, falling, mostly
empty, one long among short, and of few distinct values.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


def chunk_counts(pattern, R, rng):
    i = np.arange(R)
    return {"equal": np.full(R, 3), "rising": i * 5 // R, "falling": 5 - i * 5 // R, "few": rng.integers(0, 2, R),
            "empty": (i % 61 == 60) * 4, "one_long": 1 + (i == R - 1) * 30}[pattern]


@pytest.mark.parametrize("pattern", ["equal", "rising", "falling", "few", "empty", "one_long"])
@pytest.mark.parametrize("per_sm,past", [(48, -17), (48, 0), (64, 0), (64, -33), (64, 1), (128, 0), (128, 5)])
def test_order(per_sm, past, pattern):
    C, D = 2, 3
    R = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + past
    rng = np.random.default_rng(per_sm * 100 + past)
    lens = chunk_counts(pattern, R, rng) * C + rng.integers(0, C, R)
    off = np.zeros(R + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    tokens = rng.integers(0, 1 << 31, int(off[-1]), dtype=np.int64).astype(np.int32)
    idx = rng.integers(0, D, R).astype(np.uint32)
    digests = rng.integers(0, 256, (D, 32), dtype=np.uint8)
    kt = KeyTable(C, 4)
    ko, keys = kt.derive(tokens, off, idx, torch.from_numpy(digests).cuda())
    kt.check()
    rko, rkeys = O.derive_keys(tokens, off, C, idx, digests)
    assert np.array_equal(ko.cpu().numpy(), rko)
    assert np.array_equal(keys.cpu().numpy()[: int(rko[-1])], rkeys)
    kt.close()
