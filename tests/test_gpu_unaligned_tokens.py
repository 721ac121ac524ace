"""Chunk digests of token buffers that start at any 4-byte address: each word offset of the buffer and of the requests
in it, chunk sizes around one and several 64-byte blocks, and a last chunk that ends with the buffer."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [8, 16, 17, 32, 47, 48, 64, 80, 256])
@pytest.mark.parametrize("start", [0, 1, 2, 3])
def test_buffer_and_request_offsets(C, start):
    rng = np.random.default_rng(10 * C + start)
    lens = rng.integers(0, 5 * C, 67)
    lens[-1] = 3 * C  # the last chunk ends with the buffer
    off = np.zeros(lens.size + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    tokens = rng.integers(0, 1 << 31, int(off[-1]), dtype=np.int64).astype(np.int32)
    idx = rng.integers(0, 3, lens.size).astype(np.uint32)
    digests = rng.integers(0, 256, (3, 32), dtype=np.uint8)
    buf = torch.empty(tokens.size + start, dtype=torch.int32, device="cuda")
    buf[start:] = torch.from_numpy(tokens).cuda()
    kt = KeyTable(C, 4)
    ko, keys = kt.derive(buf[start:], off, idx, torch.from_numpy(digests).cuda())
    kt.check()
    rko, rkeys = O.derive_keys(tokens, off, C, idx, digests)
    assert np.array_equal(ko.cpu().numpy(), rko)
    assert np.array_equal(keys.cpu().numpy()[: int(rko[-1])], rkeys)
    kt.close()
