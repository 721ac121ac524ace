"""Digests of few chunks and few tree blocks, by pairs of warps: counts around a pair (16) and around the largest batch
that pairs serve (48 per SM, less the SMs of the descriptors), chunk sizes with every form of last block, and tree
levels that end inside a word."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300 import pk
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


def descriptors(D):
    return [{"model_id": "m", "weight_precision": "bf16", "weight_version": "v", "adapter_id": "a%d" % j, "kv_format": "bf16",
             "salt": "s" * j} for j in range(D)]


def check(N, C, D, seed):
    """N chunks in requests of 0 to 3, derived with the descriptors' encodings and with their digests."""
    rng = np.random.default_rng(seed)
    per = []
    while sum(per) < N:
        per.append(min(int(rng.integers(0, 4)), N - sum(per)))
    per = np.array(per + [0])
    lens = per * C + rng.integers(0, C, per.size)
    off = np.zeros(lens.size + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    tokens = rng.integers(0, 1 << 31, int(off[-1]), dtype=np.int64).astype(np.int32)
    tokens = tokens[: int(off[-1])]
    idx = rng.integers(0, D, per.size).astype(np.uint32)
    descs = descriptors(D)
    want_d = O.descriptor_digests(descs)
    rko, rkeys = O.derive_keys(tokens, off, C, idx, want_d)
    assert rkeys.shape[0] == N
    kt = KeyTable(C, 4)
    digests, ko, keys = kt.derive_enc(tokens, off, idx, descs)
    assert np.array_equal(digests.cpu().numpy(), want_d)
    assert np.array_equal(ko.cpu().numpy(), rko) and np.array_equal(keys.cpu().numpy()[:N], rkeys)
    ko, keys = kt.derive(tokens, off, idx, digests)
    assert np.array_equal(ko.cpu().numpy(), rko) and np.array_equal(keys.cpu().numpy()[:N], rkeys)
    kt.check()
    kt.close()


@pytest.mark.parametrize("N", [1, 2, 15, 16, 17, 47, 48, 49, 100])
@pytest.mark.parametrize("C", [1, 13, 14, 15, 16, 29, 30, 31, 32, 64, 256])
def test_few_chunks(N, C):
    check(N, C, 3, 1000 * N + C)


@pytest.mark.parametrize("past", [-1, 0, 1])
@pytest.mark.parametrize("D", [1, 13, 40])
def test_largest_batch_of_pairs(D, past):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    check(48 * (sms - 1 - (D + 3) // 4) + past, 1, D, 10 * D + past)


@pytest.mark.parametrize("sizes", [[0], [1], [1023], [1024, 1025, 1027, 3], [15 * 1024 + 61, 17 * 1024 + 2, 40 * 1024],
                                   [48 * 152 * 1024 - 1], [48 * 152 * 1024 + 1], [33 * 1024 + 5] * 150])
def test_tree_levels(sizes):
    rng = np.random.default_rng(len(sizes) + sizes[0])
    data = [rng.integers(0, 256, n, dtype=np.uint8) for n in sizes]
    dev = [torch.from_numpy(d).cuda() for d in data]
    scratch = torch.empty(max(pk.pk_content_scratch_bytes_batch(sizes), 16), dtype=torch.uint8, device="cuda")
    tops = torch.zeros((len(sizes), 32), dtype=torch.uint8, device="cuda")
    pk.pk_content_digests(dev, scratch, tops)
    got = tops.cpu().numpy()
    for j, d in enumerate(data):
        assert bytes(got[j]) == bytes(O.content_digest(d)), sizes[j]
