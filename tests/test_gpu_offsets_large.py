"""Chunk offsets of batches of very many requests: the two forms around the size where one takes over, and a cost that
grows no faster than the batch."""
import numpy as np
import pytest
import torch

from paper_2609_38706_gb300 import pk
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu

LIMIT = 360 * 4096  # requests up to which every tile's block reads all the others (csrc/pk_derive.cu)


def offsets(kt, off, idx, n_tokens, D=2):
    tokens = torch.zeros(n_tokens, dtype=torch.int32, device="cuda")
    ko, _ = kt.derive(tokens, off, idx, torch.zeros((D, 32), dtype=torch.uint8, device="cuda"))
    return ko.cpu().numpy(), kt.take_status()


@pytest.mark.parametrize("R", [LIMIT - 1, LIMIT, LIMIT + 1, LIMIT + 4096, 2 * LIMIT + 77])
def test_values_and_bad_requests(R):
    rng = np.random.default_rng(R)
    lens = (rng.random(R) < 0.1) * rng.integers(0, 5, R)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    idx = np.zeros(R, np.uint32)
    kt = KeyTable(2, 4)
    ko, status = offsets(kt, off, idx, int(off[-1]))
    assert status == pk.PK_OK
    assert np.array_equal(ko, np.concatenate([[0], np.cumsum(lens // 2)]))
    for at in (0, R // 2, R - 1):
        bad = idx.copy()
        bad[at] = 2
        ko, status = offsets(kt, off, bad, int(off[-1]))
        assert status == pk.PK_ERR_ARG and not ko.any()
    kt.close()


def test_cost_is_linear():
    """Four times the requests, at most six times the time (16 where every block reads every request)."""
    kt = KeyTable(16, 4)
    tokens = torch.zeros(0, dtype=torch.int32, device="cuda")
    digests = torch.zeros((1, 32), dtype=torch.uint8, device="cuda")
    keys = torch.zeros((0, 32), dtype=torch.uint8, device="cuda")
    ms = []
    for R in (1 << 21, 1 << 23):
        off = torch.zeros(R + 1, dtype=torch.int64, device="cuda")
        idx = torch.zeros(R, dtype=torch.int32, device="cuda")
        ko = torch.zeros(R + 1, dtype=torch.int64, device="cuda")
        best = float("inf")
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            pk.pk_derive_keys(kt.ctx, tokens, off, idx, digests, ko, keys, kt.status)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
    kt.check()
    kt.close()
    assert ms[1] < 6 * ms[0], ms
