"""Chunk offsets of batches around one tile (4,096 requests) and of several: values, and a bad request or descriptor
index in any tile making every offset zero."""
import numpy as np
import pytest
import torch

from paper_2609_38706_gb300 import pk
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


def derive(off, idx, n_tokens, C=3, D=2):
    kt = KeyTable(C, 4)
    tokens = torch.arange(n_tokens, dtype=torch.int32, device="cuda")
    ko, _ = kt.derive(tokens, off, idx, torch.zeros((D, 32), dtype=torch.uint8, device="cuda"))
    status = kt.take_status()
    kt.close()
    return ko.cpu().numpy(), status


@pytest.mark.parametrize("R", [0, 1, 4095, 4096, 4097, 8192, 8193, 20000])
def test_values(R):
    rng = np.random.default_rng(R)
    lens = rng.integers(0, 11, R)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ko, status = derive(off, rng.integers(0, 2, R).astype(np.uint32), max(int(off[-1]), 1))
    assert status == pk.PK_OK
    assert np.array_equal(ko, np.concatenate([[0], np.cumsum(lens // 3)]))


@pytest.mark.parametrize("R", [4096, 12289])
@pytest.mark.parametrize("where", [0.0, 0.4, 0.99])
@pytest.mark.parametrize("what", ["descriptor", "decreasing", "past the tokens"])
def test_bad_requests(R, where, what):
    rng = np.random.default_rng(R)
    lens = rng.integers(1, 11, R)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    idx = np.zeros(R, np.uint32)
    n_tokens = int(off[-1])
    at = int(where * R)
    if what == "descriptor":
        idx[at] = 2
    elif what == "decreasing":
        off[at + 1] = off[at] - 1
    else:
        off[at + 1:] = np.maximum(off[at + 1:], n_tokens + 1)
    ko, status = derive(off, idx, n_tokens)
    assert status == pk.PK_ERR_ARG and not ko.any()
