"""pk_digest_descriptors into digests at any address, as its interface allows (a slice of a packed buffer): the digests
bit-exact against the oracle, the bytes around them untouched; encodings of one block, of several, and longer than the
kernel's staging area."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300 import pk
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("start", [0, 1, 2, 4, 8, 15, 16])
def test_any_address(start):
    descs = [{"model_id": "m" * n, "weight_precision": "bf16", "weight_version": "v%d" % n, "kv_format": "bf16"}
             for n in (0, 9, 60, 500, 3000)]
    kt = KeyTable(16, 4)
    enc, off = pk.pk_descriptors_encode(descs)
    buf = torch.full((32 * len(descs) + 48,), 0xA5, dtype=torch.uint8, device="cuda")
    end = start + 32 * len(descs)
    assert buf.data_ptr() % 16 == 0
    pk.pk_digest_descriptors(kt.ctx, torch.from_numpy(enc.copy()).cuda(), torch.from_numpy(off).cuda(), buf[start:end],
                             kt.status)
    kt.check()
    got = buf.cpu().numpy()
    assert np.array_equal(got[start:end].reshape(-1, 32), O.descriptor_digests(descs))
    assert (got[:start] == 0xA5).all() and (got[end:] == 0xA5).all()
    kt.close()
