"""KeyTable.derive_lookup_store's descriptor encodings: copied in stream order without a synchronisation, so that
calls in flight keep their own; every form a field may have; none at all; refusals."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300 import pk
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu


def desc(rng, j, extra):
    d = {"model_id": "org/modèle-%d" % j, "weight_precision": "BF16",
         "weight_version": bytes(rng.integers(0, 256, 20, dtype=np.uint8)),
         "adapter_id": None if j % 3 == 0 else "a" * int(rng.integers(0, 400)), "kv_format": "float8_e5m2",
         "salt": "" if j % 2 else bytearray(b"t%d" % j)}
    if j % 5 == 2:
        del d["adapter_id"]
    if extra and j % 4 == 1:
        d["extra"] = ["x" * j, b"\x00\xff"]
    return d


def step(kt, descriptors):
    return kt.derive_lookup_store(torch.arange(8, dtype=torch.int32, device="cuda"),
                                  torch.tensor([0, 4, 8], device="cuda"), torch.zeros(2, dtype=torch.int32, device="cuda"),
                                  descriptors, torch.arange(2, dtype=torch.int32, device="cuda"))


@pytest.mark.parametrize("side_stream", [False, True])
@pytest.mark.parametrize("extra", [False, True])
def test_calls_in_flight_keep_their_encodings(side_stream, extra):
    rng = np.random.default_rng(3)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if side_stream else None
    kt = KeyTable(4, 8, stream=stream)
    batches = [[desc(rng, 10 * k + j, extra) for j in range(1 + k % 7)] for k in range(60)]
    got = []
    for b in batches:
        with torch.cuda.stream(stream):
            torch.empty(1 << 22, device="cuda").fill_(1.0)  # keeps the stream busy behind the host
        got.append(step(kt, b)[0])
    torch.cuda.synchronize()
    kt.check()
    for b, d in zip(batches, got):
        assert np.array_equal(d.cpu().numpy(), O.descriptor_digests(b))
    kt.close()


def test_no_descriptors_and_refusals():
    kt = KeyTable(4, 4)
    out = kt.derive_lookup_store(torch.zeros(0, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda"),
                                 torch.zeros(0, dtype=torch.int32, device="cuda"), [], torch.zeros(0, dtype=torch.int32, device="cuda"))
    assert out[0].shape == (0, 32)
    ok = {"weight_precision": "bf16", "kv_format": "bf16"}
    for bad in (dict(ok, weight_precision="auto"), dict(ok, kv_format=""), dict(ok, salt="s" * 4097)):
        with pytest.raises(pk.PKError) as e:
            step(kt, [ok, bad])
        with pytest.raises(pk.PKError) as want:
            pk.pk_descriptors_encode([ok, bad])
        assert e.value.code == want.value.code
    kt.close()
