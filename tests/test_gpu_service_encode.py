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


def step_inputs():
    return (torch.arange(8, dtype=torch.int32, device="cuda"), torch.tensor([0, 4, 8], device="cuda"),
            torch.zeros(2, dtype=torch.int32, device="cuda"), torch.arange(2, dtype=torch.int32, device="cuda"))


def step(kt, descriptors, inputs=None):
    tokens, off, idx, slots = inputs or step_inputs()
    return kt.derive_lookup_store(tokens, off, idx, descriptors, slots)


@pytest.mark.parametrize("side_stream", [False, True])
@pytest.mark.parametrize("extra", [False, True])
def test_calls_in_flight_keep_their_encodings(side_stream, extra):
    """60 calls enqueued behind 0.3 s of work on the table's stream.  (With appended dimensions some calls take the copies
    from pageable memory, which wait for the current stream.)"""
    rng = np.random.default_rng(3)
    stream = torch.cuda.Stream() if side_stream else None
    kt = KeyTable(4, 8, stream=stream)
    inputs = step_inputs()
    batches = [[desc(rng, 10 * k + j, extra) for j in range(1 + k % 7)] for k in range(60)]
    for b in batches[:7]:
        step(kt, b, inputs)
    # (a pinned allocation that the cache cannot serve waits for the device)
    pinned = [torch.empty(1 << k, dtype=torch.uint8, pin_memory=True) for k in range(7, 14) for _ in batches]
    del pinned
    a = torch.ones((4096, 4096), device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for _ in range(150):
            a = a @ a * 0.0 + 1.0
        done = torch.cuda.Event()
        done.record()
    got = [step(kt, b, inputs) for b in batches]
    assert extra or not done.query()
    torch.cuda.synchronize()
    kt.check()
    for b, out in zip(batches, got):
        assert np.array_equal(out[0].cpu().numpy(), O.descriptor_digests(b))
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
