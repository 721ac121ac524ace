"""KeyTable.derive_lookup_store on a table with a stream of its own: inputs that the current stream is still making when
the call returns, and inputs and outputs dropped while the table's stream has not reached the call."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_38706_gb300.service import KeyTable

pytestmark = pytest.mark.gpu

C = 4
DESCS = [{"model_id": "m%d" % j, "weight_precision": "bf16", "kv_format": "bf16"} for j in range(3)]


def backlog():
    """About 0.3 s of work on the current stream, and the event of its end."""
    a = torch.ones((4096, 4096), device="cuda")
    for _ in range(150):
        a = a @ a * 0.0 + 1.0
    e = torch.cuda.Event()
    e.record()
    return e


def inputs(seed, R=37):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 9 * C, R)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    return (rng.integers(0, 1 << 31, int(off[-1]), dtype=np.int64).astype(np.int32), off,
            rng.integers(0, len(DESCS), R).astype(np.int32))


def check(out, tokens, off, idx):
    d = O.descriptor_digests(DESCS)
    ko, keys = O.derive_keys(tokens, off, C, idx.view(np.uint32), d)
    assert np.array_equal(out[0].cpu().numpy(), d) and np.array_equal(out[1].cpu().numpy(), ko)
    assert np.array_equal(out[2].cpu().numpy()[:int(ko[-1])], keys)


def test_inputs_still_being_made():
    torch.cuda.synchronize()
    kt = KeyTable(C, 10, stream=torch.cuda.Stream())
    tokens, off, idx = inputs(1)
    made = [torch.from_numpy(x).cuda() for x in (tokens, off, idx)]
    late = [torch.zeros_like(x) for x in made]
    slots = torch.arange(tokens.size // C, dtype=torch.int32, device="cuda")
    kt.derive_lookup_store(*late, DESCS, slots)  # (pinned buffers and kernels are there)
    torch.cuda.synchronize()
    done = backlog()
    for a, b in zip(late, made):
        a.copy_(b)
    out = kt.derive_lookup_store(*late, DESCS, slots)
    assert not done.query()
    torch.cuda.synchronize()
    kt.check()
    check(out, tokens, off, idx)
    kt.close()


def overwrite_freed():
    for n in (32, 96, 148, 296, 512, 2048, 1 << 16):
        torch.full((n,), 0x7F, dtype=torch.uint8, device="cuda")


def test_memory_is_kept():
    """Host inputs (whose device copies the call drops), outputs dropped and their memory asked for again."""
    torch.cuda.synchronize()
    own = torch.cuda.Stream()
    kt = KeyTable(C, 14, stream=own)
    batches = [inputs(10 + k) for k in range(12)]
    # Every kernel loaded and every pinned buffer allocated beforehand: both may wait for the device.
    kt.derive_lookup_store(*batches[0][:3], DESCS, np.arange(batches[0][0].size // C, dtype=np.uint32))
    overwrite_freed()
    pinned = [torch.empty(256, dtype=torch.uint8, pin_memory=True) for _ in range(len(batches))]
    del pinned
    torch.cuda.synchronize()
    with torch.cuda.stream(own):
        done = backlog()
    kept = []
    for k, (tokens, off, idx) in enumerate(batches):
        out = kt.derive_lookup_store(tokens, off, idx, DESCS, np.arange(tokens.size // C, dtype=np.uint32))
        if k % 2:
            kept.append((out, batches[k]))
        del out
        overwrite_freed()
    assert not done.query()
    torch.cuda.synchronize()
    kt.check()
    for out, b in kept:
        check(out, *b)
    kt.close()
