"""Performance cases: the calls that a user of the key library makes, over the range of sizes they are made at.

Kinds of case (`kind`):
  service   KeyTable.derive_lookup_store, the whole hot path through the convenience layer: descriptors as dicts,
            tokens on the device, outputs allocated by the call.  What a small worker or router does per batch.
  step      pk_derive_lookup_store with the caller's own buffers, what an engine's scheduler calls per batch of
            prompts: descriptor digests, chunk digests, chained keys, lookup, insertion of the misses.  The first
            pass on a state stores the misses of a half-shared batch; the passes after it find every key.
  budget    the same call on a store of fixed budget that cycles through more provenances than fit, followed by the
            eviction: every pass misses, inserts and evicts.
  lookup    pk_lookup alone: half of each request's keys are in the table.
  churn     pk_store of a new generation of keys and pk_evict of the oldest one.
  content   pk_content_digests of an adapter's tensors.
  strings   pk_key_strings: the fixed-width text keys of a connector.

Every output is a whole number or a byte (hashes, slots, counts, results), so every tolerance is "exact", and there
is no error against 64-bit arithmetic to state (`exact` is None).
"""
import math

import numpy as np
import torch

from paper_2609_38706_gb300 import pk
from paper_2609_38706_gb300.service import KeyTable

VOCAB = 152064
OPS = 1384  # 32-bit operations of one SHA-256 compression: 64 rounds x 14 + 48 schedule words x 10 + 8
VERSION = "0123456789abcdef0123456789abcdef01234567"


def listed():
    return [
        # A worker's small batch through the convenience layer (the repository's tiny configuration): latency.
        dict(name="service_tiny", kind="service", R=8, T=512, C=256, D=4, cap=6, ragged=False),
        # Multi-adapter serving: 1,024 prompts of 4,096 tokens under 32 provenances, the chunk of a store connector.
        dict(name="step_multi_adapter", kind="step", R=1024, T=4096, C=256, D=32, cap=20, ragged=False),
        # The same as prompts really come: lengths spread over 1:16, packed back to back, so no request's start is aligned.
        dict(name="step_ragged", kind="step", R=900, T=16000, C=256, D=32, cap=20, ragged=True),
        # An engine's own paged cache: blocks of 16 tokens, the largest batch.
        dict(name="step_small_block", kind="step", R=16384, T=2048, C=16, D=16, cap=23, ragged=False),
        # Blocks of 16 tokens again, an ordinary batch with uneven prompts.
        dict(name="step_small_block_ragged", kind="step", R=5000, T=4093, C=16, D=16, cap=21, ragged=True),
        # Few very long prompts: one chain of 512 chunks each.
        dict(name="step_long_context", kind="step", R=64, T=131072, C=256, D=4, cap=22, ragged=False),
        # Many prompts that share a prefix under 16 provenances, the largest table.
        dict(name="step_sweep", kind="step", R=4096, T=8192, C=256, D=16, cap=24, ragged=False),
        # A store of fixed budget under more provenances than fit: 64 prompts a step, every one missed and evicted again.
        dict(name="budget_thrash", kind="budget", R=64, k=8, C=256, D=4, P=512, cap=14),
        # A scheduler asking which prefixes are cached, without storing.
        dict(name="lookup_half_hit", kind="lookup", R=16384, k=128, cap=23, ragged=False),
        # A store node taking a new generation of keys and giving up the oldest one.
        dict(name="churn_store_evict", kind="churn", n=262144, G=6, cap=22),
        # Content identity of an adapter of about 40 MB.
        dict(name="content_adapter", kind="content", n=16, size=7500000),
        # Text keys of a store connector: 150-byte rows.
        dict(name="strings_150", kind="strings", n=1000003, width=150, prefix=66),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["service", "budget", "lookup", "churn", "content", "strings"])
    if kind == "step":
        C = rng.choice([8, 16, 16, 32, 64, 128, 256, 256, 512])
        tokens = _log_int(rng, 4 * C, 16 << 20)
        R = _log_int(rng, max(1, -(-tokens // (512 * C))), max(1, min(16384, tokens // (2 * C))))
        T = tokens // R
        ragged = rng.random() < 0.75
        n = int((_lengths(R, T, ragged) // C).sum())
        cap = min(24, max(8, math.ceil(math.log2(4 * n + 64)) + rng.choice([0, 0, 1, 2])))
        return dict(kind="step", R=R, T=T, C=C, D=min(R, rng.choice([1, 4, 16, 32, 64])), cap=cap, ragged=ragged)
    if kind == "service":
        C = rng.choice([16, 64, 256])
        return dict(kind="service", R=_log_int(rng, 1, 64), T=_log_int(rng, 4 * C, 8192), C=C, D=rng.choice([1, 2, 4, 8]),
                    cap=16, ragged=True)
    if kind == "budget":
        return dict(kind="budget", R=rng.choice([8, 16, 32, 64, 128]), k=_log_int(rng, 2, 24), C=rng.choice([64, 256]),
                    D=rng.choice([2, 3, 4]), P=512, cap=16)
    if kind == "lookup":
        R, k = _log_int(rng, 1, 16384), _log_int(rng, 2, 128)
        return dict(kind="lookup", R=R, k=k, cap=max(8, math.ceil(math.log2(4 * R * k))), ragged=rng.random() < 0.5)
    if kind == "churn":
        n = _log_int(rng, 1000, 200000)
        return dict(kind="churn", n=n, G=rng.randint(2, 6), cap=math.ceil(math.log2(12 * n)))
    if kind == "content":
        n = _log_int(rng, 1, 200)
        return dict(kind="content", n=n, size=_log_int(rng, 1000, min(1 << 26, (1 << 28) // n)))
    width = rng.randint(32, 256)
    return dict(kind="strings", n=_log_int(rng, 1000, 1000000), width=width, prefix=rng.randint(0, width - 22))


# ---------------------------------------------------------------------------
# sizes and inputs
# ---------------------------------------------------------------------------
def _lengths(R, T, ragged):
    """Request lengths, the same multiset for every seed: all T, or spread over T/16 .. T (evenly in the logarithm)."""
    if not ragged or R == 1:
        return np.full(R, T, np.int64)
    return np.maximum(T * 16.0 ** (-(np.arange(R) + 0.5) / R), 1).astype(np.int64)


def _bytes(g, *shape):
    n = int(np.prod(shape))
    return torch.randint(-(1 << 62), 1 << 62, ((n + 7) // 8,), generator=g, device="cuda").view(torch.uint8)[:n].view(shape)


def _descriptors(D):
    return [dict(model_id="synthetic/model-7b", weight_precision=("bf16", "fp8_e4m3")[j % 2], weight_version=VERSION,
                 adapter_id="adapter-%02d" % (j // 2 % 8), kv_format="fp8_e4m3", salt="tenant-%d" % (j // 16))
            for j in range(D)]


def _off(lens):
    return torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)).cuda()


def _tokens(g, rs, lens, templates, shared):
    """Prompts of `lens` tokens packed back to back; half of them start with one of the templates (its first `shared`
    tokens), the rest is random."""
    R, n = len(lens), int(lens.sum())
    off = _off(lens)
    t = torch.from_numpy(rs.integers(0, len(shared), R)).cuda()
    upto = shared[t] * torch.from_numpy((rs.random(R) < 0.5).astype(np.int64)).cuda()
    tok = torch.randint(0, VOCAB, (n,), generator=g, device="cuda", dtype=torch.int32)
    req = torch.repeat_interleave(torch.arange(R, device="cuda"), torch.from_numpy(lens).cuda(), output_size=n)
    pos = torch.arange(n, device="cuda") - off[req]
    at = torch.nonzero(pos < upto[req]).view(-1)
    tok[at] = templates.view(-1)[t[req[at]] * templates.shape[1] + pos[at]]
    return tok, off


def _new(n, dtype=torch.int32, fill=0):
    return torch.full((n,), fill, dtype=dtype, device="cuda")


def _step_buffers(s, R, n):
    s.update(key_off=_new(R + 1, torch.int64), keys=torch.zeros((n, 32), dtype=torch.uint8, device="cuda"),
             hit=_new(R), slots=_new(n), result=_new(n), slot_out=_new(n), status=_new(1))


def _encoded(D):
    enc, off = pk.pk_descriptors_encode(_descriptors(D))
    return (torch.from_numpy(enc.copy()).cuda(), torch.from_numpy(off.copy()).cuda(),
            torch.zeros((D, 32), dtype=torch.uint8, device="cuda"))


def prepare(case, seed):
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    rs = np.random.default_rng(seed)
    kind = case["kind"]
    s = dict(kind=kind, case=case)
    if kind in ("step", "service"):
        R, T, C, D = case["R"], case["T"], case["C"], case["D"]
        base = _lengths(R, T, case["ragged"])
        n_keys = int((base // C).sum())
        templates = torch.randint(0, VOCAB, (min(R, 64), T), generator=g, device="cuda", dtype=torch.int32)
        shared = torch.from_numpy(rs.integers(T // 8, T + 1, len(templates))).cuda()
        kt = KeyTable(C, case["cap"])
        idx = torch.from_numpy(rs.integers(0, D, R).astype(np.int32)).cuda()
        s.update(kt=kt, desc_idx=idx, descriptors=_descriptors(D), n_keys=n_keys)
        # The table: the keys of an earlier batch of the same templates, then other keys, such that it is about
        # 0.6 full (the 64-entry one 0.5) once the batch is stored.
        lens = rs.permutation(base)
        tok, off = _tokens(g, rs, lens, templates, shared)
        pidx = torch.from_numpy(rs.integers(0, D, R).astype(np.int32)).cuda()
        load = 0.5 if case["cap"] <= 6 else 0.6
        fill = int(load * (1 << case["cap"])) - 2 * n_keys
        if fill >= 0:
            ko, pkeys = kt.derive(tok, off, pidx, kt.digests(s["descriptors"]))
            kt.store(pkeys[:n_keys], torch.arange(n_keys, dtype=torch.int32, device="cuda"))
        if fill > 0:
            kt.store(_bytes(g, fill, 32), torch.arange(n_keys, n_keys + fill, dtype=torch.int32, device="cuda"))
        kt.check("prepare")
        lens = rs.permutation(base)
        s["tokens"], s["tok_off"] = _tokens(g, rs, lens, templates, shared)
        cap = s["tokens"].numel() // C
        s["new_slots"] = torch.arange(1 << 24, (1 << 24) + cap, dtype=torch.int32, device="cuda")
        if kind == "step":
            s["enc"], s["enc_off"], s["digests"] = _encoded(D)
            _step_buffers(s, R, cap)
    elif kind == "budget":
        R, k, C, D, P = (case[x] for x in ("R", "k", "C", "D", "P"))
        kt = KeyTable(C, case["cap"])
        n, steps = R * k, D * P // R
        s.update(kt=kt, steps=steps, pool=torch.randint(0, VOCAB, (P, k * C), generator=g, device="cuda", dtype=torch.int32),
                 tok_off=torch.arange(R + 1, dtype=torch.int64, device="cuda") * (k * C), budget=P * k + P * k // 8,
                 desc_idx=[_new(R, fill=d) for d in range(D)], at=0,
                 new_slots=torch.arange(steps * n, dtype=torch.int32, device="cuda"), freed=_new(steps * n),
                 ones=_new(n, fill=1))
        s["enc"], s["enc_off"], s["digests"] = _encoded(D)
        _step_buffers(s, R, n)
        kt.attach_stamps()
        s.update(evicted=_new(n), n_evicted=_new(1, torch.int64))
        for _ in range(steps):  # one cycle: the store is at its budget from then on
            _serve(s)
        kt.check("prepare")
    elif kind == "lookup":
        R, k = case["R"], case["k"]
        lens = rs.permutation(_lengths(R, k, case["ragged"]))
        n = int(lens.sum())
        kt = KeyTable(16, case["cap"])
        keys = _bytes(g, n, 32)
        off = _off(lens)
        pos = torch.arange(n, device="cuda") - torch.repeat_interleave(off[:-1], torch.from_numpy(lens).cuda(), output_size=n)
        first = torch.from_numpy(rs.integers(0, lens + 1)).cuda()
        have = pos < torch.repeat_interleave(first, torch.from_numpy(lens).cuda(), output_size=n)
        mine = keys[have]
        kt.store(mine, torch.arange(len(mine), dtype=torch.int32, device="cuda"))
        fill = int(0.6 * (1 << case["cap"])) - len(mine)
        if fill > 0:
            kt.store(_bytes(g, fill, 32), torch.arange(len(mine), len(mine) + fill, dtype=torch.int32, device="cuda"))
        kt.check("prepare")
        s.update(kt=kt, keys=keys, key_off=off, hit=_new(R), slots=_new(n), status=_new(1))
    elif kind == "churn":
        n, G = case["n"], case["G"]
        kt = KeyTable(16, case["cap"])
        kt.attach_stamps()
        s.update(kt=kt, keys=_bytes(g, (G + 1) * n, 32),  # pages come off the free list in no order
                 new_slots=torch.randperm((G + 1) * n, generator=g, dtype=torch.int32, device="cuda"),
                 result=_new(n), slot_out=_new(n), status=_new(1), evicted=_new(n), n_evicted=_new(1, torch.int64),
                 freed=_new((G + 1) * n), ones=_new(n, fill=1), at=0)
        for _ in range(G):
            _churn(s)
        kt.check("prepare")
    elif kind == "content":
        sizes = rs.permutation(_lengths(case["n"], case["size"], True))
        s["data"] = [_bytes(g, int(x)) for x in sizes]
        s["scratch"] = torch.zeros(pk.pk_content_scratch_bytes_batch([int(x) for x in sizes]), dtype=torch.uint8, device="cuda")
        s["tops"] = torch.zeros((case["n"], 32), dtype=torch.uint8, device="cuda")
    else:
        s["keys"] = _bytes(g, case["n"], 32)
        s["prefix"] = bytes(rs.integers(33, 127, case["prefix"], dtype=np.uint8))
        s["out"] = torch.zeros((case["n"], case["width"]), dtype=torch.uint8, device="cuda")
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _serve(s):
    case = s["case"]
    R, D, P = case["R"], case["D"], case["P"]
    step = s["at"] % s["steps"]
    s["at"] += 1
    row = step * R % P
    n = s["keys"].shape[0]
    pk.pk_derive_lookup_store(s["kt"].ctx, s["pool"][row:row + R], s["tok_off"], s["desc_idx"][step * R // P], s["enc"],
                              s["enc_off"], s["digests"], s["key_off"], s["keys"], s["new_slots"][step * n:(step + 1) * n],
                              s["hit"], s["slots"], s["result"], s["slot_out"], s["status"])
    pk.pk_evict(s["kt"].ctx, s["budget"], s["budget"], s["kt"].evict_scratch, s["evicted"], s["n_evicted"], s["status"])


def _churn(s):
    n, G = s["case"]["n"], s["case"]["G"]
    gen = s["at"] % (G + 1)
    s["at"] += 1
    pk.pk_store(s["kt"].ctx, s["keys"][gen * n:(gen + 1) * n], s["new_slots"][gen * n:(gen + 1) * n], s["result"],
                s["slot_out"], s["status"])
    pk.pk_evict(s["kt"].ctx, G * n, G * n, s["kt"].evict_scratch, s["evicted"], s["n_evicted"], s["status"])


def run(s):
    kind = s["kind"]
    if kind == "step":
        pk.pk_derive_lookup_store(s["kt"].ctx, s["tokens"], s["tok_off"], s["desc_idx"], s["enc"], s["enc_off"], s["digests"],
                                  s["key_off"], s["keys"], s["new_slots"], s["hit"], s["slots"], s["result"], s["slot_out"],
                                  s["status"])
        n = s["n_keys"]
        return [s["digests"], s["key_off"], s["keys"][:n], s["hit"], s["slots"][:n], s["result"], s["slot_out"], s["status"]]
    if kind == "service":
        digests, key_off, keys, hit, slots, result, slot_out = s["kt"].derive_lookup_store(
            s["tokens"], s["tok_off"], s["desc_idx"], s["descriptors"], s["new_slots"])
        n = s["n_keys"]
        return [digests, key_off, keys[:n], hit, slots[:n], result, slot_out]
    if kind == "budget":
        _serve(s)
        s["freed"].index_add_(0, s["evicted"], s["ones"])  # the program's count of how often each page was given up
        return [s["keys"], s["hit"], s["slots"], s["result"], s["slot_out"], s["n_evicted"], s["freed"], s["status"]]
    if kind == "lookup":
        pk.pk_lookup(s["kt"].ctx, s["keys"], s["key_off"], s["hit"], s["slots"], s["status"])
        return [s["hit"], s["slots"], s["status"]]
    if kind == "churn":
        _churn(s)
        s["freed"].index_add_(0, s["evicted"], s["ones"])
        return [s["result"], s["slot_out"], s["n_evicted"], s["freed"], s["status"]]
    if kind == "content":
        pk.pk_content_digests(s["data"], s["scratch"], s["tops"])
        return [s["tops"]]
    pk.pk_key_strings(s["keys"], s["prefix"], s["case"]["width"], s["out"])
    return [s["out"]]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("step", "service", "budget"):
        C = case["C"]
        lens = np.full(case["R"], case["k"] * C) if kind == "budget" else _lengths(case["R"], case["T"], case["ragged"])
        n = int((lens // C).sum())
        # tokens, offsets, indices; keys written; an entry sector, the new slot and three results per key
        b = 4 * int(lens.sum()) + 24 * case["R"] + 32 * n + (32 + 4 + 12) * n
        if kind == "budget":  # stamps of the table read; the entries and stamps inserted and removed
            b += (8 << case["cap"]) + 2 * 40 * n + 4 * n
        return dict(bytes=b, flops=OPS * n * ((4 * C + 9 + 63) // 64 + 2))
    if kind == "lookup":
        n = int(_lengths(case["R"], case["k"], case["ragged"]).sum())
        return dict(bytes=(16 + 32 + 4) * n + 12 * case["R"], flops=0)
    if kind == "churn":  # key, slot, entry, stamp and two results per new key; the table's stamps; the removed entries
        n = case["n"]
        return dict(bytes=(16 + 4 + 32 + 8 + 8) * n + (8 << case["cap"]) + (32 + 8 + 4) * n, flops=0)
    if kind == "content":
        total, blocks = 0, 0
        for x in _lengths(case["n"], case["size"], True):
            total += int(x)
            m = int(x)
            while True:
                m = max(1, -(-m // 1024))
                blocks += m
                if m == 1:
                    break
                m *= 32
        return dict(bytes=total + 32 * case["n"], flops=OPS * 17 * blocks)
    return dict(bytes=(16 + case["width"]) * case["n"], flops=0)


def tolerance(case):
    return "exact"


def exact(case, seed):
    return None  # hashes, slots and counts: no output is a rounded number
