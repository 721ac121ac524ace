"""CPU model of the two-warp protocols of a pair: the chains (csrc/pk_derive.cu, k_chain and k_chain_split) and the
digests of few messages (csrc/pk_pair.cuh, pair_schedule and pair_rounds).

Each protocol's rounds warp (R) and schedule warp (S) are written out as their
sequences of named-barrier operations and shared-memory accesses, step by step
as the kernels issue them; every interleaving of the two warps is explored and
must end with both warps done (no deadlock), no warp arriving twice in one
phase of a barrier (count 64: one arrival per warp completes a phase), no
pending arrival left at the end, and no read of a buffer overlapping the other
warp's write of it.  A mutated protocol must fail the same checks, so that the
model is shown to catch what it is meant to catch."""
import pytest

# ops: ("arrive", id) | ("sync", id) | ("w+", buf) | ("w-", buf) | ("r+", buf) | ("r-", buf)


def chain(n):
    """n steps of a pair of either chain: barriers s1 (block-1 slice 1, and block 2 of the step ready), s1b (block-1
    slices 2-3), k (k published)."""
    S = [("w+", "kw2_0"), ("w-", "kw2_0")]
    for i in range(n):
        if i > 0:
            S += [("sync", "k"), ("r+", "kpub"), ("r-", "kpub")]
        S += [("w+", "kw1_1"), ("w-", "kw1_1"), ("arrive", "s1")]
        S += [("w+", "kw1_2"), ("w-", "kw1_2"), ("w+", "kw1_3"), ("w-", "kw1_3"), ("arrive", "s1b")]
        if i + 1 < n:
            b = f"kw2_{(i + 1) & 1}"
            S += [("w+", b), ("w-", b)]
    R = []
    for i in range(n):
        R += [("sync", "s1"), ("r+", "kw1_1"), ("r-", "kw1_1"), ("sync", "s1b"), ("r+", "kw1_2"), ("r-", "kw1_2"),
              ("r+", "kw1_3"), ("r-", "kw1_3"), ("r+", f"kw2_{i & 1}"), ("r-", f"kw2_{i & 1}")]
        if i + 1 < n:
            R += [("w+", "kpub"), ("w-", "kpub"), ("arrive", "k")]
    return R, S


def ring(n, pad=False):
    """n blocks of a pair's messages through the two-stage ring: barriers filled_0/1 and read_0/1; `pad`: then the
    constant last block, from no ring.  The rounds warp reads the next block's first words before it marks a stage read."""
    S = []
    for b in range(n):
        if b >= 2:
            S += [("sync", f"read_{b & 1}")]
        S += [("w+", f"kw_{b & 1}"), ("w-", f"kw_{b & 1}"), ("arrive", f"filled_{b & 1}")]

    def first_words(b):
        return [("sync", f"filled_{b & 1}"), ("r+", f"kw_{b & 1}"), ("r-", f"kw_{b & 1}")] if b < n else []

    total = n + pad
    R = first_words(0)
    for b in range(total):
        if b < n:
            R += [("r+", f"kw_{b & 1}"), ("r-", f"kw_{b & 1}")]
        if b + 1 < total:
            R += first_words(b + 1)
        if b + 2 < n:
            R += [("arrive", f"read_{b & 1}")]
    return R, S


def ring_and_pad(n):
    return ring(n, True)


class ProtocolError(Exception):
    pass


def explore(R, S):
    """Every interleaving of the two programs; raises ProtocolError on a violation.
    State: (pc of each warp, per barrier the set of warps arrived in its current phase and its phase
    number, the phase each warp waits for, the buffers each warp is accessing)."""
    progs = (R, S)
    seen = set()

    def key(st):
        pcs, bars, waits, acc = st
        return (pcs, tuple(sorted((b, tuple(sorted(a)), p) for b, (a, p) in bars.items())), waits,
                tuple(tuple(sorted(x)) for x in acc))

    def step(st, w):
        pcs, bars, waits, acc = st
        if waits[w] is not None:
            bid, phase = waits[w]
            if bars.get(bid, (frozenset(), 0))[1] <= phase:
                return None  # still blocked
            waits = tuple(None if j == w else waits[j] for j in range(2))
            return (pcs, bars, waits, acc)
        if pcs[w] == len(progs[w]):
            return None
        op, arg = progs[w][pcs[w]]
        bars = dict(bars)
        acc = [set(acc[0]), set(acc[1])]
        new_wait = waits[w]
        if op in ("arrive", "sync"):
            arrived, phase = bars.get(arg, (frozenset(), 0))
            if w in arrived:
                raise ProtocolError(f"warp {'RS'[w]} arrives twice in phase {phase} of barrier {arg}")
            arrived = arrived | {w}
            if len(arrived) == 2:
                bars[arg] = (frozenset(), phase + 1)
            else:
                bars[arg] = (arrived, phase)
                if op == "sync":
                    new_wait = (arg, phase)
        elif op == "w+":
            if arg in acc[1 - w]:
                raise ProtocolError(f"warp {'RS'[w]} writes {arg} while the other warp accesses it")
            acc[w].add(arg)
        elif op == "r+":
            if arg in acc[1 - w]:
                raise ProtocolError(f"warp {'RS'[w]} reads {arg} while the other warp writes it")
            acc[w].add(arg)
        else:  # w- / r-
            acc[w].discard(arg)
        pcs = tuple(pcs[j] + (1 if j == w else 0) for j in range(2))
        waits = tuple(new_wait if j == w else waits[j] for j in range(2))
        return (pcs, bars, waits, (frozenset(acc[0]), frozenset(acc[1])))

    start = ((0, 0), {}, (None, None), (frozenset(), frozenset()))
    stack = [start]
    finals = 0
    while stack:
        st = stack.pop()
        k = key(st)
        if k in seen:
            continue
        seen.add(k)
        nxt = [s for s in (step(st, 0), step(st, 1)) if s is not None]
        if not nxt:
            pcs, bars, waits, _ = st
            if pcs != (len(R), len(S)) or waits != (None, None):
                raise ProtocolError(f"deadlock at R pc {pcs[0]}/{len(R)}, S pc {pcs[1]}/{len(S)}, waits {waits}")
            pending = {b: a for b, (a, _) in bars.items() if a}
            if pending:
                raise ProtocolError(f"arrivals left pending at the end: {pending}")
            finals += 1
            continue
        stack.extend(nxt)
    return len(seen), finals


@pytest.mark.parametrize("layout", [chain, ring, ring_and_pad])
@pytest.mark.parametrize("n", [1, 2, 3, 5])
def test_protocol_has_no_deadlock_double_arrival_or_race(layout, n):
    states, finals = explore(*layout(n))
    assert finals == 1 and states > len(layout(n)[0])


def _mutate(prog, i, new=None):
    p = list(prog)
    if new is None:
        del p[i]
    else:
        p[i] = new
    return p


def test_model_catches_a_missing_sync():
    """Without the rounds warp's wait for block-1 slice 2, its read can overlap the schedule warp's write."""
    R, S = chain(3)
    i = R.index(("sync", "s1b"))
    with pytest.raises(ProtocolError):
        explore(_mutate(R, i), S)


def test_model_catches_a_double_arrival():
    """The schedule warp marking the first slice of the next step without waiting for k: a second arrival in one phase
    of its barrier, or a read of k under its write."""
    R, S = chain(3)
    j = S.index(("sync", "k"))
    with pytest.raises(ProtocolError):
        explore(R, _mutate(S, j))


def test_model_catches_a_ring_stage_filled_too_early():
    """The schedule warp not waiting until a stage is read; the rounds warp marking it read before its last words."""
    R, S = ring(5)
    with pytest.raises(ProtocolError):
        explore(R, _mutate(S, S.index(("sync", "read_0"))))
    i = R.index(("arrive", "read_0"))
    early = R[:1] + [R[i]] + R[1:i] + R[i + 1:]
    with pytest.raises(ProtocolError):
        explore(early, S)


def test_model_catches_a_buffer_reused_too_early():
    """Block 2 single-buffered (always kw2_0): the schedule warp would overwrite the buffer the rounds warp
    is still reading."""
    R, S = chain(3)
    S = [(op, "kw2_0" if isinstance(a, str) and a.startswith("kw2_") else a) for op, a in S]
    R = [(op, "kw2_0" if isinstance(a, str) and a.startswith("kw2_") else a) for op, a in R]
    with pytest.raises(ProtocolError):
        explore(R, S)


def test_model_catches_a_deadlock():
    """The schedule warp waiting for k before it has marked the step's first slice (i = 0 included)."""
    R, S = chain(2)
    S = [("sync", "k")] + S
    with pytest.raises(ProtocolError):
        explore(R, S)
