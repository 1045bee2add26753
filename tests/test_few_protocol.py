"""A model of the barrier protocol of the few-token GEMM (w4a4_gemm_few_kernel,
csrc/w4a4_few.cu) under random and starving interleavings: one CTA's TMA warp,
MMA warp and epilogue, the copies (each lands at any time after it was issued,
in any order) and the cluster barriers with the other parts of K.

Every wait is a parity wait on a counted barrier. The checks:

- no schedule deadlocks, and every wait sees the phase it means;
- a stage is refilled only after the MMAs that read it, and takes partial sums
  only after every stage has been read;
- no copy is in flight when the CTA's last warp leaves: also when the MMA warp
  or the TMA warp gives up at any of its waits, in which case nothing is
  stored."""

import random

import pytest


def run(nk, stages, seed, prefer=None, mma_gives_up=None, tma_gives_up=None, drop=None):
    """One schedule. mma_gives_up / tma_gives_up: the K block at whose wait
    that warp's limit runs out. `drop` removes one wait ("empty" or "landed")."""
    full, empty = [0] * stages, [0] * stages         # completed phases
    done = [0]
    flying, landed, read = [], {}, []                # copies by K block
    state = {"abort": False, "stored": False, "exited": 0}
    barrier = {"a": 0, "b": 0}                       # arrivals of the three roles

    def parity_wait(counts, s, parity, want):
        """Steps until the phase of that parity has completed."""
        while True:
            if (counts[s] & 1) != parity:
                assert counts[s] == want, "a parity wait satisfied by another phase"
                return
            yield "blocked"

    def join(name):
        barrier[name] += 1
        while barrier[name] < 3:
            yield "blocked"

    def leave():
        state["exited"] += 1
        assert state["exited"] < 3 or not flying, "the CTA has left with a copy in flight"

    def issue(kc):
        s = kc % stages
        assert full[s] == kc // stages, "stage refilled while a copy into it was in flight"
        assert kc < stages or kc - stages in read, "stage refilled before its MMAs"
        flying.append(kc)

    def tma():
        pre, ok, issued = min(nk, stages), True, 0
        for kc in range(pre):
            issue(kc)
            yield
        issued = pre
        for kc in range(pre, nk):
            s = kc % stages
            w = parity_wait(empty, s, (kc // stages & 1) ^ 1, kc // stages)
            if drop != "empty":
                for step in w:
                    if kc == tma_gives_up or state["abort"]:
                        ok = False
                        break
                    yield step
            if not ok:
                break
            issue(kc)
            issued = kc + 1
            yield
        if not ok:
            state["abort"] = True
        yield from join("a")
        yield from join("b")
        if state["abort"] and drop != "landed":
            for kc in range(max(issued - stages, 0), issued):
                yield from parity_wait(full, kc % stages, kc // stages & 1, kc // stages + 1)
        leave()

    def mma():
        ok = True
        for kc in range(nk):
            s = kc % stages
            for step in parity_wait(full, s, kc // stages & 1, kc // stages + 1):
                if kc == mma_gives_up or state["abort"]:
                    ok = False
                    break
                yield step
            if not ok:
                break
            assert landed.get(s) == kc
            read.append(kc)                          # (the MMAs complete in order)
            empty[s] += 1
            yield
        if not ok:
            state["abort"] = True
        done[0] += 1
        yield from join("a")
        yield from join("b")
        leave()

    def epilogue():
        yield from parity_wait(done, 0, 0, 1)
        yield from join("a")
        if not state["abort"]:
            assert not flying and read == list(range(nk)), "sums into stages that were not all read"
            yield
        yield from join("b")
        if not state["abort"]:
            state["stored"] = True
        leave()

    def copies():
        while state["exited"] < 3:
            if flying:
                kc = flying.pop(rng.randrange(len(flying)))
                landed[kc % stages] = kc
                full[kc % stages] += 1
                yield
            else:
                yield "blocked"

    rng = random.Random(seed)
    roles = {"tma": tma(), "mma": mma(), "epi": epilogue(), "copies": copies()}
    stalled = 0
    while roles:
        assert stalled < 3, "deadlock"               # (a blocked step may have moved on to another wait)
        order = [r for r in prefer or () if r in roles]
        rest = [r for r in roles if r not in order]
        rng.shuffle(rest)
        for r in order + rest:                       # the first role that can proceed
            try:
                if next(roles[r]) == "blocked":
                    continue
            except StopIteration:
                del roles[r]
            stalled = 0
            break
        else:
            stalled += 1
    gave_up = state["abort"]
    assert state["stored"] != gave_up
    return gave_up


ORDERS = (None, ("tma", "mma"), ("copies", "tma"), ("mma", "epi", "tma"), ("epi", "mma", "tma"), ("copies", "mma"))


@pytest.mark.parametrize("nk", [1, 2, 5, 6, 7, 12, 33])
@pytest.mark.parametrize("stages", [3, 6])
def test_few_barrier_protocol(nk, stages):
    for prefer in ORDERS:
        for seed in range(6):
            assert not run(nk, stages, seed, prefer)


@pytest.mark.parametrize("nk,stages", [(1, 3), (3, 3), (4, 3), (7, 3), (12, 6)])
def test_giving_up_leaves_no_copy_in_flight(nk, stages):
    """A wait that runs out at any K block, of either warp, with the copies late."""
    late = (("mma", "epi", "tma"), ("tma", "mma", "epi"), None)
    for kc in range(nk):
        for prefer in late:
            for seed in range(4):
                run(nk, stages, seed, prefer, mma_gives_up=kc)
                run(nk, stages, seed, prefer, tma_gives_up=kc)
    assert run(nk, stages, 0, late[0], mma_gives_up=0)


def test_model_catches_a_missing_wait():
    """Without the TMA warp's wait for what it has issued, an MMA warp that gives
    up lets the CTA leave under its copies; without the wait for a read stage
    the ring is refilled too early."""
    with pytest.raises(AssertionError, match="left with a copy in flight"):
        run(7, 3, 0, ("mma", "epi", "tma"), mma_gives_up=0, drop="landed")
    with pytest.raises(AssertionError, match="refilled"):
        run(7, 3, 0, ("tma", "copies"), drop="empty")
