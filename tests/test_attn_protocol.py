"""A model of the barrier protocol of attn_pv_tac_kernel (csrc/attn.cu),
run under random interleavings of its three roles, for many key-chunk
counts and items per CTA.

The kernel's TMA warp, MMA warp and softmax warps communicate only through
mbarriers whose waits name a phase parity. This model replays each role's
sequence of waits and arrivals in the kernel's order, with the kernel's
entry numbering (ring entries of an item: Q, nk pass-1 K chunks, nk pass-2
K / V pairs, M's two halves, the output slot; six ring slots; three S
buffers, which pass 1 goes round and of which pass 2 alternates between the
first two; the third lies in the columns of the P V^T and TAC accumulator, so
the softmax warps hand it over when they have read an item's TAC result) and
its masks of the buffers' parities, and checks under random schedules that

- no schedule deadlocks;
- every wait sees exactly the completed-phase count it means (a parity
  wait that could be satisfied by a phase two ahead would be a bug);
- a ring slot is refilled only after its consumer released it;
- an S buffer takes new scores only after the softmax warps have finished with
  its previous use (read it in pass 1, written P over it in pass 2), the third
  one only after they have read the previous item's TAC result out of it;
- P V^T of an item starts only after they have read all of its pass-1 scores,
  and Z_hat is written over an S buffer only after the P V^T that reads it.

The softmax warps are one role here: all sixteen run the same program and
a barrier completes when the last of them arrives. MMAs complete in issue
order, so a commit is modelled at the issuing point."""

import random

import pytest

SLOTS = 6


class Bar:
    def __init__(self):
        self.phases = 0          # completed phases

    def arrive(self):
        self.phases += 1


def run(nk, items_per_cta, seed, prefer=None, drop=None):
    """One schedule: each step runs the first role of `prefer` (a priority
    order) whose next step can proceed, else a random one among those that
    can. A priority order starves the roles at its end, where a missing
    wait shows at once. `drop` removes one wait of the MMA warp: "p" (for P(j)
    before P V^T(j)), "s" (for the S buffer before Q K^T) or "handover" (the
    same, only where Q K^T takes the third buffer over from the previous item's
    TAC result)."""
    my = items_per_cta
    E = 3 * nk + 4                                   # ring entries per item
    bars = {}

    def bar(name):
        return bars.setdefault(name, Bar())

    full = lambda g: ("full", g % SLOTS)
    empty = lambda g: ("empty", g % SLOTS)
    # a wait for phase number `want - 1` to have completed
    W = lambda name, want: ("wait", name, want)
    A = lambda name: ("arrive", name)
    filled, consumed = {}, {}                       # ring: per-slot use counts
    s_written, s_done = [0, 0, 0], [0, 0, 0]         # scores written / finished with, per buffer
    tac_written, tac_read = [0], [0]                 # TAC results in the third buffer's columns
    pass1_read = [0]                                 # pass-1 scores read, over all items

    def tma():
        for i in range(my):
            for u in range(E):
                g = i * E + u
                yield W(empty(g), g // SLOTS)        # the slot's previous use released
                assert consumed.get(g % SLOTS, 0) == g // SLOTS, "ring slot refilled before release"
                filled[g % SLOTS] = g // SLOTS + 1
                yield A(full(g))
        G = my * E
        for g in range(max(G - SLOTS, 0), G):        # every slot given back before exit
            yield W(empty(g), g // SLOTS + 1)

    def release(g):
        consumed[g % SLOTS] = consumed.get(g % SLOTS, 0) + 1
        return A(empty(g))

    def mma():
        uses, mask = [0, 0, 0], 0                    # uses of each S buffer, and the kernel's parity mask of them

        def used(b):
            nonlocal mask
            uses[b] += 1
            mask ^= 1 << b
            assert all((mask >> k & 1) == uses[k] & 1 for k in range(3))

        def scores(b):                               # Q K^T writes buffer b
            assert s_done[b] == s_written[b], "S buffer overwritten before its previous use was consumed"
            assert b != 2 or tac_read[0] == tac_written[0], "third S buffer written before the TAC result was read"
            s_written[b] += 1

        for i in range(my):
            gq, g0 = i * E, i * E + 1
            yield W("q_full", i + 1)                 # Q in TMEM: its ring slot is free again
            yield release(gq)

            def qk(g, b, handover=False):
                yield W(full(g), g // SLOTS + 1)
                if drop != "s" and not (drop == "handover" and handover):
                    yield W(("s_empty", b), uses[b])     # previous use of the buffer consumed
                scores(b)
                used(b)
                yield release(g)
                yield A(("s_full", b))
            for it in range(nk):                     # pass 1
                yield from qk(g0 + it, it % 3, it == 2 and i > 0)
            used(2)                                  # (the release of the TAC accumulator)
            for j in range(min(2, nk)):              # pass 2, first two chunks ahead
                yield from qk(g0 + nk + 2 * j, j)
            for j in range(nk):                      # one wait per pass-2 chunk
                gv, gk, b = g0 + nk + 2 * j + 1, g0 + nk + 2 * j + 4, j & 1
                more = j + 2 < nk
                if drop != "p":
                    yield W(("s_empty", b), uses[b])     # P(j) written over S(j)
                yield W(full(gv), gv // SLOTS + 1)
                if more:
                    yield W(full(gk), gk // SLOTS + 1)
                assert s_done[b] == s_written[b], "S buffer read as P(j), and overwritten, before P(j) was written"
                assert pass1_read[0] == (i + 1) * nk, "P V^T into the third S buffer before its scores were read"
                yield release(gv)                    # P V^T(j)
                if more:                             # Q K^T(j + 2) into the same buffer
                    scores(b)
                    used(b)
                    yield release(gk)
                    yield A(("s_full", b))
            yield A("pv_done")
            gm = g0 + 3 * nk
            yield W("z_full", i + 1)
            yield W(full(gm), gm // SLOTS + 1)
            yield W(full(gm + 1), (gm + 1) // SLOTS + 1)
            assert tac_read[0] == tac_written[0]
            tac_written[0] += 1
            yield release(gm)
            yield release(gm + 1)
            yield A("tac_done")
        if my:
            yield W("tac_done", my)                  # every MMA done before TMEM is freed

    def softmax():
        reads, mask = [0, 0, 0], 0                   # scores taken from each buffer, and the kernel's mask

        def wait_scores(b):
            nonlocal mask
            yield W(("s_full", b), reads[b] + 1)
            assert (mask >> b & 1) == reads[b] & 1 and s_written[b] == reads[b] + 1
            reads[b] += 1
            mask ^= 1 << b

        def put_q(i):
            gq = i * E
            yield W(full(gq), gq // SLOTS + 1)
            yield A("q_full")
        if my:
            yield from put_q(0)
        for i in range(my):
            g0 = i * E + 1
            for it in range(nk):                     # pass 1: read S, arrive
                yield from wait_scores(it % 3)
                s_done[it % 3] += 1
                pass1_read[0] += 1
                yield A(("s_empty", it % 3))
            for j in range(nk):                      # pass 2: read S, write P over it, arrive
                yield from wait_scores(j & 1)
                s_done[j & 1] += 1
                yield A(("s_empty", j & 1))
            yield W("pv_done", i + 1)                # Z_hat over the second S buffer, after every P V^T
            if i + 1 < my:
                yield from put_q(i + 1)
            yield A("z_full")
            go = g0 + 3 * nk + 2                     # the output boxes' slot
            yield W("tac_done", i + 1)
            yield W(full(go), go // SLOTS + 1)
            tac_read[0] += 1
            yield A(("s_empty", 2))                  # the third S buffer is the MMA warp's again
            yield release(go)

    rng = random.Random(seed)
    roles = {"tma": tma(), "mma": mma(), "softmax": softmax()}
    cur = {k: next(v, None) for k, v in roles.items()}

    def ready(step):
        return step[0] == "arrive" or bar(step[1]).phases >= step[2]

    while any(c is not None for c in cur.values()):
        live = [k for k, c in cur.items() if c is not None and ready(c)]
        assert live, f"deadlock at {cur}"
        k = next((r for r in prefer or () if r in live), None) or rng.choice(live)
        step = cur[k]
        if step[0] == "arrive":
            bar(step[1]).arrive()
        else:
            # a parity wait is sound only if the barrier is not two phases on
            assert bar(step[1]).phases in (step[2], step[2] + 1) or step[2] == 0, \
                f"{k} waits for phase {step[2] - 1} of {step[1]}, which has completed {bar(step[1]).phases}"
        cur[k] = next(roles[k], None)


@pytest.mark.parametrize("nk", [1, 2, 3, 4, 5, 6, 7, 8, 16, 64])
@pytest.mark.parametrize("items", [1, 2, 3])
def test_attention_barrier_protocol(nk, items):
    orders = (None, ("tma", "mma"), ("mma", "tma"), ("softmax",), ("softmax", "mma"), ("mma", "softmax"))
    for prefer in orders:
        for seed in range(6 if nk < 64 else 2):
            run(nk, items, seed, prefer)


def test_model_catches_a_missing_wait():
    """The model is not vacuous: without the MMA warp's wait for P(j)
    (P V^T(j) and Q K^T(j + 2) issued before the softmax warps have written
    P over S(j)), a schedule that runs the MMA warp ahead trips the
    S-buffer check, for every chunk count that has a pass-2 Q K^T."""
    for nk in (3, 4, 8):
        with pytest.raises(AssertionError, match="before P\\(j\\) was written"):
            run(nk, 1, 0, prefer=("mma", "tma"), drop="p")
        run(nk, 1, 0, prefer=("mma", "tma"))


def test_model_catches_a_missing_s_wait():
    """Without Q K^T's wait for its S buffer (scores written into a buffer
    whose previous scores the softmax warps have not read yet), the same
    schedule trips the check: with two chunks where pass 2 comes round to the
    first buffer, from four on within pass 1."""
    for nk in (2, 3, 4, 8):
        with pytest.raises(AssertionError, match="previous use was consumed"):
            run(nk, 2, 0, prefer=("mma", "tma"), drop="s")
        run(nk, 2, 0, prefer=("mma", "tma"))


def test_model_catches_a_missing_handover():
    """Without the wait of the next item's third Q K^T for the epilogue's
    release, a schedule that starves the softmax warps writes scores over a
    TAC result they have not read."""
    for nk in (3, 4, 7, 64):
        with pytest.raises(AssertionError, match="before the TAC result was read"):
            run(nk, 2, 0, prefer=("mma", "tma"), drop="handover")
        run(nk, 2, 0, prefer=("mma", "tma"))
