"""The hand-off of the 256-channel F-stage (ppf_correct_ws256_kernel) between its
FIR threads and its two groups of FFT threads, checked on the host.

Agents on counting barriers with the semantics of bar.sync / bar.arrive, in
random interleavings. Group g takes the rounds b = g mod 2; FULL[q] and EMPTY[q]
belong to row buffer q = b mod NB and have two parties, the FIR threads and the
group whose rounds use that buffer.

  FP32, split FP16  NB = 4. A buffer is the round's rows (overwritten in place by
                    the group's P1 between its two own barriers) and its table of
                    anchors; both are free at EMPTY[q], from round 4 on.
  FP16, BF16        NB = 2. The table of factors has an EMPTY of its own
                    (EMPTYF[q]): the FIR threads wait for it in the middle of a
                    round, and the group arrives there after it has read the
                    factors, which is after it gave the rows back.

Every interleaving must finish, every read must see its own round's data, and
no barrier may be left half arrived."""
import random

import pytest


def fir(rounds, nb, table_apart, wait_table=True):
    for b in range(rounds):
        q = b % nb
        if b >= nb:
            yield "sync", ("EMPTY", q)
        if not table_apart:
            yield "write", ("table", q, b)
        yield "write", ("rows", q, b)
        if table_apart:
            if b >= nb and wait_table:
                yield "sync", ("EMPTYF", q)
            yield "write", ("table", q, b)
            yield "write", ("rows", q, b)             # second half of the round's outputs
        yield "arrive", ("FULL", q)


def group(g, rounds, nb, table_apart, wait_table=True, table_with_rows=False):
    for b in range(g, rounds, 2):
        q, again = b % nb, b + nb < rounds
        yield "sync", ("FULL", q)
        yield "read", ("rows", q, b)
        yield "write", ("rows", q, ("P1", b))
        yield "read", ("rows", q, ("P1", b))
        if table_apart:
            if again:
                yield "arrive", ("EMPTY", q)
                if table_with_rows and wait_table:
                    yield "arrive", ("EMPTYF", q)
            yield "read", ("table", q, b)
            if again and wait_table and not table_with_rows:
                yield "arrive", ("EMPTYF", q)
        else:
            yield "read", ("table", q, b)
            if again:
                yield "arrive", ("EMPTY", q)


def simulate(agents, seed):
    rng = random.Random(seed)
    count, generation, memory, waiting = {}, {}, {}, {}

    def arrive(key):
        count[key] = count.get(key, 0) + 1
        if count[key] == 2:
            count[key], generation[key] = 0, generation.get(key, 0) + 1

    ops = {k: next(a, None) for k, a in enumerate(agents)}
    while any(op is not None for op in ops.values()):
        ready = [k for k, op in ops.items() if op is not None and
                 (k not in waiting or generation.get(waiting[k][0], 0) >= waiting[k][1])]
        if not ready:
            return "deadlock"
        k = rng.choice(ready)
        kind, arg = ops[k]
        if k in waiting:                              # its sync has completed
            del waiting[k]
        elif kind == "sync":
            target = generation.get(arg, 0) + 1
            arrive(arg)
            if generation.get(arg, 0) < target:
                waiting[k] = (arg, target)
                continue
        elif kind == "arrive":
            arrive(arg)
        elif kind == "write":
            memory[arg[:2]] = arg[2]
        elif memory.get(arg[:2]) != arg[2]:
            return "stale"
        ops[k] = next(agents[k], None)
    return "partial" if any(count.values()) else "ok"


def outcomes(rounds, nb, apart, fir_kw={}, group_kw={}):
    return {simulate([fir(rounds, nb, apart, **fir_kw), *(group(g, rounds, nb, apart, **group_kw) for g in (0, 1))], seed)
            for seed in range(200)}


@pytest.mark.parametrize("nb,apart", [(4, False), (2, True)])
@pytest.mark.parametrize("rounds", [1, 2, 3, 4, 5, 6, 9, 64])
def test_handoff_completes_and_reads_its_own_round(rounds, nb, apart):
    assert outcomes(rounds, nb, apart) == {"ok"}


@pytest.mark.parametrize("planted", [(dict(wait_table=False), dict(wait_table=False)),   # the table's own wait missing
                                     ({}, dict(table_with_rows=True))])                  # released before it is read
def test_planted_mistakes_are_caught(planted):
    assert outcomes(12, 2, True, *planted) - {"ok"}


def test_two_buffers_without_a_wait_are_caught():
    """Four buffers' rule (EMPTY from round 4 on) on two buffers overwrites rows in use."""
    def hasty(rounds):
        for op, arg in fir(rounds, 2, False):
            if op != "sync":
                yield op, arg
    seen = {simulate([hasty(9), group(0, 9, 2, False), group(1, 9, 2, False)], s) for s in range(200)}
    assert seen - {"ok"}
