"""The barrier protocol of the shared-row-tile attention (attention_umma.cu, `kpar`) as a model: two softmax groups, an MMA
issuer per group, one score buffer and barrier per three key tiles, K / V tiles that arrive in any order.  A wait by
parity passes when the barrier has completed an odd number of phases more (or fewer) than the waiter believes, which no
run on a GPU shows reliably; here the order of events is drawn at random."""
import os
import random
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_06295_b200", "csrc")
STAGES = 6


class Barrier:
    """mbarrier with one arrival per phase: wait(parity) passes iff the phase of that parity is the last completed."""

    def __init__(self):
        self.done = 0

    def passed(self, parity):
        return self.done & 1 != parity


def issuer(i, first_scores, n_tiles, kv, p_full, queue):
    for t in first_scores:
        yield lambda t=t: kv[t % STAGES].passed(t // STAGES & 1)
        queue.append(("S", t))
    for u, t in enumerate(range(i, n_tiles, 2)):
        yield lambda u=u: p_full[i].passed(u & 1)
        queue.append(("O", t))
        if t + 3 < n_tiles:
            yield lambda t=t: kv[(t + 3) % STAGES].passed((t + 3) // STAGES & 1)
            queue.append(("S", t + 3))


def group(i, n_tiles, s_full, o_full, p_full, read):
    for u, t in enumerate(range(i, n_tiles, 2)):
        yield lambda t=t: s_full[t % 3].passed(t // 3 & 1)
        read.append(t)
        yield lambda: True                                   # the softmax: anything may happen meanwhile
        if u:
            yield lambda u=u: o_full[i].passed((u - 1) & 1)
        p_full[i].done += 1


def run(start, n_tiles, rng):
    """One run; returns the tiles whose scores a group took before they were complete, or None if it got stuck."""
    kv, s_full, o_full, p_full = ([Barrier() for _ in range(k)] for k in (STAGES, 3, 2, 2))
    queues, read = ([], []), []
    complete = [set(), set()]                                # S and O tiles
    actors = [issuer(i, start[i], n_tiles, kv, p_full, queues[i]) for i in (0, 1)]
    actors += [group(i, n_tiles, s_full, o_full, p_full, read) for i in (0, 1)]
    waits = [next(a) for a in actors]
    weight = [rng.choice((1, 1, 20)) for _ in range(4)]      # some runs have a slow actor, or slow products
    arrived, early, slow_copy = set(), [], rng.random() < 0.5
    while any(w is not None for w in waits) or queues[0] or queues[1]:
        moves = [("actor", k) for k, w in enumerate(waits) if w is not None and w() for _ in range(weight[k])]
        moves += [("mma", i) for i in (0, 1) if queues[i] for _ in range(1 if slow_copy else 5)]   # in order per issuer
        moves += [("copy", t) for t in range(n_tiles) if t not in arrived and
                  (t < STAGES or t - STAGES in complete[1])]                                        # any order
        if not moves:
            return None
        what, k = rng.choice(moves)
        if what == "actor":
            before = len(read)
            waits[k] = next(actors[k], None)
            early += [t for t in read[before:] if t not in complete[0]]
        elif what == "mma":
            kind, t = queues[k].pop(0)
            complete[kind == "O"].add(t)
            (o_full[t & 1] if kind == "O" else s_full[t % 3]).done += 1
        else:
            arrived.add(k)
            kv[k % STAGES].done += 1
    return early


@pytest.mark.parametrize("n_tiles", [4, 5, 8, 13, 24])
def test_groups_only_read_complete_scores(n_tiles):
    one_issuer = ((0, 1, 2), ())
    for seed in range(500):
        assert run(one_issuer, n_tiles, random.Random(seed)) == []


def test_the_model_finds_a_start_shared_by_the_issuers():
    """S(0) and S(2) from one issuer, S(1) from the other: group 1 may wait for S(3) before S(0) is complete."""
    early = [run(((0, 2), (1,)), 8, random.Random(seed)) for seed in range(500)]
    assert any(early) and {t for e in early for t in e or ()} >= {3}


def test_the_kernel_starts_with_one_issuer():
    src = open(os.path.join(CSRC, "attention_umma.cu")).read()
    end = src.index("int buf = ")                              # the issuers' walk over the tiles; their start precedes it
    startup = re.sub(r"//[^\n]*", "", src[src.rindex("if (kpar)", 0, end):end])
    assert re.search(r"for \(int t = 0; t < 3 && ok && i == 0; \+\+t\)", startup)
    assert startup.count("issue_s(") == 1 and "tile_ready(t)" in startup
