"""The K/V ring of the two-tile refresh kernel: every copy into a slot is ordered after the MMAs that read it.

A model of refresh_tc_kernel's roles as a graph of what comes before what: each stream's MMAs complete in issue
order, a stream's turn starts once the other's P V is issued (its last MMAs of S may still be to come), P(t) is
written after S(t) has completed, and tile T is copied after `done[T - ahead]`. Who arrives on `done` is read from
the kernel's source: B's softmax alone (a count of one) leaves A's reads of a slot unordered with the next copy.
"""

import os
import re

import pytest

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_2609_05821_gb300", "csrc", "refresh_tc.cu")


def _releasers():
    with open(SRC) as f:
        src = f.read()
    count = int(re.search(r"mbar_init\(&s\.done\[i\], (\d+)\)", src).group(1))
    commits = "mma_commit_if(frees, &s.done[" in src
    assert "mbar_arrive_if(releases, &s.done[" in src and count == 1 + commits
    return "AB" if commits else "B"


def _model(items, stages, releasers):
    """Edges (event -> events it comes after) of a CTA that takes items of (key tiles of A, of B)."""
    ahead = (stages - 1) // 2
    after = {}
    edge = lambda e, *before: after.setdefault(e, set()).update(b for b in before if b)
    base, last_mma, last_issue, prev_turn = 0, {"A": None, "B": None}, {"A": None, "B": None}, {"A": None, "B": None}
    reads = {}  # slot -> MMAs that read its present content, in program order of the copies

    def mma(x, name, *before):
        issue, done = ("issue", x, name), ("done", x, name)
        edge(issue, last_issue[x], *before)
        edge(done, issue, last_mma[x])
        last_issue[x], last_mma[x] = issue, done
        return done

    for nt_a, nt in items:
        n_t = {"A": nt_a, "B": nt}
        for t in range(-1, nt):
            for x in "AB":
                T = base + t + 1
                handed = prev_turn["B" if x == "A" else "A"]
                p_v = None
                if 0 <= t < n_t[x]:
                    p_v = mma(x, ("PV", base + t), ("copied", "V", base + t), ("done", x, ("S", base + t)), handed)
                    reads.setdefault(("V", base + t), []).append(p_v)
                # the turn passes once P V is issued; the MMAs of S may follow
                edge(("turn", x, base, t), last_issue[x], handed)
                prev_turn[x] = ("turn", x, base, t)
                if t + 1 < n_t[x]:
                    s = mma(x, ("S", T), ("copied", "K", T), handed)
                    reads.setdefault(("K", T), []).append(s)
                if t + 1 < nt:
                    if x == "A" and "A" in releasers:
                        edge(("free", T), last_mma["A"], prev_turn["A"])
                    if x == "B":
                        edge(("free", T), ("done", "B", ("S", T)))
        base += nt
    for T in range(base):
        for what in "KV":
            edge(("copied", what, T), ("free", T - ahead) if T >= ahead else None)
    return after, reads, base


def _before(after, e, memo):
    """Everything that comes before event e."""
    if e not in memo:
        memo[e] = set()
        for b in after.get(e, ()):
            memo[e] |= {b} | _before(after, b, memo)
    return memo[e]


ITEMS = [[(4, 4), (3, 7)], [(0, 5), (2, 2), (0, 1)], [(1, 6), (0, 3), (5, 5)], [(1, 1)] * 8, [(9, 10), (1, 9)]]


def _unordered(items, stages, releasers):
    after, reads, n = _model(items, stages, releasers)
    bad, memo = [], {}
    slot = lambda what, T: (2 * T + (what == "V")) % stages
    order = [(w, T) for T in range(n) for w in "KV"]
    for i, (w, T) in enumerate(order):
        old = next(((v, U) for v, U in reversed(order[:i]) if slot(v, U) == slot(w, T)), None)
        if old:
            here = _before(after, ("copied", w, T), memo)
            bad += [(old, (w, T)) for r in reads.get(old, []) if r not in here]
    return bad


@pytest.mark.parametrize("stages", (5,))
@pytest.mark.parametrize("items", ITEMS)
def test_copies_follow_the_reads_of_their_slot(items, stages):
    assert not _unordered(items, stages, _releasers())


def test_one_stream_alone_does_not_free_a_slot():
    assert _unordered(ITEMS[0], 5, "B")
