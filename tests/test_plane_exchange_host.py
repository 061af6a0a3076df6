"""The pivot-column exchange of the coarse plane factorisation, as an order of
reads and writes between CTAs (no GPU).

At step k every CTA waits at barrier k, arrives at barrier k + 1 (the owner of
column k + 1 after storing it into buffer (k + 1) mod 3 of every CTA) and reads
buffer k mod 3. What a CTA did before an arrive happens before what follows the
wait of another only if the arrive releases and the wait acquires; that order has
to cover both the store before its reads and the reads before the store that
reuses their buffer. The qualifiers are taken from the kernel's source."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1912_06934_gb300", "csrc",
                   "coarse_planes.cu")


def _ordered(nct, m, owner_arrive, other_arrive, wait):
    """Whether every conflicting pair of accesses is ordered, by vector clocks."""
    clock = [[0] * nct for _ in range(nct)]  # clock[c][d]: the last event of d that c is after
    sent = [[0] * nct for _ in range(nct)]   # what the pending barrier carries
    last = [[] for _ in range(3)]            # accesses of a buffer since its last store: (CTA, event)
    fine = True

    def access(c, buf, store):
        nonlocal fine
        clock[c][c] += 1
        seen = last[buf] if store else last[buf][:1]
        fine = fine and all(clock[c][d] >= e for d, e in seen)
        last[buf] = [(c, clock[c][c])] if store else last[buf] + [(c, clock[c][c])]

    def arrive(c, kind):
        sent[c] = list(clock[c]) if kind == "release" else [0] * nct

    for c in range(nct):
        if c == 0:
            access(0, 0, True)
        arrive(c, owner_arrive)
    for k in range(m):
        carried = [max(s[d] for s in sent) for d in range(nct)]
        for c in range(nct):
            if wait == "acquire":
                clock[c] = [max(a, b) for a, b in zip(clock[c], carried)]
        for c in range(nct):  # before the step's reads, as far ahead as a CTA may run
            if k + 1 < m:
                own = c == (k + 1) % nct
                if own:
                    access(c, (k + 1) % 3, True)
                arrive(c, owner_arrive if own else other_arrive)
        for c in range(nct):
            access(c, k % 3, False)
    return fine


def _qualifiers():
    text = open(SRC).read()
    kinds = dict(re.findall(r"void (cluster_\w+)\(\)\s*\{\s*asm volatile\(\"barrier\.cluster\.\w+\.(\w+);\"", text))
    start = text.index(") plane_factor_kernel(")
    body = text[start:text.index("using PlaneFactorFn")]
    arrives = re.findall(r"\b(cluster_arrive\w*)\(\)", body)
    waits = re.findall(r"\b(cluster_wait\w*)\(\)", body)
    assert arrives and waits
    return [kinds[a] for a in arrives], [kinds[w] for w in waits]


@pytest.mark.parametrize("nct", [1, 2, 3, 4, 8, 16])
@pytest.mark.parametrize("m", [1, 2, 5, 40])
def test_pivot_buffers_are_ordered(nct, m):
    arrives, waits = _qualifiers()
    assert "release" in arrives  # the owner's
    for other in set(arrives):
        for w in set(waits):
            assert _ordered(nct, m, "release", other, w)


def test_the_order_needs_release_and_acquire():
    assert _ordered(4, 12, "release", "release", "acquire")
    assert not _ordered(4, 12, "release", "relaxed", "acquire")
    assert not _ordered(4, 12, "relaxed", "release", "acquire")
    assert not _ordered(4, 12, "release", "release", "relaxed")
