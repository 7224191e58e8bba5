"""Order of the replicated level's bulk copies in the resident kernel, checked on the host.

Each HSS step a CTA stores its rows of the first replicated level's right side and copies them to
every other CTA.  Its next store to those rows has to come after every receiver has them, for the
copy reads them until then.  The order of the events is read from the kernel's source; the model has
the edges that order CTAs: a copy before its receiver's wait ends, every arrival at the cluster
barrier before any wait of it ends, and a halo exchange between neighbours per pass (the fewest
passes between two restrictions: one distributed level)."""
import os

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_18694_gb300", "csrc",
                   "resident.cu")
PASSES = 5  # post-sweeps 2, HSS right side, second pre-sweep, residual


def restrict_events():
    """(event, ...) of restrict_pass on a CTA that has not given up, in program order"""
    text = open(SRC).read()
    body = text[text.index(" restrict_pass("):]
    body = body[:body.index("\n}\n")]
    marks = {"wait": "barrier.cluster.wait", "store": "M.b - M.W + at, acc", "copy": "cp.async.bulk",
             "received": "(&hd.mbr[copies & 1], "}
    at = {e: body.index(m) for e, m in marks.items()}
    assert all(body.count(m) == 1 for m in marks.values())
    return sorted(at, key=at.get)


@pytest.mark.parametrize("cs", [2, 16])
def test_copied_rows_are_overwritten_after_every_receiver_has_them(cs):
    order = restrict_events() + ["arrive"] + [f"pass{q}" for q in range(PASSES)]
    after = {}  # event -> events it comes before

    def edge(a, b):
        after.setdefault(a, []).append(b)

    for r in range(cs):
        chain = [(r, t, e) for t in range(2) for e in order]
        for a, b in zip(chain, chain[1:]):
            edge(a, b)
        for t in range(2):
            for d in range(cs):
                if d != r:
                    edge((r, t, "copy"), (d, t, "received"))
                if t == 0:
                    edge((r, 0, "arrive"), (d, 1, "wait"))
            for q in range(PASSES):  # a pass ends with the rows that the neighbours sent in it
                nxt = (t, f"pass{q + 1}") if q + 1 < PASSES else (t + 1, order[0])
                for d in (r - 1, r + 1):
                    if 0 <= d < cs:
                        edge((r, t, f"pass{q}"), (d, *nxt))
    for d in range(cs):
        seen, todo = set(), [(d, 0, "received")]
        while todo:
            for b in after.get(todo.pop(), []):
                if b not in seen:
                    seen.add(b)
                    todo.append(b)
        assert all((s, 1, "store") in seen for s in range(cs)), d
