"""The hand-over between the two warp groups of the tensor-core prefill, on the CPU: every
interleaving of a small model of a run of fast segments.

Two builder threads (the loader, which waits and arrives for its group, and any other) and the
issuing state thread pass the segments on as the kernel's builder_run and state_run do: built ->
decision -> go.  Both builder threads read the decision on the segment before, after a barrier of
their group; a thread that reads another answer than its partner goes to the CTA-wide barrier
alone, and neither barrier ever completes (a hang: they are no bounded waits)."""
import os
import re

import pytest

import paper_2609_15030_gb300 as hs

CSRC = os.path.join(os.path.dirname(hs.__file__), "csrc")
END = 8


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _steps(s, words, fast):
    """The states one step on from s = (loader, builder, issuer, built, go, decisions), each
    thread a (segment, program counter)."""
    loader, other, issuer, built, go, dec = s
    last = len(fast) - 1
    at_barrier = lambda t: t[1] in (0, 2, 7)
    past = lambda t: (t[0], END if t[1] == 7 else t[1] + 1)
    out = []
    if at_barrier(loader) and at_barrier(other):       # a barrier of the builders completes
        out.append((past(loader), past(other), issuer, built, go, dec))
    for me in (0, 1):
        k, pc = t = s[me]
        n_built = built
        if pc in (1, 6):                               # the loader's wait for "go"
            if me == 0 and (pc == 6 or k > 0) and go < k + (pc == 6):
                continue
            t = (k, pc + 1)
        elif pc == 3:                                  # the decision on the segment before
            t = (k, 4 if k == 0 or dec[(k - 1) % words] else END)
        elif pc == 4:                                  # the loader hands the segment over
            n_built += me == 0
            t = (k, 6 if k == last else 5)
        elif pc == 5:
            t = (k + 1, 0)
        else:
            continue
        out.append((t, other, issuer, n_built, go, dec) if me == 0 else
                   (loader, t, issuer, n_built, go, dec))
    k, pc = issuer
    if pc == 0 and built > k:                          # judge segment k
        dec = dec[:k % words] + (fast[k],) + dec[k % words + 1:]
        out.append((loader, other, (k, 1), built, go, dec))
    elif pc == 1:
        out.append((loader, other, (k, END) if k == last or not fast[k] else (k + 1, 0),
                    built, go + 1, dec))
    return out


def _stuck(words, fast):
    """The states in which no thread can move and not all stand at the CTA-wide barrier."""
    seen, todo, stuck = set(), [((0, 0), (0, 0), (0, 0), 0, 0, (1,) * words)], []
    while todo:
        s = todo.pop()
        if s in seen:
            continue
        seen.add(s)
        nxt = _steps(s, words, fast)
        if not nxt and any(t[1] != END for t in s[:3]):
            stuck.append(s)
        todo += nxt
    return stuck


@pytest.mark.parametrize("stop", range(1, 8))
def test_every_builder_thread_reads_the_same_decision(stop):
    """Runs of 1 to 7 segments whose last is fast or not, and runs stopped with one more
    segment built ahead."""
    m = re.search(r"constexpr int kDecisions = (\d+);", _source("gla_chunk_common.cuh"))
    words = int(m.group(1)) if m else 1
    for fast in ((1,) * stop, (1,) * (stop - 1) + (0,), (1,) * (stop - 1) + (0, 1)):
        assert _stuck(words, fast) == []
    if stop > 1:                                       # the model sees the fault of a single word
        assert _stuck(1, (1,) * (stop - 1) + (0, 1))
