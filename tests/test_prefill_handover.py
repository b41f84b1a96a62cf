"""Orders that the tensor-core prefill's warps must keep, on the CPU: every interleaving of a
small model of the hand-over in a run of fast segments, the order of two tensor-core products on
the same columns, and where the time limit of a wait starts.

The hand-over: two builder threads (the loader, which waits and arrives for its group, and any other) and the
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


def _body(src, name):
    """The text of a function from its name to the closing brace in column 0."""
    at = src.index(f" {name}(")
    return src[at:src.index("\n}", at)]


def test_products_on_the_same_columns_have_one_shape():
    """Tensor-core products execute in issue order only on the same accumulator with the same
    shape.  The exact path's update accumulates onto D_O while S^T Q~^T may still run: the
    accumulators both write have one instruction descriptor, and no other overlaps them (S^T
    starts where D_O's 64 columns end)."""
    src = _source("gla_chunk_common.cuh")
    product = re.compile(r"mma_tf32_ts\(tmem \+ (\w+),.*?((?:Geo<D>::)?IDT_\w+)", re.S)
    first = dict(product.findall(_body(src, "exact_issue_sq")))
    second = dict(product.findall(_body(src, "exact_issue_update")))
    assert first.keys() & second.keys() == {"TM_O0"}
    assert first["TM_O0"] == second["TM_O0"] == "IDT_N64"
    assert re.search(r"IDT_N64 = idesc_tf32\(128, 64, ", src)
    assert second == {"TM_O0": "IDT_N64", "TM_S": "Geo<D>::IDT_ST"}
    column = lambda name: int(re.search(rf"constexpr uint32_t {name} = (\d+);", src).group(1))
    assert column("TM_O0") + 64 <= column("TM_S")


def test_output_pass_time_limit_starts_after_the_kernel_before():
    """In the output pass the state warps wait, without a limit, for the scan, while the builders
    already work.  Every bounded wait of theirs on the state warps (bar_go) follows the loader's own
    wait for the scan: a slow scan is not reported as a wait that ran out."""
    kernel = _source("gla_chunked_tc.cu")
    waits = re.findall(r"(\w+)\(\w+, (?:\w+, )?bar_go, (\w+)\)", kernel)
    assert sorted(waits) == [("wait_all", "ph_stall"), ("wait_group", "ph_go")]   # the first: a test hook
    go = kernel[kernel.index("auto wait_go = "):]
    go = go[:go.index("};")]
    assert re.search(r"if \(RESTART && tid == kLoader\)\s*pdl_wait\(\);\s*return wait_group\(1, kLoader, bar_go", go)
    assert kernel.count("wait_go()") == 2
