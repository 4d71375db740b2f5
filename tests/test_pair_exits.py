"""The softmax warp pair of the attention kernel leaves together.

Two warps share 64-thread named barriers, which have no time limit, while their
bounded mbarrier waits can end differently in the two: one sees the abort flag,
the other its barrier complete.  So no warp may leave its loops on the outcome of
a wait that it has not exchanged at a pair barrier.  Checked without a GPU: a
model of the two warps' control flow runs over every combination of wait
outcomes, and the kernel's source is held to the rule the model needs.
"""
import itertools
import os
import re

import pytest

ATTN = os.path.join(os.path.dirname(__file__), "..", "paper_2506_02780_gb300", "csrc", "attn.cu")


def _warp(segments, outcome, shared_advance):
    """One softmax warp over segments of the given tile counts: yields each pair
    barrier with what it exchanges there and receives the partner's value;
    outcome(where) is how its wait at that place ends."""
    s = 0
    while True:
        ok = True
        for t in range(segments[s]):
            got = outcome(("scores", s, t))
            if not (yield (s, t), got) or not got:
                ok = False
                break
            if t > 0 and not outcome(("rescale", s, t)):
                ok = False                    # stays with its partner until the segment's end
        have = ok and outcome(("last product", s))
        if shared_advance:
            have = have and outcome(("segment", s + 1))
        if not (yield (s, "end"), have) or not have:
            return
        s += 1
        if not shared_advance and not outcome(("segment", s)):
            return
        if s == len(segments):                # the published end of the walk
            return


def _hangs(segments, outcomes, shared_advance):
    """Run two warps in lockstep; True when one waits at a pair barrier that its partner
    never reaches, or meets it at another one."""
    warps = [_warp(segments, o, shared_advance) for o in outcomes]
    sent = [None, None]
    while True:
        at = []
        for w, v in zip(warps, sent):
            try:
                at.append(w.send(v))
            except StopIteration:
                at.append(None)
        if at[0] is None or at[1] is None:
            return at[0] is not at[1]
        if at[0][0] != at[1][0]:
            return True
        sent = [at[1][1], at[0][1]]


def _places(segments):
    for s, n in enumerate(segments):
        for t in range(n):
            yield ("scores", s, t)
            if t > 0:
                yield ("rescale", s, t)
        yield ("last product", s)
        yield ("segment", s + 1)


def _any_hang(segments, shared_advance):
    """Each warp's waits end well up to one place and badly there (or never); a later
    wait can end either way, since an abort flag does not undo a completed barrier."""
    places = list(_places(segments))
    for fail0, fail1 in itertools.product([None, *places], repeat=2):
        for later in itertools.product((False, True), repeat=2):
            def outcome(fail, late):
                failed = False

                def f(place):
                    nonlocal failed
                    if failed:
                        return late
                    failed = place == fail
                    return not failed
                return f
            if _hangs(segments, [outcome(fail0, later[0]), outcome(fail1, later[1])], shared_advance):
                return True
    return False


@pytest.mark.parametrize("segments", [(1,), (3,), (1, 2), (2, 1, 3)])
def test_exchanged_exits_leave_no_partner_behind(segments):
    assert not _any_hang(segments, shared_advance=True)


def test_a_segment_wait_decided_alone_would():
    assert _any_hang((1, 2), shared_advance=False)


def test_the_kernel_exchanges_every_exit():
    src = re.sub(r"//[^\n]*", "", open(ATTN).read()[open(ATTN).read().index("softmax: one query row"):])
    soft = src[:src.index("__syncthreads()")]
    # the walk takes its first segment behind a CTA barrier and later ones without a wait
    assert re.search(r"for \(bool more = first\(false\); more && ok; more = next_published\(\)\)", soft)
    assert not re.search(r"\b(next|receive)\(", soft)
    bars = [m.start() for m in re.finditer(r"bar\.sync %0, 64", soft)]
    assert len(bars) == 2
    # the scores' wait goes out with the row maxima, those for the last product and the
    # next segment with the sums; the remaining one, before a rescale, only clears ok
    scores, rescale, last, segment = (m.start() for m in re.finditer(r"\bwait\(", soft))
    assert scores < soft.index("got ? __float_as_uint(tmax) : kFail") < bars[0] < rescale
    assert rescale < last < segment < soft.index("s_xok[nseg & 1][qd][hf] = have") < bars[1]
    # the ways out: a failed exchange of the scores, or !ok after the segment's end,
    # where a warp that alone lost ok has told its partner (have starts with ok)
    (out,) = (m.start() for m in re.finditer(r"\b(break|return)\b", soft))
    assert "got && other != kFail" in soft[bars[0]:out] and out < rescale
    assert "const bool have = ok &&" in soft and soft[bars[1]:].count("if (!both) ok = false;") == 1
