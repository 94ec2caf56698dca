"""A wait of the decode kernel that gives up in some warps of a group and not in others: all four warps must leave, together.

Run on a model on the CPU (a GPU test would need a wait that never completes while copies and MMAs are in flight). The order of waits,
votes, barriers and arrivals, and what a wait that gave up does, are read from the kernel's source; the warps of one group are
interleaved over it, with every choice of the warps and of the wait that give up."""
from __future__ import annotations

import itertools
import os
import random
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2608_08081_b200", "csrc", "iq_decode_kernel.cuh")
STAGES = 3


def _body(text, opening):
    """The text between the braces that the first match of `opening` ends with."""
    m = re.search(opening, text)
    assert m, opening
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[m.end():i - 1], i


TOKEN = re.compile(r"mbar_wait_\w+\(&?(?P<wait>s_bar|o_bar)\b|(?P<slot>next_slot\(\))|(?P<vote>group_bar_or\()|(?P<sync>group_bar_sync\()"
                   r"|mbar_arrive\((?P<arrive>\w+)\)|(?P<ktile>\bk_tile\()")


def _tokens(text):
    out = []
    for m in TOKEN.finditer(text):
        statement = text[m.start():].split(";")[0]
        if m["wait"] or m["slot"]:  # a wait that gave up: the warp votes at once, goes on to the next vote, or leaves
            goes_on = "failed |=" in text[:m.start()].rsplit("\n", 1)[1]
            out.append(("wait", m["wait"] or "full", "vote" if "give_up()" in statement else "go on" if goes_on else "leave"))
        elif m["vote"]:  # whether a warp that gave up before votes for leaving
            named = re.search(r"\bexceed\)", statement) and re.search(r"bool exceed = [^;]*\bfailed;", text)
            out.append(("vote", bool(re.search(r"\bfailed\)", statement) or named)))
        elif m["sync"]:
            out.append(("sync",))
        else:
            out.append(("arrive", m["arrive"] or "k_ready"))
    return out


def _program(path):
    """What a compute warp does: at the first slot, when it opens a segment, in a block, when it closes the segment, when it gives up."""
    text = re.sub(r"//[^\n]*", "", open(SOURCE).read())
    text = text[text.index("if (!control) {"):text.index("allow_dependent_launch();\n  if (__syncthreads_or")]
    opening = _tokens(_body(text, r"auto open_segment = [^{]*\{")[0])
    close = _body(text, r"auto close_segment = [^{]*\{")[0]
    plain, end = _body(close, r"if constexpr \(!ARGMAX\) \{")
    closes = [_tokens(plain), _tokens(close[end:])]
    give_up = _tokens(_body(text, r"auto give_up = [^{]*\{")[0]) if "auto give_up" in text else []
    first = re.search(r"\n[^\n]*next_slot\(\);?[^\n]*\n\s*(if \(failed\)[^\n]*\n\s*)?if constexpr \(I8\) \{", text)
    assert first
    int8, end = _body(text, r"if constexpr \(I8\) \{\s*constexpr int NLR")
    segments = int8 if path == "int8" else _body(text[end:], r"^ else \{")[0]
    block, end = _body(segments, r"while \(more\) \{")
    behind = re.match(r"\s*if \((\w+)\) break;", segments[end:])[1]  # who leaves behind the blocks: warps that gave up, or that left a block
    block = _tokens(block)
    assert [t[1] for t in block if t[0] == "wait"] == ["s_bar", "full", "o_bar"] and [t[0] for t in block][1] == "vote"
    assert opening == [("sync",)] and all(1 <= len(c) <= 2 for c in closes) and behind in ("failed", "more")
    return dict(first_vote="group_bar_or" in first[0], opening=opening if path == "int8" else [], block=block, closes=closes, give_up=len(give_up),
                behind=behind)


class _Left(Exception):
    pass


def _warp(prog, close, segments, raises, own_operand):
    """One warp as a generator of requests; returns True if it gave up."""
    gave_up = False

    def wait(bar, n, then):
        nonlocal gave_up
        if not (yield ("wait", bar, n)):
            gave_up = True
            if then == "vote":
                for _ in range(prog["give_up"]):
                    yield ("vote", True)
            if then != "go on":
                raise _Left

    try:
        ok = yield ("wait", "full", 0)
        if prog["first_vote"]:
            if (yield ("vote", not ok)):
                return True
        elif not ok:
            return True
        n = 0
        for blocks in segments:
            if own_operand:
                for _ in prog["opening"]:
                    yield ("sync",)
            yield ("arrive", "k_ready", n)
            for i in range(blocks):
                raised = None
                for t in prog["block"]:
                    if t[0] == "wait":
                        yield from wait(t[1], n + (t[1] == "full"), t[2])
                    elif t[0] == "vote" and raised is None:
                        raised = yield ("vote", raises[n] or (t[1] and gave_up))
                    elif t[0] == "vote":  # behind a vote that passed: on leaving
                        if raised and (yield ("vote", t[1] and gave_up)):
                            raise _Left
                    elif t[0] == "sync":
                        if raised:
                            yield ("sync",)
                    elif t[1] == "p_ready":
                        yield ("arrive", "p_ready", n)
                    elif i + 1 < blocks:  # the next block of the segment
                        yield ("arrive", "k_ready", n + 1)
                n += 1
            if prog["behind"] == "failed" and gave_up:
                raise _Left
            if close[0][0] == "sync":
                yield ("sync",)
            elif (yield ("vote", close[0][1] and gave_up)):
                for _ in close[1:]:
                    yield ("vote", True)
                raise _Left
        return False
    except _Left:
        return True


def _run(prog, close, segments, raises, own_operand, gives_up, rng):
    """Interleaves four warps; gives_up: (warp, number of its wait) pairs. Returns what the warps returned; None: one never leaves."""
    warps = [_warp(prog, close, segments, raises, own_operand) for _ in range(4)]
    asks = [next(w) for w in warps]
    waits, result = [0] * 4, [None] * 4
    arrived, at_barrier = {}, []
    control_left = []  # the last MMAs that the control warp issued, over whatever was there, when its own wait gave up

    def done(bar, n):
        full = lambda kind, i: len(arrived.get((kind, i), ())) == 4  # noqa: E731
        if control_left:
            return (bar, n) in control_left or bar == "full" and n < STAGES or n < control_left[0][1]
        if bar == "full":  # a slot is staged again once the scores of the block after its last one have been issued
            return n < STAGES or full("k_ready", n - STAGES + 1)
        return full("k_ready" if bar == "s_bar" else "p_ready", n)

    def answer(w, value):
        try:
            asks[w] = warps[w].send(value)
        except StopIteration as e:
            asks[w], result[w] = None, e.value

    while any(a is not None for a in asks):
        ready, stuck = [], []
        for w, a in enumerate(asks):
            if a is None or w in at_barrier:
                continue
            (stuck if a[0] == "wait" and not done(a[1], a[2]) and (w, waits[w]) not in gives_up else ready).append(w)
        if not ready and not stuck:
            return None  # everybody that is left stands at a barrier
        if not ready and not control_left and rng.random() < 0.5:  # nothing moves: a wait runs out, the control warp's ...
            control_left.append(max((asks[v][1:] for v in stuck if asks[v][1] != "full"), key=lambda x: x[1], default=("full", 0)))
            continue
        w = rng.choice(ready or stuck)  # ... or one of these warps'
        a = asks[w]
        if a[0] == "wait":
            ok = bool(ready) and (w, waits[w]) not in gives_up
            waits[w] += 1
            answer(w, ok)
        elif a[0] == "arrive":
            arrived.setdefault(a[1:], set()).add(w)
            answer(w, None)
        else:
            assert all(asks[v][0] == a[0] for v in at_barrier), "a vote and a plain barrier meet"
            at_barrier.append(w)
            if len(at_barrier) == 4:
                value = any(asks[v][1] for v in at_barrier) if a[0] == "vote" else None
                everybody, at_barrier = at_barrier, []
                for v in everybody:
                    answer(v, value)
    return result


@pytest.mark.parametrize("argmax", [0, 1])
@pytest.mark.parametrize("path", ["int8", "fp16"])
def test_a_group_leaves_together(path, argmax):
    prog = _program(path)
    rng = random.Random(7)
    for segments, own_operand in itertools.product([(), (1,), (3,), (1, 2), (2, 1, 1)], [False, True]):
        blocks = sum(segments)
        for style in ("never", "always", "mixed"):
            raises = [style == "always" or (style == "mixed" and rng.random() < 0.5) for _ in range(blocks)]
            args = (prog, prog["closes"][argmax], segments, raises, own_operand)
            assert _run(*args, set(), rng) == [False] * 4
            for number in range(3 * blocks + 1):
                for mask in range(1, 16):
                    assert _run(*args, {(w, number) for w in range(4) if mask >> w & 1}, rng) == [True] * 4, (segments, style, number, mask)
            for _ in range(50):  # warps that give up at different waits
                some = {(w, rng.randrange(3 * blocks + 1)) for w in range(4) if rng.random() < 0.6}
                assert _run(*args, some, rng) == [bool(some)] * 4, (segments, style, some)
