"""Every wait of a kernel on another thread, warp or block is bounded by the handle's limit (oras_options.wait_ms): the
wait functions have no default for it, and every call passes one that comes from the handle."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1605_04521_gb300", "csrc")
WAITS = ("mbar_wait", "wait_counter", "grid_wait")


def sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f)) as s:
                yield f, re.sub(r"//[^\n]*", "", s.read())


def arguments(text, at):
    """The text between the parenthesis at `at` and the one that closes it."""
    depth, i = 0, at
    while True:
        depth += {"(": 1, ")": -1}.get(text[i], 0)
        i += 1
        if depth == 0:
            return text[at + 1:i - 1]


def test_every_wait_takes_the_handles_limit():
    calls = 0
    for f, text in sources():
        for m in re.finditer(r"\b(%s)(?=\()" % "|".join(WAITS), text):
            args = arguments(text, m.end())
            last = re.split(r",(?![^(]*\))", args)[-1].strip()
            if re.match(r"uint64_t ", last):               # the declaration
                assert "=" not in last, (f, m.group(1), last)
                continue
            calls += 1
            assert re.fullmatch(r"(a\.)?(wait_ns|limit_ns)|drain_limit\((a\.)?wait_ns\)", last), (f, m.group(1), last)
    assert calls > 15
