"""Rules that the CUDA sources keep and no run can show: a kernel that may be
placed while the launch before it runs reads nothing before its own wait, and
a barrier handed to a function is passed by the whole block at once."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_08692_gb300", "csrc")


def _sources():
    out = {}
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".hpp")):
            text = open(os.path.join(CSRC, name)).read()
            out[name] = re.sub(r"//[^\n]*", "", text)
    return out


def _body(text, at):
    """The braced block that opens at or after `at`."""
    start = text.index("{", at)
    depth = 0
    for k in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[start + 1:k]
    raise AssertionError("unbalanced braces")


def _depth(body, at):
    return body.count("{", 0, at) - body.count("}", 0, at)


def test_every_trigger_has_its_wait():
    """griddepcontrol.launch_dependents stands in follow_launch alone, which
    waits for the launch before in every thread that passes it."""
    found = 0
    for name, text in _sources().items():
        for m in re.finditer(r"griddepcontrol\.launch_dependents", text):
            head = text.rindex("__device__", 0, m.start())
            body = _body(text, head)
            assert "griddepcontrol.wait" in body, (name, text[head:m.start()])
            assert "if" not in body, (name, text[head:m.start()])
            found += 1
    assert found == 1


def test_chained_kernels_wait_before_they_read():
    chained, definitions = set(), {}
    for text in _sources().values():
        for m in re.finditer(r"launch_chained\(([^;]*);", text):
            chained |= set(re.findall(r"\bk_\w+", m.group(1)))
        for m in re.finditer(r"auto\* kernel =([^;]*);\s*return launch_chained", text):
            chained |= set(re.findall(r"\bk_\w+", m.group(1)))
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
            definitions[m.group(1)] = _body(text, m.end())
    assert len(chained) >= 9 and chained <= set(definitions)
    for name in chained:
        body = definitions[name]
        at = body.find("follow_launch();")
        assert at >= 0 and _depth(body, at) == 0, name
        before = body[:at]
        assert not re.search(r"\b(if|for|while|return)\b|E\.|->", before), (name, before)


def test_shared_emission_meets_at_one_barrier():
    """emit_shared's two warps take different branches; the barrier between
    them stands outside both, once."""
    text = _sources()["shower_cycle.cuh"]
    body = _body(text, text.index("emit_shared("))
    calls = [m.start() for m in re.finditer(r"\bsync\(\);", body)]
    assert len(calls) == 1 and _depth(body, calls[0]) == 0
    assert "__syncthreads" not in body
