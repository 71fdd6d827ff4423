"""Kernels that may start beside the previous one (they call wait_for_previous): no
pointer parameter is __restrict__ and nothing is read with __ldg, but for the
constants written before any such launch. Either would tell the compiler that the
memory does not change while the kernel runs, which starts before its inputs are
written."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0908_3749_gb300", "csrc")
CONSTANTS = ("LogEntry", "ExpEntry", "bconst")


def _close(text, at, pair):
    depth = 0
    for j in range(at, len(text)):
        depth += (text[j] == pair[0]) - (text[j] == pair[1])
        if depth == 0:
            return j
    raise ValueError("unbalanced")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__", text):
            name = re.compile(r"\b(k_\w+)\(").search(text, m.end())
            end = _close(text, name.end() - 1, "()")
            body = text.index("{", end)
            yield (os.path.basename(path), name.group(1), text[name.end():end],
                   text[body:_close(text, body, "{}") + 1])


def test_overlapped_kernels_read_their_inputs_behind_the_wait():
    found = []
    for path, name, params, body in _kernels():
        if "wait_for_previous()" not in body:
            continue
        found.append(name)
        for p in params.split(","):
            assert "__restrict__" not in p or any(c in p for c in CONSTANTS), (path, name, p.strip())
        assert "__ldg" not in body, (path, name)
    assert {"k_conv", "k_wgrad", "k_update", "k_step", "k_step_pipe", "k_step2", "k_step_tc", "k_step_lanes"} <= set(found)
