"""The rules a kernel that overlaps its predecessor in the stream keeps, read
off the sources: no read-only pointer to data an overlapping launch may write
(the compiler may move such loads over the wait), and no way out that passes
by the wait (a launch that ends before the one it overlaps lets later launches
overlap that one too)."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_29692_gb300", "csrc")
WAIT = re.compile(r"pdl_wait\(\);|griddepcontrol\.wait")
# tables filled at context creation, and a state that is final before the launch
# ahead starts (the gradient pass, launched without overlap, lies in between)
FINAL = {("k_line_search", "sc"), ("k_line_search", "rank"), ("k_line_support", "psi")}


def kernels():
    """(name, parameters, body) of every kernel that waits for its predecessor."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__ void(?: __launch_bounds__\((?:[^()]|\([^()]*\))*\))?\s+(\w+)\(", text):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            params, start = text[m.end():i - 1], text.index("{", i)
            j, depth = start + 1, 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                j += 1
            body = text[start:j]
            if WAIT.search(body):
                yield m.group(1), params, body


def test_no_read_only_pointer_to_data_of_an_overlapping_launch():
    found = [(name, p) for name, params, _ in kernels()
             for p in re.findall(r"const [\w:<> ]+\*\s*__restrict__ (\w+)", params)]
    assert len(list(kernels())) >= 8
    assert sorted(set(found) - FINAL) == []


def test_a_converged_step_waits_before_it_returns():
    seen = 0
    for name, _, body in kernels():
        for m in re.finditer(r"converged\)\s*(\{[^}]*return;|return;)", body):
            # a wait in the block of the return, or ahead of it: for sure, or whenever there is a step record
            ahead = re.search(r"[;{]\s+(?:if \(gate\) )?(?:asm volatile\(\")?(?:pdl_wait|griddepcontrol\.wait)", body[:m.start()])
            assert ahead or WAIT.search(m.group(1)), name
            seen += 1
    assert seen >= 5
