"""Block barriers in the CUDA sources: no __syncthreads() stands under an `if` (or its `else`) whose condition
depends on the thread. A barrier that a block's threads reach at different places of the text is undefined in
CUDA C++, whatever the hardware makes of it. Conditions on kernel arguments, template arguments or the block
are fine, and so are loops."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_04491_gb300", "csrc")
SOURCES = sorted(os.path.basename(f) for ext in ("cu", "cuh", "h") for f in glob.glob(os.path.join(CSRC, "*." + ext)))


def conditional_barriers(text):
    """Lines of the __syncthreads() calls under a run-time condition that depends on threadIdx."""
    blank = lambda m: re.sub(r"[^\n]", " ", m.group())
    text = re.sub(r"//[^\n]*|/\*.*?\*/|\"(\\.|[^\"\\\n])*\"", blank, text, flags=re.S)
    kernels = [m.start() for m in re.finditer(r"__global__|__device__", text)] + [len(text)]
    stack, found, start, condition = [], [], 0, None     # start: where the current statement begins
    for m in re.finditer(r"[{};]|__syncthreads\s*\(", text):
        head = text[start:m.start()].strip()
        if m.group() == ";" and head.count("(") > head.count(")"):
            continue                                     # inside a for's parentheses
        branch = re.match(r"(else\b\s*)?(if\b(?!\s*constexpr)(?P<c>.*))?", head, flags=re.S)
        if branch.group("c"):
            condition = branch.group("c")
        under = condition if branch.group() else None    # a plain else: the condition of its if
        if m.group() == "{":
            stack.append(under)
            start = m.end()
        elif m.group() in "};":
            if m.group() == "}" and stack:
                condition = stack.pop()
            start = m.end()
        else:
            begin = max(k for k in [0] + kernels if k <= m.start())
            per_thread = {"threadIdx"}
            for _ in range(3):                           # names assigned from it, and from those
                for name, value in re.findall(r"(\w+)\s*=(?!=)([^;,]*)", text[begin:m.start()]):
                    if per_thread & set(re.findall(r"\w+", value)):
                        per_thread.add(name)
            if any(c and per_thread & set(re.findall(r"\w+", c)) for c in stack + [under]):
                found.append(text.count("\n", 0, m.start()) + 1)
    return found


@pytest.mark.parametrize("name", SOURCES)
def test_no_barrier_under_a_condition(name):
    with open(os.path.join(CSRC, name)) as f:
        assert conditional_barriers(f.read()) == []


def test_the_search_finds_them():
    fine = ("for (int i = 0; i < n; ++i) { if (threadIdx.x) x = 1; __syncthreads(); }",
            "if constexpr (L > threads) { __syncthreads(); }",
            "if (n > 0) { int i = threadIdx.x; if (i) f(); __syncthreads(); }",
            "if (blockIdx.x == 0) { __syncthreads(); return; } __syncthreads();")
    wrong = ("if (threadIdx.x < 32) { f(); __syncthreads(); }",
             "int t = threadIdx.x, w = t / 32; if (w < 3) __syncthreads();",
             "int w = threadIdx.x / 32; if (w < 3) { f(); } else { for (;;) { __syncthreads(); } }")
    for body in fine:
        assert conditional_barriers("__global__ void k() {\n" + body + "\n}") == [], body
    for body in wrong:
        assert conditional_barriers("__global__ void k() {\n" + body + "\n}") == [2], body
