"""Where warps of a role meet at a named barrier inside a loop, a warp whose bounded wait ran out must keep meeting the others: two warps
may see the same wait end differently (complete, or the abort flag of another role first), and one that leaves the loop early leaves
the others at a barrier without a limit.  Read from the sources: such a wait cannot be made to fail on a device at will."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2411_09909_b200", "csrc", "*.cu")))


def strip(text):
    return re.sub(r"//[^\n]*", "", text)


def loops_around(text, at):
    """(head, body) of every loop whose braces enclose position `at`, innermost first."""
    depth, found = 0, []
    for i in range(at, -1, -1):
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth:
                depth -= 1
                continue
            head = re.search(r"\b(for|while)\s*\(([^{}]*)\)\s*$", text[:i])
            if head:
                end, d = i, 0
                while True:
                    d += {"{": 1, "}": -1}.get(text[end], 0)
                    if d == 0:
                        break
                    end += 1
                found.append((head.group(0), text[i:end]))
    return found


def early_exits(body):
    """`break` or `return` at a failed wait that leaves this loop: not inside a nested loop or lambda."""
    depth, skip, out = 0, [], []
    for m in re.finditer(r"[{}]|if \(!ok\)\s*(?:break|return)", body):
        if m.group() == "{":
            before = body[:m.start()].rstrip()
            depth += 1
            if depth > 1 and (re.search(r"\b(for|while)\s*\([^{}]*\)$", before) or re.search(r"\]\s*(\([^{}]*\))?$", before)):
                skip.append(depth)
        elif m.group() == "}":
            if skip and skip[-1] == depth:
                skip.pop()
            depth -= 1
        elif not skip:
            out.append(m.group())
    return out


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_warp_leaves_others_at_a_named_barrier(path):
    text = strip(open(path).read())
    # a barrier, or the call of a lambda that is one
    names = re.findall(r"auto (\w+) = \[[^\]]*\] \{ asm volatile\(\"bar\.sync", text)
    spots = [m.start() for m in re.finditer("|".join([r"bar\.sync"] + [rf"\b{n}\(\);" for n in names]), text)]
    for at in spots:
        for head, body in loops_around(text, at):
            assert not re.search(r"\bok\b", head), head
            assert not early_exits(body), head


def test_the_kernels_that_meet_are_seen():
    seen = {os.path.basename(p): len(re.findall(r"bar\.sync", strip(open(p).read()))) for p in SOURCES}
    assert {k for k, v in seen.items() if v} == {"attention_fp4.cu", "gemm_fp4.cu", "gemm_rows.cu"}
