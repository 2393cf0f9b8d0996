"""Every wait of the kernels is bounded, so every one can run out: whoever waits has to look at how it ended.  Read from the sources, since a
wait that runs out inside a kernel at work is nothing to bring about on a GPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_19602_b200", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
WAITS = ("mbar_wait", "mbar_wait_warp", "mbar_wait_slow", "mbar_try")


def block(text, at):
    """The text between the brace at `at` and the one that closes it."""
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at + 1:i]
    raise AssertionError("a brace is not closed")


def without_conditions(text):
    """The beginning of a statement less the if (..), for (..), while (..), else and do before it."""
    while True:
        text = text.strip()
        m = re.match(r"(else|do)\b", text) or re.match(r"(if|for|while)\s*(constexpr\s*)?(?=\()", text)
        if not m:
            return text
        end = m.end()
        if m.group(1) in ("if", "for", "while"):
            depth = 0
            for end in range(m.end(), len(text)):
                depth += {"(": 1, ")": -1}.get(text[end], 0)
                if depth == 0:
                    break
            else:
                return text                          # the call stands in the condition
            end += 1
        text = text[end:]


def dropped(text):
    text = re.sub(r"//[^\n]*", "", text)
    names = set(WAITS)
    for m in re.finditer(r"auto (\w+) = \[[^\]]*\]\s*(\([^)]*\))?\s*\{", text):
        body = block(text, m.end() - 1)
        if "return" in body and any(re.search(rf"\b{w}\(", body) for w in WAITS):
            names.add(m.group(1))
    found = []
    for m in re.finditer(rf"\b(?:tc::)?({'|'.join(sorted(names))})\(", text):
        start = max(text.rfind(c, 0, m.start()) for c in ";{}")
        # (the semicolons of a for's head are inside its brackets)
        while text[start] == ";" and text.count("(", text.rfind("\n", 0, start), start) > text.count(")", text.rfind("\n", 0, start), start):
            start = max(text.rfind(c, 0, start) for c in ";{}")
        if without_conditions(text[start + 1:m.start()]) == "":
            found.append((m.group(1), text[m.start():m.start() + 60].split("\n")[0]))
    return found


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_result_of_a_bounded_wait_is_dropped(path):
    assert dropped(open(path).read()) == []


def test_a_dropped_result_is_seen():
    waits = "auto final = [&](int t) { const bool ok = mbar_wait_warp(bar, 0); return ok; };\n"
    assert not dropped(waits + "if (have && final(1)) { x = 1; }\nok = ok && final(0);\nwhile (!mbar_try(a, 0) && go()) {}\nreturn tc::mbar_wait(a, 1);")
    for call in ("final(0);", "if (have) final(0);", "else final(0);", "for (int i = 0; i < n; ++i) tc::mbar_wait(a, i);", "{ mbar_try(a, 0); }"):
        assert len(dropped(waits + call)) == 1, call
