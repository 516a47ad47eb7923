"""Full-mask warp collectives in the CUDA sources, read as text (no GPU).

A value that other warps change (a volatile load) may differ between the lanes
of one warp: the lanes need not execute the load together.  A branch on such a
value must not enclose a full-mask collective, and must not leave a loop (or a
function) that has one: lanes that part there wait in different collectives.
The value is to be read by one lane and broadcast."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2112_06154_gb300", "csrc")
KEYWORDS = {"if", "for", "while", "switch", "do", "else", "return", "sizeof"}
COLLECTIVE = re.compile(r"__(?:shfl|ballot|any|all|match|reduce|syncwarp)\w*\s*\(")
SHARED_READ = re.compile(r"\*\s*\(\s*volatile\b|\bld_acquire\s*\(")
ONE_LANE = re.compile(r"\b(?:lane|tid|threadIdx\.x)\s*==\s*0\b")


def strip(text):
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    text = re.sub(r"//[^\n]*", " ", text)
    text = re.sub(r'"(?:\\.|[^"\\])*"', '""', text)
    return re.sub(r"^\s*#(?:[^\n]*\\\n)*[^\n]*", " ", text, flags=re.M)


def closing(s, i):
    """Index of the bracket that closes the one at i."""
    pairs, depth = {"(": ")", "{": "}", "[": "]"}, 0
    for j in range(i, len(s)):
        if s[j] in "({[":
            depth += 1
        elif s[j] in pairs.values():
            depth -= 1
            if depth == 0:
                return j
    raise ValueError("unbalanced brackets")


def functions(s):
    """(name, body start, body end) of every function definition."""
    head, at, out = re.compile(r"(\w+)\s*\(([^(){};]*(?:\([^()]*\)[^(){};]*)*)\)\s*(?:const\s*)?\{"), 0, []
    while (m := head.search(s, at)):
        end = closing(s, m.end() - 1)
        if m.group(1) in KEYWORDS:
            at = m.end()
            continue
        out.append((m.group(1), m.end(), end))
        at = end
    return out


def statement(s, i):
    """(start, end, head, condition, bodies) of the statement at i."""
    while s[i].isspace():
        i += 1
    word = re.match(r"\w+", s[i:])
    word = word.group(0) if word else ""
    if s[i] == "{":
        return i, closing(s, i) + 1, "{", "", [(i + 1, closing(s, i))]
    if word in ("if", "for", "while", "switch"):
        p = s.index("(", i)
        q = closing(s, p)
        b = statement(s, q + 1)
        end, bodies = b[1], [(b[0], b[1])]
        rest = re.match(r"\s*else\b", s[end:])
        if word == "if" and rest:
            e = statement(s, end + rest.end())
            bodies.append((e[0], e[1]))
            end = e[1]
        return i, end, word, s[p + 1:q], bodies
    if word == "do":
        b = statement(s, i + 2)
        w = s.index("(", b[1])
        q = closing(s, w)
        return i, s.index(";", q) + 1, "do", s[w + 1:q], [(b[0], b[1])]
    j = i
    while s[j] != ";":
        j = closing(s, j) + 1 if s[j] in "({[" else j + 1
    return i, j + 1, "", "", []


def findings(text):
    s = strip(text)
    funcs = functions(s)
    calls = {n: s[b:e] for n, b, e in funcs}
    collective = {n for n, body in calls.items() if COLLECTIVE.search(body)}
    while True:  # and what calls one
        more = {n for n, body in calls.items() if n not in collective
                and any(re.search(r"\b%s\s*(?:<[^;()]*>)?\(" % c, body) for c in collective)}
        if not more:
            break
        collective |= more

    def has(part):
        return bool(COLLECTIVE.search(part)) or any(
            re.search(r"\b%s\s*(?:<[^;()]*>)?\(" % c, part) for c in collective)

    out = []
    for name, b, e in funcs:
        tainted = set()

        def parted(cond):
            return bool(SHARED_READ.search(cond)) or any(re.search(r"\b%s\b" % v, cond) for v in tainted)

        def walk(i, end, loop, one_lane, cond_parted):
            while i < end and s[i:end].strip():
                st, en, kind, cond, bodies = statement(s, i)
                i = en
                src = s[st:en]
                if kind == "{":
                    walk(bodies[0][0], bodies[0][1], loop, one_lane, cond_parted)
                    continue
                if kind in ("if", "for", "while", "switch", "do"):
                    single = one_lane or bool(ONE_LANE.search(cond))
                    apart = not single and parted(cond)
                    if apart and has("".join(s[x:y] for x, y in bodies)):
                        out.append((name, " ".join(src.split())[:90]))
                    for x, y in bodies:
                        walk(x, y, src if kind in ("for", "while", "do") else loop, single,
                             False if kind in ("for", "while", "do") else cond_parted or apart)
                    continue
                jump = re.match(r"(break|continue|return)\b", src)
                if jump and cond_parted:
                    around = s[b:e] if jump.group(1) == "return" else loop
                    if has(around):
                        out.append((name, "parted " + src))
                if not one_lane:
                    for v in re.finditer(r"\b(\w+)\s*(?:\[[^\]]*\])?\s*=(?!=)([^;]*)", src):
                        if SHARED_READ.search(v.group(2)):
                            tainted.add(v.group(1))

        walk(b, e, "", False, False)
    return out


def test_the_reading_finds_both_forms():
    loop = ("__global__ void k(int* s) { for (;;) { const int t = *(volatile int*)s; "
            "%s } }")
    assert findings(loop % "if (x > t) { y = __shfl_sync(kFull, x, 0); }")
    assert findings(loop % "if (t) break; y = __ballot_sync(kFull, x);")
    assert findings("__device__ void f() { __syncwarp(); } __global__ void k(int* s) "
                    "{ for (;;) { f(); if (*(volatile int*)s > 3) break; } }")
    assert not findings(loop % "const int y = __shfl_sync(kFull, x, 0); if (lane == 0 && y > t) *s = y;")
    assert not findings("__global__ void k(int* s) { for (;;) { int t = 0; if (lane == 0) "
                        "t = *(volatile int*)s; if (__shfl_sync(kFull, t, 0)) break; } }")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_no_collective_under_a_value_other_warps_change(name):
    with open(os.path.join(CSRC, name)) as f:
        assert findings(f.read()) == []
