"""Order of the shared-memory reductions of the persistent class steps where one block takes every kind of
row: the accesses of one step are read from the kernel's source in program order and replayed with
vector clocks, every warp at its own pace between barriers.  Two accesses of a word, one a write, that no
barrier orders are a race."""
from __future__ import annotations

import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2312_04876_gb300", "csrc", "sweep.cu")
WARPS = 16


def between(text, start, end):
    a = text.index(start)
    return text[a:text.index(end, a)]


def kernel_ops():
    """(operations of a row of a multi-warp group, those after a kind's last row, the kinds' group sizes)."""
    src = open(SRC).read()
    row = between(src, "__device__ __forceinline__ void sweep_row(", "\n}\n")
    # the branches of groups within a warp
    row, cut = re.subn(r"\} else \{\s*team_sync<G, T>\(\);[^}]*\}", "}", row)
    assert cut == 1
    tokens = {"bar": r"team_any<G, T>\(|team_sync<G, T>\(", "wh": r"sh\.red_h\[warp\] =", "rh": r"sh\.red_h\[gi",
              "ws": r"sh\.red_s\[warp\] =", "rs": r"sh\.red_s\[gi", "wc": r"sh\.red_c\[warp\] =", "rc": r"sh\.red_c\[gi"}
    pattern = "|".join(f"(?P<{k}>{v})" for k, v in tokens.items())
    ops = [m.lastgroup for m in re.finditer(pattern, row)]
    assert ops.count("bar") >= 4 and {"wh", "rh", "ws", "rs", "wc", "rc"} <= set(ops)
    rows = between(src, "auto rows = [&]", "\n      };")
    after = ["bar"] * len(re.findall(r"team_sync<G, T>\(\)", rows[rows.index("sweep_rows<"):]))
    hubs = between(src[src.index("auto rows = [&]"):], "if constexpr (HUBS) {", "} else {")
    kinds = [int(g) for g in re.findall(r"rows\(Role<(\d+),", hubs)]
    assert len(kinds) >= 4
    return ops, after, [g for g in kinds if g > 32]


def races(ops, after, kinds, rows_a_kind):
    clock = [[0] * WARPS for _ in range(WARPS)]
    writes, reads, found = {}, {}, []

    def before(w, stamp):  # the access at stamp = (warp, time) happened before warp w's next one
        return clock[w][stamp[0]] >= stamp[1]

    def access(w, word, write):
        clock[w][w] += 1
        others = [writes[word]] if word in writes else []
        if write:
            others += reads.get(word, [])
        for o in others:
            if o[0] != w and not before(w, o):
                found.append((word, o[0], w))
        if write:
            writes[word], reads[word] = (w, clock[w][w]), []
        else:
            reads.setdefault(word, []).append((w, clock[w][w]))

    for g in kinds:
        n = g // 32
        for op in ops * rows_a_kind + after:
            for base in range(0, WARPS, n):
                group = range(base, base + n)
                if op == "bar":
                    join = [max(c) for c in zip(*(clock[w] for w in group))]
                    for w in group:
                        clock[w] = list(join)
                else:
                    for w in group:
                        for i in ([w] if op[0] == "w" else group):
                            access(w, (op[1], i), op[0] == "w")
    return found


@pytest.mark.parametrize("rows_a_kind", [1, 2])
def test_kinds_of_rows_of_one_block_do_not_race(rows_a_kind):
    ops, after, kinds = kernel_ops()
    assert races(ops, after, kinds, rows_a_kind) == []


def test_the_replay_sees_a_missing_barrier():
    ops, _, kinds = kernel_ops()
    assert races(ops, [], kinds, 1)


def rounds_of_an_insertion(lg):
    """Rounds that the giant rows' table insertion takes where every claim but the last free slot's is lost to
    another key: the kernel's probe, one lane, buckets of four slots (as read, `from` on)."""
    mask = (1 << lg) - 1
    taken, s, frm, load, view, rounds = set(), 0, 0, True, set(), 0
    while True:
        rounds += 1
        if load:
            view = set(taken)
        j = next((t for t in range(frm, 4) if s + t not in view), 4)
        load = False
        if j < 4:
            if s + j not in taken and len(taken) == mask:
                return rounds
            taken.add(s + j)  # another key, just before
            frm = j + 1
        else:
            s, frm, load = (s + 4) & mask, 0, True


@pytest.mark.parametrize("lg", [6, 7, 10, 14])
def test_the_pool_insertion_has_rounds_for_its_worst_case(lg):
    put = between(open(SRC).read(), "bool pool_put(", "\n}\n")
    limit, = re.findall(r"__any_sync\(0xffffffffu, left\) && p (<=?) ([^;]+); p\+\+", put)
    names = dict(re.findall(r"const unsigned (\w+) = ([^;]+);", put))
    bound = limit[1]
    while bound in names and bound != "mask":
        bound = names[bound]
    allowed = eval(bound.replace("/", "//"), {"mask": (1 << lg) - 1}) + (limit[0] == "<=")
    assert rounds_of_an_insertion(lg) <= allowed
