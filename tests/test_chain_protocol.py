"""Who waits for whom inside a CTA of the reverse chain (csrc/tile_chain.cu), explored on the CPU in every order that the warps may run in.

The model has two of the epilogue warps (warp 0, which adds up the dot products, and another), the copy warp and the MMA warp, and the
steps of a chunk that touch the once-per-chunk barriers.  An mbarrier wait names the parity of a phase: it blocks while that phase is
the barrier's current one - and again once the barrier has completed one phase more."""
import pathlib
import re

import pytest

SOURCE = pathlib.Path(__file__).resolve().parent.parent / "paper_2608_21308_b200" / "csrc" / "tile_chain.cu"
CHUNKS = 3

# The statements the programs below stand for, in the order of the source
STATEMENTS = [
    "if (G.issuer() || n == 0) G.await(&sh.ops, n, 405);",
    "if (G.copier()) G.await(&sh.scaled, n, 410);",
    "if (ph == 0 && st == LAST && tk == 0 && nres < NMAT && G.copier()) G.await(&sh.ops, n, 411);",
    "P.before = &sh.phb;",
    "P.before = &sh.zb;",
    "if (!NORMED) G.signal(&sh.ops);",
    "G.signal(&sh.ops);",
    "if (lane == 0) { sh.dots[n & 1][warp][0] = pw; sh.dots[n & 1][warp][1] = pm; sh.dots[n & 1][warp][2] = pb; }",
    "G.signal(&sh.scaled);",
    "if (tk == tbn - 1) G.signal(&sh.phb);",
    "G.signal(&sh.zb);",
    "G.await(&sh.scaled, n, 409);  // every warp's share of the dot products",
    "for (int w = 0; w < 16; ++w) x += sh.dots[n & 1][w][lane];",
    "if (!NORMED) G.signal(&sh.ops);",
]


def dots_slot(n):
    return n & 1


def scaled_wait(n, at):  # chunks whose `scaled` the copy warp waits for at this point of chunk n
    return [n] if at == "rows" else []


def programs(resident, sets):
    """`sets` accumulator sets; as many jobs (products with an epilogue) between the chunk's two cluster barriers."""
    per_chunk = 6 + sets

    def consume(j):
        return [("await", f"full{j % sets}", j // sets), ("signal", f"empty{j % sets}")]

    def issue(j):
        return ([("await", f"empty{j % sets}", j // sets - 1)] if j >= sets else []) + [("use",), ("signal", f"full{j % sets}")]

    def epilogue(w):
        p = [("signal", "ops")]
        for n in range(CHUNKS):
            j = n * per_chunk
            p += [("write", dots_slot(n), w, n), ("signal", "scaled")] + consume(j) + [("signal", "phb")] + consume(j + 1)
            p += [("arrive",), ("cluster",), ("arrive",)] + sum((consume(j + 2 + e) for e in range(sets)), [])
            p += [("cluster",)] + consume(j + 2 + sets) + [("signal", "zb")] + sum((consume(j + 3 + sets + e) for e in range(3)), [])
            p += [("await", "scaled", n), ("read", dots_slot(n), n)] if w == 0 else []
            p += [("signal", "ops")]
        return p

    copy, mma = [], []
    for n in range(CHUNKS):
        j = n * per_chunk
        copy += [("arrive",)] + ([("await", "ops", 0)] if n == 0 else []) + [("await", "scaled", m) for m in scaled_wait(n, "head")]
        copy += ([] if resident else [("await", "ops", n)]) + [("load",), ("await", "phb", n)] + [("load",)] * (1 + sets)
        copy += [("await", "scaled", m) for m in scaled_wait(n, "rows")]
        copy += [("cluster",), ("arrive",), ("cluster",), ("load",), ("load",), ("await", "zb", n), ("load",), ("load",)]
        mma += [("arrive",), ("await", "ops", n)] + sum((issue(j + e) for e in range(2 + sets)), [])
        mma += [("cluster",), ("arrive",), ("cluster",)] + sum((issue(j + 2 + sets + e) for e in range(4)), [])
    return [epilogue(0), epilogue(1), copy, mma]


def explore(progs):
    """What goes wrong in some order of the warps' steps."""
    faults = set()
    counts = {"ops": 2, "scaled": 2, "phb": 2, "zb": 2, "full0": 1, "full1": 1, "empty0": 2, "empty1": 2}
    names = sorted(counts)
    # positions; arrivals per barrier so far; arrivals at and waits of the CTA-wide barrier per warp; loads under way; dots[slot][warp]
    start = ((0,) * 4, (0,) * len(names), (0,) * 4, (0,) * 4, 0, ((-1, -1), (-1, -1)))
    seen, todo = {start}, [start]
    while todo:
        pos, arr, carr, cwait, loads, dots = todo.pop()
        moved = False
        for i, prog in enumerate(progs):
            if pos[i] == len(prog):
                continue
            op = prog[pos[i]]
            a, ca, cw, ld, dt = list(arr), list(carr), list(cwait), loads, [list(x) for x in dots]
            if op[0] == "signal":
                a[names.index(op[1])] += 1
            elif op[0] == "await":
                b = names.index(op[1])
                if (arr[b] // counts[op[1]]) & 1 == op[2] & 1:
                    continue
            elif op[0] == "arrive":
                ca[i] += 1
            elif op[0] == "cluster":
                if min(carr) <= cwait[i]:
                    continue
                cw[i] += 1
            elif op[0] == "load":
                ld += 1
            elif op[0] == "use":
                if loads == 0:
                    continue
                ld -= 1
            elif op[0] == "write":
                dt[op[1]][op[2]] = op[3]
            elif dots[op[1]] != (op[2], op[2]):
                faults.add(f"sum of chunk {op[2]} takes the dot products of chunks {dots[op[1]]}")
            moved = True
            nxt = (pos[:i] + (pos[i] + 1,) + pos[i + 1:], tuple(a), tuple(ca), tuple(cw), ld, tuple(tuple(x) for x in dt))
            if nxt not in seen:
                seen.add(nxt)
                todo.append(nxt)
        if not moved and any(p < len(progs[i]) for i, p in enumerate(pos)):
            faults.add(f"every warp waits, at {[progs[i][p] if p < len(progs[i]) else 'end' for i, p in enumerate(pos)]}")
    return faults


def test_the_model_is_of_this_source():
    lines = [x.strip() for x in SOURCE.read_text().splitlines()]
    assert [x for x in lines if re.search(r"\bsh\.(dots|ops|phb|scaled|zb)\b", x)] == STATEMENTS


def test_dot_products_of_two_chunks_do_not_meet():
    assert not [f for f in explore(programs(True, 2)) if f.startswith("sum")]


@pytest.mark.parametrize("sets", [1, 2])
@pytest.mark.parametrize("resident", [True, False])
def test_no_wait_is_overtaken(resident, sets):
    assert not explore(programs(resident, sets))
