"""Host-side checks of the several-steps-per-launch 2D path (no GPU).

Launches of a pass overlap: the kernel lets the next launch start, and the
next one takes tensor memory before it waits for this one.  The order of those
operations is read from the kernel's source, and every interleaving of the
CTAs of three launches that share an SM is walked through: none may end with
CTAs that wait for each other.
"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_15744_gb300", "csrc")


def _events():
    """What a CTA of tile2d_tmem_kernel does, in program order."""
    text = open(os.path.join(CSRC, "step2d_tile_kernels.cuh")).read()
    body = text[text.index("tile2d_tmem_kernel(Tile2DArgs a)"):]
    body = re.sub(r"//[^\n]*", "", body[:body.index("\n}\n")])
    marks = {"alloc": "tcgen05.alloc", "free": "tcgen05.dealloc", "trigger": "let_next_start();",
             "wait": "wait_for_previous();", "barrier": r"pts.init("}
    assert all(body.count(m) == 1 for m in marks.values())
    return sorted(marks, key=lambda k: body.index(marks[k]))


def _stuck(order, launches, slots):
    """A state in which CTAs remain and none can go on, or None.  One CTA per
    launch on the SM; only warp 0 allocates and frees, the other warps run
    ahead of it up to a barrier.  A launch starts when the one before has
    triggered (any warp); `slots` CTAs hold tensor memory at a time."""
    warp0, rest = order, [e for e in order if e not in ("alloc", "free")]
    start = tuple((0, 0) for _ in range(launches))

    def done(pc):
        return pc[0] == len(warp0) and pc[1] == len(rest)

    def passed(pc, what):   # by any warp
        return warp0.index(what) < pc[0] or (what in rest and rest.index(what) < pc[1])

    def moves(s):
        held = sum(passed(pc, "alloc") and not passed(pc, "free") for pc in s)
        for i, pc in enumerate(s):
            if i and not passed(s[i - 1], "trigger"):
                continue
            for w, prog in enumerate((warp0, rest)):
                if pc[w] == len(prog):
                    continue
                e, ok = prog[pc[w]], True
                if e == "alloc":
                    ok = held < slots
                elif e == "wait":
                    ok = i == 0 or done(s[i - 1])
                elif e in ("barrier", "free"):   # the other warps must have come as far
                    other, q = pc[1 - w], (rest, warp0)[w]
                    ok = other >= (q.index("barrier") if e == "barrier" else len(q))
                if ok:
                    new = (pc[0] + 1, pc[1]) if w == 0 else (pc[0], pc[1] + 1)
                    yield s[:i] + (new,) + s[i + 1:]

    seen, todo = {start}, [start]
    while todo:
        s = todo.pop()
        nxt = list(moves(s))
        if not nxt and not all(done(pc) for pc in s):
            return s
        for n in nxt:
            if n not in seen:
                seen.add(n)
                todo.append(n)
    return None


def test_overlapping_launches_never_wait_for_each_others_tensor_memory():
    order = _events()
    for launches in (2, 3, 4, 5):
        for slots in (1, 2):   # 512 columns: one density CTA, or two with 256 each
            assert _stuck(order, launches, slots) is None, (order, launches, slots)


def test_the_walk_finds_the_circular_wait():
    # triggered before the columns are held: a later launch can take them first
    early = ["alloc", "trigger", "barrier", "wait", "free"]
    assert all(_stuck(early, n, 1) is not None for n in (2, 3))
    # waiting before allocating, as the 3D pair kernel does, is sound as well
    assert _stuck(["trigger", "wait", "alloc", "barrier", "free"], 4, 1) is None
