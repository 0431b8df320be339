"""How a CTA pair of the GEMM kernel ends (csrc/gemm.cuh), over every order in which its warps can come to it, on the CPU.

The order of the steps is read from the source.  A model of the two CTAs, each with the warp that gives tensor memory back and one
that stands for its other roles, is then walked through all of its states: whoever gives up, and whenever, everybody has to retire.
A wait on an mbarrier may give up at any time (its limit, or the CTA's abort flag); a cluster barrier waits for every warp that has not
retired; the pair's deallocation may wait until the other CTA has issued its own."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STEPS = [(r"warp_mbar_wait\(tmem_free", "wait tmem_free"), (r"warp_mbar_wait\(peer_free", "wait peer_free"),
         (r"mbar_arrive_cluster_relaxed\(peer_free", "arrive"), (r"tmem_dealloc_pair", "dealloc"), (r"cluster_sync_all", "barrier")]


def _steps(code):
    found = [(m.start(), name) for pattern, name in STEPS for m in re.finditer(pattern, code)]
    return [name for _, name in sorted(found)]


def _source_order():
    """(the deallocating warp's steps when all went well, everybody's steps behind a wait that ran out)"""
    src = open(os.path.join(ROOT, "paper_2609_31551_b200", "csrc", "gemm.cuh")).read()
    src = re.sub(r"//[^\n]*", "", src)
    end = src.rindex("if (!ok) {")
    good = src[src.rindex("if (warp == kTmemWarp && ok) {", 0, end):end]
    return _steps(good), _steps(src[end:])


def _stuck(good, failed):
    """The first reachable state in which somebody has not retired and nobody can move (None: there is none)."""
    gone = ("gone", 0)
    # a warp: (program, position); the other roles' warp is running, retired, or in the failure path (it deallocates nothing)
    start = ((("good", 0), ("good", 0)), ("run", "run"), frozenset(), frozenset(), frozenset())
    programs = {"good": good, "failed": failed}
    seen, stack = {start}, [start]
    while stack:
        state = stack.pop()
        tmem, other, arrived, freeing, met = state
        moves = []

        def tmem_to(c, pos, arrived=arrived, freeing=freeing, met=met):
            program, at = pos
            t = list(tmem)
            t[c] = gone if program != "gone" and at == len(programs[program]) else pos
            moves.append((tuple(t), other, arrived, freeing, met))

        def barrier_passes():
            waiting = {("tmem", c) for c in (0, 1) if tmem[c] != gone} | {("other", c) for c in (0, 1) if other[c] != "gone"}
            return waiting <= met

        for c in (0, 1):
            if tmem[c] != gone:
                program, at = tmem[c]
                step = programs[program][at]
                nxt = (program, at + 1)
                if step.startswith("wait"):
                    tmem_to(c, ("failed", 0))
                    if step == "wait tmem_free" or c in arrived:
                        tmem_to(c, nxt)
                elif step == "arrive":
                    tmem_to(c, nxt, arrived=arrived | {1 - c})
                elif step == "dealloc":
                    if c not in freeing:
                        tmem_to(c, (program, at), freeing=freeing | {c})
                    elif 1 - c in freeing:
                        tmem_to(c, nxt)
                elif step == "barrier":
                    if ("tmem", c) not in met:
                        tmem_to(c, (program, at), met=met | {("tmem", c)})
                    elif barrier_passes():
                        tmem_to(c, nxt)
            if other[c] == "run":
                for to, more in (("gone", set()), ("failed", {("other", c)} if "barrier" in failed else set())):
                    o = list(other)
                    o[c] = to
                    moves.append((tmem, tuple(o), arrived, freeing, met | more))
            elif other[c] == "failed" and ("barrier" not in failed or barrier_passes()):
                o = list(other)
                o[c] = "gone"
                moves.append((tmem, tuple(o), arrived, freeing, met))
        if not moves and not (tmem == (gone, gone) and other == ("gone", "gone")):
            return state
        for m in moves:
            if m not in seen:
                seen.add(m)
                stack.append(m)
    return None


def test_the_model_finds_a_pair_that_never_retires():
    good = ["wait tmem_free", "arrive", "wait peer_free", "dealloc"]
    # one CTA waits in its deallocation for the other, which gave up behind its own arrival and stands at the barrier
    assert _stuck(good, ["barrier", "dealloc"]) is not None
    assert _stuck(good, ["dealloc", "barrier"]) is None


def test_a_pair_retires_whoever_gives_up():
    good, failed = _source_order()
    assert good == ["wait tmem_free", "arrive", "wait peer_free", "dealloc"]
    assert sorted(failed) == ["barrier", "dealloc"]
    assert _stuck(good, failed) is None, f"the failure path {failed} can wait for a warp that waits for it"
