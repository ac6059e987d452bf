"""Hand-over of a step's exponent inside k_apply_tc64, as an ordering argument on the CPU.

The digit warps write the exponent of step s to slot s mod 4; the epilogue group of the
step reads it.  A slot is safe if every read is ordered before the write that reuses it.
The orders that exist are each role's program order and the barriers; the epilogue's is
taken from the source, so that a read moved behind the arrival is found here."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2401_06277_gb300", "csrc")
STEPS, SLOTS = 16, 4


def epilogue_order(source):
    """Positions of the exponent's read and of the arrival that frees the accumulators."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, source)).read())
    body = src[src.index("void epilogue("):src.index("__global__")]
    return body.index("sexp["), body.index("mbar_arrive(C.free")


def ordered(read_first):
    """Pairs (step, step) of read and reuse that nothing orders."""
    after = {}

    def edge(a, b):
        after.setdefault(a, []).append(b)

    for s in range(STEPS):
        first, second = ("read", "free") if read_first else ("free", "read")
        edge(("done", s), (first, s))
        edge((first, s), (second, s))
        edge((second, s), ("done_seen", s + 2))        # the group's next step
        edge(("done_seen", s), (first, s))
        edge(("free", s), ("mma", s + 2))              # the accumulators are used again
        edge(("write", s), ("mma", s))
        edge(("mma", s), ("mma", s + 1))
        edge(("mma", s), ("done", s))
        edge(("done", s), ("write", s + 2))            # the digit planes are used again
        edge(("write", s), ("write", s + 1))
    loose = []
    for s in range(STEPS - SLOTS):
        seen, todo = set(), [("read", s)]
        while todo:
            for b in after.get(todo.pop(), ()):
                if b not in seen:
                    seen.add(b)
                    todo.append(b)
        if ("write", s + SLOTS) not in seen:
            loose.append((s, s + SLOTS))
    return loose


def test_operator_reads_the_exponent_before_its_slot_can_be_reused():
    read, free = epilogue_order("sv_apply_tc64.cu")
    assert ordered(read < free) == []


def test_the_argument_needs_that_order():
    assert ordered(False) != []


@pytest.mark.parametrize("slots", [5, 8])
def test_exponents_of_cells_are_read_before_their_slot_is_written_again(slots):
    """Per row pair, written when the pair is read (before the waits of its step q - 1),
    used by the steps q - 1 and q before their arrival: six slots are needed, eight are kept."""
    after = {}

    def edge(a, b):
        after.setdefault(a, []).append(b)

    for s in range(STEPS):
        edge(("read", s), ("free", s))
        edge(("free", s), ("mma", s + 2))
        edge(("mma", s), ("done", s))
        edge(("mma", s), ("mma", s + 1))
        edge(("done", s), ("waited", s + 2))           # a digit warp, in its step s + 2
        edge(("waited", s), ("write", s + 2))          # then the next row pair, that of step s + 1
    loose = []
    for q in range(STEPS - slots):
        seen, todo = set(), [("read", q)]
        while todo:
            for b in after.get(todo.pop(), ()):
                if b not in seen:
                    seen.add(b)
                    todo.append(b)
        if ("write", q + slots) not in seen:
            loose.append(q)
    assert (loose == []) == (slots >= 6)
    src = open(os.path.join(CSRC, "sv_apply_tc64.cu")).read()
    assert "cexp[((q & 7) * 2 + a) * WCOLS + col] =" in src and "pexp[((q & 7) * 4 + 2 * a) * WCOLS + col] =" in src


@pytest.mark.parametrize("slots", [5, 8])
def test_sweep_reads_the_exponents_of_cells_before_their_slot_is_written_again(slots):
    """The sweep: six chains a step, chains c and c + 3 take turns in an accumulator, the
    epilogue reads the pairs s .. s + 2 after the last of them.  Pair q is written at the
    begin of step q - 2, each step waiting for all chains of the step before it."""
    after = {}

    def edge(a, b):
        after.setdefault(a, []).append(b)

    for s in range(STEPS):
        for c in range(6):
            edge(("done", s, c), ("free", s, c))
            edge(("free", s, c), ("free", s, c + 1) if c < 5 else ("read", s))
            use_next = ("mma", s, c + 3) if c < 3 else ("mma", s + 1, c - 3)
            edge(("free", s, c), use_next)
            edge(("mma", s, c), ("done", s, c))
            edge(("done", s, c), ("waited", s + 1))
        edge(("read", s), ("free", s + 2, 0))          # the group's next step
        edge(("waited", s), ("write", s + 3))
    loose = []
    for q in range(2, STEPS - slots - 2):
        for s in (q - 2, q - 1, q):                    # the steps that use pair q
            seen, todo = set(), [("read", s)]
            while todo:
                for b in after.get(todo.pop(), ()):
                    if b not in seen:
                        seen.add(b)
                        todo.append(b)
            if ("write", q + slots) not in seen:
                loose.append((q, s))
    assert (loose == []) == (slots == 8)
    src = open(os.path.join(CSRC, "sv_vanka_tc64.cu")).read()
    assert "cexp[((q & 7) * 2 + a) * WCOLS + col] =" in src and "pexp[((q & 7) * 4 + 2 * a) * WCOLS + col] =" in src
