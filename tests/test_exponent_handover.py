"""Hand-over of a step's exponent inside k_apply_tc64, as an ordering argument on the CPU.

The digit warps write the exponent of step s to slot s mod 4; the epilogue group of the
step reads it.  A slot is safe if every read is ordered before the write that reuses it.
The orders that exist are each role's program order and the barriers; the epilogue's is
taken from the source, so that a read moved behind the arrival is found here."""
import os
import re

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
