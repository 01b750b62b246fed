"""The room of a sibling group's piece list (apply_oct.cu, apply_oct_tc.cu): the kernels hold
OCT_TERM_PIECES entries per term in shared memory, counted here apart from the kernels' tables."""
import itertools
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0706_0747_gb300", "csrc")


def products(dims, classes):
    """Disjoint products of per-direction sets (core, off, both) whose translations have a number of
    core directions in `classes`."""
    classes = frozenset(classes)
    if not classes:
        return []
    if classes == frozenset(range(dims + 1)):
        return [("both",) * dims]
    core = frozenset(s - 1 for s in classes if s > 0)
    off = frozenset(s for s in classes if s < dims)
    if core == off:
        return [("both",) + p for p in products(dims - 1, core)]
    return [("core",) + p for p in products(dims - 1, core)] + [("off",) + p for p in products(dims - 1, off)]


def test_every_schedule_fits_the_piece_list():
    most = 0
    for n in range(5):
        for classes in itertools.combinations(range(4), n):
            pieces = products(3, classes)
            for v in itertools.product((True, False), repeat=3):  # each class's translations exactly once
                hits = sum(all(s == "both" or (s == "core") == c for s, c in zip(p, v)) for p in pieces)
                assert hits == (sum(v) in classes)
            most = max(most, len(pieces))
            if 3 in classes:  # leaf and internal siblings, J_m > j: the core for the leaves alone
                most = max(most, len(products(3, set(classes) - {3})) + 1)
    with open(os.path.join(CSRC, "oct_pieces.cuh")) as f:
        room = int(re.search(r"#define OCT_TERM_PIECES (\d+)", f.read()).group(1))
    assert most <= room
    for name in ("apply_oct.cu", "apply_oct_tc.cu"):
        with open(os.path.join(CSRC, name)) as f:
            assert "OCT_TERM_PIECES * (size_t)M * sizeof(uint32_t)" in f.read(), name
