"""CPU: which pairs of eigenvectors the refined eigensolver of dmrg_truncate corrects in its one
first-order step.  The step leaves an off-diagonal of about g E (E = g / gap), so a pair is taken
only where that is below the rounding of the largest eigenvalue (1e-16) and E is small; the rest
of a block's pairs have to be rounding themselves or the block goes to the FP64 solver.  The
numbers checked lie off the rule's two lines by a factor, so that rounding decides nothing."""
import math

import numpy as np
import pytest

from tests.test_lib_cpu import lib  # noqa: F401  (fixture)


@pytest.mark.parametrize("gm", [1.0, 3e-7, 4e12])
def test_first_order_step_leaves_rounding_only(lib, gm):  # noqa: F811
    accepts = lib.dmrg_test_refine_accepts
    taken = 0
    for gap in gm * np.logspace(-14, 0, 57):
        for E in np.logspace(-14, 0, 57):
            left = E * E * gap / gm  # what the step leaves, of the largest eigenvalue
            for g, d in ((E * gap, gap), (-E * gap, gap), (E * gap, -gap)):
                if left > 1.1e-16 or E > 1.1e-5:
                    assert not accepts(g, d, gm), (g, d, gm)
                elif left < 0.9e-16 and E < 0.9e-5:
                    assert accepts(g, d, gm), (g, d, gm)
                    taken += 1
    assert taken > 0


def test_what_is_not_a_number_is_not_taken(lib):  # noqa: F811
    accepts = lib.dmrg_test_refine_accepts
    for g, gap, gm in ((math.nan, 1.0, 1.0), (1e-12, math.nan, 1.0), (1e-12, 1.0, math.nan), (1e-12, 0.0, 1.0),
                       (math.inf, 1.0, 1.0)):
        assert not accepts(g, gap, gm)
