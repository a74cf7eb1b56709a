"""The stack's projections at the edges of their tilings against the oracle: a width
that ends inside a 32-feature piece, rows that take more token tiles than the fewest,
an unsplit residual over several rounds of tiles, split K with its reduces, and a last
round in narrower tiles."""
import dataclasses

import numpy as np
import pytest

import jet_synth
from test_gpu_stack import SMALL, _check_rows, _gpu_stack, _oracle_stack

pytestmark = pytest.mark.gpu

# requests, candidates, tokens a candidate, D, Dff, Hl, dv
CASES = [
    (2, 2, 3, 1040, 320, 2, 64),
    (1, 1, 1, 256, 192, 2, 32),
    (13, 5, 5, 272, 64, 2, 160),
    (60, 4, 4, 512, 1088, 4, 64),
    (3, 3, 4, 1536, 2048, 8, 128),
    (8, 2, 3, 128, 9984, 2, 32),
]


@pytest.mark.parametrize("R,C,m,D,Dff,Hl,dv", CASES)
def test_projection_tilings(jet, R, C, m, D, Dff, Hl, dv):
    w = dataclasses.replace(SMALL, D=D, Hl=Hl, dv=dv)
    spec = jet_synth.StackSpec(("linear", "full"), Dff)
    p = jet_synth.custom_problem(w, [9 + r % 7 for r in range(R)], [C] * R, [m] * (R * C),
                                 np.arange(R * C * m) * 7 % w.V, seed=160 + R)
    got, _ = _gpu_stack(jet, p, spec, "delta")
    _check_rows(got, _oracle_stack(p, spec, "delta"), len(spec.kinds))
