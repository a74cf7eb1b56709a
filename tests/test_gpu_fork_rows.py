"""The fork's outputs without forked states (the form that reads the prefix
state once for a batch of fed tokens) against the oracle: candidates up to the
batch's 16 fed tokens and one beyond it, batches split between candidates,
more candidates than a warp has lanes, a request with nothing fed."""
import dataclasses

import numpy as np
import pytest

import jet_synth
from gpu_common import check_fork, oracle_layout, run_problem

pytestmark = pytest.mark.gpu

CASES = [
    ([1, 1, 2, 17, 16, 2, 1, 9, 9], [4, 4, 1]),     # 16 fed tokens on few CTAs: stepped
    ([2] * 40 + [1] * 3, [40, 3]),                  # 40 candidates: more than a warp; none fed
    ([1, 18, 3, 2], [3, 1]),                        # 17 fed tokens: the state-stepping form
    ([3] * 28 + [4] * 12, [1] * 40),                # 2.3 tokens a request: stepped
    ([3] * 27 + [4] * 13, [1] * 40),                # and one more in all: by products
    ([6] * 2, [1] * 2),                             # five, few CTAs: stepped
    ([1, 1, 2, 17, 16, 2, 1, 9, 9] * 16, [4, 4, 1] * 16),  # the first on more CTAs: by products
]


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("rule", ["delta", "gla"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_fork_outputs_without_states(jet, case, rule, dtype):
    lens, counts = CASES[case]
    w = dataclasses.replace(jet_synth.WORKLOADS["ordinal_hybrid"], V=4096, D=256, Hl=2,
                            dv=128 * (1 + case % 2), dtype=dtype)
    ids = np.random.default_rng(case).integers(0, w.V, size=int(np.sum(lens)))
    p = jet_synth.custom_problem(w, [3] * len(counts), counts, lens, ids, seed=70 + case)
    got, _ = run_problem(jet, p, keep_fork=False, rule=rule)
    check_fork(oracle_layout(p), p, got, list(range(p.R)), rule=rule)
