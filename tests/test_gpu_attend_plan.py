"""The scoring attention's split and deal of work against the oracle: a few long
prefixes cut into many chunks, a prefix just past the shortest chunk, more items
than CTAs of uneven length (several a CTA, dealt back and forth), and more than 32
requests of one to many chunks (the combine meets rows that are already written
and chunks that a request does not have), long uneven chunks from the longest-first
list, and a deal that passes over windows of 32 requests."""
import dataclasses

import numpy as np
import pytest

import jet_synth
from gpu_common import TOL_ATTN_BF16, check_attention, oracle_layout, run_problem

pytestmark = pytest.mark.gpu

CASES = [
    ([5000], dict(Hq=16, Hkv=2, d=256)),
    ([193], dict(Hq=8, Hkv=2, d=64)),
    ([2049, 100, 700], dict(Hq=32, Hkv=8, d=128)),
    ([1 + 37 * i % 900 for i in range(90)], dict(Hq=24, Hkv=4, d=64)),
    ([4000] + [50 + 61 * i for i in range(32)], dict(Hq=32, Hkv=8, d=128)),
    ([600 + 230 * i for i in range(20)], dict(Hq=8, Hkv=8, d=64)),
    ([60 + 7 * (i % 3) for i in range(300)], dict(Hq=4, Hkv=4, d=64)),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_attention_plan(jet, case):
    pl, over = CASES[case]
    w = dataclasses.replace(jet_synth.WORKLOADS["tiny"], dtype="bf16", **over)
    rng = np.random.default_rng(case)
    lens = rng.integers(1, 6, size=3 * len(pl))
    p = jet_synth.custom_problem(w, pl, [3] * len(pl), lens, [1] * int(lens.sum()),
                                 seed=140 + case)
    got, _ = run_problem(jet, p)
    rows = list(range(p.N)) if p.N <= 60 else sorted(rng.choice(p.N, 60, replace=False).tolist())
    check_attention(oracle_layout(p), p, got["o"], rows, TOL_ATTN_BF16)
