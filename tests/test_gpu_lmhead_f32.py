"""The float32 LM head's tiles on the GPU against the oracle: rows around the
8- and 16-row tiles, vocabularies around the 128-entry tile, hidden sizes
around the 32-element K slice and its ring of stages, a row with more targets
than a warp has lanes, tiles on one CTA and on two."""
import dataclasses

import numpy as np
import pytest

import jet_synth
import oracle as O
from gpu_common import oracle_layout, run_problem

pytestmark = pytest.mark.gpu

# (candidate lengths of the one request, V, D): N = 1 + sum (m - 1) rows
CASES = [
    ([1], 1, 8),
    ([1] * 40, 127, 40),          # one row, 40 targets
    ([8, 1], 128, 32),            # 8 rows: the small tile, full
    ([9], 129, 200),              # 9 rows: the large tile, mostly empty
    ([8, 9], 300, 192),           # 16 rows, as many K slices as stages
    ([12, 7], 1000, 520),         # 18 rows: two row tiles
    ([8, 1], 9900, 72),           # too many tiles for two CTAs a tile, 8 rows
    ([12, 7], 5000, 40),          # the same with two row tiles
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_f32_lm_head_tiles(jet, case):
    lens, V, D = CASES[case]
    w = dataclasses.replace(jet_synth.WORKLOADS["tiny"], V=V, D=D)
    ids = np.random.default_rng(case).integers(0, V, size=int(np.sum(lens)))
    ids[0], ids[-1] = 0, V - 1
    p = jet_synth.custom_problem(w, [5], [len(lens)], lens, ids, seed=60 + case)
    got, _ = run_problem(jet, p)
    lay = oracle_layout(p)
    H, W = p.f32("hidden").astype(np.float64), p.f32("w_lm").astype(np.float64)
    ell = O.token_logprobs(lay, p.f32("hidden"), p.f32("w_lm"), np.arange(lay["T"]))
    # a float32 logit is a sum of D products in eight chains of at most D / 8 + 4
    # terms, then 8 more: each rounding at most 2^-24 of the sum of magnitudes;
    # l differs by at most the logit's and the log-sum-exp's error (plus 2^-22 of
    # the values themselves for the exp, log and subtraction)
    mag = (np.abs(H) @ np.abs(W).T).max()
    tol = 2 * (D / 8 + 16) * 2.0 ** -24 * mag + 8 * 2.0 ** -22 * (1 + np.abs(ell).max())
    assert np.abs(got["ell"] - ell).max() <= tol
    s = O.candidate_scores(lay, ell)
    assert np.abs(got["s"] - s).max() <= tol * max(lens) + 2.0 ** -22 * np.abs(s).max()
