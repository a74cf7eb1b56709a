"""Prefill attention on SM pairs (head dimensions 128 and 256) against the
oracle: prefixes around the 128-key tile and the pair's query block, more items
than pairs of one tile each (every role runs ahead of the others), short prefixes
that leave a pair's second half empty and run on single SMs, and a running maximum
that keeps growing, so that the output accumulator is rescaled for some of a warp's
vectors and not for others - also in the scoring step's attention, which shares
that rule."""
import dataclasses

import numpy as np
import pytest

import jet_synth
import oracle as O
from gpu_common import TOL_ATTN_BF16, oracle_layout, run_problem
from test_gpu_prefill import _prefill

pytestmark = pytest.mark.gpu

CASES = [
    ([127, 128, 129, 31, 32, 33, 1], dict(Hq=16, Hkv=2, d=256)),  # 32-position blocks
    ([256, 41, 42, 43, 84, 85], dict(Hq=24, Hkv=4, d=256)),       # 42-position blocks
    ([255, 257, 384], dict(Hq=2, Hkv=2, d=128)),                  # g = 1: 256-position blocks
    ([3, 130, 2], dict(Hq=128, Hkv=1, d=128)),                    # g = 128: two positions
    (list(range(1, 120)) * 2, dict(Hq=16, Hkv=4, d=256)),         # single SMs: half of it empty
]


def _problem(pl, over, seed):
    w = dataclasses.replace(jet_synth.WORKLOADS["tiny"], dtype="bf16", **over)
    R = len(pl)
    return jet_synth.custom_problem(w, pl, [1] * R, [1] * R, [0] * R, seed=seed)


def _check(p, got, rows, tol):
    w = p.work
    ref = O.prefill_attention(p.prefix_len, p.f32("q_pre"), p.f32("k_pre"), p.f32("v_pre"),
                              w.Hq, w.Hkv, rows=rows)
    assert np.abs(got[rows] - ref).max() <= tol


@pytest.mark.parametrize("case", range(len(CASES)))
def test_prefill_pair_blocks(jet, case):
    pl, over = CASES[case]
    p = _problem(pl, over, 110 + case)
    got = _prefill(jet, p)
    rng = np.random.default_rng(case)
    rows = range(p.total_prefix) if p.total_prefix <= 600 else \
        sorted(set(rng.integers(0, p.total_prefix, 300).tolist()) | {0, p.total_prefix - 1})
    _check(p, got, list(rows), TOL_ATTN_BF16)


SHORT = [
    ([48] * 240, dict(Hq=16, Hkv=4, d=256)),        # pairs: 960 items of one tile
    ([60] * 90, dict(Hq=8, Hkv=2, d=128)),          # pairs: 180 items of one tile
    ([16] * 64, dict(Hq=32, Hkv=8, d=128)),         # half of a pair's block: single SMs
    ([17, 31, 1] * 40, dict(Hq=16, Hkv=4, d=128)),  # single SMs
    ([21] * 90, dict(Hq=24, Hkv=4, d=256)),         # single SMs
]


@pytest.mark.parametrize("case", range(len(SHORT)))
def test_prefill_of_many_short_prefixes(jet, case):
    pl, over = SHORT[case]
    p = _problem(pl, over, 200 + case)
    rows = np.random.default_rng(case).integers(0, p.total_prefix, 300).tolist()
    _check(p, _prefill(jet, p), sorted(set(rows) | {0, p.total_prefix - 1}), _bar(p))


def _grow(p, tensor="k_pre"):
    """Scale every request's keys by 1 + position / 8: the scores' spread grows
    along the prefix, so the running maxima keep growing by more than 2^8."""
    k = p.f32(tensor)
    pos = np.concatenate([np.arange(P) for P in p.prefix_len])
    k = k * (1.0 + pos / 8.0)[:, None, None].astype(np.float32)
    p._cache[(tensor, k.shape)] = jet_synth.f32_to_bf16_bits(k).reshape(k.shape)


def _bar(p):
    # the weights are rounded to bf16 in the numerator and summed as rounded:
    # each is off by at most 2^-9 of itself, which moves the average by at most
    # 2 x 2^-9 max |v|; the output's own rounding adds 2^-9 |o|
    return 3 * 2.0 ** -9 * np.abs(p.f32("v_pre")).max()


@pytest.mark.parametrize("d", [64, 128, 256])
def test_prefill_growing_maximum(jet, d):
    p = _problem([700, 300], dict(Hq=8, Hkv=2, d=d), 120)
    _grow(p)
    got = _prefill(jet, p)
    _check(p, got, sorted(np.random.default_rng(d).integers(0, 1000, 200).tolist()), _bar(p))


def test_scoring_attention_growing_maximum(jet):
    w = dataclasses.replace(jet_synth.WORKLOADS["tiny"], dtype="bf16", Hq=8, Hkv=2, d=256)
    lens = [4, 3, 2, 5]
    p = jet_synth.custom_problem(w, [900, 333], [2, 2], lens, [1] * sum(lens), seed=121)
    _grow(p)
    got, _ = run_problem(jet, p)
    lay = oracle_layout(p)
    ref = O.cascade_attention(lay, p.f32("q"), p.f32("k_pre"), p.f32("v_pre"), p.f32("k_cand"),
                              p.f32("v_cand"), w.Hq, w.Hkv)
    assert np.abs(got["o"] - ref).max() <= _bar(p)
