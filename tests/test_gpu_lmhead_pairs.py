"""The LM head of more than 256 rows against the oracle, on CTA pairs (from 16 K
slices on) and on single CTAs: rows just past one token tile and at uneven shares of
16- and 32-row blocks, odd numbers of vocabulary tiles, and limits on the SMs it may
use (few and odd ones leave single CTAs), which must not change a result."""
import dataclasses

import numpy as np
import pytest

import jet_synth
import oracle as O
from gpu_common import TOL_LOGPROB, dims_for, oracle_layout

pytestmark = pytest.mark.gpu

# (rows of the one request - a shared row and one candidate's fed tokens, V, D): single
# CTAs, then pairs in both formats, in bf16 alone (15 and 16 K slices are D 960 and 961
# there, twice that in e4m3), and in neither
CASES = [(257, 300, 72), (272, 129, 64), (400, 1000, 200), (513, 640, 136), (529, 127, 64),
         (257, 300, 1928), (272, 129, 2048), (400, 1000, 1992), (513, 640, 1928),
         (529, 127, 2048), (609, 300, 968), (609, 300, 960)]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("lm", ["bf16", "e4m3"])
def test_lm_head_pairs(jet, case, lm):
    import torch
    from oracle import e4m3 as Q
    from paper_2609_33874_gb300 import step as S
    N, V, D = CASES[case]
    D = (D + 15) // 16 * 16 if lm == "e4m3" else D
    w = dataclasses.replace(jet_synth.WORKLOADS["tiny"], V=V, D=D, dtype="bf16", w_std=0.1)
    ids = np.random.default_rng(case).integers(0, V, size=N)
    ids[0], ids[-1] = 0, V - 1
    p = jet_synth.custom_problem(w, [3], [1], [N], ids, seed=130 + case)
    lay = oracle_layout(p)
    host = jet.jet_layout_build(p.prefix_len, p.n_cand, p.cand_len, p.target_ids, V)
    hidden = jet_synth.torch_tensor(p, "hidden", device="cuda")
    w_lm = jet_synth.torch_tensor(p, "w_lm", device="cuda")
    if lm == "e4m3":
        ref = Q.token_logprobs_e4m3(lay, p.f32("hidden"), *Q.quantize_rows(p.f32("w_lm")),
                                    np.arange(lay["T"]))
        w_lm = S.quantize_lm_head(w_lm)
    else:
        ref = O.token_logprobs(lay, p.f32("hidden"), p.f32("w_lm"), np.arange(lay["T"]))
    first = None
    for sms in (0, 1, 2, 5, 9):
        dims = dims_for(jet, w)
        dims.max_sms = sms
        step = S.ScoringStep(host, dims, jet.DECIDE_ARGMAX, lm=lm)
        step.score(hidden, w_lm)
        torch.cuda.synchronize()
        assert jet.jet_device_status() == 0
        ell = step.tok_logprob.cpu().numpy()
        assert np.abs(ell - ref).max() <= TOL_LOGPROB
        # the same products summed in the same order, whatever the split
        first = ell if first is None else first
        np.testing.assert_array_equal(ell, first)
