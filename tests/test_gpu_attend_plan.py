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
from gpu_common import (TOL_ATTN_BF16, TOL_ATTN_F32, build_step, check_attention, oracle_layout,
                        run_problem)

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


LONG = [600 + 230 * i for i in range(20)]
LONGER = [100] + LONG[1:10] + [LONG[10] - 1030] + LONG[11:19] + [LONG[19] + 1530]
OTHER_WORDS = [
    # prefixes of the sizes and of the words (as many keys), the request past the plan
    ("bf16", [128, 100], [150, 78], 0, dict(Hq=8, Hkv=2, d=64)),            # one chunk
    ("bf16", [500, 460, 300], [300, 360, 600], 2, dict(Hq=16, Hkv=2, d=128)),  # split chunks
    ("bf16", LONG, LONGER, 19, dict(Hq=8, Hkv=8, d=64)),                    # the work list
    ("f32", [128, 100], [150, 78], 0, dict(Hq=8, Hkv=2, d=64)),
]


@pytest.mark.parametrize("case", range(len(OTHER_WORDS)))
def test_words_of_another_batch_stay_in_the_workspace(jet, case):
    # a layout whose words hold a longer prefix than the sizes that the workspace was
    # planned for: that request is left out and reported, nothing is written past the
    # plan's bytes, and the other requests get their answers
    import torch
    dtype, planned, worded, long, over = OTHER_WORDS[case]
    w = dataclasses.replace(jet_synth.WORKLOADS["tiny"], dtype=dtype, **over)
    R = len(planned)

    def problem(pl):
        return jet_synth.custom_problem(w, pl, [2] * R, [3] * (2 * R), [1] * (6 * R), seed=180 + case)

    step, _, _ = build_step(jet, problem(planned))
    p = problem(worded)
    x = {n: jet_synth.torch_tensor(p, n, device="cuda")
         for n in ("q", "k_pre", "v_pre", "k_cand", "v_cand")}
    words = jet.jet_layout_build(p.prefix_len, p.n_cand, p.cand_len, p.target_ids, w.V).words
    step.layout.words.copy_(torch.from_numpy(words.copy()).to(step.layout.words.device))
    need = jet.jet_workspace_bytes(step.host_layout.sizes, step.dims)
    ws = torch.full((need + (8 << 20),), 0x5A, dtype=torch.uint8, device="cuda")
    jet.jet_prefix_attend(step.layout, step.dims, x["q"], x["k_pre"], x["v_pre"], x["k_cand"],
                          x["v_cand"], step.o, ws, ws_bytes=need)
    torch.cuda.synchronize()
    assert jet.jet_device_status() == 10  # JET_ERR_DEVICE
    assert bool((ws[need:] == 0x5A).all())
    lay = oracle_layout(p)
    rows = [n for n in range(p.N) if lay["row_req"][n] != long]
    rows = rows[:30] + rows[-10:]
    check_attention(lay, p, step.o.float().cpu().numpy(), sorted(set(rows)),
                    TOL_ATTN_BF16 if dtype == "bf16" else TOL_ATTN_F32)


SPLIT = [
    ("bf16", 500, dict(Hq=16, Hkv=2, d=128)),   # chunks of 192 keys
    ("bf16", 6000, dict(Hq=8, Hkv=2, d=64)),
    ("bf16", 100, dict(Hq=8, Hkv=2, d=256)),    # one chunk, written directly
    ("f32", 100, dict(Hq=8, Hkv=2, d=64)),      # four chunks
]


@pytest.mark.parametrize("case", range(len(SPLIT)))
@pytest.mark.parametrize("what", ["nan_key", "inf_value"])
def test_non_finite_inputs_reach_the_output(jet, case, what):
    # a NaN key makes the outputs of its kv head's query heads NaN, an infinite value
    # its column of them non-finite, also where the prefix is split and where the
    # chunk of that key has no weight left against the others
    import torch
    dtype, P, over = SPLIT[case]
    w = dataclasses.replace(jet_synth.WORKLOADS["tiny"], dtype=dtype, **over)
    p = jet_synth.custom_problem(w, [P], [2], [3, 2], [1] * 5, seed=190 + case)
    step, x, w_lm = build_step(jet, p)
    at, g = P // 3, w.Hq // w.Hkv
    if what == "nan_key":
        x["k_pre"][at, 1, 5] = float("nan")
    else:
        x["v_pre"][at, 1, 5] = float("inf")
        # the last key's score is larger by 416, 600 powers of two of weight
        x["q"][:, :, 0] = 16.0
        x["k_pre"][:, :, 0] = 0.0
        x["k_pre"][P - 1, :, 0] = 26.0 * w.d ** 0.5
    jet.jet_prefix_attend(step.layout, step.dims, x["q"], x["k_pre"], x["v_pre"], x["k_cand"],
                          x["v_cand"], step.o, step.ws)
    torch.cuda.synchronize()
    assert jet.jet_device_status() == 0
    o = step.o.float().cpu()
    assert torch.isfinite(o[:, :g]).all()  # the other kv head's
    if what == "nan_key":
        assert torch.isnan(o[:, g:]).all()
    else:
        assert not torch.isfinite(o[:, g:, 5]).any()
        assert torch.isfinite(o[:, g:, :5]).all() and torch.isfinite(o[:, g:, 6:]).all()
