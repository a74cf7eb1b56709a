"""The chunked prefix scan with more (request, head) items than SMs, so that a CTA
works through several in turn, against the oracle: prefixes around the chunk edges
and of uneven length, with and without a start state, both rules."""
import dataclasses

import numpy as np
import pytest

import jet_synth
import oracle as O
from gpu_common import TOL_FORK_REL
from test_gpu_prefill import _check_scan_out

pytestmark = pytest.mark.gpu

EDGES = [1, 63, 64, 65, 128, 130, 200, 2]
CASES = [
    (20, 8),   # a few CTAs have a second item
    (58, 8),   # three or four items a CTA
    (9, 40),   # few requests, many heads
]


@pytest.mark.parametrize("rule", ["delta", "gla"])
@pytest.mark.parametrize("R,Hl", CASES)
def test_scan_items(jet, R, Hl, rule):
    import torch
    w = dataclasses.replace(jet_synth.WORKLOADS["ordinal_hybrid"], Hl=Hl, dtype="bf16")
    pl = [EDGES[i % len(EDGES)] + 64 * (i % 3) for i in range(R)]
    p = jet_synth.custom_problem(w, pl, [1] * R, [1] * R, [0] * R, seed=170 + R)
    hl = jet.jet_layout_build(p.prefix_len, p.n_cand, p.cand_len, p.target_ids, w.V)
    dims = jet.make_dims(jet.DTYPE_BF16, Hl=w.Hl, dk=w.dk, dv=w.dv, D=w.D)
    t = [jet_synth.torch_tensor(p, n, device="cuda")
         for n in ("lq_pre", "lk_pre", "lv_pre", "alpha_pre", "beta_pre")]
    for with_init in (False, True):
        s_init = jet_synth.torch_tensor(p, "s_prefix", device="cuda") if with_init else None
        o = torch.empty(p.total_prefix, w.Hl, w.dv, dtype=torch.bfloat16, device="cuda")
        s_out = torch.empty(R, w.Hl, w.dk, w.dv, dtype=torch.float32, device="cuda")
        jet.jet_prefill_state(hl.to_device("cuda"), dims, *t, o, s_out, s_init=s_init,
                              rule=jet.RULES[rule])
        torch.cuda.synchronize()
        assert jet.jet_device_status() == 0
        ref_o, ref_s = O.prefill_state(p.prefix_len, p.f32("s_prefix") if with_init else None,
                                       *(p.f32(n) for n in ("lq_pre", "lk_pre", "lv_pre",
                                                            "alpha_pre", "beta_pre")), rule)
        rel = np.abs(s_out.cpu().numpy() - ref_s).max() / np.abs(ref_s).max()
        assert rel <= TOL_FORK_REL, f"state error {rel}"
        _check_scan_out(o.float().cpu().numpy(), ref_o, True)
