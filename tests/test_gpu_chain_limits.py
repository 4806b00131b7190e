"""One sequence at the edges of the one-sequence chain kernel, against the oracle: the widest feed-forward layer that it takes, and the
widths at which the fusion FC is cut in two."""
from dataclasses import replace

import numpy as np
import pytest

import hivis_inputs as hi
from tests.harness import LOGIT_RTOL, LOGIT_RTOL_F32, Case, check_draft_parity, check_kv_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_widest_feed_forward_layer(dtype):
    """Greedy and drawn, in one launch; operands are fp32, so the logits are those of an fp32 program in either type (sums of 24832
    products: some 800 in a lane's chain, then a tree)."""
    import torch
    base = hi.workload("c1_tiny_f32_b1")
    wl = hi.scaled(base, dims=replace(base.dims, ffn=24832, dtype=dtype))
    case = Case(wl)
    try:
        dr, k, V = case.drafter, wl.k, wl.dims.vocab
        res = check_draft_parity(case, rtol=LOGIT_RTOL_F32 if dtype == "f32" else LOGIT_RTOL)
        check_kv_parity(case, res["ref"])
        case.gpu_restore()
        n = dr.launch_count()
        case.gpu_draft()
        assert dr.launch_count() == n + 1
        case.gpu_restore()
        u = torch.rand((1, k, V), device="cuda", generator=torch.Generator(device="cuda").manual_seed(3)).clamp_(1e-6, 1 - 1e-6)
        ids, logits = dr.draft_sampled(1, k, 1.0, u, case.d_resid)
        drawn = logits.double() - torch.log(-torch.log(u.double()))
        top = drawn.topk(2, -1)
        clear = top.values[..., 0] - top.values[..., 1] > 1e-4
        assert bool(clear.any()) and bool((ids == top.indices[..., 0])[clear].all())
        ref = case.oracle_run(forced=ids.cpu().numpy())
        err = np.abs(logits[0].cpu().numpy() - ref[0]["logits"]).max(-1) / np.abs(ref[0]["logits"]).max(-1)
        assert err.max() <= (LOGIT_RTOL_F32 if dtype == "f32" else LOGIT_RTOL)
        dr.status()
    finally:
        case.close()


@pytest.mark.parametrize("dtype,d", [("f32", 1000), ("f32", 1024), ("f32", 1280), ("f32", 2560), ("bf16", 2048), ("bf16", 2560)])
def test_fusion_in_two_parts(dtype, d):
    """The part of the hidden half that is used behind the LM head is whole chunks of 4 KB: none of it, all of it, some of it (fp32 1280
    and 2560: 1024 and 2048 columns)."""
    base = hi.workload("c1_tiny_f32_b1")
    wl = hi.scaled(base, dims=replace(base.dims, d=d, vocab=1000, dtype=dtype), k=4)
    case = Case(wl)
    try:
        res = check_draft_parity(case, rtol=LOGIT_RTOL_F32 if dtype == "f32" else LOGIT_RTOL)
        check_kv_parity(case, res["ref"])
        case.drafter.status()
    finally:
        case.close()
