"""Calls captured into a CUDA graph: every replay gives what the calls give, and so does an eager call after the capture."""
import pytest

import hivis_inputs as hi
from tests.harness import Case

pytestmark = pytest.mark.gpu


def turns():
    """name -> (workload, sequences, what a turn drafts)."""
    return {"fp32, one sequence": ("c1_tiny_f32_b1", 1, "draft"), "one sequence": ("mini_mha_b1", 1, "draft"),
            "one sequence, drawn": ("mini_mha_b1", 1, "sampled"), "5 sequences": ("mini_mha_b5_ragged", 5, "draft"),
            "5 sequences, drawn": ("mini_mha_b5_ragged", 5, "sampled"), "16 sequences": ("mini_gqa_b16_ragged", 16, "draft"),
            "20 sequences": ("mini_mha_b5_ragged", 20, "draft"), "40 sequences": ("mini_gqa_b16_ragged", 40, "draft"),
            "tree": ("mini_mha_b1", 1, "tree"), "fp32 tree": ("c1_tiny_f32_b1", 1, "tree")}


@pytest.mark.parametrize("pairs", [3, 40])
@pytest.mark.parametrize("name", turns())
def test_captured_turns_replay(name, pairs):
    import torch
    base, B, what = turns()[name]
    wl = hi.scaled(hi.workload(base), batch=B, k=3, text_len=None, text_len_range=(50, 70))
    case = Case(wl, max_len=160)
    try:
        dr = case.drafter
        case.gpu_prefill()
        rows = [int(n) - 1 for n in case.lens]
        ids, hidden = case.d_ids[:pairs].contiguous(), case.d_hidden[:pairs].contiguous()
        uniforms = torch.rand((B, 3, wl.dims.vocab), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
        uniforms.clamp_(1e-6, 1 - 1e-6)

        def turn():
            dr.set_kv_len_batch(rows, restore_pending=True)
            dr.prefill(ids, hidden, [0, pairs], slots=[0], start_pos=[2], resid0=case.d_resid[0])
            if what == "tree":
                return dr.draft_tree(0, 4, 3, 20, case.d_resid)
            if what == "sampled":
                return dr.draft_sampled(B, 3, 1.0, uniforms, case.d_resid)
            return dr.draft(B, 3, case.d_resid, want_logits=True)

        def same(got):
            torch.cuda.synchronize()
            return all(torch.equal(x, y) for x, y in zip(got, want))
        want = [t.clone() for t in turn()]
        g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=s):
            out = turn()
        assert same(turn())                       # nothing has been replayed yet
        for _ in range(3):
            for t in out:
                t.zero_()
            g.replay()
            assert same(out)
            assert same(turn())
        del g
        dr.status()
    finally:
        case.close()
