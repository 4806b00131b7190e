"""Projected residual rows, in one pass over the projection for several rows."""
from types import SimpleNamespace

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 2, 4, 5, 8])
@pytest.mark.parametrize("d", [264, 2560])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_a_projection_that_is_exact(dtype, d, rows):
    """A projection that permutes and doubles is exact in either type, so a drafter that projects the rows gives, bit for bit, what
    one gives that is handed the permuted and doubled rows."""
    import torch
    from paper_2509_23928_b200 import Drafter
    D = SimpleNamespace(d=d, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=512, vocab=640, rms_eps=1e-5, rope_base=10000.0, dtype=dtype)
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(d + rows)
    new = lambda *shape: torch.empty(shape, dtype=t, device="cuda").normal_(0.0, 0.02, generator=gen)
    qw, kvw = 256, 128
    W = {"embed": new(640, d), "lm_head": new(640, d), "fc": new(d, 2 * d), "norm1": 1 + new(d), "wq": new(qw, d), "wk": new(kvw, d),
         "wv": new(kvw, d), "wo": new(d, qw), "norm2": 1 + new(d), "w_gate": new(512, d), "w_up": new(512, d), "w_down": new(d, 512)}
    perm = torch.randperm(d, device="cuda", generator=gen)
    P = torch.zeros((d, d), dtype=t, device="cuda")
    P[torch.arange(d, device="cuda"), perm] = 2.0
    resid, ids, hidden = new(rows, d), torch.arange(6, dtype=torch.int32, device="cuda"), new(6, d)
    out = []
    for weights, r in (({**W, "resid_proj": P}, resid), (W, 2 * resid[:, perm].contiguous())):
        dr = Drafter(D, weights, max_batch=1, max_len=32, max_k=8)
        dr.prefill(ids, hidden, [0, 6], resid0=r[0].contiguous())
        got = dr.draft(1, 8, r, want_logits=True)
        out.append((*got, *dr.read_kv(0, 0, 13)))
        dr.status()
        dr.close()
    assert all(torch.equal(x, y) for x, y in zip(*out))


@pytest.mark.parametrize("rows", [1, 3, 4, 6])
@pytest.mark.parametrize("d", [264, 2560])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_a_dense_projection(dtype, d, rows):
    """With a fusion FC of zeros the fused input is the projected row itself.  A row is a chain of d / 32 fused multiply-adds a lane and
    five additions across the lanes, each rounded once: (d / 32 + 5) * 2^-24 of the sum of the products' sizes, and as much again where
    a lane's turns do not come out even."""
    import torch
    from paper_2509_23928_b200 import Drafter
    D = SimpleNamespace(d=d, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=512, vocab=640, rms_eps=1e-5, rope_base=10000.0, dtype=dtype)
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(d + rows)
    new = lambda *shape: torch.empty(shape, dtype=t, device="cuda").normal_(0.0, 0.02, generator=gen)
    W = {"embed": new(640, d), "lm_head": new(640, d), "fc": torch.zeros((d, 2 * d), dtype=t, device="cuda"), "norm1": 1 + new(d),
         "wq": new(256, d), "wk": new(128, d), "wv": new(128, d), "wo": new(d, 256), "norm2": 1 + new(d), "w_gate": new(512, d),
         "w_up": new(512, d), "w_down": new(d, 512), "resid_proj": new(d, d)}
    resid, ids, hidden = new(rows, d), torch.arange(6, dtype=torch.int32, device="cuda"), new(6, d)
    dr = Drafter(D, W, max_batch=1, max_len=32, max_k=8)
    P, r = W["resid_proj"].double(), resid.double()
    want, size = r @ P.T, r.abs() @ P.abs().T
    for s in range(rows):
        dr.prefill(ids, hidden, [0, 6], start_pos=[0])
        dr.draft(1, s + 1, resid)
        got = dr.tap("u", 1)[0].double()
        assert bool(((got - want[s]).abs() <= 2 * (d / 32 + 5) * 2.0 ** -24 * size[s]).all()), s
    dr.status()
    dr.close()
