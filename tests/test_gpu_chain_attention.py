"""The attention of the one-sequence chain kernel against the definition in 64 bits, from the query projection and the cache that the
step itself left."""
from types import SimpleNamespace

import pytest

pytestmark = pytest.mark.gpu
# "many heads": more units than CTAs, so a CTA stages one after the other (n up to 128; longer caches are not staged)
SHAPES = {"heads of 128": (20, 4, 128), "heads of 64": (12, 2, 64), "few heads": (4, 2, 64), "many heads": (336, 48, 64)}


# lengths: one row; the edges of a warp's block and of a split; units that are staged and units that are not (more than 128 rows: 1000
# rows in 7 splits); 18 and 31 splits, more than a CTA has warps
@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 65, 225, 257, 560, 897, 1000])
@pytest.mark.parametrize("heads", SHAPES)
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_one_sequence(dtype, heads, n):
    """fp32 throughout: a score is a chain of up to 128 products (2^-24 of the sum of their sizes each, a few units), the angles and
    exponentials are fp32 functions, the output a sum over the rows: 3e-5 of the largest output covers them several times over, a row
    or a part left out is 1e-3 or more."""
    import torch
    from paper_2509_23928_b200 import Drafter
    hq, hkv, dh = SHAPES[heads]
    d, half = 256, dh // 2
    D = SimpleNamespace(d=d, n_q_heads=hq, n_kv_heads=hkv, head_dim=dh, ffn=512, vocab=640, rms_eps=1e-5, rope_base=10000.0, dtype=dtype)
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(n)
    new = lambda *shape, std=0.02: torch.empty(shape, dtype=t, device="cuda").normal_(0.0, std, generator=gen)
    qw, kvw = hq * dh, hkv * dh
    W = {"embed": new(640, d), "lm_head": new(640, d), "fc": new(d, 2 * d), "norm1": 1 + new(d), "wq": new(qw, d, std=0.08), "wk": new(kvw, d, std=0.08),
         "wv": new(kvw, d), "wo": new(d, qw), "norm2": 1 + new(d), "w_gate": new(512, d), "w_up": new(512, d), "w_down": new(d, 512)}
    dr = Drafter(D, W, max_batch=1, max_len=1024, max_k=4)
    ids = torch.randint(0, 640, (n,), dtype=torch.int32, device="cuda", generator=gen)
    dr.prefill(ids, new(n, d, std=1.0), [0, n], start_pos=[0])
    freq = D.rope_base ** (-torch.arange(half, dtype=torch.float64, device="cuda") / half)
    for k in (1, 3):
        dr.set_kv_len_batch([n - 1], restore_pending=True)
        dr.draft(1, k, None)
        p = n - 1 + k - 1
        q, got = dr.tap("q", 1).double().view(hq, dh), dr.tap("attn", 1).double().view(hq, dh)
        lo, hi, a = q[:, :half], q[:, half:], p * freq
        rot = torch.cat([lo * a.cos() - hi * a.sin(), hi * a.cos() + lo * a.sin()], -1)
        key, val = (x.double().view(p + 1, hkv, dh).repeat_interleave(hq // hkv, 1) for x in dr.read_kv(0, 0, p + 1))
        want = torch.einsum("hn,nhd->hd", torch.softmax(torch.einsum("hd,nhd->hn", rot, key) / dh ** 0.5, -1), val)
        assert float((got - want).abs().max()) <= 3e-5 * float(want.abs().max())
    dr.status()
    dr.close()
