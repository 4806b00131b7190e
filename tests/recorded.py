"""Outputs that are kept bit for bit: digests of small seeded runs, compared with tests/golden/recorded_outputs.json.

What is recorded hangs on the order in which long sums are added: the cached rows are rounded to bf16 after sums over thousands of
terms, and the list of a draft tree (or a token drawn by inverse CDF) is decided by differences far below the precision of the
logits.  Another order is as accurate, but changes which rows round up and which of two nodes of equal standing is kept, so a
change of order is a change of results.  `python tests/recorded.py` on a B200 prints the digests of the package on the path.
"""
import hashlib
import json
import os
import sys
from types import SimpleNamespace

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "recorded_outputs.json")


def dims(d, hq, hkv, dh, ffn, vocab):
    return SimpleNamespace(d=d, n_q_heads=hq, n_kv_heads=hkv, head_dim=dh, ffn=ffn, vocab=vocab, rms_eps=1e-5, rope_base=10000.0,
                           dtype="bf16")


# long sums on few rows, with heads of 128 and of 64; and one whose sums are too short to be split evenly over the chip
SHAPES = {"wide128": dims(2560, 20, 4, 128, 1024, 2048), "wide64": dims(2048, 12, 2, 64, 1024, 2048),
          "narrow": dims(256, 4, 2, 64, 512, 2048)}


class Run:
    """A drafter with seeded weights, and the generator that its inputs come from."""

    def __init__(self, shape, seed, batch=1, rows=400, bias=False, project=False):
        import torch
        from paper_2509_23928_b200 import Drafter
        D, self.torch = SHAPES[shape], torch
        self.gen = torch.Generator(device="cuda").manual_seed(seed)
        qw, kvw = D.n_q_heads * D.head_dim, D.n_kv_heads * D.head_dim
        W = {"embed": self.normal(D.vocab, D.d), "lm_head": self.normal(D.vocab, D.d), "fc": self.normal(D.d, 2 * D.d),
             "norm1": 1 + self.normal(D.d), "wq": self.normal(qw, D.d), "wk": self.normal(kvw, D.d), "wv": self.normal(kvw, D.d),
             "wo": self.normal(D.d, qw), "norm2": 1 + self.normal(D.d), "w_gate": self.normal(D.ffn, D.d),
             "w_up": self.normal(D.ffn, D.d), "w_down": self.normal(D.d, D.ffn)}
        if bias:
            W.update(bq=self.normal(qw), bk=self.normal(kvw), bv=self.normal(kvw))
        if project:
            W["resid_proj"] = self.normal(D.d, D.d)
        self.dims, self.batch = D, batch
        self.dr = Drafter(D, W, max_batch=batch, max_len=rows, max_k=8)
        self.resid = self.normal(4, D.d)

    def normal(self, *shape, std=0.02):
        return self.torch.empty(shape, dtype=self.torch.bfloat16, device="cuda").normal_(0.0, std, generator=self.gen)

    def prefill(self, counts):
        n = sum(counts)
        ids = self.torch.randint(0, self.dims.vocab, (n,), dtype=self.torch.int32, device="cuda", generator=self.gen)
        cu = [sum(counts[:i]) for i in range(len(counts) + 1)]
        self.dr.prefill(ids, self.normal(n, self.dims.d, std=1.0), cu, start_pos=[0] * len(counts), resid0=self.resid[0])

    def rows(self, counts):
        parts = [t for b, n in enumerate(counts) if n > 1 for t in self.dr.read_kv(b, 0, n - 1)]
        return digest(*parts)


def digest(*tensors):
    h = hashlib.sha256()
    for t in tensors:
        h.update(t.cpu().contiguous().numpy().tobytes())
    return h.hexdigest()[:16]


# pairs of one prefix build: one pass, several, the edges of the GEMMs' tiles; enough for tiles of 256 weight rows
BUILDS = [[2], [9], [16], [17], [33], [64], [65], [118], [257], [1, 3, 7, 2, 4, 5, 20], [100, 1, 200, 64], [390] * 7]


def prefix_rows(shape, bias, project):
    r = Run(shape, 11, batch=8, bias=bias, project=project)
    out = {}
    for counts in BUILDS:
        r.prefill(counts)
        out["+".join(map(str, counts))] = r.rows(counts)
    r.dr.status()
    return out


def projected_rows(shape):
    """What a projected residual row adds to u, at every step of a chain of one sequence (and the chain's logits)."""
    r = Run(shape, 12, project=True)
    r.prefill([1])
    ids, logits = r.dr.draft(1, 5, r.resid, want_logits=True)
    u = r.dr.tap("u", 1)
    r.dr.status()
    return digest(u, ids, logits)


def trees(shape, project):
    r = Run(shape, 13, project=project)
    out = {}
    for n, topk, depth, keep in ((5, 4, 3, 20), (33, 10, 6, 60), (150, 12, 5, 80), (300, 2, 8, 17)):
        r.prefill([n])
        toks, parents, scores, count = r.dr.draft_tree(0, topk, depth, keep, r.resid)
        out[f"{n} rows, top {topk}, depth {depth}, {keep} kept"] = digest(toks, parents, scores, count[:1],
                                                                      *r.dr.read_kv(0, n - 1, 1 + (depth - 1) * topk))
    r.dr.status()
    return out


RECORDS = {
    "prefix_wide128": lambda: prefix_rows("wide128", False, False),
    "prefix_wide128_bias": lambda: prefix_rows("wide128", True, False),
    "prefix_wide64_bias": lambda: prefix_rows("wide64", True, False),
    "projected_rows": lambda: projected_rows("wide128"),
    "tree_narrow": lambda: trees("narrow", False),
    "tree_wide128": lambda: trees("wide128", False),
    "tree_wide64_projected": lambda: trees("wide64", True),
}


if __name__ == "__main__":
    print(json.dumps({name: RECORDS[name]() for name in (sys.argv[1:] or RECORDS)}, indent=1))
