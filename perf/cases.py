"""The work that users of the drafter library have it do, as measurable cases.

A server that decodes with a drafter makes the same few calls over and over, and every case is one turn of them:

  open     requests arrive: the prefix of every sequence is built from its prompt (a slot that served another request
           before is started again at row 0) and the first chain is drafted.
  round    the steady state of greedy speculative decoding: the rows of the tokens the target accepted last time are
           rebuilt from its true features, k tokens are drafted, and they are verified against the target's logits.
  sampled  the same round at temperature 1: tokens drawn from the drafter's distribution, verified by speculative sampling.
  tree     the same round for one sequence with a draft tree in place of the chain.
  score    a drafter is evaluated on recorded continuations, many sequences at a time: the rows of the last window are
           built from recorded features, then the next window is run with the recorded tokens and its logits are kept.

Every turn starts from cached rows that a prefill truncates to (start_pos), so that a case can be run again and again on
the same state.  Chains also return the logits of every step: they are what a caller that wants more than the tokens gets.
"""
import math

import torch

from paper_2509_23928_b200 import Drafter


class Dims:
    """What the drafter is told about a model."""

    def __init__(self, d, n_q_heads, n_kv_heads, head_dim, ffn, vocab, rms_eps, dtype, logits):
        self.d, self.n_q_heads, self.n_kv_heads, self.head_dim, self.ffn, self.vocab = d, n_q_heads, n_kv_heads, head_dim, ffn, vocab
        self.rms_eps, self.rope_base, self.dtype = rms_eps, 10000.0, dtype
        self.logits = torch.bfloat16 if logits == "bf16" else torch.float32      # element type of the target's logits
        self.torch = torch.bfloat16 if dtype == "bf16" else torch.float32
        self.size = 2 if dtype == "bf16" else 4
        self.qw, self.kvw = n_q_heads * head_dim, n_kv_heads * head_dim

    def prefix_params(self):
        return 2 * self.d * self.d + 2 * self.kvw * self.d

    def step_params(self):
        d = self.d
        return 2 * d * d + (self.qw + 2 * self.kvw) * d + d * self.qw + 3 * d * self.ffn + self.vocab * d


SHAPES = {
    # the smallest drafter of the repository's configurations, in fp32
    "tiny": Dims(256, 4, 4, 64, 688, 1024, 1e-5, "f32", "f32"),
    # the two full-size ones
    "llava": Dims(4096, 32, 32, 128, 11008, 32000, 1e-5, "bf16", "bf16"),
    "qwen": Dims(3584, 28, 4, 128, 18944, 152064, 1e-6, "bf16", "bf16"),
    # a smaller one of no particular model: five query heads per KV head, and a vocabulary whose rows are not aligned
    "mid": Dims(2560, 20, 4, 128, 6912, 50257, 1e-6, "bf16", "bf16"),
}


def _case(op, shape, batch, k, lo, hi, name=None, **more):
    c = {"op": op, "shape": shape, "batch": batch, "k": k, "text_lo": lo, "text_hi": hi, "bias": False, "project": False}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one short sequence of a tiny fp32 drafter, where launches and grid barriers are all there is
        _case("round", "tiny", 1, 4, 32, 32, "round_tiny_f32_b1"),
        # one user, interactive: the case the method is quoted on
        _case("round", "llava", 1, 5, 128, 128, "round_llava_b1"),
        # a small server's batch, every sequence of its own length
        _case("round", "llava", 16, 5, 64, 512, "round_llava_b16_ragged"),
        # the same batch for a drafter that keeps 576 visual positions in its cache: attention over long caches
        _case("round", "llava", 16, 5, 704, 704, "round_llava_b16_visual"),
        # grouped KV heads, QKV biases, a large vocabulary, longer chains
        _case("round", "qwen", 8, 7, 256, 256, "round_qwen_b8", bias=True),
        # decoding at temperature 1
        _case("sampled", "llava", 16, 5, 128, 128, "sampled_llava_b16"),
        # the paper's own setting: a top-10 tree of depth 6 with 60 nodes kept, residual rows projected
        _case("tree", "llava", 1, 6, 128, 128, "tree_llava_b1", topk=10, keep=60, project=True),
        # one request arrives with a short question
        _case("open", "llava", 1, 5, 117, 117, "open_llava_b1"),
        # a few requests of uneven lengths
        _case("open", "mid", 5, 3, 37, 411, "open_mid_b5_ragged"),
        # a batch of requests
        _case("open", "qwen", 8, 7, 256, 256, "open_qwen_b8", bias=True),
        # the largest: a batch whose prompts hold 2048 visual positions each
        _case("open", "llava", 16, 5, 2176, 2176, "open_llava_b16_visual"),
        # as many sequences as a context takes, evaluated on recorded continuations
        _case("score", "llava", 64, 5, 64, 512, "score_llava_b64_ragged"),
    ]


def _spread(rng, lo, hi):
    """A whole number of [lo, hi], spread evenly over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["round", "round", "sampled", "tree", "open", "open", "score"])
    shape = rng.choice(["llava", "llava", "qwen", "mid", "tiny"])
    k = rng.randint(1, 8)
    more = {"bias": rng.random() < 0.3, "project": rng.random() < 0.25}
    if op == "tree":
        batch, k = 1, rng.randint(2, 8)
        more["topk"] = rng.randint(2, 12)
        more["keep"] = rng.randint(8, 80)
    elif op == "score":
        batch = _spread(rng, 2, 64)
    elif op == "sampled" and shape == "tiny":
        batch = 1                                  # (drawing is for bf16 drafters, or for one sequence)
    else:
        batch = _spread(rng, 1, 16)
    longest = 2048 if op == "open" else 1024 if batch <= 16 else 512
    hi = _spread(rng, 4, longest)
    lo = hi if rng.random() < 0.4 else rng.randint(1 + hi // 8, hi)
    return _case(op, shape, batch, k, lo, hi, **more)


# ------------------------------------------------------------------------------------------------------------ state
def _lengths(case, gen):
    return torch.randint(case["text_lo"], case["text_hi"] + 1, (case["batch"],), generator=gen).tolist()


def _accepted(case, gen):
    """How many drafted tokens the target took, per sequence: P(n) ~ 0.75^n."""
    w = 0.75 ** torch.arange(case["k"] + 1, dtype=torch.float64)
    return torch.multinomial(w, case["batch"], replacement=True, generator=gen).tolist()


def _starts(counts):
    cu = [0]
    for n in counts:
        cu.append(cu[-1] + n)
    return cu


def _inputs(case, seed):
    """Everything that a turn is given, drawn from the seed alone; and the two generators, for what follows the draft."""
    D = SHAPES[case["shape"]]
    op, B, k = case["op"], case["batch"], case["k"]
    host = torch.Generator().manual_seed(seed)                       # lengths and accept counts
    gen = torch.Generator(device="cuda").manual_seed(seed)           # everything on the GPU

    def normal(*shape, std=1.0, mean=0.0, dtype=D.torch):
        return torch.empty(shape, dtype=dtype, device="cuda").normal_(mean, std, generator=gen)

    def tokens(n):
        return torch.randint(0, D.vocab, (n,), dtype=torch.int32, device="cuda", generator=gen)

    d, F, V = D.d, D.ffn, D.vocab
    W = {"embed": normal(V, d, std=0.02), "lm_head": normal(V, d, std=0.02), "fc": normal(d, 2 * d, std=0.02),
         "norm1": normal(d, std=0.02, mean=1.0), "wq": normal(D.qw, d, std=0.02), "wk": normal(D.kvw, d, std=0.02),
         "wv": normal(D.kvw, d, std=0.02), "wo": normal(d, D.qw, std=0.02), "norm2": normal(d, std=0.02, mean=1.0),
         "w_gate": normal(F, d, std=0.02), "w_up": normal(F, d, std=0.02), "w_down": normal(d, F, std=0.02)}
    if case["bias"]:
        W.update(bq=normal(D.qw, std=0.02), bk=normal(D.kvw, std=0.02), bv=normal(D.kvw, std=0.02))
    if case["project"]:
        W["resid_proj"] = normal(d, d, std=0.02)
    T = _lengths(case, host)
    x = {"W": W, "T": T, "resid": normal(4, d, std=0.02), "normal": normal, "host": host}
    # the prompts: the rows [0, T) of every slot where the turn does not build them itself
    cu = _starts(T if op == "open" else [t + 1 for t in T])
    x["prompt"] = (tokens(cu[-1]), normal(cu[-1], d), cu)
    if op != "open":
        # the pairs of the last turn, which every turn builds again
        n = [k] * B if op == "score" else [a + 1 for a in _accepted(case, host)]
        cu = _starts(n)
        x["pairs"] = (tokens(cu[-1]), normal(cu[-1], d), cu)
    if op == "score":
        x["recorded"] = tokens(B * k).view(B, k)
    if op == "sampled":
        x["uniforms"] = torch.empty((B, k, V), device="cuda").uniform_(1e-6, 1.0 - 1e-6, generator=gen)
        x["u_accept"] = torch.empty((B, k), device="cuda").uniform_(0.0, 1.0, generator=gen)
        x["u_sample"] = torch.empty((B,), device="cuda").uniform_(0.0, 1.0, generator=gen)
    return x


def prepare(case, seed):
    D = SHAPES[case["shape"]]
    op, B, k, V = case["op"], case["batch"], case["k"], D.vocab
    x = _inputs(case, seed)
    T, host, normal = x["T"], x["host"], x["normal"]
    extra = 1 + (k - 1) * case["topk"] if op == "tree" else k
    dr = Drafter(D, x.pop("W"), max_batch=B, max_len=max(T) + 2 * k + 2 + extra, max_k=max(8, k))
    st = {"op": op, "B": B, "k": k, "drafter": dr, "resid": x["resid"]}
    ids, hidden, cu = x["prompt"]
    if op == "open":
        st.update(ids=ids, hidden=hidden, cu=cu, start=[0] * B)
        return st
    dr.prefill(ids, hidden, cu, start_pos=[0] * B, resid0=st["resid"][0])
    ids, hidden, cu = x["pairs"]
    st.update(ids=ids, hidden=hidden, cu=cu, start=T)
    if op == "score":
        st["recorded"] = x["recorded"]
        return st
    # the target's logits: they follow the draft for a while, as a target's do
    dr.prefill(st["ids"], st["hidden"], cu, start_pos=T, resid0=st["resid"][0])
    if op == "sampled":
        st.update(uniforms=x["uniforms"], u_accept=x["u_accept"], u_sample=x["u_sample"])
        draft_logits = dr.draft_sampled(B, k, 1.0, st["uniforms"], st["resid"])[1]
        st["target"] = torch.cat([draft_logits + normal(B, k, V, dtype=torch.float32), normal(B, 1, V, dtype=torch.float32)], 1).to(D.logits)
        return st
    if op == "tree":
        toks, parents, _, count = dr.draft_tree(0, case["topk"], k, case["keep"], st["resid"])
        toks, parents, count = toks.tolist(), parents.tolist(), int(count[0])
        st["topk"], st["keep"] = case["topk"], case["keep"]
        st["target"] = normal(count + 1, V, dtype=D.logits)
        at, left = -1, _accepted(case, host)[0]
        for i in range(count):                                       # a parent comes before its children
            if left and parents[i] == at:
                st["target"][at + 1, toks[i]] = 12.0
                at, left = i, left - 1
        return st
    drafted = dr.draft(B, k, st["resid"]).tolist()
    st["target"] = normal(B, k + 1, V, dtype=D.logits)
    for b, n in enumerate(_accepted(case, host)):
        for j in range(min(n + 1, k)):
            st["target"][b, j, drafted[b][j]] = 12.0 if j < n else -12.0
    return st


def run(state):
    dr, B, k, resid = state["drafter"], state["B"], state["k"], state["resid"]
    dr.prefill(state["ids"], state["hidden"], state["cu"], start_pos=state["start"], resid0=resid[0])
    if state["op"] == "open":
        ids, logits = dr.draft(B, k, resid, want_logits=True)
        return {"ids": ids, "logits": logits}
    if state["op"] == "score":
        _, logits = dr.draft(B, k, resid, forced_ids=state["recorded"], want_logits=True)
        return {"logits": logits}
    if state["op"] == "tree":
        toks, parents, scores, count = dr.draft_tree(0, state["topk"], k, state["keep"], resid)
        n, path, nxt, rows = dr.verify_tree(0, k, state["target"])
        return {"tokens": toks, "parents": parents, "scores": scores, "count": count, "accepted": n, "path": path, "next": nxt, "rows": rows}
    if state["op"] == "sampled":
        ids, logits = dr.draft_sampled(B, k, 1.0, state["uniforms"], resid)
        n, nxt, rows = dr.verify_sampled(ids, logits, state["target"], 1.0, state["u_accept"], state["u_sample"])
    else:
        ids, logits = dr.draft(B, k, resid, want_logits=True)
        n, nxt, rows = dr.verify(ids, state["target"])
    return {"ids": ids, "logits": logits, "accepted": n, "next": nxt, "rows": rows}


def work(case):
    """Weights once per draft step (no step can start before the one before it is over, and a drafter does not fit on the
    chip), the prefix layers' weights once, every cached row once per step, hidden states, logits and draws once."""
    D = SHAPES[case["shape"]]
    op, B, k, es = case["op"], case["batch"], case["k"], D.size
    T = (case["text_lo"] + case["text_hi"]) / 2
    if op == "open":
        pairs, rows = B * (T - 1), T - 1
    else:
        n = k - 1 if op == "score" else sum(i * 0.75 ** i for i in range(k + 1)) / sum(0.75 ** i for i in range(k + 1))
        pairs, rows = B * n, T + n
    pb = (D.prefix_params() if pairs > 0 else 0) * es + (pairs + B) * D.d * es + pairs * (D.d + 2 * D.kvw) * es
    pf = 2.0 * pairs * D.prefix_params()
    nodes = B * k if op != "tree" else 1 + (k - 1) * case["topk"]
    kept = B * k if op != "tree" else 0                              # positions whose logits are handed out
    db = k * D.step_params() * es + B * k * 2 * (rows + k / 2) * D.kvw * es + 4.0 * kept * D.vocab
    df = 2.0 * nodes * D.step_params() + 4.0 * nodes * rows * D.qw
    if case["project"]:
        db += 2 * D.d * D.d * es
        df += 2.0 * 5 * D.d * D.d
    lb = 2 if D.logits == torch.bfloat16 else 4
    vb = 0.0
    if op in ("round", "sampled"):
        vb = B * (k + 1) * D.vocab * lb + (2 * 4.0 * B * k * D.vocab if op == "sampled" else 0)
    elif op == "tree":
        vb = (min(case["keep"], case["topk"] + (k - 1) * case["topk"] ** 2) + 1) * D.vocab * lb
    return {"bytes": pb + db + vb, "flops": pf + df}


def tolerance(case):
    """Measured by running the cases through the library's other kernels (the prefix built 16 pairs at a time and on the
    tensor cores, the chain in one launch and one launch per phase), which add in another order; about four times the
    largest difference seen.  fp32: 2e-7 with rounding alone.  bf16: 2e-5 when only the order of a chain's sums changes,
    1.4e-3 when the order inside the prefix changes which way rows of the cache and their operands are rounded to bf16.
    More than 16 sequences: 6e-3, since there a chain's activations are rounded to bf16 between the layers as well."""
    if SHAPES[case["shape"]].dtype == "f32":
        return {"rel": 2e-6, "differ": 0.0}
    if case["batch"] > 16:
        return {"rel": 2.5e-2, "differ": 0.01}
    return {"rel": 5e-3, "differ": 0.01}


@torch.no_grad()
def exact(case, seed):
    """The drafter's logits in 64 bits, from the definition of the step.  A chain that feeds its own tokens has such a value
    only as long as every token is decided by more than 32 or 16 bits may move a logit; a tree of near-ties has none."""
    op, B, k, D = case["op"], case["batch"], case["k"], SHAPES[case["shape"]]
    if op == "tree":
        return None
    x = _inputs(case, seed)
    W = {n: w.double() for n, w in x["W"].items() if n not in ("embed", "lm_head")}
    rho = x["resid"].double()
    if case["project"]:
        rho = rho @ W["resid_proj"].T
    half = D.head_dim // 2
    freq = D.rope_base ** (-torch.arange(half, dtype=torch.float64, device="cuda") / half)

    def norm(u, gain):
        return u * torch.rsqrt((u * u).mean(-1, keepdim=True) + D.rms_eps) * gain

    def fuse(f, ids, step):
        return torch.cat([f.double(), x["W"]["embed"][ids.long()].double()], -1) @ W["fc"].T + rho[min(step, 3)]

    def rows(h, m, heads):
        z = h @ W["w" + m].T + (W["b" + m] if case["bias"] else 0.0)
        return z.view(len(h), heads, D.head_dim)

    def rope(z, pos):
        a = pos.double()[:, None] * freq
        c, s = a.cos()[:, None], a.sin()[:, None]
        lo, hi = z[..., :half], z[..., half:]
        return torch.cat([lo * c - hi * s, hi * c + lo * s], -1)

    cached, feats, last = [], [], []                                 # per sequence: K and V; the pending pair
    for b in range(B):
        parts = [(x["prompt"], op != "open")] + ([(x["pairs"], False)] if op != "open" else [])
        ids = torch.cat([p[0][p[2][b]:p[2][b + 1] - cut] for p, cut in parts])
        hidden = torch.cat([p[1][p[2][b]:p[2][b + 1] - cut] for p, cut in parts])
        h = norm(fuse(hidden[:-1], ids[:-1], 0), W["norm1"])
        pos = torch.arange(len(h), device="cuda")
        cached.append([rope(rows(h, "k", D.n_kv_heads), pos), rows(h, "v", D.n_kv_heads)])
        feats.append(hidden[-1].double())
        last.append(ids[-1])
    f, tok = torch.stack(feats), torch.stack(last)
    pos = torch.tensor([len(c[0]) for c in cached], device="cuda")
    # what may move a logit, of the logits' root mean square: the lower half of a bf16 or fp32 number, with room for the largest of many
    sure = 6e-3 if D.dtype == "bf16" else 1e-5
    ids, logits = [], torch.empty((B, k, D.vocab), dtype=torch.float64, device="cuda")
    for s in range(k):
        u = fuse(f, tok, s)
        h = norm(u, W["norm1"])
        q, kk, vv = rope(rows(h, "q", D.n_q_heads), pos + s), rope(rows(h, "k", D.n_kv_heads), pos + s), rows(h, "v", D.n_kv_heads)
        out = []
        for b, c in enumerate(cached):
            c[0], c[1] = torch.cat([c[0], kk[b:b + 1]]), torch.cat([c[1], vv[b:b + 1]])
            g = q[b].view(D.n_kv_heads, -1, D.head_dim)
            p = torch.softmax(torch.einsum("hgd,nhd->hgn", g, c[0]) / math.sqrt(D.head_dim), -1)
            out.append(torch.einsum("hgn,nhd->hgd", p, c[1]).reshape(-1))
        y = u + torch.stack(out) @ W["wo"].T
        h = norm(y, W["norm2"])
        f = y + (torch.nn.functional.silu(h @ W["w_gate"].T) * (h @ W["w_up"].T)) @ W["w_down"].T
        for lo in range(0, D.vocab, 16384):
            logits[:, s, lo:lo + 16384] = f @ x["W"]["lm_head"][lo:lo + 16384].double().T
        if op == "score":
            tok = x["recorded"][:, s]
            continue
        z = logits[:, s] - torch.log(-torch.log(x["uniforms"][:, s].double())) if op == "sampled" else logits[:, s]
        top = z.topk(2)
        if s < k - 1 and bool((top.values[:, 0] - top.values[:, 1] < sure * logits[:, s].square().mean(-1).sqrt()).any()):
            return None
        tok = top.indices[:, 0]
        ids.append(tok.int())
    out = {"logits": logits}
    if op in ("round", "sampled"):
        out.update(accepted=None, next=None, rows=None)
    return out if op == "score" else {"ids": None, **out}
