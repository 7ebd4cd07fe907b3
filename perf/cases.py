"""The calls whose speed this library is measured by, through its public binding.

A case is a dict of plain values; ``kind`` names the entry point:

  step        eg_mla_step: the new token's append and one decode step (every
              gate mode, bf16 and fp32), either issued eagerly with its
              arguments bound once or replayed from a CUDA graph
  layer       eg_mla_layer_decode: one decode step through a whole attention
              layer, from the hidden state to the output projection
  prefill     eg_mla_prefill: packed prompts, attention and cache write
  r0          eg_mla_decode_r0: decode with the gate after the up-projection
  gate_table  eg_mla_gate_table: the gate of every vocabulary entry

Sequence lengths are part of the case (log-uniform in [lo, hi], drawn from
``lens_seed``), everything else is drawn on the GPU from the seed of the state.
Value distributions are those of the package's synthetic workloads.
"""
import math
import random

import torch

from paper_2509_16686_gb300 import _lib

DEV = "cuda"
PAGE = 64
D_ROPE = 64


def _case(**kw):
    c = dict(kind="step", dtype="bf16", gate="mul_ln", batch=1, lo=1, hi=1, lens_seed=0, heads=16, d_nope=128,
             d_rope=D_ROPE, d_c=256, vocab=32000, ids="uniform", permuted=True, affine=True, graph=False,
             n_embd=0, d_e=0)
    c.update(kw)
    return c


def listed():
    return [
        # a handful of short chats: the latency of a step's launches
        _case(name="step_small", batch=4, lo=60, hi=700, lens_seed=1, graph=True),
        # the ordinary serving batch: 32 sequences of 4K tokens, contiguous pages
        _case(name="step_4k", batch=32, lo=4096, hi=4096, permuted=False, affine=False, graph=True),
        # long context: 8 sequences of 32K tokens, pages permuted over one pool
        _case(name="step_32k", batch=8, lo=32768, hi=32768, affine=False),
        # a mixed batch: 128 sequences between 128 and 16384 tokens, Zipf ids
        _case(name="step_ragged", batch=128, lo=128, hi=16384, lens_seed=3, d_c=192, vocab=50000, ids="zipf",
              affine=False),
        # the plain MLA model (gate off) on the same kind of batch
        _case(name="step_mla", gate="none", batch=128, lo=128, hi=16384, lens_seed=3, d_c=512, vocab=50000,
              ids="zipf", affine=False),
        # single precision, the setting of a numerical check against training
        _case(name="step_fp32", dtype="fp32", batch=8, lo=100, hi=3000, lens_seed=4, d_c=256),
        # one of the 24 attention layers of a decode step: 64 sequences of 8K
        _case(name="layer_8k", kind="layer", batch=64, lo=8192, hi=8192, vocab=50000, permuted=False, affine=False,
              n_embd=2048),
        # the prompt of one user, not a multiple of any tile
        _case(name="prefill_one", kind="prefill", batch=1, lo=777, hi=777),
        # a full prefill batch
        _case(name="prefill_4k", kind="prefill", batch=8, lo=4096, hi=4096, affine=False),
        # prompts as they arrive
        _case(name="prefill_ragged", kind="prefill", batch=16, lo=128, hi=4096, lens_seed=6, d_c=192, vocab=50000,
              ids="zipf", affine=False),
        # the paper's literal gate placement
        _case(name="r0_4k", kind="r0", batch=8, lo=4096, hi=4096),
        # the gate table at model load, or per step where it is not stored
        _case(name="gate_table", kind="gate_table", vocab=32000, d_e=256),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "mla", "fp32", "layer", "layer", "prefill", "prefill", "r0",
                       "gate_table"])
    lens_seed = rng.randrange(1 << 20)
    common = dict(lens_seed=lens_seed, ids=rng.choice(["uniform", "zipf"]), permuted=rng.random() < 0.7,
                  affine=rng.random() < 0.5, vocab=_log_int(rng, 1000, 50000))

    def lens(tokens, longest):
        """A batch and a range of lengths with at most `tokens` tokens in all."""
        batch = _log_int(rng, 1, 128)
        hi = _log_int(rng, 16, max(16, min(longest, tokens // batch)))
        return dict(batch=batch, lo=rng.choice([hi, max(1, hi // 128), max(1, hi // 3)]), hi=hi)

    if kind == "step":
        return _case(**common, **lens(400000, 32768), d_c=rng.choice([192, 256]),
                     gate=rng.choice(["mul_ln", "mul_ln", "mul_ln", "mul", "add_ln", "none"]),
                     d_nope=rng.choice([64, 128, 128]), graph=rng.random() < 0.5)
    if kind == "mla":
        return _case(**common, **lens(300000, 32768), d_c=512, gate="none", graph=rng.random() < 0.5)
    if kind == "fp32":
        return _case(**common, **lens(10000, 4096), dtype="fp32", heads=rng.choice([4, 12, 16]),
                     d_nope=rng.choice([32, 64, 128]), d_rope=rng.choice([16, 64]),
                     d_c=rng.choice([64, 128, 256, 512]), gate=rng.choice(["mul_ln", "mul_ln", "none"]))
    if kind == "layer":
        return _case(kind="layer", **common, **lens(400000, 16384), d_c=rng.choice([192, 256]),
                     n_embd=rng.choice([768, 1024, 2048]))
    if kind == "prefill":
        longest = _log_int(rng, 16, 4096)
        batch = _log_int(rng, 1, max(1, min(32, 32768 // longest)))
        return _case(kind="prefill", **common, batch=batch, lo=rng.choice([longest, max(1, longest // 32)]),
                     hi=longest, d_c=rng.choice([64, 128, 192, 256, 512]), heads=rng.choice([8, 12, 16]),
                     gate=rng.choice(["mul_ln", "mul_ln", "none"]))
    if kind == "r0":
        return _case(kind="r0", **common, **lens(32768, 8192), d_c=rng.choice([192, 256]))
    return _case(kind="gate_table", **common, d_c=rng.choice([64, 128, 192, 256]),
                 d_e=rng.choice([64, 128, 256, 512]))


# ------------------------------------------------------------------ inputs
def _lengths(case):
    r = random.Random(case["lens_seed"])
    return [_log_int(r, case["lo"], case["hi"]) for _ in range(case["batch"])]


def _inputs(case, seed):
    """Everything a call reads, on the GPU, from the seed."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    scale = 0.5 if case["dtype"] == "bf16" else 1.0
    H, dn, dr, dc, V = (case[k] for k in ("heads", "d_nope", "d_rope", "d_c", "vocab"))

    def normal(shape, std=1.0, mean=0.0, dtype=dt):
        # drawn in chunks, so that a large tensor needs no second one in fp32
        n = math.prod(shape)
        out = torch.empty(n, dtype=dtype, device=DEV)
        for i in range(0, n, 1 << 26):
            m = min(1 << 26, n - i)
            out[i:i + m] = torch.randn(m, generator=g, device=DEV).mul_(std).add_(mean)
        return out.view(shape)

    def token_ids(n):
        if case["ids"] == "zipf":   # ranks with probability ~ r^-1.1
            cdf = torch.arange(1, V + 1, device=DEV, dtype=torch.float64).pow_(-1.1).cumsum(0)
            u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * cdf[-1]
            return torch.searchsorted(cdf, u).clamp_(max=V - 1).to(torch.int32)
        return torch.randint(0, V, (n,), generator=g, device=DEV, dtype=torch.int32)

    if case["kind"] == "gate_table":
        de = case["d_e"]
        return dict(emb=normal((V, de)), w_ue=normal((dc, de), de ** -0.5))

    lens = _lengths(case)
    B = len(lens)
    pages = [(n + PAGE - 1) // PAGE for n in lens]
    width = max(pages)
    need = sum(pages) if case["permuted"] else B * width
    order = torch.randperm(need, generator=g, device=DEV).to(torch.int32).cpu().tolist() if case["permuted"] else None
    table, k = [], 0
    for b, n in enumerate(pages):
        if order is None:
            table.append(list(range(b * width, (b + 1) * width)))
        else:
            table.append(order[k:k + n] + [order[-1]] * (width - n))
            k += n
    d = dict(lens=lens, block_table=torch.tensor(table, dtype=torch.int32, device=DEV),
             w_uk=normal((H, dn, dc), dc ** -0.5), w_uv=normal((H, dn, dc), dc ** -0.5),
             seq_lens=torch.tensor(lens, dtype=torch.int32, device=DEV))
    if case["affine"]:
        d.update(gamma=normal((dc,), 0.1, 1.0, torch.float32), beta=normal((dc,), 0.1, 0.0, torch.float32))
    else:
        d.update(gamma=torch.ones(dc, device=DEV), beta=torch.zeros(dc, device=DEV))
    if case["kind"] == "r0":
        d["gate_r0"] = normal((V, H * 2 * dn), 0.1, 1.0)
        d["w_ukv"] = torch.cat([d["w_uk"], d["w_uv"]], dim=1).reshape(H * 2 * dn, dc).contiguous()
        d["gamma"] = normal((H * 2 * dn,), 0.1, 1.0, torch.float32)
        d["beta"] = normal((H * 2 * dn,), 0.1, 0.0, torch.float32)
    else:
        d["gate_table"] = normal((V, dc), 0.1, 1.0)
    if case["kind"] == "prefill":
        T = sum(lens)
        cu = [0]
        for n in lens:
            cu.append(cu[-1] + n)
        d.update(q=normal((T, H, dn + dr)), c=normal((T, dc), scale), kr=normal((T, dr)), ids_new=token_ids(T),
                 cu=torch.tensor(cu, dtype=torch.int32, device=DEV),
                 c_pool=torch.zeros((need, PAGE, dc), dtype=dt, device=DEV),
                 kr_pool=torch.zeros((need, PAGE, dr), dtype=dt, device=DEV),
                 id_pool=torch.zeros((need, PAGE), dtype=torch.int32, device=DEV))
        return d
    d.update(c_pool=normal((need, PAGE, dc), scale), kr_pool=normal((need, PAGE, dr)),
             id_pool=token_ids(need * PAGE).view(need, PAGE), ids_new=token_ids(B), positions=d["seq_lens"] - 1)
    if case["kind"] == "layer":
        E = case["n_embd"]
        d.update(x=normal((B, E)), w_qkv_a=normal((H * (dn + dr) + dc + dr, E), E ** -0.5),
                 kv_norm_w=normal((dc,), 0.1, 1.0), w_o=normal((E, H * dn), (H * dn) ** -0.5))
    else:
        d.update(q=normal((B, H, dn + dr)), c_new=normal((B, dc), scale), kr_new=normal((B, dr)))
    return d


def _bytes(n):
    return torch.empty(max(int(n), 1), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    d = _inputs(case, seed)
    H, dn, dc = case["heads"], case["d_nope"], case["d_c"]
    dims = _lib.make_dims(H, dn, case["d_rope"], dn, dc, case["vocab"], dtype=case["dtype"],
                          gate=case["gate"] != "none", gate_op=case["gate"] if case["gate"] != "none" else "mul_ln")
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    kind = case["kind"]
    s = dict(d, kind=kind, dims=dims, status=status)
    if kind == "gate_table":
        s["out"] = torch.empty((case["vocab"], dc), dtype=torch.bfloat16, device=DEV)
        return s
    B, longest = len(d["lens"]), max(d["lens"])
    s["longest"] = longest
    if kind == "prefill":
        s["out"] = torch.empty((sum(d["lens"]), H, dn), dtype=torch.bfloat16, device=DEV)
        s["workspace"] = _bytes(_lib.eg_mla_prefill_workspace_size(dims, B, sum(d["lens"])))
        return s
    if kind == "r0":
        s["out"] = torch.empty((B, H, dn), dtype=torch.bfloat16, device=DEV)
        s["workspace"] = _bytes(_lib.eg_mla_decode_r0_workspace_size(dims, B, d["block_table"].shape[1],
                                                                     d["c_pool"].shape[0]))
        return s
    if kind == "layer":
        s["layer"] = _lib.make_layer_dims(case["n_embd"])
        s["out"] = torch.empty((B, case["n_embd"]), dtype=torch.bfloat16, device=DEV)
        s["workspace"] = _bytes(_lib.eg_mla_layer_workspace_size(dims, s["layer"], B))
        s["weights"] = _lib.make_layer_weights(d["w_qkv_a"], d["kv_norm_w"], d["w_o"], d["gate_table"], d["gamma"],
                                               d["beta"], d["w_uk"], d["w_uv"])
        return s
    s["out"] = torch.empty((B, H, dn), dtype=d["q"].dtype, device=DEV)
    s["workspace"] = _bytes(_lib.eg_mla_decode_workspace_size(dims, B))

    def bound():
        return _lib.bind_step(dims, d["c_pool"], d["kr_pool"], d["id_pool"], d["c_new"], d["kr_new"], d["ids_new"],
                              d["positions"], d["q"], d["block_table"], d["seq_lens"], longest, d["gate_table"],
                              d["gamma"], d["beta"], d["w_uk"], d["w_uv"], s["out"], s["workspace"], 0, status)

    s["step"] = bound()
    if case["graph"]:
        s["step"]()   # the library's first call of a shape comes before any capture
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            s["captured"] = bound()
            s["captured"]()
        s["graph"] = graph
    return s


def run(s):
    kind = s["kind"]
    if kind == "step":
        if "graph" in s:
            s["graph"].replay()
        else:
            s["step"]()
    elif kind == "layer":
        _lib.eg_mla_layer_decode(s["dims"], s["layer"], s["weights"], s["x"], s["ids_new"], s["positions"],
                                 s["c_pool"], s["kr_pool"], s["id_pool"], s["block_table"], s["seq_lens"],
                                 s["longest"], s["out"], s["workspace"], 0, s["status"])
    elif kind == "prefill":
        _lib.eg_mla_prefill(s["dims"], s["q"], s["c"], s["kr"], s["ids_new"], s["cu"], s["longest"], s["gate_table"],
                            s["gamma"], s["beta"], s["w_uk"], s["w_uv"], s["out"], s["workspace"], s["c_pool"],
                            s["kr_pool"], s["id_pool"], s["block_table"], dev_status=s["status"])
    elif kind == "r0":
        _lib.eg_mla_decode_r0(s["dims"], s["q"], s["c_pool"], s["kr_pool"], s["id_pool"], s["block_table"],
                              s["seq_lens"], s["w_ukv"], s["gate_r0"], s["gamma"], s["beta"], s["out"],
                              s["workspace"], dev_status=s["status"])
    else:
        _lib.eg_mla_gate_table(s["dims"], s["emb"], s["w_ue"], s["out"], dev_status=s["status"])
    got = {"out": s["out"], "status": s["status"]}
    if kind in ("step", "layer", "prefill"):
        got.update(c_pool=s["c_pool"], kr_pool=s["kr_pool"], id_pool=s["id_pool"])
    return got


def work(case):
    H, dn, dr, dc, V = (case[k] for k in ("heads", "d_nope", "d_rope", "d_c", "vocab"))
    e = 2 if case["dtype"] == "bf16" else 4
    kind = case["kind"]
    if kind == "gate_table":
        de = case["d_e"]
        return {"bytes": 2 * (V * de + dc * de + V * dc), "flops": 2 * V * de * dc}
    lens = _lengths(case)
    B, T = len(lens), sum(lens)
    gated = case["gate"] != "none"
    distinct = _zipf_distinct(V, T) if case["ids"] == "zipf" else V * (1 - math.exp(-T / V))
    token = (dc + dr) * e + (4 if gated else 0)
    up = 2 * H * dn * dc * e     # W_UK and W_UV
    if kind == "prefill":
        rows = T * (H * (dn + dr) + H * dn) * e + 2 * T * token + up + (distinct * dc * e if gated else 0)
        pairs = sum(n * (n + 1) // 2 for n in lens)
        return {"bytes": int(rows), "flops": 2 * T * dc * H * 2 * dn + 2 * pairs * H * (2 * dn + dr)}
    if kind == "r0":
        return {"bytes": int(T * token + distinct * H * 2 * dn * e + up + B * H * (2 * dn + dr) * e),
                "flops": 2 * T * dc * H * 2 * dn + 2 * T * H * (2 * dn + dr)}
    bytes_ = T * token + up + (distinct * dc * e if gated else 0) + B * H * (2 * dn + dr) * e
    flops = 2 * T * H * (2 * dc + dr) + 2 * B * H * dc * 2 * dn
    if kind == "layer":
        E = case["n_embd"]
        rows = H * (dn + dr) + dc + dr + H * dn
        bytes_ += rows * E * 2 + 2 * B * E * 2 - B * H * (2 * dn + dr) * e
        flops += 2 * B * rows * E
    return {"bytes": int(bytes_), "flops": flops}


def _zipf_distinct(V, T):
    """The expected number of distinct ids among T draws with probability ~ r^-1.1."""
    total = sum(r ** -1.1 for r in range(1, V + 1))
    return sum(1 - math.exp(-T * r ** -1.1 / total) for r in range(1, V + 1))


def tolerance(case):
    # about four times the distance of the path from exact()
    if case["dtype"] == "fp32":
        return {"rel": 2e-6}
    if case["kind"] == "gate_table":
        return {"rel": 7e-3}
    return {"rel": 1.2e-2}


# ------------------------------------------------------------------- exact
def _gated(case, d, c, ids):
    """The latent rows c (64 bits) under the gate, normalised where the mode says so."""
    if case["gate"] == "none":
        return c
    g = d["gate_table"].double()[ids.long()]
    if case["gate"] == "mul":
        return c * g
    z = c + g if case["gate"] == "add_ln" else c * g
    z = z - z.mean(-1, keepdim=True)
    z = z / (z.square().mean(-1, keepdim=True) + 1e-5).sqrt()
    return z * d["gamma"].double() + d["beta"].double()


def _rows(case, d, b, n):
    """Page rows of sequence b's first n tokens."""
    at = torch.arange(n, device=DEV)
    return d["block_table"][b].long()[at // PAGE] * PAGE + at % PAGE


def _rotated(x, pos):
    """Consecutive pairs of x [..., d] turned by pos * 10000^(-2i/d)."""
    n = x.shape[-1]
    w = 10000.0 ** (-torch.arange(0, n, 2, device=DEV, dtype=torch.float64) / n)
    a = pos.double()[:, None] * w
    a = a.view(a.shape[0], *([1] * (x.dim() - 2)), n // 2)
    u, v = x[..., 0::2], x[..., 1::2]
    return torch.stack([u * a.cos() - v * a.sin(), u * a.sin() + v * a.cos()], -1).flatten(-2)


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "gate_table":
        return {"out": d["emb"].double() @ d["w_ue"].double().T, "status": None}
    H, dn, dr, dc = (case[k] for k in ("heads", "d_nope", "d_rope", "d_c"))
    lens, B = d["lens"], len(d["lens"])
    scale = 1 / math.sqrt(dn + dr)
    w_uk, w_uv = d["w_uk"].double(), d["w_uv"].double()
    got = {"status": None}

    if kind == "prefill":
        out = torch.empty((sum(lens), H, dn), dtype=torch.float64, device=DEV)
        pools = [d[k].view(-1, d[k].shape[-1]) for k in ("c_pool", "kr_pool")] + [d["id_pool"].view(-1)]
        at = 0
        for b, n in enumerate(lens):
            here = slice(at, at + n)
            rows = _rows(case, d, b, n)
            for pool, new in zip(pools, (d["c"], d["kr"], d["ids_new"])):
                pool[rows] = new[here]
            z = _gated(case, d, d["c"][here].double(), d["ids_new"][here])
            kr = d["kr"][here].double()
            for h in range(H):
                k = torch.cat([z @ w_uk[h].T, kr], -1)
                s = (d["q"][here, h].double() @ k.T).mul_(scale)
                s.masked_fill_(torch.ones(n, n, dtype=torch.bool, device=DEV).triu_(1), -math.inf)
                out[here, h] = s.softmax(-1) @ (z @ w_uv[h].T)
            at += n
        return dict(got, out=out, c_pool=d["c_pool"].double(), kr_pool=d["kr_pool"].double(), id_pool=d["id_pool"])

    c_pool, kr_pool = d["c_pool"].double(), d["kr_pool"].double()
    ids = d["id_pool"].view(-1)
    c_rows, kr_rows = c_pool.view(-1, dc), kr_pool.view(-1, dr)
    if kind == "layer":
        pos = d["positions"]
        p = d["x"].double() @ d["w_qkv_a"].double().T
        nq = H * (dn + dr)
        q = p[:, :nq].reshape(B, H, dn + dr)
        q = torch.cat([q[..., :dn], _rotated(q[..., dn:], pos)], -1)
        c_new = p[:, nq:nq + dc]
        c_new = c_new / (c_new.square().mean(-1, keepdim=True) + 2.0 ** -23).sqrt() * d["kv_norm_w"].double()
        kr_new = _rotated(p[:, nq + dc:], pos)
    else:
        q = d["q"].double()
    if kind == "step":
        c_new, kr_new = d["c_new"].double(), d["kr_new"].double()
    out = torch.empty((B, H, dn), dtype=torch.float64, device=DEV)
    for b, n in enumerate(lens):
        rows = _rows(case, d, b, n)
        if kind != "r0":
            c_rows[rows[-1]], kr_rows[rows[-1]], ids[rows[-1]] = c_new[b], kr_new[b], d["ids_new"][b]
        c, kr, i = c_rows[rows], kr_rows[rows], ids[rows]
        if kind == "r0":
            z = (c @ d["w_ukv"].double().T) * d["gate_r0"][i.long()].double()
            z = z - z.mean(-1, keepdim=True)
            z = z / (z.square().mean(-1, keepdim=True) + 1e-5).sqrt()
            z = (z * d["gamma"].double() + d["beta"].double()).view(n, H, 2, dn)
            s = torch.einsum("hd,nhd->hn", q[b, :, :dn], z[:, :, 0]) + q[b, :, dn:] @ kr.T
            out[b] = torch.einsum("hn,nhd->hd", (s * scale).softmax(-1), z[:, :, 1])
            continue
        z = _gated(case, d, c, i)
        qa = torch.einsum("hd,hdc->hc", q[b, :, :dn], w_uk)
        s = (qa @ z.T + q[b, :, dn:] @ kr.T) * scale
        out[b] = torch.einsum("hc,hdc->hd", s.softmax(-1) @ z, w_uv)
    if kind == "r0":
        return dict(got, out=out)
    if kind == "layer":
        out = out.reshape(B, -1) @ d["w_o"].double().T
    return dict(got, out=out, c_pool=c_pool, kr_pool=kr_pool, id_pool=d["id_pool"])
