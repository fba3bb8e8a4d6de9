"""The measured workloads of this library: what a video speculative-decoding program asks of it, call by call and as a whole step.

A program uses the library at two rates.  Once per prompt it scores the visual tokens (`hippo_attention_mass` per target layer,
then `hippo_select_tokens`) and prunes the draft cache (`hippo_gather_kv`); these calls are issued one by one.  Per decoding
round it drafts tokens (one `hippo_draft_attention` per draft layer and token), verifies them (`hippo_verify_attention` per
target layer, or all layers in one `hippo_verify_attention_layers`) and accepts (`hippo_accept`); the attention legs are
captured once into CUDA graphs and replayed, as `paper_2601_08273_b200/vpsd.py` and `bench.py` do, acceptance is a plain call.

Shapes are those of `workloads.CONFIGS` (a tiny fp32 case, 7B-class 6k tokens, 32k tokens, eight ragged sequences on a
shuffled paged cache, 70B-class 64k tokens); values are drawn as there: N(0,1) embeddings, queries, keys and values, power-law
attention mass with inflated frame borders, N(0,3) logits with the draft model close to the target.  `draw` spreads the sizes
over the ranges between and around them.
"""
import math

import numpy as np
import torch

from paper_2601_08273_b200 import binding as hb
from paper_2601_08273_b200 import workloads as W
from paper_2601_08273_b200.step import HippoStep

PAGE = hb.PAGE_SIZE
BIG_BYTES = 21.6e9      # K and V of the largest listed pass (65,801 keys, 80 layers)


# ------------------------------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------------------------------

def listed():
    return [
        # the whole step on the tiny fp32 configuration (256 visual tokens): nothing but launches and latency
        _step("step_tiny_fp32", 0),
        # the whole step at 32k tokens: selection, gather, 7 x 28 draft calls beside 36 verification layers, acceptance
        _step("step_32k", 2),
        # selection once per prompt: 6k tokens (the paper's 32 frames of 14 x 14), ...
        dict(name="select_6k", kind="select", batch=1, tokens=32 * 196, spread=0, grid_h=14, grid_w=14, dim=3584, keep_pct=10, dtype="bf16"),
        # ... eight ragged sequences with partial last frames in one call, ...
        dict(name="select_ragged_8", kind="select", batch=8, tokens=8 * 10272, spread=4544, grid_h=14, grid_w=14, dim=3584, keep_pct=10, dtype="bf16"),
        # ... and the longest video
        dict(name="select_64k", kind="select", batch=1, tokens=65536, spread=0, grid_h=16, grid_w=16, dim=8192, keep_pct=10, dtype="bf16"),
        # one target layer's share of the attention mass that the selection fuses in (once per layer and prompt)
        dict(name="mass_32k", kind="mass", batch=1, tokens=32768, spread=0, l_txt=256, q_heads=32, kv_heads=8, head_dim=128, dtype="bf16"),
        # pruning the draft cache of eight ragged sequences, page ids shuffled, 28 layers, 10 % of the visual tokens and all text
        dict(name="gather_ragged_8", kind="gather", batch=8, tokens=8 * 10272, spread=4544, n_text=128, layers=28, kv_heads=2, head_dim=64,
             keep_pct=10, paged=True, dtype="bf16"),
        # one draft token: 28 layers over the pruned cache of a 6k-token video (755 keys), ...
        dict(name="draft_token_6k", kind="draft", batch=1, q_len=1, kv=627 + 128 + 3, spread=0, layers=28, q_heads=14, kv_heads=2, head_dim=64,
             paged=False, dtype="bf16"),
        # ... and of a 32k-token one
        dict(name="draft_token_32k", kind="draft", batch=1, q_len=1, kv=3277 + 256 + 4, spread=0, layers=28, q_heads=16, kv_heads=2, head_dim=64,
             paged=False, dtype="bf16"),
        # verification with one call per layer (an engine whose other operators sit between the layers): eight ragged sequences
        dict(name="verify_calls_ragged_8", kind="verify_calls", batch=8, q_len=6, kv=10406, spread=4544, layers=28, q_heads=28, kv_heads=4,
             head_dim=128, paged=True, dtype="bf16"),
        # verification of all layers in one call: the longest video, 80 layers
        dict(name="verify_layers_64k", kind="verify_layers", batch=1, q_len=6, kv=65536 + 256 + 6, spread=0, layers=80, q_heads=64, kv_heads=8,
             head_dim=128, paged=False, dtype="bf16"),
        # acceptance at batch 1, seven draft tokens, sampling mode
        dict(name="accept_g7", kind="accept", batch=1, gamma=7, vocab=152064, noise=1.0, greedy=False),
    ]


def _step(name, index):
    c = W.CONFIGS[index]
    return dict(name=name, kind="step", config=index, frames=c.frames, n_text=c.n_text, gamma=c.gamma, target_layers=c.tgt_layers,
                draft_layers=c.dft_layers, keep_pct=c.keep_pct)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["select", "select", "mass", "gather", "draft", "draft", "verify_calls", "verify_layers", "accept", "step"])
    grid = rng.choice([(14, 14), (16, 16), (8, 8), (14, 14), (16, 16), (12, 20)])
    if kind == "select":
        batch = rng.choice([1, 1, 1, 2, 8])
        dim = 8 * _log_int(rng, 1024 / 8, 1024)
        tokens = _log_int(rng, 256 * batch, 65536)
        fp32 = tokens * dim <= 3e7 and rng.random() < 0.3       # fp32 storage is for small checks
        return dict(kind=kind, batch=batch, tokens=tokens, spread=int(rng.uniform(0, 0.5) * tokens / batch), grid_h=grid[0], grid_w=grid[1],
                    dim=dim, keep_pct=rng.choice([5, 10, 25, 50]), dtype="fp32" if fp32 else "bf16")
    if kind == "mass":
        heads, group = rng.choice([(4, 7), (8, 4), (8, 8), (2, 7)])
        batch = rng.choice([1, 1, 4])
        tokens = _log_int(rng, 512 * batch, 65536)
        return dict(kind=kind, batch=batch, tokens=tokens, spread=int(rng.uniform(0, 0.3) * tokens / batch), l_txt=rng.randint(16, 256),
                    q_heads=heads * group, kv_heads=heads, head_dim=128, dtype="bf16")
    if kind == "gather":
        batch = rng.choice([1, 1, 8])
        tokens = _log_int(rng, 2048 * batch, 65536 if batch == 1 else 100000)
        return dict(kind=kind, batch=batch, tokens=tokens, spread=int(rng.uniform(0, 0.4) * tokens / batch), n_text=rng.randint(16, 256), layers=28,
                    kv_heads=rng.choice([2, 4]), head_dim=64, keep_pct=rng.choice([5, 10, 25, 50]), paged=rng.random() < 0.5, dtype="bf16")
    if kind == "draft":
        batch = rng.choice([1, 1, 1, 8])
        heads, group = rng.choice([(2, 7), (2, 8), (4, 7)])
        kv = _log_int(rng, 100, 33000 if batch == 1 else 4000)
        return dict(kind=kind, batch=batch, q_len=rng.choice([1, 1, 1, 2]), kv=kv, spread=int(rng.uniform(0, 0.5) * kv) if batch > 1 else 0,
                    layers=28, q_heads=heads * group, kv_heads=heads, head_dim=64, paged=batch > 1 or rng.random() < 0.3, dtype="bf16")
    if kind in ("verify_calls", "verify_layers"):
        heads, group = rng.choice([(4, 7), (8, 4), (8, 8)])
        batch = rng.choice([1, 1, 1, 4, 8])
        gamma = rng.choice([1, 3, 5, 7, 8])
        kv = _log_int(rng, 1000, 66000 if batch == 1 else 13000)
        layers = rng.choice([28, 36, 80])
        per_layer = kv * batch * 2 * heads * 128 * 2
        layers = max(1, min(layers, int(BIG_BYTES / (2 if kind == "verify_calls" else 1) / per_layer)))
        return dict(kind=kind, batch=batch, q_len=gamma + 1, kv=kv, spread=int(rng.uniform(0, 0.4) * kv) if batch > 1 else 0, layers=layers,
                    q_heads=heads * group, kv_heads=heads, head_dim=128, paged=batch > 1 or rng.random() < 0.3, dtype="bf16")
    if kind == "accept":
        return dict(kind=kind, batch=rng.choice([1, 1, 1, 2, 4, 8]), gamma=rng.choice([1, 3, 5, 7, 8]),
                    vocab=rng.choice([152064, 151936, 128256, _log_int(rng, 1000, 152064)]), noise=rng.choice([0.1, 0.5, 1.0, 3.0]),
                    greedy=rng.random() < 0.3)
    index = rng.choice([0, 1, 1, 2])
    c = W.CONFIGS[index]
    return dict(kind="step", config=index, frames=_log_int(rng, 2 if index == 0 else 8, c.frames), n_text=rng.randint(16, c.n_text),
                gamma=rng.choice([3, 4, 5, 7]), target_layers=c.tgt_layers, draft_layers=c.dft_layers, keep_pct=rng.choice([5, 10, 25]))


# ------------------------------------------------------------------------------------------------------------------------
# shared pieces
# ------------------------------------------------------------------------------------------------------------------------

def _lengths(total, batch, spread):
    """`batch` lengths around total / batch, within +- spread / 2: the same ones for every seed, so that outputs keep their shapes."""
    mean = total // batch
    if batch == 1 or spread < 2:
        return [mean] * batch
    r = np.random.default_rng([total, batch, spread])
    half = min(spread // 2, mean - 1)
    return [int(mean + x) for x in r.integers(-half, half + 1, size=batch)]


def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 16 + salt)
    return g


def _torch_dtype(case):
    return torch.float32 if case["dtype"] == "fp32" else torch.bfloat16


def _normal(shape, dtype, gen):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=gen)


def _mass(lengths, grid_h, grid_w, gen):
    """Attention mass: power law over a random order of the tokens, four times as much on the frame borders, sums to 1."""
    out = []
    for n in lengths:
        rank = torch.randperm(n, generator=gen, device="cuda").double() + 1
        cell = torch.arange(n, device="cuda") % (grid_h * grid_w)
        y, x = cell // grid_w, cell % grid_w
        border = (y == 0) | (y == grid_h - 1) | (x == 0) | (x == grid_w - 1)
        w = rank ** -1.1 * torch.where(border, 4.0, 1.0)
        out.append((w / w.sum()).float())
    return torch.cat(out)


def _table(caps, paged, seed):
    """(page table tensor or None, pages per row, pages in the pool) for the capacities; shuffled page ids when paged."""
    t, pool = W.make_page_table(caps, np.random.default_rng([seed, 77]) if paged else None)
    if not paged and len(caps) == 1:
        return None, t.shape[1], pool
    return torch.from_numpy(t).cuda(), t.shape[1], pool


class _Captured:
    """`fn` as a CUDA graph, captured after one eager pass (the library's one-time set-up happens there).  Holds `fn`, and through it
    every buffer that the graph works on, for as long as it can be replayed."""

    def __init__(self, fn):
        self.fn = fn
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            fn()
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph):
            fn()

    def replay(self):
        self.graph.replay()


# ------------------------------------------------------------------------------------------------------------------------
# one kind of work each: prepare_*(case, seed) -> state with a "run" function in it
# ------------------------------------------------------------------------------------------------------------------------

def _prepare_select(case, seed):
    lengths = _lengths(case["tokens"], case["batch"], case["spread"])
    gen = _gen(seed, 1)
    gh, gw = case["grid_h"], case["grid_w"]
    embeds = _normal((sum(lengths), case["dim"]), _torch_dtype(case), gen)
    mass = _mass(lengths, gh, gw, gen)
    k = [W.keep_count(n, case["keep_pct"]) for n in lengths]
    kept = torch.empty(max(sum(k), 1), dtype=torch.int32, device="cuda")
    fused = torch.empty(sum(lengths), dtype=torch.float32, device="cuda")
    ws = hb.new_workspace(hb.hippo_select_workspace_bytes(lengths, gh, gw))

    def run():
        return hb.hippo_select_tokens(embeds, mass, lengths, k, gh, gw, kept_idx=kept, fused_score=fused, workspace=ws)

    return run


def _prepare_mass(case, seed):
    lengths = _lengths(case["tokens"], case["batch"], case["spread"])
    gen = _gen(seed, 2)
    dt, D, Hkv, Hq = _torch_dtype(case), case["head_dim"], case["kv_heads"], case["q_heads"]
    table, mpps, pool = _table([n + case["l_txt"] for n in lengths], case["batch"] > 1, seed)
    u = torch.nn.functional.normalize(_normal((D,), torch.float32, gen), dim=0)
    # text-to-visual attention that follows a power law over the keys: queries and keys share a direction (workloads.mass_inputs)
    q = (_normal((case["batch"], case["l_txt"], Hq, D), torch.float32, gen) + 4.0 * u).to(dt)
    rank = torch.randperm(pool * PAGE, generator=gen, device="cuda").reshape(pool, 1, PAGE, 1).float() + 1
    keys = _normal((pool, Hkv, PAGE, D), torch.float32, gen)
    keys += (-1.1 * torch.log(rank)) * math.sqrt(D) / 4.0 * u
    keys = keys.to(dt)
    values = torch.empty_like(keys)         # a cache has both; only the keys are read
    kv = hb.KVCache(keys, values, table, mpps)
    mass = torch.zeros(sum(lengths), dtype=torch.float32, device="cuda")
    ws = hb.new_workspace(hb.hippo_attention_mass_workspace_bytes(lengths, case["l_txt"], Hq, Hkv, D, hb.HIPPO_DTYPE_BF16))
    weight = 1.0 / (Hq * case["l_txt"])

    def run():
        mass.zero_()
        return hb.hippo_attention_mass(q, kv, lengths, weight, mass, workspace=ws)

    return run


def _prepare_gather(case, seed):
    lengths = _lengths(case["tokens"], case["batch"], case["spread"])
    gen = _gen(seed, 3)
    dt, L, h, d = _torch_dtype(case), case["layers"], case["kv_heads"], case["head_dim"]
    ctx = [n + case["n_text"] for n in lengths]
    k = [W.keep_count(n, case["keep_pct"]) for n in lengths]
    n_keep = [x + case["n_text"] for x in k]
    offs = np.concatenate([[0], np.cumsum(n_keep)]).astype(np.int32)
    keep = torch.empty(int(offs[-1]), dtype=torch.int32, device="cuda")
    for b, n in enumerate(lengths):         # kept visual tokens ascending, then every text position
        vis = torch.randperm(n, generator=gen, device="cuda")[:k[b]].sort().values
        keep[offs[b]:offs[b + 1]] = torch.cat([vis, torch.arange(n, ctx[b], device="cuda")]).int()
    offsets = torch.from_numpy(offs).cuda()
    st, s_mpps, s_pool = _table(ctx, case["paged"], seed)
    dt_, d_mpps, d_pool = _table([n + 8 for n in n_keep], case["paged"], seed)
    src_k, src_v = (_normal((L, s_pool, h, PAGE, d), dt, gen) for _ in range(2))
    dst_k, dst_v = (torch.zeros((L, d_pool, h, PAGE, d), dtype=dt, device="cuda") for _ in range(2))
    src, dst = hb.KVCache(src_k[0], src_v[0], st, s_mpps), hb.KVCache(dst_k[0], dst_v[0], dt_, d_mpps)
    s_stride, d_stride = (x[0].numel() * x.element_size() for x in (src_k, dst_k))
    total = int(offs[-1])

    def run():
        hb.hippo_gather_kv(L, src, s_stride, dst, d_stride, case["batch"], keep, offsets, total)
        return dst_k, dst_v

    return run


def _attention_state(case, seed):
    """Per-layer caches, queries and outputs of an attention leg; kv is the mean length of a sequence."""
    lengths = _lengths(case["kv"] * case["batch"], case["batch"], case["spread"])
    lengths = [max(n, case["q_len"]) for n in lengths]
    gen = _gen(seed, 4)
    dt, L, H, D = _torch_dtype(case), case["layers"], case["kv_heads"], case["head_dim"]
    table, mpps, pool = _table(lengths, case["paged"] or case["batch"] > 1, seed)
    k, v = (_normal((L, pool, H, PAGE, D), dt, gen) for _ in range(2))
    q = _normal((L, case["batch"], case["q_len"], case["q_heads"], D), dt, gen)
    out = torch.empty_like(q)
    caches = [hb.KVCache(k[l], v[l], table, mpps) for l in range(L)]
    return lengths, torch.tensor(lengths, dtype=torch.int32, device="cuda"), caches, q, out


def _prepare_draft(case, seed):
    lengths, kv_len, caches, q, out = _attention_state(case, seed)
    ws = hb.new_workspace(hb.hippo_attention_workspace_bytes(case["batch"], case["q_len"], case["q_heads"], case["kv_heads"], case["head_dim"]))
    most = max(lengths)

    def token():
        for l, kv in enumerate(caches):
            hb.hippo_draft_attention(q[l], kv, kv_len, most, out=out[l], workspace=ws)

    g = _Captured(token)

    def run():
        g.replay()
        return out

    return run


def _prepare_verify_calls(case, seed):
    lengths, kv_len, caches, q, out = _attention_state(case, seed)
    ws = hb.new_workspace(hb.hippo_attention_workspace_bytes(case["batch"], case["q_len"], case["q_heads"], case["kv_heads"], case["head_dim"]))
    most = max(lengths)

    def leg():
        for l, kv in enumerate(caches):
            hb.hippo_verify_attention(q[l], kv, kv_len, most, out=out[l], workspace=ws, kv_len_host=lengths)

    g = _Captured(leg)

    def run():
        g.replay()
        return out

    return run


def _prepare_verify_layers(case, seed):
    lengths, kv_len, caches, q, out = _attention_state(case, seed)
    ws = hb.new_workspace(hb.hippo_verify_attention_layers_workspace_bytes(case["layers"], case["batch"], case["q_len"], case["q_heads"],
                                                                           case["kv_heads"], case["head_dim"]))
    most = max(lengths)
    qs, outs = list(q), list(out)

    def leg():
        hb.hippo_verify_attention_layers(qs, caches, kv_len, most, outs, workspace=ws, kv_len_host=lengths)

    g = _Captured(leg)

    def run():
        g.replay()
        return out

    return run


def _prepare_accept(case, seed):
    B, g, V = case["batch"], case["gamma"], case["vocab"]
    gen = _gen(seed, 5)
    target = 3.0 * _normal((B, g + 1, V), torch.float32, gen)
    draft = target[:, :g] + case["noise"] * _normal((B, g, V), torch.float32, gen)
    tokens = torch.multinomial(torch.softmax(draft.reshape(B * g, V), dim=-1), 1, generator=gen).int().reshape(B, g)
    u = torch.rand((B, g), generator=gen, device="cuda")
    ur = torch.rand((B,), generator=gen, device="cuda")
    n_acc = torch.empty(B, dtype=torch.int32, device="cuda")
    out = torch.empty((B, g + 1), dtype=torch.int32, device="cuda")
    ws = hb.new_workspace(hb.hippo_accept_workspace_bytes(B, g, V))
    mode = hb.HIPPO_ACCEPT_GREEDY if case["greedy"] else hb.HIPPO_ACCEPT_SAMPLE

    def run():
        return hb.hippo_accept(target, draft, tokens, u, ur, n_accepted=n_acc, out_tokens=out, workspace=ws, mode=mode)

    return run


def _step_config(case, seed):
    return W.CONFIGS[case["config"]].replace(seed=seed, frames=case["frames"], n_text=case["n_text"], gamma=case["gamma"], keep_pct=case["keep_pct"])


def _prepare_step(case, seed):
    st = HippoStep(_step_config(case, seed), target_layers=case["target_layers"], draft_layers=case["draft_layers"])
    g = _Captured(st.run)

    def run():
        g.replay()
        return {"kept": st.keep_idx, "fused": st.fused, "draft_k": st.dst_k, "draft_v": st.dst_v, "draft_out": st.out_d,
                "verify_out": st.out_t, "n_accepted": st.n_accepted, "tokens": st.out_tokens}

    return run


_PREPARE = {"select": _prepare_select, "mass": _prepare_mass, "gather": _prepare_gather, "draft": _prepare_draft,
            "verify_calls": _prepare_verify_calls, "verify_layers": _prepare_verify_layers, "accept": _prepare_accept, "step": _prepare_step}


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def run(state):
    return state()


# ------------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------------------------------

def _select_work(tokens, grid_h, grid_w, dim, esize):
    """Each embedding read once; per full frame the crops' distinct dot products, a norm and a temporal dot product per token."""
    pairs = 0
    for y in range(0, grid_h, 5):
        for x in range(0, grid_w, 5):
            m = min(5, grid_h - y) * min(5, grid_w - x)
            pairs += m * (m - 1) // 2
    dots = tokens / (grid_h * grid_w) * pairs + 2 * tokens
    return tokens * (dim * esize + 8), 2.0 * dots * dim


def _attention_work(case):
    esize = 4 if case["dtype"] == "fp32" else 2
    keys, rows = case["kv"] * case["batch"] * case["layers"], case["q_len"] * case["q_heads"]
    io = 2 * case["layers"] * case["batch"] * rows * case["head_dim"] * esize
    return keys * 2 * case["kv_heads"] * case["head_dim"] * esize + io, 4.0 * keys * rows * case["head_dim"]


def work(case):
    kind = case["kind"]
    if kind == "select":
        b, f = _select_work(case["tokens"], case["grid_h"], case["grid_w"], case["dim"], 4 if case["dtype"] == "fp32" else 2)
    elif kind == "mass":
        b = case["tokens"] * (case["kv_heads"] * case["head_dim"] * 2 + 4) + case["batch"] * case["l_txt"] * case["q_heads"] * case["head_dim"] * 2
        f = 2.0 * case["tokens"] * case["l_txt"] * case["q_heads"] * case["head_dim"]       # the logits, formed once
    elif kind == "gather":
        kept = case["tokens"] * case["keep_pct"] / 100 + case["batch"] * case["n_text"]
        b, f = 2 * kept * case["layers"] * 2 * case["kv_heads"] * case["head_dim"] * 2, 0.0
    elif kind in ("draft", "verify_calls", "verify_layers"):
        b, f = _attention_work(case)
    elif kind == "accept":
        rows = case["gamma"] + 1 if case["greedy"] else 2 * case["gamma"] + 1
        b, f = case["batch"] * rows * case["vocab"] * 4, 0.0
    else:
        c = _step_config(case, 0)
        n_v = c.frames * c.grid_h * c.grid_w
        e = 4 if c.dtype == "fp32" else 2
        keep, ctx = W.keep_count(n_v, c.keep_pct) + c.n_text, n_v + c.n_text
        b, f = _select_work(n_v, c.grid_h, c.grid_w, c.embed_dim, e)
        b += 2 * keep * case["draft_layers"] * 2 * c.dft_kv_heads * c.dft_head_dim * e                               # gather
        b += c.gamma * keep * case["draft_layers"] * 2 * c.dft_kv_heads * c.dft_head_dim * e                         # draft tokens
        b += (ctx + c.gamma + 1) * case["target_layers"] * 2 * c.tgt_kv_heads * c.tgt_head_dim * e                   # verification
        b += (2 * c.gamma + 1) * c.vocab * 4                                                                         # acceptance
        f += 4.0 * c.gamma * keep * case["draft_layers"] * c.dft_q_heads * c.dft_head_dim
        f += 4.0 * (c.gamma + 1) * ctx * case["target_layers"] * c.tgt_q_heads * c.tgt_head_dim
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    kind = case["kind"]
    if kind in ("gather", "accept"):
        return "exact"                                   # bytes copied; token ids and counts
    if kind == "select":
        # fp64 scores rounded once to fp32; a kept list shifts where two scores tie to the last bit
        return {"rel": 3e-7, "max": 2e-6, "differ": 0.01}
    if kind == "mass":
        return {"rel": 3e-6, "max": 1e-5}                # fp32 sums of up to 65,536 exponentials of fp32 logits (3e-7 off fp64 at 32k)
    if case.get("config") == 0:
        return {"rel": 2e-6, "max": 2e-5, "differ": 0.01}    # fp32 storage and arithmetic
    # bf16 outputs, probabilities rounded to bf16 for the second contraction: two work splits differ by rel 2.9e-3, max 1.5e-2
    return {"rel": 1e-2, "max": 0.06, "differ": 0.01}
