"""The work that a user of this framework has it do, as cases that can be timed and compared.

Every case goes through the package's public entry points with the shapes of the package's own
workloads (synth.WORKLOADS) or generic sizes between them: selection from a given candidate memory and
from visual tokens (with the cross-modal encoder), with one token per round, with groups of tokens,
with a pointer decoder of two layers and with the training aggregates; the gather and the projector;
the prefill of short, ordinary and long batches; generation steps; and the whole pipeline.

Weights and inputs are drawn on the GPU from the seed with the distributions that synth states next to
its shapes (N(0, 1) visual tokens, N(0, 0.02) text embeddings and weights).  Few decoder layers stand for
the 28 or 32 of a whole model: every layer does the same work on other weights, and a rounding travels
through fewer of them."""
import dataclasses
import math

import torch
import torch.nn.functional as F

from paper_2609_13804_gb300 import binding as sp
from paper_2609_13804_gb300 import synth

DEV = "cuda"
TAU, BETA = 0.25, 0.99  # pointer temperature and discount of the training aggregates

# Selector and language-model shapes of the package's workloads, by the workload they come from.
_W = {n: f() for n, f in synth.WORKLOADS.items()}
SHAPES = {"small": _W["llava15-576-1layer"], "llava": _W["llava15-7b-b16"], "qwen": _W["qwen25vl-varres-b8"]}


# ----------------------------------------------------------------------------- cases

def listed():
    return [
        # One image asked about on its own: visual tokens and prompt in, kept indices out, through the
        # encoder.  The smallest call: launches and the rounds' latency count.
        _select("one image encoded", "small", images=1, n_vis=576, n_txt=32, k_max=64, encode=True),
        # The batch of the headline workload, from a memory that an encoder of the user's own made, with
        # a STOP that ends some of the images early.
        _select("batch of images", "llava", images=16, n_vis=576, k_max=192, stop=True),
        # Multi-tile images of 3,328 tokens, one episode each, five tokens a round: the keys of an
        # episode are larger than the shared memory of its cluster.
        _select("tiled images", "qwen", images=4, n_vis=3328, g=5, k_max=160),
        # A pointer decoder of two layers, images of uneven sizes.
        _select("two-layer pointer decoder", "llava", images=4, n_vis=576, k_max=64, dec_layers=2, ragged=True),
        # High-resolution images in groups of 576 candidates, encoded: the largest encoder call.
        _select("any-resolution encoded", "llava", images=8, n_vis=2880, n_txt=64, group=576, g=5, k_max=32,
                encode=True),
        # The training-time forward: rollout with aggregates, soft top-k, noise gate.
        {"name": "training forward", "kind": "train", "dims": "llava", "images": 8, "n_vis": 576, "k_max": 96,
         "ragged": True},
        # The kept rows of a batch gathered and projected into the packed language-model input.
        {"name": "gather and project", "kind": "project", "dims": "llava", "images": 16, "n_vis": 576, "n_txt": 48,
         "kept": 64},
        # The prefill of a pruned batch (about 1,800 packed tokens), writing the cache generation reads.
        {"name": "prefill pruned batch", "kind": "prefill", "dims": "llava", "seqs": 16, "tokens": 160,
         "ragged": True, "layers": 2, "kv": True},
        # Unpruned multi-tile prefixes with grouped-query heads and 3-D rotary positions.
        {"name": "prefill long", "kind": "prefill", "dims": "qwen", "seqs": 4, "tokens": 3424, "ragged": False,
         "layers": 1, "kv": False},
        # One pruned image and its prompt: fewer rows than a tile, bound by the weights.
        {"name": "prefill one short", "kind": "prefill", "dims": "llava", "seqs": 1, "tokens": 97, "ragged": False,
         "layers": 2, "kv": True},
        # Generation after that batch's prefill: steps chained on the device.
        {"name": "decode batch", "kind": "decode", "dims": "llava", "seqs": 16, "context": 160, "ragged": True,
         "layers": 4, "steps": 4},
        # Visual tokens in, hidden states out: encoder, selection, gather, projector, prefill.
        {"name": "pipeline", "kind": "pipeline", "dims": "llava", "images": 4, "n_vis": 576, "n_txt": 48, "g": 1,
         "k_max": 96, "stop": True, "layers": 2},
    ]


def _select(name, dims, *, images, n_vis, k_max, n_txt=0, group=0, g=1, encode=False, dec_layers=1, ragged=False,
            stop=False):
    c = {"kind": "select", "dims": dims, "images": images, "n_vis": n_vis, "n_txt": n_txt, "group": group, "g": g,
         "k_max": k_max, "encode": encode, "dec_layers": dec_layers, "ragged": ragged, "stop": stop}
    return dict(c, name=name) if name else c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["select", "select", "encode", "tiles", "deep", "train", "project", "prefill", "long", "decode",
                       "decode", "pipeline"])
    odd = rng.random() < 0.5
    if kind == "select":
        return _select("", rng.choice(["small", "llava"]), images=_log(rng, 1, 16), n_vis=rng.randint(100, 1010),
                       g=rng.choice([1, 1, 2, 5]), k_max=_log(rng, 16, 96), ragged=odd, stop=rng.random() < 0.5)
    if kind == "encode":
        if rng.random() < 0.5:
            return _select("", "small", images=_log(rng, 1, 4), n_vis=rng.randint(100, 700), n_txt=rng.randint(1, 64),
                           k_max=_log(rng, 8, 64), encode=True, ragged=odd)
        return _select("", "llava", images=_log(rng, 1, 8), n_vis=rng.randint(700, 2880), n_txt=rng.randint(8, 64),
                       group=576, g=5, k_max=_log(rng, 8, 32), encode=True, ragged=odd)
    if kind == "tiles":
        return _select("", "qwen", images=_log(rng, 1, 4), n_vis=rng.randint(2100, 3328), g=5, k_max=_log(rng, 40, 160),
                       ragged=odd)
    if kind == "deep":
        return _select("", rng.choice(["small", "llava"]), images=_log(rng, 1, 4), n_vis=rng.randint(64, 576),
                       k_max=_log(rng, 8, 56), dec_layers=2, ragged=odd)
    if kind == "train":
        return {"kind": "train", "dims": rng.choice(["small", "llava"]), "images": _log(rng, 1, 16),
                "n_vis": rng.randint(100, 1010), "k_max": _log(rng, 16, 96), "ragged": odd}
    if kind == "project":
        return {"kind": "project", "dims": "llava", "images": _log(rng, 1, 32), "n_vis": rng.randint(200, 2880),
                "n_txt": rng.randint(0, 96), "kept": _log(rng, 8, 192)}
    if kind == "prefill":
        return {"kind": "prefill", "dims": rng.choice(["small", "llava", "qwen"]), "seqs": _log(rng, 1, 16),
                "tokens": _log(rng, 17, 640), "ragged": odd, "layers": rng.choice([1, 2]), "kv": rng.random() < 0.5}
    if kind == "long":
        return {"kind": "prefill", "dims": rng.choice(["llava", "qwen"]), "seqs": _log(rng, 1, 4),
                "tokens": rng.randint(1000, 3400), "ragged": odd, "layers": 1, "kv": rng.random() < 0.5}
    if kind == "decode":
        seqs = _log(rng, 1, 48)
        return {"kind": "decode", "dims": rng.choice(["llava", "qwen"]), "seqs": seqs,
                "context": _log(rng, 16, min(4096, 16384 // seqs)), "ragged": odd, "layers": rng.choice([2, 3]),
                "steps": rng.randint(2, 4)}
    return {"kind": "pipeline", "dims": rng.choice(["small", "llava"]), "images": _log(rng, 1, 8),
            "n_vis": rng.randint(100, 700), "n_txt": rng.randint(4, 64), "g": rng.choice([1, 5]),
            "k_max": _log(rng, 16, 96), "stop": odd, "layers": rng.choice([1, 2])}


# ----------------------------------------------------------------------------- sizes (from the case alone)

def _spread(n, count, ragged):
    """Sizes of the images or sequences: all n, or spread over 0.35 n .. n."""
    if not ragged:
        return [n] * count
    return [max(1, int(n * (0.35 + 0.65 * ((0.618034 * (i + 1)) % 1.0)))) for i in range(count)]


def _vis(case):
    return _spread(case["n_vis"], case["images"], case.get("ragged", False))


def _txt(case):
    return [case.get("n_txt", 0)] * case["images"]


def _episodes(n_vis, group):
    """(first row, candidates) of every episode."""
    out, r = [], 0
    for n in n_vis:
        gs = group or n
        out += [(r + s, min(gs, n - s)) for s in range(0, n, gs)]
        r += n
    return out


def _kept(case):
    """Kept tokens of every image of a projector case: 1/4 .. 7/4 of the mean."""
    n, k = case["n_vis"], case["kept"]
    return [min(n, max(1, int(k * (0.25 + 1.5 * ((0.618034 * (i + 1)) % 1.0))))) for i in range(case["images"])]


def _shapes(case):
    w = SHAPES[case["dims"]]
    encode = case.get("encode", False) or case["kind"] == "pipeline"
    s = dataclasses.replace(w.selector, n_enc_layers=w.selector.n_enc_layers if encode else 0,
                            n_dec_layers=case.get("dec_layers", 1))
    mrope = (16, 24, 24) if case["dims"] == "qwen" and case["kind"] == "prefill" else (0, 0, 0)
    return s, dataclasses.replace(w.model, n_layers=case.get("layers", 1), mrope_section=mrope)


# ----------------------------------------------------------------------------- inputs (from the seed alone)

class _Draw:
    def __init__(self, seed):
        self.gen = torch.Generator(device=DEV).manual_seed(seed)

    def f32(self, *shape, std=0.02):
        return torch.randn(shape, device=DEV, generator=self.gen) * std

    def bf16(self, *shape, std=0.02):
        return self.f32(*shape, std=std).to(torch.bfloat16)


def _norm(n, r):
    return 1 + r.f32(n, std=0.1), r.f32(n, std=0.1)


def _selector_weights(s, r):
    D, h, ffn = s.D, s.h, s.enc_ffn
    w = {"W_p": r.bf16(D, s.D_text), "s_stop": r.f32(D), "s_start": r.f32(D), "W_in": r.f32(h, D),
         "Wk_p": r.f32(h, D), "enc": [], "lower": []}
    for n in ("Wq_s", "Wk_s", "Wv_s", "Wo_s", "Wq_p"):
        w[n] = r.f32(h, h)
    for n, size in (("ln_text", D), ("ln1", h), ("ln2", h)):
        w[n + "_g"], w[n + "_b"] = _norm(size, r)
    for _ in range(s.n_enc_layers):
        L = {"Wqkv": r.bf16(3 * D, D), "Wo": r.bf16(D, D), "W1": r.bf16(ffn, D), "W2": r.bf16(D, ffn)}
        for n in ("ln1", "ln2"):
            L[n + "_g"], L[n + "_b"] = _norm(D, r)
        w["enc"].append(L)
    for _ in range(s.n_dec_layers - 1):
        L = {n: r.f32(h, h) for n in ("Wq_s", "Wk_s", "Wv_s", "Wo_s", "Wq_c", "Wo_c")}
        L.update({n: r.f32(h, D) for n in ("Wk_c", "Wv_c")}, W1=r.bf16(4 * h, h), W2=r.bf16(h, 4 * h))
        for n in ("ln1", "ln2", "ln3"):
            L[n + "_g"], L[n + "_b"] = _norm(h, r)
        w["lower"].append(L)
    return w


def _model_weights(m, r):
    qkv, dq = (m.n_heads + 2 * m.n_kv_heads) * m.head_dim, m.n_heads * m.head_dim
    layers = [{"Wqkv": r.bf16(qkv, m.d), "Wo": r.bf16(m.d, dq), "Wgu": r.bf16(2 * m.ffn, m.d),
               "Wdown": r.bf16(m.d, m.ffn), "attn_norm": 1 + r.f32(m.d, std=0.1), "mlp_norm": 1 + r.f32(m.d, std=0.1)}
              for _ in range(m.n_layers)]
    head = {"final_norm": 1 + r.f32(m.d, std=0.1), "proj_W1": None, "proj_W2": None}
    if m.proj_kind == "linear":
        head["proj_W1"] = r.bf16(m.d, m.proj_in)
    elif m.proj_kind == "mlp2":
        head["proj_W1"], head["proj_W2"] = r.bf16(m.proj_hidden, m.proj_in), r.bf16(m.d, m.proj_hidden)
    return layers, head


def _stop_bias(case, s, r):
    """STOP switched off (a fixed budget of k_max tokens), zero (training), or at a level that the best
    remaining logit falls below after some rounds: the logits of these weights have a standard deviation
    of about 0.0004 sqrt(D h)."""
    E = len(_episodes(_vis(case), case.get("group", 0)))
    if case["kind"] == "train":
        return torch.zeros(E, device=DEV)
    if not case["stop"]:
        return torch.full((E,), -1e30, device=DEV)
    level = 2.2 + 0.5 * torch.rand(E, device=DEV, generator=r.gen)
    return level * (4e-4 * math.sqrt(s.D * s.h))


def _inputs(case, seed):
    """Everything a case's pass reads, as tensors (the caches and packed inputs of the later stages in
    place of the stages before them)."""
    r, kind = _Draw(seed), case["kind"]
    s, m = _shapes(case)
    i = {}
    if kind in ("select", "train", "pipeline"):
        i["sel"] = _selector_weights(s, r)
        n_vis, n_txt = sum(_vis(case)), sum(_txt(case))
        if case.get("encode") or kind == "pipeline":
            i["X"], i["E_text"] = r.bf16(n_vis, s.D, std=1.0), r.bf16(n_txt, s.D_text)
        else:
            i["H"] = r.f32(n_vis, s.D, std=1.0)
        i["stop_bias"] = _stop_bias(case, s, r)
        if kind == "train":
            i["X"], i["noise"] = r.bf16(n_vis, s.D, std=1.0), r.bf16(n_vis, s.D, std=1.0)
    if kind in ("project", "prefill", "decode", "pipeline"):
        i["layers"], i["head"] = _model_weights(m, r)
    if kind == "project":
        n, B = case["n_vis"], case["images"]
        i["X"], i["text"] = r.bf16(n * B, m.proj_in, std=1.0), r.bf16(sum(_txt(case)), m.d)
        kept = _kept(case)
        i["idx"] = torch.full((B, max(kept)), -1, dtype=torch.int32, device=DEV)
        for b, k in enumerate(kept):
            i["idx"][b, :k] = torch.randperm(n, device=DEV, generator=r.gen)[:k].sort().values
        i["count"] = torch.tensor(kept, dtype=torch.int32, device=DEV)
    if kind == "prefill":
        lens = _spread(case["tokens"], case["seqs"], case["ragged"])
        i["x"] = r.bf16(sum(lens), m.d, std=0.5)
        i["cu"] = torch.tensor([sum(lens[:b]) for b in range(len(lens) + 1)], dtype=torch.int32, device=DEV)
        i["pos"] = torch.cat([torch.arange(n, dtype=torch.int32, device=DEV) for n in lens])
        if sum(m.mrope_section):
            i["pos3"] = torch.cat([_grid_positions(n) for n in lens])
    if kind == "decode":
        B, steps, W = case["seqs"], case["steps"], m.n_kv_heads * m.head_dim
        lens = _spread(case["context"], B, case["ragged"])
        i["lens"] = torch.tensor(lens, dtype=torch.int32, device=DEV)
        # keys and values have the spread that a projection of unit-RMS rows by N(0, 0.02) gives them
        i["kv"] = r.bf16(m.n_layers, 2, B, case["context"] + steps, W, std=0.02 * math.sqrt(m.d))
        i["x"] = r.bf16(steps, B, m.d, std=0.5)
    return i


def _grid_positions(n):
    """(t, h, w, unused) of a sequence: a grid of 32 columns, the last 1/32 of it text after it."""
    vis, q = n - n // 32, torch.arange(n, dtype=torch.int32, device=DEV)
    start = max(32, -(-vis // 32))
    p = torch.stack([torch.zeros_like(q), q // 32, q % 32, torch.zeros_like(q)], 1)
    t = (start + q - vis)[:, None] * torch.tensor([1, 1, 1, 0], dtype=torch.int32, device=DEV)
    return torch.where((q < vis)[:, None], p, t).contiguous()


def prepare(case, seed):
    s, m = _shapes(case)
    i = _inputs(case, seed)
    st = {"case": case, "in": i}
    if "sel" in i:
        st["selector"] = sp.Selector(s, i["sel"], DEV)
    if "layers" in i:
        st["model"] = sp.Model(m, None, None, DEV, max_pos=4352,
                               device_weights={"layers": i["layers"], "head": i["head"]})
    if case["kind"] == "prefill" and case["kv"]:
        st["kv"] = sp.kv_cache(st["model"], case["seqs"], case["tokens"] + 16)
    if case["kind"] == "decode":
        st["lens"] = i["lens"].clone()
    if case["kind"] == "pipeline":
        st["pipe"] = sp.Pipeline(st["selector"], st["model"], _vis(case), _txt(case), group_size=0, g=case["g"],
                                 k_max=case["k_max"])
        st["pipe"].hidden.zero_()  # the rows past the packed length stay as they are
    return st


# ----------------------------------------------------------------------------- one pass

def run(st):
    return {"select": _run_select, "train": _run_train, "project": _run_project, "prefill": _run_prefill,
            "decode": _run_decode, "pipeline": _run_pipeline}[st["case"]["kind"]](st)


def _run_select(st):
    c, i = st["case"], st["in"]
    # a user that encodes takes the kept indices and the memory; the traces are the other calls' outputs
    o = sp.sp_select(st["selector"], _vis(c), _txt(c), stop_bias=i["stop_bias"], X=i.get("X"), E_text=i.get("E_text"),
                     H=i.get("H"), group_size=c["group"], g=c["g"], k_max=c["k_max"], traces=not c["encode"],
                     memory=c["encode"], ws=st.get("ws"))
    st["ws"] = o["_ws"]
    return {k: v for k, v in o.items() if k not in ("_ws", "k_cap")}


def _run_train(st):
    c, i, n_vis = st["case"], st["in"], _vis(st["case"])
    o = sp.sp_select(st["selector"], n_vis, _txt(c), stop_bias=i["stop_bias"], H=i["H"], k_max=c["k_max"],
                     train=(TAU, BETA), ws=st.get("ws"))
    st["ws"] = o["_ws"]
    a = sp.sp_soft_topk(n_vis, score=o["score"], kbar=o["kbar"], tau=TAU)
    x = sp.sp_vp_gate(X=i["X"], noise=i["noise"], alpha=a["alpha"])
    return {"idx": o["idx"], "count": o["count"], "score": o["score"], "kbar": o["kbar"], "alpha": a["alpha"],
            "k": a["k"], "gated": x}


def _run_project(st):
    c, i, m = st["case"], st["in"], st["model"]
    n_vis, n_txt = _vis(c), _txt(c)
    o = st["out"] = sp.sp_compact(n_vis, n_txt, X=i["X"], text=i["text"], idx=i["idx"], count=i["count"],
                                  k_cap=i["idx"].shape[1], index_mode=True, out=st.get("out"))
    if "ws" not in st:
        st["ws"] = sp.workspace(sp.lib().sp_project_workspace(m.handle, o["rows_cap"]), DEV)
    sp.sp_project(m, vis_row_map=o["vis_row_map"], vis_cu=o["vis_cu"], packed=o["packed"], rows_cap=o["rows_cap"],
                  B=len(n_vis), X=i["X"], vis_src=o["vis_src"], ws=st["ws"])
    return {k: o[k] for k in ("packed", "cu_seqlens", "pos", "vis_src", "vis_row_map", "vis_cu")}


def _run_prefill(st):
    c, i = st["case"], st["in"]
    o = sp.sp_prefill(st["model"], x=i["x"], cu_seqlens=i["cu"], pos=i["pos"], B=c["seqs"], T_cap=i["x"].shape[0],
                      max_seqlen_cap=c["tokens"], ws=st.get("ws"), hidden=st.get("hidden"), kv=st.get("kv"),
                      pos3=i.get("pos3"))
    st["ws"], st["hidden"] = o["_ws"], o["hidden"]
    return {"hidden": o["hidden"], "kv": st["kv"]} if c["kv"] else {"hidden": o["hidden"]}


def _run_decode(st):
    c, i = st["case"], st["in"]
    st["lens"].copy_(i["lens"])  # generation starts behind the prefix again
    hidden = st.setdefault("hidden", [None] * c["steps"])
    for t in range(c["steps"]):
        o = sp.sp_decode(st["model"], x=i["x"][t], lens=st["lens"], kv=i["kv"], max_len_cap=i["kv"].shape[3],
                         ws=st.get("ws"), hidden=hidden[t])
        st["ws"], hidden[t] = o["_ws"], o["hidden"]
    return {"hidden": list(hidden), "kv": i["kv"], "lens": st["lens"]}


def _run_pipeline(st):
    p, i = st["pipe"], st["in"]
    p(i["X"], i["E_text"], i["stop_bias"])
    return {"idx": p.idx, "count": p.count, "cu_seqlens": p.cu, "hidden": p.hidden}


# ----------------------------------------------------------------------------- work

def _select_work(case, s):
    n_vis = _vis(case)
    N, L, D, h = sum(n_vis), sum(_txt(case)), s.D, s.h
    E = len(_episodes(n_vis, case.get("group", 0)))
    rounds = -(-case["k_max"] // case.get("g", 1))
    # per candidate: decoder token, folded key, query, key and value; per lower layer its cross key and value
    flops = 2.0 * N * (2 * s.n_dec_layers * h * D + 3 * h * h)
    nbytes = 4.0 * (2 * s.n_dec_layers * h * D + 3 * h * h) + 4.0 * N * D
    # per round: pointer logits, attention over the history (half of k_max long on average)
    flops += rounds * (2.0 * N * h + E * 2.0 * case["k_max"] * h)
    lower = s.n_dec_layers - 1
    flops += lower * rounds * (4.0 * N * h + E * (2.0 * 8 * h * h + 2.0 * 3 * h * h))
    nbytes += lower * (2.0 * 8 * h * h + 4.0 * 3 * h * h)
    if s.n_enc_layers:
        T = [v + t for v, t in zip(n_vis, _txt(case))]
        P = 4 * D * D + 2 * D * s.enc_ffn
        flops += 2.0 * L * D * s.D_text + s.n_enc_layers * (2.0 * sum(T) * P + 4.0 * D * sum(t * t for t in T))
        nbytes += 2.0 * (N * D + L * s.D_text + D * s.D_text + s.n_enc_layers * P)
    return nbytes, flops


def _layers_work(m, rows, pairs, layers):
    """Decoder layers over `rows` rows that attend to `pairs` (query, key) pairs."""
    P = m.d * (m.n_heads + 2 * m.n_kv_heads) * m.head_dim + m.d * m.n_heads * m.head_dim + 3 * m.d * m.ffn
    return 2.0 * layers * P, layers * (2.0 * rows * P + 4.0 * m.n_heads * m.head_dim * pairs)


def work(case):
    kind = case["kind"]
    s, m = _shapes(case)
    if kind == "select":
        b, f = _select_work(case, s)
    elif kind == "train":
        b, f = _select_work(case, s)
        b += 6.0 * sum(_vis(case)) * s.D
    elif kind == "project":
        rows = sum(_kept(case))
        P = m.proj_in * m.proj_hidden + m.proj_hidden * m.d
        b = 2.0 * P + 2.0 * rows * (m.proj_in + m.d) + 4.0 * sum(_txt(case)) * m.d
        f = 2.0 * rows * P
    elif kind == "prefill":
        lens = _spread(case["tokens"], case["seqs"], case["ragged"])
        b, f = _layers_work(m, sum(lens), sum(n * (n + 1) / 2 for n in lens), m.n_layers)
        b += 6.0 * sum(lens) * m.d
        if case["kv"]:
            b += 4.0 * m.n_layers * sum(lens) * m.n_kv_heads * m.head_dim
    elif kind == "decode":
        lens = _spread(case["context"], case["seqs"], case["ragged"])
        b = f = 0.0
        for t in range(case["steps"]):
            pairs = sum(n + t + 1 for n in lens)
            wb, wf = _layers_work(m, case["seqs"], pairs, m.n_layers)
            b += wb + 4.0 * m.n_layers * pairs * m.n_kv_heads * m.head_dim
            f += wf
    else:
        b, f = _select_work(case, s)
        rows = case["images"] * case["k_max"]
        n = case["k_max"] + case["n_txt"]
        wb, wf = _layers_work(m, case["images"] * n, case["images"] * n * (n + 1) / 2, m.n_layers)
        P = m.proj_in * m.proj_hidden + m.proj_hidden * m.d if m.proj_kind == "mlp2" else m.proj_in * m.d
        b, f = b + wb + 2.0 * P + 4.0 * case["images"] * n * m.d, f + wf + 2.0 * rows * P
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times the error against exact() measured on a GB300 (relative, 2-norm): 1.1e-5 to 3.8e-5
    in the logits' gaps (2.5e-5 in the margins, which are differences of them), 1.5e-3 in the encoder's memory,
    1.7e-3 in the noise gate's 16-bit rows, 2.3e-3 behind the projector, 3.5e-3 behind one decoder layer
    and 8.3e-3 behind two to four.  Whole values differ where two tokens' logits are the same to rounding."""
    kind = case["kind"]
    if kind == "select" and not case["encode"]:
        return {"rel": 1.5e-4, "max": 2e-3, "differ": 0.01}
    if kind in ("select", "train"):
        return {"rel": 6e-3, "max": 0.05, "differ": 0.01}
    if kind == "project":
        return {"rel": 1e-2, "max": 0.1}
    return {"rel": 0.015 if case["layers"] == 1 else 0.03, "max": 0.2, "differ": 0.01 if kind == "pipeline" else 0.0}


# ----------------------------------------------------------------------------- the same in 64 bits

def exact(case, seed):
    kind, i = case["kind"], _inputs(case, seed)
    s, m = _shapes(case)
    if kind == "select":
        if case["encode"]:  # which tokens are kept hangs on the 16-bit encoder's roundings; the memory does not
            return {"idx": None, "count": None, "err": None, "memory": _exact_encoder(case, s, i)}
        r = _exact_rollout(case, s, i, None)
        # (the margins are differences of nearly equal logits: what they say is in the gaps too)
        return {"idx": None, "count": None, "err": None, "order": None, "ep_count": None, "rounds": None,
                "margin": None, "gap": r["gap"]}
    if kind == "train":
        r = _exact_rollout(case, s, i, (TAU, BETA))
        k = r["kbar"].sum() / case["images"]
        alpha = torch.cat([_exact_soft_topk(v, k, TAU) for v in r["score"].split(_vis(case))])
        gated = alpha.sqrt()[:, None] * i["X"].double() + (1 - alpha).clamp(min=0).sqrt()[:, None] * i["noise"].double()
        return {"idx": None, "count": None, "score": r["score"], "kbar": r["kbar"], "alpha": alpha, "k": k.reshape(1),
                "gated": gated}
    if kind == "project":
        return _exact_project(case, m, i)
    if kind == "prefill":
        return _exact_prefill(case, m, i)
    if kind == "decode":
        return _exact_decode(case, m, i)
    return None  # which tokens the pipeline keeps hangs on the 16-bit encoder's roundings


def _lin(x, w):
    return x @ w.double().T


def _ln(x, L, n, eps):
    return F.layer_norm(x, x.shape[-1:], L[n + "_g"].double(), L[n + "_b"].double(), eps)


def _exact_encoder(case, s, i):
    n_vis, n_txt, out, v0, t0 = _vis(case), _txt(case), [], 0, 0
    w = i["sel"]
    for n, L in zip(n_vis, n_txt):
        text = _ln(_lin(i["E_text"][t0:t0 + L].double(), w["W_p"]), w, "ln_text", s.ln_eps)
        x = torch.cat([i["X"][v0:v0 + n].double(), s.g_text * text])
        for B in w["enc"]:
            q, k, v = _lin(_ln(x, B, "ln1", s.ln_eps), B["Wqkv"]).split(s.D, 1)
            x = x + _lin(_attend(q, k, v, s.enc_heads, s.enc_heads, s.enc_head_dim, False), B["Wo"])
            x = x + _lin(F.gelu(_lin(_ln(x, B, "ln2", s.ln_eps), B["W1"])), B["W2"])
        out.append(x[:n])
        v0, t0 = v0 + n, t0 + L
    return torch.cat(out)


def _attend(q, k, v, heads, kv_heads, dh, causal):
    o = torch.empty_like(q)
    mask = torch.ones(len(q), len(k), dtype=torch.bool, device=q.device).triu(1 + len(k) - len(q)) if causal else None
    for a in range(heads):
        c = a * kv_heads // heads
        p = q[:, a * dh:(a + 1) * dh] @ k[:, c * dh:(c + 1) * dh].T / math.sqrt(dh)
        p = torch.softmax(p.masked_fill_(mask, -math.inf) if causal else p, 1)
        o[:, a * dh:(a + 1) * dh] = p @ v[:, c * dh:(c + 1) * dh]
    return o


def _exact_rollout(case, s, i, train):
    """Every episode's rounds, one by one: the gap trace and the training aggregates."""
    w, g, k_max, h = i["sel"], case.get("g", 1), case["k_max"], s.h
    d = {k: v.double() for k, v in w.items() if torch.is_tensor(v)}
    eps_list = _episodes(_vis(case), case.get("group", 0))
    nan = torch.full((len(eps_list), k_max + 1), math.nan, dtype=torch.float64, device=DEV)
    out = {"gap": nan, "score": torch.zeros(len(i["H"]), dtype=torch.float64, device=DEV),
           "kbar": torch.zeros(len(eps_list), dtype=torch.float64, device=DEV)}
    fold = (d["Wq_p"].T @ d["Wk_p"]).T / math.sqrt(h)
    lower = [{k: v.double() for k, v in L.items()} for L in w["lower"]]
    for e, (r0, n) in enumerate(eps_list):
        M = torch.cat([i["H"][r0:r0 + n].double(), d["s_stop"][None], d["s_start"][None]])
        Y, KT = M @ d["W_in"].T, M[:n + 1] @ fold
        cross = [(M[:n + 1] @ L["Wk_c"].T, M[:n + 1] @ L["Wv_c"].T) for L in lower]
        caches = [([], []) for _ in range(len(lower) + 1)]
        free = torch.ones(n, dtype=torch.bool, device=DEV)
        new, nsel, rnd, alive, disc = [n + 1], 0, 0, 1.0, 1.0
        while nsel < k_max:
            for row in new:  # the history's new positions through every layer
                y = Y[row]
                for L, (ck, cv), cache in zip(lower, cross, caches):
                    y = y + _self(y, L, cache, s.ln_eps)
                    p = torch.softmax(ck @ (L["Wq_c"] @ _ln(y, L, "ln2", s.ln_eps)) / math.sqrt(h), 0)
                    y = y + L["Wo_c"] @ (p @ cv)
                    y = y + L["W2"] @ F.gelu(L["W1"] @ _ln(y, L, "ln3", s.ln_eps))
                last = y + _self(y, d, caches[-1], s.ln_eps) if row == new[-1] else _self(y, d, caches[-1], s.ln_eps)
            logits = KT @ _ln(last, d, "ln2", s.ln_eps)
            raw, stop = logits[n], logits[n] + i["stop_bias"][e].double()
            avail = int(n - nsel)
            if avail == 0:
                out["gap"][e, rnd] = -math.inf
                break
            vis = logits[:n].masked_fill(~free, -math.inf)
            top = vis.topk(min(g, avail))
            out["gap"][e, rnd] = top.values[0] - raw
            if train:
                disc *= train[1]
                p = torch.softmax(torch.cat([vis, stop[None]]) / train[0], 0)
                out["score"][r0:r0 + n] += alive * disc * p[:n]
                out["kbar"][e] += alive * (1 - p[n])
                alive = alive * (1 - p[n])
            if bool(stop > top.values[0]):
                break
            new = top.indices[:min(g, k_max - nsel, avail)].tolist()
            free[new] = False
            nsel, rnd = nsel + len(new), rnd + 1
    return out


def _self(y, L, cache, eps):
    """What self-attention adds to the new position; its key and value join the cache."""
    x = _ln(y, L, "ln1", eps)
    cache[0].append(L["Wk_s"] @ x)
    cache[1].append(L["Wv_s"] @ x)
    p = torch.softmax(torch.stack(cache[0]) @ (L["Wq_s"] @ x) / math.sqrt(len(y)), 0)
    return L["Wo_s"] @ (p @ torch.stack(cache[1]))


def _exact_soft_topk(score, k, tau):
    """alpha = sigmoid(2 (s - theta) / tau) with theta such that they sum to k."""
    n = len(score)
    if k <= 0 or k >= n:
        return torch.full_like(score, 0.0 if k <= 0 else 1.0)
    lo, hi = score.min() - 30 * tau, score.max() + 30 * tau
    for _ in range(80):
        mid = (lo + hi) / 2
        over = torch.sigmoid(2 * (score - mid) / tau).sum() > k
        lo, hi = torch.where(over, mid, lo), torch.where(over, hi, mid)
    return torch.sigmoid(2 * (score - (lo + hi) / 2) / tau)


def _exact_project(case, m, i):
    kept, n, L = _kept(case), case["n_vis"], case["n_txt"]
    cap = i["idx"].shape[1]
    packed = torch.zeros(sum(min(n, cap) + L for _ in kept), m.d, dtype=torch.float64, device=DEV)
    r = 0
    for b, k in enumerate(kept):
        x = i["X"][b * n + i["idx"][b, :k].long()].double()
        packed[r:r + k] = _lin(F.gelu(_lin(x, i["head"]["proj_W1"])), i["head"]["proj_W2"])
        packed[r + k:r + k + L] = i["text"][b * L:(b + 1) * L].double()
        r += k + L
    return {"packed": packed, "cu_seqlens": None, "pos": None, "vis_src": None, "vis_row_map": None, "vis_cu": None}


def _rms(x, g, eps):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * g.double()


def _angles(m, pos):
    """cos and sin per rotation pair: pos [T], or [T, 4] with a component per section."""
    inv = m.rope_theta ** (-torch.arange(0, m.head_dim, 2, dtype=torch.float64, device=DEV) / m.head_dim)
    if pos.dim() == 1:
        a = pos.double()[:, None] * inv
    else:
        sec = torch.repeat_interleave(torch.arange(3, device=DEV), torch.tensor(m.mrope_section, device=DEV))
        a = pos.double()[:, sec] * inv
    return a.cos()[:, None], a.sin()[:, None]


def _rotate(x, heads, cs):
    T = len(x)
    a, b = x.view(T, heads, -1).chunk(2, -1)
    return torch.cat([a * cs[0] - b * cs[1], b * cs[0] + a * cs[1]], -1).reshape(T, -1)


def _exact_layer(m, L, x, cs, attend):
    """One decoder layer; attend(q, k, v) gives the attention's output from the rows' rotated q and k."""
    dq, W = m.n_heads * m.head_dim, m.n_kv_heads * m.head_dim
    q, k, v = _lin(_rms(x, L["attn_norm"], m.rms_eps), L["Wqkv"]).split([dq, W, W], 1)
    x = x + _lin(attend(_rotate(q, m.n_heads, cs), _rotate(k, m.n_kv_heads, cs), v), L["Wo"])
    a = _rms(x, L["mlp_norm"], m.rms_eps)
    act = F.silu(_lin(a, L["Wgu"][:m.ffn])) * _lin(a, L["Wgu"][m.ffn:])
    return x + _lin(act, L["Wdown"])


def _exact_prefill(case, m, i):
    lens, S, W = _spread(case["tokens"], case["seqs"], case["ragged"]), case["tokens"] + 16, m.n_kv_heads * m.head_dim
    x, cs = i["x"].double(), _angles(m, i.get("pos3", i["pos"]))
    kv = torch.zeros(m.n_layers, 2, len(lens), S, W, dtype=torch.float64, device=DEV) if case["kv"] else None
    for l, L in enumerate(i["layers"]):
        def attend(q, k, v):
            out = []
            for b, (qs, ks, vs) in enumerate(zip(q.split(lens), k.split(lens), v.split(lens))):
                out.append(_attend(qs, ks, vs, m.n_heads, m.n_kv_heads, m.head_dim, True))
                if kv is not None:
                    kv[l, 0, b, :lens[b]], kv[l, 1, b, :lens[b]] = ks, vs
            return torch.cat(out)
        x = _exact_layer(m, L, x, cs, attend)
    out = {"hidden": _rms(x, i["head"]["final_norm"], m.rms_eps)}
    return dict(out, kv=kv) if kv is not None else out


def _exact_decode(case, m, i):
    lens, hidden, kv = i["lens"].tolist(), [], i["kv"].double()
    for t in range(case["steps"]):
        x = i["x"][t].double()
        cs = _angles(m, torch.tensor(lens, device=DEV))
        for l, L in enumerate(i["layers"]):
            def attend(q, k, v):
                out = []
                for b, n in enumerate(lens):
                    kv[l, 0, b, n], kv[l, 1, b, n] = k[b], v[b]
                    out.append(_attend(q[b:b + 1], kv[l, 0, b, :n + 1], kv[l, 1, b, :n + 1], m.n_heads, m.n_kv_heads,
                                       m.head_dim, False))
                return torch.cat(out)
            x = _exact_layer(m, L, x, cs, attend)
        hidden.append(_rms(x, i["head"]["final_norm"], m.rms_eps))
        lens = [n + 1 for n in lens]
    return {"hidden": hidden, "kv": kv, "lens": None}
