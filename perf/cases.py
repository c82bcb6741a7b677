"""What this framework is used for, as cases whose time and outputs can be measured.

Two kinds of work, both through ``kvec.KvecSelector``, the framework's Python entry point:

* ``select``: the end of a prefill.  A program holds every layer's window queries, keys and values and a
  selector made for its model; a pass resets the coverage state (a new prompt) and asks for the eviction
  selection, either of all layers in one call or (``call = "layer"``) of one layer, as a prefill that evicts
  layer by layer does.  Options: the window rows' log-sum-exp supplied by the caller (``lse``), every position
  a candidate (``all_positions``), the head-wise adaptive fill (``head_budget`` with ``ada_floor``), the scores
  behind the selection read back (``scores``).
* ``decode``: one decoding step of attention over compacted caches, for every layer of a token, either as
  plain calls or (``graph``) replayed from a CUDA graph, as serving loops run it.

Inputs are Gaussian queries, keys and values in bf16 with a planted attention sink and salient positions that
layers and heads share in part (``synth``), the stand-in this repository uses for prompts of trained models.
"""
import math

import torch

from paper_2606_29563_gb300 import kvec, synth

HEAD_DIM = 128
WINDOW, OBS_WINDOW, EXT_WINDOW, POOL = 32, 16, 32, 7
MAX_TOKENS = 83_000 * 32          # layers x tokens of the largest listed case


def _select(name, q_heads, kv_heads, layers, lens, budget, **options):
    case = {"name": name, "kind": "select", "q_heads": q_heads, "kv_heads": kv_heads, "layers": layers,
            "lens": lens, "budget": budget, "max_seqlen": 0, "call": "layers", "lam": 1.0, "lse": False,
            "all_positions": False, "head_budget": False, "ada_floor": 0.2, "scores": False,
            "salient": 0.01, "lognormal": 0.0}
    case.update(options)
    return case


def _decode(name, q_heads, kv_heads, layers, lens, cap, graph):
    return {"name": name, "kind": "decode", "q_heads": q_heads, "kv_heads": kv_heads, "layers": layers,
            "lens": lens, "cap": cap, "graph": graph}


def _text(lens):
    return ",".join(str(int(n)) for n in lens)


# Eight ragged prompts of 4096 to 16384 tokens: the batch that bench.py times by default.
RAGGED8 = _text(synth.WORKLOADS["llama8b_ragged8_b256"].seqlens)
# Sixteen chat-sized prompts, some of them shorter than the budget (every token of those is kept).
SHORT16 = "1873,301,2954,96,777,1502,2411,640,3071,255,1190,2048,431,1667,129,2733"


def listed():
    return [
        # The smallest call: one layer of a small multi-head model, where launches are all there is.
        _select("layer_mha8_1k", 8, 8, 1, "1024", 128, call="layer", lam=0.0, salient=0.04),
        # One layer of an 8B model per call: a prefill that evicts as it goes.
        _select("layer_llama8b_8k", 32, 8, 1, "8192", 512, call="layer"),
        # One layer together with the scores behind its choice, at an odd length: what a study of the selection
        # reads, and the case whose floating-point scores are compared with 64 bits.
        _select("scores_qwen7b_11k", 28, 4, 1, "11003", 512, call="layer", scores=True),
        # A whole prefill of one prompt, the framework's ordinary call, at three lengths and two models.
        _select("prefill_llama8b_8k", 32, 8, 32, "8192", 512),
        _select("prefill_llama8b_32k", 32, 8, 32, "32768", 128, salient=0.005, lognormal=0.5),
        _select("prefill_qwen7b_16k", 28, 4, 28, "16384", 512),
        # Batched prefills: many short prompts on a server whose handle allows long ones, and the largest case.
        _select("prefill_llama8b_short16", 32, 8, 32, SHORT16, 256, max_seqlen=16384),
        _select("prefill_llama8b_ragged8", 32, 8, 32, RAGGED8, 256),
        # The same batch when the prefill's attention hands over its rows' log-sum-exp.
        _select("prefill_lse_ragged8", 32, 8, 32, RAGGED8, 256, lse=True),
        # Head-wise adaptive budgets over a whole prefill.
        _select("prefill_adaptive_8k", 32, 8, 32, "8192", 512, head_budget=True),
        # One generated token of one sequence: 32 layers' attention over 512 kept rows, replayed from a graph.
        _decode("decode_token_b1", 32, 8, 32, "512", 512, True),
        # Decoding for a full server: 64 sequences of up to 2048 cached rows (kept ones and decoded ones).
        _decode("decode_b64_2k", 32, 8, 4, _text(1024 + (i * 389) % 1025 for i in range(64)), 2048, False),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    # Heads of 7B to 70B models and of small multi-head ones.
    q_heads, kv_heads = rng.choice([(32, 8), (32, 8), (28, 4), (8, 8), (16, 16), (40, 8), (64, 8)])
    layers = rng.choice([1, 2, 8, 28, 32, 32])
    if rng.random() < 0.25:
        batch = _log_int(rng, 1, 64)
        cap = _log_int(rng, 32, 4096)
        lens = [rng.randint(max(1, cap // 3), cap) for _ in range(batch)]
        layers = max(1, min(layers, int(20e9 / (batch * kv_heads * cap * 4 * HEAD_DIM)) // 8))
        return {k: v for k, v in _decode("", q_heads, kv_heads, layers, _text(lens), cap, rng.random() < 0.5).items()
                if k != "name"}
    batch = rng.choice([1, 1, 2, 4, 8, 16])
    heads = max(kv_heads / 8, q_heads / 32)        # work per token against the largest listed case's
    top = min(32768, int(MAX_TOKENS / (layers * batch * heads)))
    longest = _log_int(rng, 256, top)
    lens = [longest] + [rng.randint(max(WINDOW, longest // 4), longest) for _ in range(batch - 1)]
    budget = _log_int(rng, 48, min(2048, max(64, longest // 2)))
    case = _select("", q_heads, kv_heads, layers, _text(lens), budget)
    if layers == 1:
        case["call"] = "layer"
    option = rng.choice(["", "", "", "lse", "all_positions", "head_budget"])
    if option:
        case[option] = True
    if option == "head_budget":                    # its outputs have room for one head taking every shared slot
        case["lens"] = _text(lens[:2])
    # A handle sized for the prompt, or for the server's longest one.
    case["max_seqlen"] = rng.choice([0, 0, 32768])
    del case["name"]
    return case


# ------------------------------------------------------------------------------------------------ inputs

def _lens(case):
    return [int(n) for n in case["lens"].split(",")]


def _workload(case, seed):
    return synth.Workload(
        name="case", layers=case["layers"], seqlens=tuple(_lens(case)), num_q_heads=case["q_heads"],
        num_kv_heads=case["kv_heads"], window=WINDOW, obs_window=OBS_WINDOW, ext_window=EXT_WINDOW,
        pool_kernel=POOL, budget=case["budget"], lam=case["lam"], all_positions=int(case["all_positions"]),
        head_budget=int(case["head_budget"]), ada_floor=case["ada_floor"], salient_frac=case["salient"],
        p_share=0.7, carry=0.6, lognormal_sigma=case["lognormal"], seed=int(seed) % (1 << 31))


def _logits(wl, x, s, dtype):
    """scale * <q, k> of sequence s's window rows, [H_kv][g][w][L], -inf where the key comes after the row."""
    g, w, cu = wl.group, wl.window, wl.cu_seqlens
    L = cu[s + 1] - cu[s]
    q = x["q_obs"][s].to(dtype).view(w, wl.num_kv_heads, g, HEAD_DIM).permute(1, 2, 0, 3)
    k = x["k"][cu[s]:cu[s + 1]].to(dtype).permute(1, 2, 0)
    logits = torch.matmul(q.reshape(wl.num_kv_heads, g * w, HEAD_DIM), k).view(wl.num_kv_heads, g, w, L)
    logits *= 1.0 / math.sqrt(HEAD_DIM)
    rows = torch.arange(w, device=k.device)
    hidden = (torch.arange(w, device=k.device)[None, :] > rows[:, None])   # keys of the window part
    logits[..., L - w:].masked_fill_(hidden, -math.inf)
    return logits


def _lse(wl, x):
    out = torch.empty(wl.batch, wl.window, wl.num_q_heads, dtype=torch.float32, device="cuda")
    for s in range(wl.batch):
        lse = torch.logsumexp(_logits(wl, x, s, torch.float32), dim=3)     # [H_kv][g][w]
        out[s] = lse.permute(2, 0, 1).reshape(wl.window, wl.num_q_heads)
    return out


def _select_inputs(case, seed):
    wl = _workload(case, seed)
    structure = [synth.salient_structure(wl, b, wl.layers) for b in range(wl.batch)]
    return wl, [synth.make_layer(wl, l, "cuda", structure) for l in range(wl.layers)]


def _decode_inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    lens = _lens(case)
    draw_bf16 = lambda *shape: torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32).to(torch.bfloat16)
    cache = (len(lens), case["kv_heads"], case["cap"], HEAD_DIM)
    q = [draw_bf16(len(lens), case["q_heads"], HEAD_DIM) for _ in range(case["layers"])]
    k = [draw_bf16(*cache) for _ in range(case["layers"])]
    v = [draw_bf16(*cache) for _ in range(case["layers"])]
    return q, k, v, torch.tensor(lens, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    if case["kind"] == "decode":
        q, k, v, lens = _decode_inputs(case, seed)
        sel = kvec.KvecSelector(kvec.make_params(case["q_heads"], case["kv_heads"], max_batch=lens.numel(),
                                                 max_seqlen=max(case["cap"], WINDOW), max_layers=case["layers"]))
        state = {"case": case, "sel": sel, "q": q, "k": k, "v": v, "lens": lens,
                 "out": torch.empty(case["layers"], lens.numel(), case["q_heads"], HEAD_DIM, device="cuda")}
        if case["graph"]:
            _decode_token(state)
            torch.cuda.synchronize()
            state["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(state["graph"]):
                _decode_token(state)
            state["out"].zero_()
        return state
    wl, xs = _select_inputs(case, seed)
    sel = kvec.KvecSelector(kvec.params_from_workload(wl, max_seqlen=case["max_seqlen"] or None))
    cap = kvec.kvec_output_capacity(sel.params, wl.budget)
    idx = torch.empty(wl.layers, wl.batch, wl.num_kv_heads, cap, dtype=torch.int32, device="cuda")
    out_k = torch.empty(*idx.shape, HEAD_DIM, dtype=torch.bfloat16, device="cuda")
    out_v = torch.empty_like(out_k)
    cu = torch.tensor(wl.cu_seqlens, dtype=torch.int32).pin_memory()
    return {"case": case, "wl": wl, "sel": sel, "cu": cu, "cu_dev": cu.cuda(),
            "q": [x["q_obs"] for x in xs], "k": [x["k"] for x in xs], "v": [x["v"] for x in xs],
            "lse": [_lse(wl, x) for x in xs] if case["lse"] else None,
            "coverage": sel.new_state(wl.batch), "views": {}, "idx": idx, "out_k": out_k, "out_v": out_v,
            "outs": [(idx[l], out_k[l], out_v[l]) for l in range(wl.layers)]}


# ------------------------------------------------------------------------------------------------ one pass

def _decode_token(state):
    for l in range(len(state["q"])):
        state["sel"].decode_attention(state["q"][l], state["k"][l], state["v"][l], state["lens"], out=state["out"][l])


def run(state):
    case = state["case"]
    if case["kind"] == "decode":
        if case["graph"]:
            state["graph"].replay()
        else:
            _decode_token(state)
        return {"out": state["out"]}
    wl, sel, coverage = state["wl"], state["sel"], state["coverage"]
    kvec.kvec_reset(sel.handle, coverage.data_ptr(), wl.batch, torch.cuda.current_stream().cuda_stream)
    if case["call"] == "layer":
        for l in range(wl.layers):
            sel.select_layer(state["cu"], state["cu_dev"], state["q"][l], state["k"][l], state["v"][l], coverage,
                             wl.budget, outs=state["outs"][l], lse=state["lse"][l] if state["lse"] else None)
    else:
        sel.select_layers(state["cu"], state["cu_dev"], state["q"], state["k"], state["v"], coverage, wl.budget,
                          state["outs"], lses=state["lse"])
    got = {"idx": state["idx"], "k": state["out_k"], "v": state["out_v"], "coverage": coverage}
    if case["scores"]:
        got.update(_scores(state))
    return got


class _DeviceArray:
    """A device pointer as torch takes it, without a copy; it keeps the memory's owner."""

    def __init__(self, ptr, shape, owner):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (int(ptr), False), "version": 3,
                                         "strides": None}


def _scores(state):
    """Copies of the last layer's scores, which the selector overwrites, cut to the candidates of each sequence."""
    wl, view = state["wl"], kvec.kvec_debug_scores(state["sel"].handle)
    heads, row, views = wl.num_kv_heads, view.max_seqlen, state["views"]
    key = (view.P_O, view.P_Oext, view.Pprime, view.I, view.sigma)
    if key not in views:                           # a program wraps the pointers once
        array = lambda ptr, *shape: torch.as_tensor(_DeviceArray(ptr, shape, state["sel"]), device="cuda")
        cut = lambda t: [t[s, ..., :n - WINDOW] for s, n in enumerate(wl.seqlens)]
        views[key] = {"P_O": cut(array(view.P_O, wl.batch, heads, row)),
                      "P_Oext": cut(array(view.P_Oext, wl.batch, heads, row)),
                      "Pprime": cut(array(view.Pprime, wl.batch, heads, row)),
                      "I": cut(array(view.I, wl.batch, row)), "sigma": [array(view.sigma, wl.batch, heads)]}
    return {name: [t.clone() for t in parts] for name, parts in views[key].items()}


# ------------------------------------------------------------------------------------------------ what it takes

def work(case):
    lens, hq, hkv, layers = _lens(case), case["q_heads"], case["kv_heads"], case["layers"]
    row = 2 * HEAD_DIM
    if case["kind"] == "decode":
        rows = sum(lens) * hkv
        return {"bytes": layers * (2 * rows * row + len(lens) * hq * (row + 4 * HEAD_DIM)),
                "flops": layers * 4 * HEAD_DIM * rows * (hq // hkv)}
    # Keys and window queries read once; the kept keys and values read and written with their positions.
    kept = sum(min(n, case["budget"]) for n in lens) * hkv
    layer = sum(lens) * hkv * row + len(lens) * WINDOW * hq * row + kept * (4 * row + 4)
    if case["lse"]:
        layer += len(lens) * WINDOW * hq * 4
    return {"bytes": layers * layer, "flops": layers * 2 * HEAD_DIM * WINDOW * hq * sum(lens)}


def tolerance(case):
    if case["kind"] == "decode":
        # fp32 sums over up to 4096 rows, measured against 64 bits: 3.3e-7.
        return {"rel": 1.2e-6}
    if case["scores"]:
        # fp32 scores, measured against 64 bits: 3.3e-7; positions as below.
        return {"rel": 1.4e-6, "differ": 0.01}
    # A selection with other roundings swaps tokens whose scores tie to within them, about one kept row in ten
    # thousand, and what lies between the two moves by one place in the sorted outputs.
    return {"rel": 0.03, "max": 0.99, "differ": 0.01}


# ------------------------------------------------------------------------------------------------ in 64 bits

def _pool(p):
    """Max-pool of width POOL along the last axis, neighbours past the ends left out."""
    halo = POOL // 2
    padded = torch.nn.functional.pad(p, (halo, halo), value=-math.inf)
    return padded.unfold(-1, POOL, 1).amax(-1)


def exact(case, seed):
    """Decode outputs, and the scores of a first layer; selected positions and copied rows have no 64-bit value."""
    if case["kind"] == "decode":
        q, k, v, lens = _decode_inputs(case, seed)
        g, out = case["q_heads"] // case["kv_heads"], []
        for l in range(case["layers"]):
            rows = []
            for s, n in enumerate(lens.tolist()):
                qs = q[l][s].double().view(case["kv_heads"], g, HEAD_DIM)
                a = torch.softmax(torch.matmul(qs, k[l][s, :, :n].double().transpose(1, 2)) / math.sqrt(HEAD_DIM), -1)
                rows.append(torch.matmul(a, v[l][s, :, :n].double()).reshape(case["q_heads"], HEAD_DIM))
            out.append(torch.stack(rows))
        return {"out": torch.stack(out)}
    if not case["scores"]:
        return None
    got = {"idx": None, "k": None, "v": None, "coverage": None}
    wl, xs = _select_inputs(case, seed)
    got.update({name: [] for name in ("P_O", "P_Oext", "Pprime", "I")})
    got["sigma"] = [torch.zeros(wl.batch, wl.num_kv_heads, dtype=torch.float64)]
    for s, L in enumerate(_lens(case)):
        a = torch.softmax(_logits(wl, xs[0], s, torch.float64), -1).sum(1)[..., :L - WINDOW]   # [H_kv][w][candidates]
        p_o, p_e = _pool(a[:, WINDOW - OBS_WINDOW:].mean(1)), _pool(a[:, WINDOW - EXT_WINDOW:].mean(1))
        importance = _pool(a[:, WINDOW - OBS_WINDOW:].amax(0).mean(0))
        sigma = p_o.std(1)
        extended = torch.zeros(wl.num_kv_heads, dtype=torch.bool, device="cuda")
        extended[torch.argsort(sigma)[:wl.num_ext_heads]] = True
        got["P_O"].append(p_o)
        got["P_Oext"].append(p_e)
        got["I"].append(importance)
        got["Pprime"].append(torch.where(extended[:, None], p_e, p_o) + wl.lam * importance)   # n_t = 0
        got["sigma"][0][s] = sigma.cpu()
    return got
