"""Performance cases of the MI hook: what a serving engine or an analysis script has it do, over the sizes it is used at.

Three paths through the public entry points:

  hook    probes, steering vectors and projections of a decode step or of a prefill batch (contexts without SAE
          weight sets): `set_slot_map` / `set_request_map`, `apply`
  sae     sparse-autoencoder apps, alone or beside probes and steering in one batch: `set_slot_map`, `apply`
  static  the SAE function for callers that may not allocate: `sae_apply_static`

A case says whether the program replays a CUDA graph that it captured once (`graph`), as an engine's decode step
does, or calls eagerly.  Every pass installs the step's slot map, as every step of continuous batching does.

SAE passes begin with a copy into `hidden` that stands for the layer in front of the hook: the SAE function is
applied in place, and without that copy the next pass would work on the output of this one.  The copy is not part
of `work`.  Probes, steering and projections do not need it (their cost does not depend on the values).
"""
import numpy as np
import torch

import paper_2607_22595_b200 as mix

EDITS = 16          # edited features per SAE app (half of them features that fire on one of the app's rows)


# ------------------------------------------------------------------------------------------ the cases
def _hook(name, d, T, live, layers=1, probes=0, wide_probes=0, classes=1, steers=0, projects=0, hooked=0.75, request=1,
          chain=False, gated=False, graph=True, two_level=False):
    """request: longest request in tokens (1: a pure decode step)."""
    c = dict(path="hook", d=d, T=T, live=live, layers=layers, probes=probes, wide_probes=wide_probes, classes=classes,
             steers=steers, projects=projects, hooked=hooked, request=request, chain=chain, gated=gated, graph=graph,
             two_level=two_level)
    return dict(name=name, **c) if name else c


def _sae(name, d, d_sae, sets, act, k, T, live, requests, error=True, weights="bf16", tiled=False, graph=True, readout=False,
         probes=0, classes=1, steers=0, share=1.0):
    """share: part of the live rows that carry an SAE app; of the others, a third each are probe, steering and plain rows
    (all plain where there are no probes or steering vectors)."""
    c = dict(path="sae", d=d, d_sae=d_sae, sets=sets, act=act, k=k, T=T, live=live, requests=requests, error=error,
             weights=weights, tiled=tiled, graph=graph, readout=readout, probes=probes, classes=classes, steers=steers,
             share=share)
    return dict(name=name, **c) if name else c


def _static(name, rows, d, d_sae, act, k, error=True):
    c = dict(path="static", rows=rows, d=d, d_sae=d_sae, act=act, k=k, error=error)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one hooked layer, a handful of requests, called eagerly with the map already on the device: a notebook or
        # a small server; nothing but latency
        _hook("decode_8_rows_eager", d=4096, T=8, live=7, probes=3, steers=2, graph=False),
        # a decode step with every layer hooked (32 contexts), one graph: the step of the decode configuration
        # (256 one-token requests, 64 probes, 32 steering vectors, a quarter of the rows plain)
        _hook("decode_step_32_layers", d=4096, T=256, live=256, layers=32, probes=64, steers=32),
        # several apps on each row (probe, gated steering, five-class probe), a few layers, the map given in its
        # two-level form (token -> request -> slot) as an engine holds it
        _hook("decode_chained_gated", d=5120, T=192, live=187, layers=4, probes=6, wide_probes=6, classes=5, steers=6,
              chain=True, gated=True, two_level=True),
        # a chunked-prefill batch with every kind of app on its requests, ragged lengths
        _hook("prefill_all_kinds", d=5120, T=16384, live=15873, probes=8, wide_probes=8, classes=16, steers=8, projects=4,
              hooked=0.7, request=2048),
        # the smallest SAE call (the tiny configuration): 64 tokens of 8 requests, eagerly, selected features read out
        _sae("sae_tiny_eager", d=512, d_sae=4096, sets=1, act="topk", k=32, T=64, live=64, requests=8, graph=False, readout=True,
             share=0.5, probes=2, steers=2),
        # the everyday one: one dictionary of 16 k features on a decode batch, features read out, weights as they come
        _sae("sae_decode_16k", d=4096, d_sae=16384, sets=1, act="topk", k=64, T=128, live=91, requests=91, readout=True),
        # four wide dictionaries side by side, one per group of requests (the SAE-heavy configuration)
        _sae("sae_four_sets_65k", d=4096, d_sae=65536, sets=4, act="topk", k=64, T=512, live=512, requests=32, tiled=True),
        # the same kind of batch with 8-bit encoder and input, at sizes that fill no tile evenly
        _sae("sae_three_sets_fp8_input", d=4224, d_sae=49408, sets=3, act="topk", k=50, T=600, live=555, requests=40,
             weights="fp8_input"),
        # chunked prefill + decode with all three primitives (the mixed configuration)
        _sae("mixed_prefill_jumprelu", d=5120, d_sae=32768, sets=2, act="jumprelu", k=0, T=8192, live=8192, requests=64,
             probes=8, classes=16, steers=8, share=0.23),
        # reconstruction instead of editing: the residual is replaced by what the sparse dictionary makes of it, as
        # when a dictionary's loss is measured
        _sae("reconstruct_jumprelu", d=2304, d_sae=24576, sets=1, act="jumprelu", k=0, T=1024, live=1000, requests=10, error=False,
             graph=False),
        # the widest dictionaries (the replay configuration's shape), 8-bit encoder weights, a graph captured for more
        # rows than are live
        _sae("sae_131k_fp8_weights", d=8192, d_sae=131072, sets=2, act="topk", k=128, T=2048, live=1337, requests=50,
             weights="fp8", probes=64, steers=16, share=0.6),
        # the call that allocates nothing, at the largest size it takes
        _static("static_128_rows", rows=128, d=4096, d_sae=8192, act="topk", k=64),
    ]


def _log(rng, lo, hi, step=1):
    """Spread over the logarithm of [lo, hi], in multiples of `step`."""
    x = lo * (hi / lo) ** rng.random()
    return max(lo, min(hi, int(round(x / step)) * step))


def _draw(rng):
    path = rng.choice(["decode", "decode", "chain", "prefill", "sae", "sae", "sae", "mixed", "reconstruct", "static"])
    d = 64 * _log(rng, 12, 128)                            # 768 .. 8192
    if path == "decode":
        T = _log(rng, 1, 2048)
        layers = _log(rng, 1, 32)
        return _hook(None, d=d, T=T, live=T - rng.randrange(T // 4 + 1), layers=layers, probes=_log(rng, 1, 64),
                     wide_probes=rng.choice([0, 4]), classes=rng.randrange(2, 17), steers=_log(rng, 1, 32),
                     projects=rng.choice([0, 2]), hooked=rng.choice([0.25, 0.75, 1.0]), gated=rng.random() < 0.3,
                     graph=layers > 1 or rng.random() < 0.5)
    if path == "chain":
        T = _log(rng, 8, 1024)
        return _hook(None, d=d, T=T, live=T - rng.randrange(T // 4 + 1), layers=_log(rng, 1, 16), probes=rng.randrange(1, 9),
                     wide_probes=rng.randrange(1, 9), classes=rng.randrange(2, 17), steers=rng.randrange(1, 9), chain=True,
                     gated=rng.random() < 0.5, two_level=rng.random() < 0.5)
    if path == "prefill":
        T = _log(rng, 2049, 32768)
        return _hook(None, d=d, T=T, live=T - rng.randrange(T // 8 + 1), probes=rng.randrange(0, 9), wide_probes=rng.randrange(0, 9),
                     classes=rng.randrange(2, 33), steers=rng.randrange(1, 9), projects=rng.randrange(0, 5),
                     hooked=rng.choice([0.3, 0.7, 1.0]), request=_log(rng, 1, 2048), graph=rng.random() < 0.5)
    weights = rng.choice(["bf16", "bf16", "bf16", "fp8", "fp8_input"])
    if weights != "bf16":
        d = max(768, d // 128 * 128)
    act = rng.choice(["topk", "topk", "jumprelu", "relu"])
    k = _log(rng, 16, 128) if act == "topk" else 0
    if path == "sae":
        T = _log(rng, 1, 2048)
        return _sae(None, d=d, d_sae=256 * _log(rng, 8, 512), sets=_log(rng, 1, 8), act=act, k=k, T=T,
                    live=T - rng.randrange(T // 4 + 1), requests=_log(rng, 1, 64), error=act != "topk" or rng.random() < 0.7,
                    weights=weights, tiled=weights == "bf16" and rng.random() < 0.5, graph=rng.random() < 0.7,
                    readout=act == "topk" and rng.random() < 0.5)
    if path == "mixed":
        T = _log(rng, 1024, 8192)
        return _sae(None, d=d, d_sae=256 * _log(rng, 16, 256), sets=rng.randrange(1, 4), act=act, k=k, T=T,
                    live=T - rng.randrange(T // 8 + 1), requests=_log(rng, 8, 128), weights=weights,
                    tiled=weights == "bf16" and rng.random() < 0.5, probes=rng.randrange(1, 9), classes=rng.choice([1, 4, 16]),
                    steers=rng.randrange(1, 9), share=rng.choice([0.1, 0.25, 0.5]))
    if path == "reconstruct":
        T = _log(rng, 16, 1024)
        act = rng.choice(["relu", "jumprelu", "topk"])
        return _sae(None, d=64 * _log(rng, 12, 64), d_sae=256 * _log(rng, 16, 128), sets=1, act=act, k=64 if act == "topk" else 0, T=T, live=T - rng.randrange(T // 8 + 1), requests=_log(rng, 1, 16), error=False, graph=rng.random() < 0.3)
    act = rng.choice(["topk", "jumprelu", "relu"])
    return _static(None, rows=_log(rng, 1, 128), d=64 * _log(rng, 8, 64), d_sae=256 * _log(rng, 4, 32), act=act,
                   k=_log(rng, 8, 64) if act == "topk" else 0, error=rng.random() < 0.7)


def _cost(case):
    w = work(case)
    return w["bytes"] / 6e12 + w["flops"] / 1.2e15


def _room(case):
    """Bytes of device memory a state takes, roughly."""
    if case["path"] != "sae":
        return 0
    rows = case["T"] + 128 * case["sets"] + 128
    per = case["d"] * case["d_sae"] * (2 + _code_bytes(case) * (2 if case["tiled"] or case["weights"] != "bf16" else 1))
    return case["sets"] * per + rows * (4 * case["d_sae"] + 4 * case["d"])


def draw(rng):
    dearest = max(_cost(c) for c in listed())
    while True:
        case = _draw(rng)
        if _cost(case) <= dearest and _room(case) <= 20 << 30:
            return case


# ------------------------------------------------------------------------------------------ what a pass cannot do without
def _code_bytes(case):
    return 2 if case["weights"] == "bf16" else 1


def _kind_rows(case):
    """Rows of each kind in one batch: fixed by the case (which rows they are comes from the seed)."""
    live = case["live"]
    if case["path"] == "hook":
        kinds = [k for k in ("probes", "wide_probes", "steers", "projects") if case[k]]
        n = round(case["hooked"] * live)
        if case["chain"]:
            return {"chain": n, "plain": live - n}
        rows = {k: n // len(kinds) + (i < n % len(kinds)) for i, k in enumerate(kinds)}
    else:
        n = max(1, round(case["share"] * live))
        rest = live - n
        rows = {"sae": n}
        if case["probes"]:
            rows["probes"] = rest // 3
        if case["steers"]:
            rows["steers"] = rest // 3
    rows["plain"] = live - sum(rows.values())
    return rows


def _active(case):
    """Features a row's reconstruction sums over."""
    return case["k"] if case["act"] == "topk" else case["d_sae"] // 256


def _sae_work(case, rows, sets, code_bytes):
    d, S = case["d"], case["d_sae"]
    sets = min(sets, rows)
    flops = 2.0 * rows * d * S
    nbytes = sets * S * (code_bytes * d + 4.0) + rows * 4.0 * d
    terms = EDITS if case["error"] else EDITS + _active(case)
    flops += 2.0 * rows * terms * d
    touched = EDITS * min(rows, case.get("requests", 1)) if case["error"] else rows * terms
    nbytes += 2.0 * d * min(touched, sets * S)
    return nbytes, flops


def work(case):
    d = case["d"]
    if case["path"] == "static":
        nbytes, flops = _sae_work(case, case["rows"], 1, 2)
        return {"bytes": nbytes, "flops": flops}
    rows = _kind_rows(case)
    nbytes, flops = 4.0 * case["live"], 0.0
    if case["path"] == "sae":
        nbytes, flops = _sae_work(case, rows["sae"], case["sets"], _code_bytes(case))
        nbytes += 4.0 * case["live"]
        if case["readout"]:
            nbytes += 8.0 * rows["sae"] * case["k"]
    for kind, n in rows.items():
        if kind in ("plain", "sae") or not n:
            continue
        if kind == "chain":
            used = [(case["probes"], 1), (case["wide_probes"], case["classes"]), (case["steers"], 1)]
            nbytes += 4.0 * d * n + sum(2.0 * d * c * min(n, m) for m, c in used) + 4.0 * n * (1 + case["classes"])
            flops += 2.0 * n * d * (2 + case["classes"])
            continue
        C = case["classes"] if kind == "wide_probes" or (kind == "probes" and case["path"] == "sae") else 1
        writes = kind in ("steers", "projects")
        nbytes += n * (4.0 * d if writes else 2.0 * d + 4.0 * C) + 2.0 * d * C * min(n, case[kind])
        flops += 2.0 * n * d * C * (2 if kind == "projects" else 1)
    layers = case.get("layers", 1)
    return {"bytes": nbytes * layers, "flops": max(flops, 1.0) * layers}


def tolerance(case):
    # bf16 hidden states (2^-9 relative rounding; the few elements whose fp32 value sits on a rounding boundary may go
    # either way) and fp32 scores through the hardware exponential.  Features are selected by fp32 pre-activations: one
    # that lies within their rounding of a threshold, or of the k-th value, may be in or out (a whole decoder row of the
    # rows that are rebuilt from their features), and near-ties may change places in the read-out
    if case["path"] == "hook":
        return {"rel": 1e-3, "max": 2e-2}
    if case["error"]:
        return {"rel": 3e-3, "max": 0.1, "differ": 2e-3}
    return {"rel": 1e-2, "max": 0.5, "differ": 2e-3}


# ------------------------------------------------------------------------------------------ inputs
def _normal(shape, std, gen, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=gen)


def _requests(rng, rows, n):
    """`rows` tokens cut into at most n ragged requests (none empty)."""
    n = max(1, min(n, rows))
    return 1 + rng.multinomial(rows - n, rng.dirichlet(np.full(n, 2.0))) if rows else np.zeros(0, dtype=np.int64)


def _lay_out(rng, T, parts):
    """parts: (length, slot) of every request; contiguous token ranges in a random order -> token_slot, token_req, req_slot."""
    order = rng.permutation(len(parts))
    token_slot, token_req, t = np.full(T, -1, np.int32), np.full(T, -1, np.int32), 0
    for r in order:
        n, slot = parts[r]
        token_slot[t:t + n] = slot
        token_req[t:t + n] = r
        t += n
    return token_slot, token_req, np.array([s for _, s in parts], np.int32)


def _state(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return gen, np.random.default_rng(seed)


def _captured(body):
    """A CUDA graph of body(), captured once, as an engine does at start-up."""
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        body()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            body()
    torch.cuda.current_stream().wait_stream(stream)
    return graph


def _prepare_hook(case, seed):
    gen, rng = _state(case, seed)
    d, T, L, C = case["d"], case["T"], case["layers"], case["classes"]
    n_p, n_w, n_s, n_r = case["probes"], case["wide_probes"], case["steers"], case["projects"]
    hidden = _normal((L, T, d), 1.0, gen)
    hidden[:, :, torch.randint(0, d, (max(d // 1000, 1),), generator=gen, device="cuda")] *= 20.0     # outlier channels
    cols = (1 if n_p else 0) + C if case["chain"] else (C if n_w else 1)
    scores = torch.zeros((L, T, cols), dtype=torch.float32, device="cuda")
    earlier = torch.rand((T, 1), generator=gen, device="cuda")          # what a probe at an earlier layer wrote
    first = {"probes": 0, "wide_probes": n_p, "steers": n_p + n_w, "projects": n_p + n_w + n_s}
    n_slots = n_p + n_w + n_s + n_r
    contexts = []
    for layer in range(L):
        m = mix.Mix(d_model=d, T_max=T, n_slots_max=n_slots, C_max=cols, flags=mix.MIX_FLAG_SLOT_CHAINS if case["chain"] else 0)
        narrow, wide, bias = _normal((max(n_p, 1), 1, d), d ** -0.5, gen), _normal((max(n_w, 1), C, d), d ** -0.5, gen), torch.zeros(C, device="cuda")
        vectors = _normal((n_s + n_r + 1, d), d ** -0.5, gen)
        for i in range(n_p):
            m.register_probe(i, narrow[i], bias[:1], mix.MIX_ACT_SIGMOID)
        for i in range(n_w):
            m.register_probe(first["wide_probes"] + i, wide[i], bias, mix.MIX_ACT_SOFTMAX)
        for i in range(n_s):
            m.register_steer(first["steers"] + i, vectors[i], float(rng.uniform(1.0, 8.0)))
            if case["gated"]:
                m.set_gate(first["steers"] + i, earlier, column=0, threshold=0.5)
        for i in range(n_r):
            m.register_project(first["projects"] + i, vectors[n_s + i], 1.0)
        if case["chain"]:                                                # probe -> steering -> wide probe
            for i in range(n_p):
                m.set_chain(i, first["steers"] + i % n_s)
            for i in range(n_s):
                m.set_chain(first["steers"] + i, first["wide_probes"] + i % n_w)
        contexts.append(m)
    parts = []
    for kind, n in _kind_rows(case).items():
        lengths = _requests(rng, n, -(-n * 4 // max(case["request"], 4)) if case["request"] > 1 else n)
        for i, length in enumerate(lengths):
            head = "probes" if kind == "chain" else kind
            parts.append((int(length), -1 if kind == "plain" else first[head] + i % case[head]))
    token_slot, token_req, req_slot = _lay_out(rng, T, parts)
    s = dict(path="hook", contexts=contexts, hidden=hidden, scores=scores, live=case["live"], graph=None, requests=None, earlier=earlier)
    live = case["live"]
    if case["two_level"]:
        s["requests"] = tuple(torch.from_numpy(a).cuda() for a in (token_req[:live].copy(), req_slot))
    elif case["graph"]:
        s["map"] = torch.from_numpy(token_slot[:live].copy()).pin_memory()
    else:
        s["map"] = torch.from_numpy(token_slot[:live].copy()).cuda()
    _install_map(s)

    def body():
        for layer, m in enumerate(contexts):
            m.apply(hidden[layer], scores[layer])

    s["body"] = body
    if case["graph"]:
        keep = hidden.clone()
        s["graph"] = _captured(body)
        hidden.copy_(keep)
    return s


def _install_map(s):
    for m in s["contexts"]:
        if s["requests"] is not None:
            m.set_request_map(s["requests"][0], s["requests"][1], s["live"])
        else:
            m.set_slot_map(s["map"], s["live"])


ACTS = {"relu": mix.MIX_SAE_RELU, "jumprelu": mix.MIX_SAE_JUMPRELU, "topk": mix.MIX_SAE_TOPK}


def _dictionary(gen, d, S, act, error, weights):
    """An SAE weight set.  W_enc ~ N(0, 1/d), decoder rows of unit length, biases around -0.1; the dictionaries that
    replace the residual are sparse (about one feature in 256 fires), those that only edit need not be."""
    scale = theta = None
    if weights == "bf16":
        W_enc = _normal((S, d), d ** -0.5, gen)
    else:
        W_enc, scale = torch.empty((S, d), dtype=torch.uint8, device="cuda"), torch.empty(S, device="cuda")
        for r in range(0, S, 16384):
            x = _normal((min(16384, S - r), d), d ** -0.5, gen, torch.float32)
            scale[r:r + 16384] = x.abs().amax(dim=1) / 448.0
            W_enc[r:r + 16384] = (x / scale[r:r + 16384, None]).to(torch.float8_e4m3fn).view(torch.uint8)
    W_dec = _normal((S, d), d ** -0.5, gen)
    b_enc = _normal((S,), 0.02, gen, torch.float32) - 0.1
    if act == "jumprelu":
        lo, hi = (0.05, 0.3) if error else (2.3, 2.8)
        theta = torch.rand(S, generator=gen, device="cuda") * (hi - lo) + lo
    elif act == "relu" and not error:
        b_enc -= 2.5
    return dict(W_enc=W_enc, b_enc=b_enc, W_dec=W_dec, theta=theta, w_scale=scale)


def _firing(row, w, n):
    """n features with the largest pre-activations on a row."""
    W = w["W_enc"]
    z = torch.empty(W.shape[0], device="cuda")
    for r in range(0, W.shape[0], 32768):
        part = W[r:r + 32768]
        if part.dtype == torch.uint8:
            part = part.view(torch.float8_e4m3fn).to(torch.bfloat16)
        z[r:r + 32768] = (part @ row).float()
    if w["w_scale"] is not None:
        z *= w["w_scale"]
    return torch.topk(z + w["b_enc"], n).indices


def _edits(rng, S, firing):
    """EDITS features, half of them firing ones; the first half of the list is set to a value, the second switched off."""
    some = rng.permutation(firing)[:EDITS // 2]
    idx = np.unique(np.concatenate([some, rng.integers(0, S, 4 * EDITS)]), return_index=True)
    idx = np.concatenate([some, rng.integers(0, S, 4 * EDITS)])[np.sort(idx[1])][:EDITS].astype(np.int32)
    rng.shuffle(idx)
    mode = np.where(np.arange(EDITS) < EDITS // 2, mix.MIX_EDIT_CLAMP, mix.MIX_EDIT_ABLATE).astype(np.uint8)
    return idx, np.where(mode == mix.MIX_EDIT_CLAMP, rng.uniform(2.0, 8.0, EDITS), 0.0).astype(np.float32), mode


def _prepare_sae(case, seed):
    gen, rng = _state(case, seed)
    d, S, T, G, C = case["d"], case["d_sae"], case["T"], case["sets"], case["classes"]
    fresh = _normal((T, d), 1.0, gen)
    hidden = fresh.clone()
    rows = _kind_rows(case)
    n_p, n_s = case["probes"], case["steers"]
    lengths = _requests(rng, rows["sae"], case["requests"])
    slots = len(lengths)                                                 # one app per request
    flags = {"bf16": 0, "fp8": mix.MIX_FLAG_FP8_W_ENC, "fp8_input": mix.MIX_FLAG_FP8_W_ENC | mix.MIX_FLAG_FP8_ACT}[case["weights"]]
    m = mix.Mix(d_model=d, T_max=T, n_slots_max=n_p + n_s + slots, n_groups_max=G, C_max=C, k_max=case["k"], r_max=EDITS,
                d_sae_max=S, flags=flags | (mix.MIX_FLAG_RETILE_W_ENC if case["tiled"] else 0))
    sets = [_dictionary(gen, d, S, case["act"], case["error"], case["weights"]) for _ in range(G)]
    for g, w in enumerate(sets):
        m.register_sae_weights(g, S, ACTS[case["act"]], case["k"], w["W_enc"], w["b_enc"], w["W_dec"], theta=w["theta"], w_scale=w["w_scale"])
    probe_w, bias, vectors = _normal((max(n_p, 1), C, d), d ** -0.5, gen), torch.zeros(C, device="cuda"), _normal((max(n_s, 1), d), d ** -0.5, gen)
    for i in range(n_p):
        m.register_probe(i, probe_w[i], bias, mix.MIX_ACT_SIGMOID if C == 1 else mix.MIX_ACT_SOFTMAX)
    for i in range(n_s):
        m.register_steer(n_p + i, vectors[i], float(rng.uniform(1.0, 8.0)))
    parts = [(int(n), n_p + n_s + i) for i, n in enumerate(lengths)]
    for kind, first, many in (("probes", 0, n_p), ("steers", n_p, n_s), ("plain", -1, 1)):
        if rows.get(kind):
            for i, n in enumerate(_requests(rng, rows[kind], case["requests"])):
                parts.append((int(n), first + i % many if kind != "plain" else -1))
    token_slot = _lay_out(rng, T, parts)[0]
    firing = [_firing(fresh[t], sets[g], max(case["k"], 32)) for g in range(G) for t in [int(np.argmax(token_slot == n_p + n_s + g))]]
    firing = torch.stack(firing).cpu().numpy()
    for i in range(slots):
        idx, val, mode = _edits(rng, S, firing[i % G])
        m.register_sae_app(n_p + n_s + i, i % G, idx, val, mode, case["error"])
    s = dict(path="sae", contexts=[m], hidden=hidden, fresh=fresh, scores=None, live=case["live"], graph=None, requests=None, sets=sets,
             probe_w=probe_w, readout=None)
    if n_p:
        s["scores"] = torch.zeros((T, C), dtype=torch.float32, device="cuda")
    if case["readout"]:
        s["readout"] = (torch.zeros((T, case["k"]), dtype=torch.int32, device="cuda"), torch.zeros((T, case["k"]), device="cuda"))
        m.set_feature_out(*s["readout"])
    token_slot = torch.from_numpy(token_slot[:case["live"]].copy())
    s["map"] = token_slot.pin_memory() if case["graph"] else token_slot.cuda()
    _install_map(s)

    def body():
        hidden.copy_(fresh)
        m.apply(hidden, s["scores"])

    s["body"] = body
    if case["graph"]:
        s["graph"] = _captured(body)
    return s


def _prepare_static(case, seed):
    gen, rng = _state(case, seed)
    d, S, k = case["d"], case["d_sae"], case["k"]
    fresh = _normal((case["rows"], d), 1.0, gen)
    w = _dictionary(gen, d, S, case["act"], case["error"], "bf16")
    idx, val, mode = _edits(rng, S, _firing(fresh[0], w, 32).cpu().numpy())
    s = dict(path="static", hidden=fresh.clone(), fresh=fresh, w=w, act=ACTS[case["act"]], d_sae=S, k=k, edits=(idx, val, mode), error=case["error"],
             readout=None)
    if k:
        s["readout"] = (torch.zeros((case["rows"], k), dtype=torch.int32, device="cuda"), torch.zeros((case["rows"], k), device="cuda"))
    return s


def prepare(case, seed):
    return {"hook": _prepare_hook, "sae": _prepare_sae, "static": _prepare_static}[case["path"]](case, seed)


def run(state):
    s = state
    if s["path"] == "static":
        s["hidden"].copy_(s["fresh"])
        w, (idx, val, mode), out = s["w"], s["edits"], s["readout"] or (None, None)
        mix.sae_apply_static(s["hidden"], s["d_sae"], s["act"], s["k"], w["W_enc"], w["b_enc"], w["W_dec"], idx, val, mode, s["error"],
                             theta=w["theta"], topk_idx=out[0], topk_val=out[1])
        return {"hidden": s["hidden"], "features": s["readout"]}
    _install_map(s)
    if s["graph"] is not None:
        s["graph"].replay()
    else:
        s["body"]()
    if s["path"] == "hook":
        return {"hidden": s["hidden"], "scores": s["scores"]}
    return {"hidden": s["hidden"], "scores": s["scores"], "features": s["readout"]}
