"""GPU: slot chains (several apps applied in order to one row in one mix_apply) against the oracle and,
bit for bit, against the same apps applied by separate calls."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import mi_hook as O

from parity import CANARY_F32, CANARY_I32, HIDDEN_TOL_FRAC, TOPK_TIE_TOL, run_gpu

pytestmark = pytest.mark.gpu
DEV = "cuda"
SCORE_TOL = 2e-3        # a probe behind a write inherits the +-1 bf16 ulp the written row may differ by


def _mixlib():
    import paper_2607_22595_b200 as mixlib
    return mixlib


def check_chain_parity(wh, out, scale_with_output=False, expect_status=0):
    ref = O.apply_chain_hook(wh)
    hmax = float(np.abs(O.bf16_to_f64(wh.hidden)).max())
    if scale_with_output:      # an app's output may dwarf the hidden state (see parity.check_parity)
        hmax = max([hmax] + [float(np.abs(ref.y[t]).max()) for t in range(wh.T_max) if ref.modified[t]])
    sb = out["scores"].view(np.uint32)
    redo = {}
    for t in range(wh.T_max):
        if t in ref.topk:                         # TopK ids: equal up to near-ties at the k-th value
            K_ref, k = ref.topk[t], len(ref.topk[t])
            K_gpu = out["topk_idx"][t, :k].astype(np.int64)
            if set(K_gpu.tolist()) != set(K_ref.tolist()):
                redo[t] = K_gpu
    if redo:
        ref2 = O.apply_chain_hook(wh, list(redo), topk_override=redo)
        for t in redo:
            assert np.abs(ref2.y[t] - ref.y[t]).max() <= 10 * TOPK_TIE_TOL * max(1.0, hmax), "row %d: not a near-tie" % t
            ref.y[t], ref.n_active[t] = ref2.y[t], ref2.n_active[t]
    n_mod = n_scores = 0
    for t in range(wh.T_max):
        if not ref.modified[t]:
            assert np.array_equal(out["hidden"][t], wh.hidden[t]), "row %d must be bit-identical" % t
        else:
            err = np.abs(O.bf16_to_f64(out["hidden"][t]) - ref.y[t]).max()
            assert err <= HIDDEN_TOL_FRAC * hmax, "row %d hidden off by %g" % (t, err)
            n_mod += 1
        cols = ref.scores[t]
        for c in range(out["scores"].shape[1]):
            if c in cols:
                got = float(out["scores"][t, c])
                assert abs(got - cols[c]) <= SCORE_TOL * max(1.0, abs(cols[c])), "row %d col %d: %g vs %g" % (t, c, got, cols[c])
                n_scores += 1
            else:
                assert sb[t, c] == CANARY_F32, "row %d col %d was written" % (t, c)
        if t in ref.n_active and t in ref.topk:
            assert int(out["n_active"][t]) == ref.n_active[t]
        elif t not in ref.n_active:
            assert int(out["n_active"][t]) == int(CANARY_I32)
    if expect_status is not None:
        assert out["status"] == expect_status
    return dict(modified=n_mod, scores=n_scores, swaps=len(redo))


@pytest.mark.parametrize("graph", [False, True])
def test_chained_workload_matches_oracle(graph):
    w = W.make_chained(DEV)
    out = run_gpu(w, flags=_mixlib().MIX_FLAG_SLOT_CHAINS, graph=graph)
    st = check_chain_parity(W.host(w), out)
    assert st["modified"] > 150 and st["scores"] > 300


def test_chained_large_batch_and_conditional_graph():
    # T_max above the one-CTA-per-row limit of the unchained kernels; SAE chain inside a graph IF node
    w = W.make_chained(DEV, T=2600, d=320, d_sae=1024, k=8, C=7)
    out = run_gpu(w, flags=_mixlib().MIX_FLAG_SLOT_CHAINS, graph=True, conditional=True)
    check_chain_parity(W.host(w), out)


def test_chain_equals_separate_calls_bit_for_bit():
    """chain 0 -> 1 -> 2 -> 3 in one call == four contexts, one app each, applied one after the other."""
    mixlib = _mixlib()
    w = W.make_chained(DEV)
    slot = np.where(np.arange(w.T_max) % 3 == 0, -1, 0).astype(np.int32)       # two thirds of the rows start chain 0
    wc = W.Workload("c", w.d_model, w.T_max, w.T_max, w.hidden, slot, w.apps, w.groups, w.n_slots_max, w.n_groups_max,
                    w.C_max, w.k_max, w.r_max, w.d_sae_max, chains=w.chains)
    a = run_gpu(wc, flags=mixlib.MIX_FLAG_SLOT_CHAINS)
    h = w.hidden.clone()
    C = w.C_max
    scores = torch.from_numpy(np.full((w.T_max, C), CANARY_F32, dtype=np.uint32).view(np.float32)).cuda()
    col = 0
    for s in O.chain_slots(W.host(wc), 0):
        app = w.apps[s]
        one = W.Workload("one", w.d_model, w.T_max, w.T_max, h, slot.copy(), {0: app},
                         w.groups if app.kind == W.KIND_SAE else {}, n_slots_max=1,
                         n_groups_max=w.n_groups_max if app.kind == W.KIND_SAE else 0, C_max=C, k_max=w.k_max,
                         r_max=w.r_max, d_sae_max=w.d_sae_max)
        m = W.make_context(mixlib.Mix, one)
        sc = torch.zeros((w.T_max, C), dtype=torch.float32, device=DEV)
        m.apply(h, sc)
        torch.cuda.synchronize()
        if app.kind == W.KIND_PROBE:
            n = app.W.shape[0]
            rows = torch.from_numpy(slot == 0).cuda()
            scores[rows, col:col + n] = sc[rows, :n]
            col += n
        assert m.get_status() == 0
        m.destroy()
    assert np.array_equal(a["hidden"], W.bits(h))
    got, want = a["scores"], scores.cpu().numpy()
    assert np.array_equal(got.view(np.uint32) == CANARY_F32, want.view(np.uint32) == CANARY_F32)
    live = want.view(np.uint32) != CANARY_F32
    # the probes run in different kernels (different summation order): equal to rounding, not bitwise
    assert np.abs(got[live] - want[live]).max() <= 1e-5


def test_chain_links_can_change_between_replays():
    mixlib = _mixlib()
    w = W.make_chained(DEV)
    m = W.make_context(mixlib.Mix, w, flags=mixlib.MIX_FLAG_SLOT_CHAINS)
    out = run_gpu(w, mix=m, graph=True)
    check_chain_parity(W.host(w), out)
    # cut chain 0 after its steering app, and let the projection run alone
    m.set_chain(1, -1)
    m.set_chain(4, -1)
    w2 = W.Workload(w.name, w.d_model, w.T_max, w.T_live, w.hidden, w.token_slot, w.apps, w.groups, w.n_slots_max,
                    w.n_groups_max, w.C_max, w.k_max, w.r_max, w.d_sae_max, chains={0: 1, 2: 3, 6: 1})
    out2 = run_gpu(w2, mix=m, graph=True)
    check_chain_parity(W.host(w2), out2)
    m.destroy()


def test_set_chain_error_codes():
    mixlib = _mixlib()
    w = W.make_chained(DEV)
    plain = W.make_context(mixlib.Mix, W.Workload(w.name, w.d_model, w.T_max, w.T_live, w.hidden, w.token_slot, w.apps,
                                                  w.groups, w.n_slots_max, w.n_groups_max, w.C_max, w.k_max, w.r_max,
                                                  w.d_sae_max))
    with pytest.raises(mixlib.MixError) as e:
        plain.set_chain(0, 1)                                  # context created without the flag
    assert e.value.code == -1
    plain.destroy()
    m = W.make_context(mixlib.Mix, w, flags=mixlib.MIX_FLAG_SLOT_CHAINS)
    for bad in [(3, 0),       # an SAE app can only end a chain
                (2, 0),       # cycle 0 -> 1 -> 2 -> 0
                (7, 0),       # 7 -> 0 -> 1 -> 2 -> 3: five apps
                (7, 7)]:      # a slot cannot follow itself
        with pytest.raises(mixlib.MixError) as e:
            m.set_chain(*bad)
        assert e.value.code == -1, bad
    with pytest.raises(mixlib.MixError) as e:
        m.set_chain(0, 99)
    assert e.value.code == -2
    # class columns: chain 0 -> 1 -> 2 writes 1 + 5 of the C_max = 7 columns; a 7-class probe in slot 2
    # is fine on its own but no longer fits behind the probe of slot 0
    g = torch.Generator(device=DEV); g.manual_seed(1)
    wide = torch.randn((7, w.d_model), generator=g, device=DEV).to(torch.bfloat16)
    with pytest.raises(mixlib.MixError) as e:
        m.register_probe(2, wide, None, mixlib.MIX_ACT_SOFTMAX)
    assert e.value.code == -1
    # the failed calls changed nothing: the original chains still give the oracle's result
    out = run_gpu(w, mix=m)
    check_chain_parity(W.host(w), out)
    # unregistering a slot removes the links that point to it
    m.unregister_app(1)
    w4 = W.Workload(w.name, w.d_model, w.T_max, w.T_live, w.hidden, w.token_slot,
                    {s: a for s, a in w.apps.items() if s != 1}, w.groups, w.n_slots_max, w.n_groups_max, w.C_max,
                    w.k_max, w.r_max, w.d_sae_max, chains={2: 3, 4: 5})
    out = run_gpu(w4, mix=m)
    ref_rows_slot1 = np.nonzero(w.token_slot[:w.T_live] == 1)[0]
    assert np.array_equal(out["hidden"][ref_rows_slot1], W.bits(w.hidden)[ref_rows_slot1])
    m.destroy()


# ------------------------------------------------------------------ seeded random chains
def _random_chained_workload(seed):
    from test_gpu_fuzz import random_workload
    w = random_workload(seed)
    rng = np.random.default_rng(seed + 77)
    light = [s for s, a in w.apps.items() if a.kind in (W.KIND_PROBE, W.KIND_STEER, W.KIND_PROJECT)]
    sae = [s for s, a in w.apps.items() if a.kind == W.KIND_SAE]
    rng.shuffle(light)
    chains, C_need = {}, w.C_max
    i = 0
    while i < len(light):
        n = int(rng.integers(1, 4))                                   # 1..3 light apps, then maybe an SAE app
        members = light[i:i + n]
        i += n
        if sae and rng.random() < 0.5:
            members = members + [int(rng.choice(sae))]
        classes = sum(w.apps[s].W.shape[0] for s in members if w.apps[s].kind == W.KIND_PROBE)
        if classes > 64 or len(members) < 2:
            continue
        for a, b in zip(members[:-1], members[1:]):
            chains[a] = b
        C_need = max(C_need, classes)
    return W.Workload(w.name + "c", w.d_model, w.T_max, w.T_live, w.hidden, w.token_slot, w.apps, w.groups, w.n_slots_max,
                      w.n_groups_max, C_need, w.k_max, w.r_max, w.d_sae_max, chains=chains)


@pytest.mark.parametrize("seed", range(16))
def test_random_chains(seed):
    mixlib = _mixlib()
    w = _random_chained_workload(3000 + seed)
    out = run_gpu(w, flags=mixlib.MIX_FLAG_SLOT_CHAINS, graph=bool(seed % 2), conditional=bool(seed % 4 == 1))
    check_chain_parity(W.host(w), out, scale_with_output=True, expect_status=None)
    assert out["status"] & ~mixlib.MIX_STATUS_TOPK_GENERAL == 0


@pytest.mark.parametrize("d", [64, 2048, 2112, 4096, 4160, 6144, 6208, 8192])
@pytest.mark.parametrize("T", [9, 2049])
def test_every_width_chained_and_one_by_one(d, T):
    """The hook kernels of every row width, at the edges of the widths: a probe, a steering vector, a projection and a five-class
    probe on one row, the third and the last gated -- in a chain, and one context each (small contexts; above 2048 rows the
    chain's vectors stay in the caller's memory).  Scores against float64: a sum of n = d products in fp32 is within n 2^-24 of
    the sum of their magnitudes, whatever its order."""
    mixlib = _mixlib()
    g = torch.Generator(device=DEV); g.manual_seed(d + T)
    h = torch.randn((T, d), generator=g, device=DEV).to(torch.bfloat16)
    w1 = (torch.randn((1, d), generator=g, device=DEV) * d ** -0.5).to(torch.bfloat16)
    w5 = (torch.randn((5, d), generator=g, device=DEV) * d ** -0.5).to(torch.bfloat16)
    v, r = [(torch.randn((d,), generator=g, device=DEV) * d ** -0.5).to(torch.bfloat16) for _ in range(2)]
    bias = torch.randn(5, generator=g, device=DEV)
    gate = torch.randn((T, 1), generator=g, device=DEV)
    slots = torch.where(torch.arange(T, device=DEV) % 4 == 3, -1, 0).to(torch.int32)

    def register(m, first, kinds):
        for i, kind in enumerate(kinds):
            s = first + i
            if kind == "probe":
                m.register_probe(s, w1, bias[:1], mixlib.MIX_ACT_NONE)
            elif kind == "steer":
                m.register_steer(s, v, 1.5)
            elif kind == "project":
                m.register_project(s, r, 0.75)
            else:
                m.register_probe(s, w5, bias, mixlib.MIX_ACT_NONE)
            if kind in ("project", "wide"):
                m.set_gate(s, gate, column=0, threshold=0.0)

    kinds = ["probe", "steer", "project", "wide"]
    m = mixlib.Mix(d_model=d, T_max=T, n_slots_max=4, C_max=6, flags=mixlib.MIX_FLAG_SLOT_CHAINS)
    register(m, 0, kinds)
    for s in range(3):
        m.set_chain(s, s + 1)
    m.set_slot_map(slots, T)
    chained, scores = h.clone(), torch.full((T, 6), 7.0, device=DEV)
    m.apply(chained, scores)
    torch.cuda.synchronize()
    assert m.get_status() == 0
    m.destroy()
    hooked = slots == 0
    opened = hooked & (gate[:, 0] >= 0)
    one, one_scores, before = h.clone(), torch.full((T, 6), 7.0, device=DEV), {}
    for kind in kinds:
        before[kind] = one.clone()
        m = mixlib.Mix(d_model=d, T_max=T, n_slots_max=1, C_max=5)
        register(m, 0, [kind])
        m.set_slot_map(slots, T)
        sc = torch.full((T, 5), 7.0, device=DEV)
        m.apply(one, sc)
        torch.cuda.synchronize()
        assert m.get_status() == 0
        m.destroy()
        if kind == "probe":
            one_scores[:, 0] = sc[:, 0]
        elif kind == "wide":
            one_scores[:, 1:] = sc
    if T <= 2048:
        assert torch.equal(chained, one) and torch.equal(scores, one_scores)
    assert torch.equal(chained[~hooked], h[~hooked]) and bool((scores[~hooked] == 7.0).all()) and bool((scores[~opened][:, 1:] == 7.0).all())
    for sc, row in ((scores, chained), (one_scores, before["wide"])):
        for col, Wm, x, rows in ((0, w1, h, hooked), (1, w5, row, opened)):
            x64, W64 = x[rows].double(), Wm.double()
            want = x64 @ W64.T + bias[:Wm.shape[0]].double()
            bound = (d + 1) * 2.0 ** -24 * (x64.abs() @ W64.abs().T + bias[:Wm.shape[0]].abs().double())
            assert bool(((sc[rows, col:col + Wm.shape[0]].double() - want).abs() <= bound).all())
    steered = (h.double() + 1.5 * v.double()).float().to(torch.bfloat16)
    assert bool(((before["project"] - steered)[hooked].abs() <= steered[hooked].abs() * 2.0 ** -7 + 1e-30).all())
    # Rows: the write is one fp32 operation per element whatever the kernel, so where the projection's gate is closed a chained row has the
    # same bits.  Where it is open, the two dot products may differ by twice the bound above, and a bf16 rounding may fall to either side.
    assert torch.equal(chained[hooked & ~opened], one[hooked & ~opened])
    s64, r64 = before["project"][opened].double(), r.double()
    err = 0.75 * (d + 1) * 2.0 ** -24 * (s64.abs() @ r64.abs())[:, None] * r64.abs()
    projected = s64 - 0.75 * (s64 @ r64)[:, None] * r64
    for got in (chained, one):
        diff = (got[opened].double() - projected).abs()
        assert bool((diff <= err + projected.abs() * (2.0 ** -8 + 2.0 ** -22) + 1e-30).all())


# ------------------------------------------------------------------ gates on scores of the same chain
# app: (kind, gate), gate: (column of the chain's scores, comparison, threshold) or None; "p1" and "p2" have one class, "wide" has five
OWN_GATES = {
    "write on a raw logit": [("p1", None), ("steer", (0, W.GATE_GE, 0.0))],
    "write on a softmax class": [("steer", None), ("wide", None), ("project", (3, W.GATE_LT, 0.2))],
    "read on a read on a read": [("p1", None), ("wide", (0, W.GATE_GE, 0.0)), ("p2", (2, W.GATE_GE, 0.2)), ("steer", (6, W.GATE_LT, 0.0))],
    "two on one, the second on its opposite": [("project", None), ("p2", None), ("steer", (0, W.GATE_GE, 0.0)), ("p1", (0, W.GATE_LT, 0.0))],
    "own column and a later probe's": [("p1", (0, W.GATE_GE, 0.0)), ("steer", (2, W.GATE_GE, 0.2)), ("wide", None)],
}
CLASSES = {"p1": 1, "p2": 1, "wide": 5}


@pytest.mark.parametrize("d,T", [(64, 9), (2112, 64), (8192, 21), (320, 2049)])
@pytest.mark.parametrize("form", sorted(OWN_GATES))
def test_a_gate_on_a_score_of_its_own_chain_is_decided_as_separate_calls_decide_it(form, d, T):
    """Separate calls that write the same score buffer decide a gate on what an earlier probe of the chain has just written there,
    or, where that probe's gate was closed or the probe comes later, on what was there before.  The buffer holds the opposite
    decisions to begin with.  Above 2048 rows the kernels add in another order: there a row counts if its gated scores lie
    further from their thresholds than two such sums may differ (n = d products of fp32: 2 n 2^-24 times the sum of their
    magnitudes, which is at most the product of the norms, here below twice the row's), and a written row is equal to one rounding
    to bf16 per write."""
    mixlib = _mixlib()
    apps = OWN_GATES[form]
    C = 7
    g = torch.Generator(device=DEV); g.manual_seed(d + T)
    rnd = lambda *shape: torch.randn(shape, generator=g, device=DEV)
    h = rnd(T, d).to(torch.bfloat16)
    Wt = {k: (rnd(n, d) * d ** -0.5).to(torch.bfloat16) for k, n in CLASSES.items()}
    bias = {k: rnd(n) for k, n in CLASSES.items()}
    v, r = [(rnd(d) * d ** -0.5).to(torch.bfloat16) for _ in range(2)]
    slots = torch.where(torch.arange(T, device=DEV) % 4 == 3, -1, 0).to(torch.int32)

    def register(m, s, kind, gate, buf):
        if kind in CLASSES:
            m.register_probe(s, Wt[kind], bias[kind], mixlib.MIX_ACT_SOFTMAX if kind == "wide" else mixlib.MIX_ACT_NONE)
        elif kind == "steer":
            m.register_steer(s, v, 1.5)
        else:
            m.register_project(s, r, 0.75)
        if gate is not None:
            m.set_gate(s, buf, column=gate[0], cmp=gate[1], threshold=gate[2])

    def buffer(old):              # the scores, and room behind them for a call whose first column is not the buffer's
        flat = torch.zeros((T + 1) * C, device=DEV)
        flat[:T * C] = old.flatten()
        return flat

    def separate(old):
        flat, x, col = buffer(old), h.clone(), 0
        for kind, gate in apps:
            m = mixlib.Mix(d_model=d, T_max=T, n_slots_max=1, C_max=C)
            register(m, 0, kind, gate, flat[:T * C].view(T, C))
            m.set_slot_map(slots, T)
            m.apply(x, flat[col:col + T * C].view(T, C))
            torch.cuda.synchronize()
            assert m.get_status() == 0
            m.destroy()
            col += CLASSES.get(kind, 0)
        return x, flat[:T * C].view(T, C)

    def chained(old, graph):
        flat, x = buffer(old), h.clone()
        scores = flat[:T * C].view(T, C)
        m = mixlib.Mix(d_model=d, T_max=T, n_slots_max=len(apps), C_max=C, flags=mixlib.MIX_FLAG_SLOT_CHAINS)
        for s, (kind, gate) in enumerate(apps):
            register(m, s, kind, gate, scores)
        for s in range(len(apps) - 1):
            m.set_chain(s, s + 1)
        m.set_slot_map(slots, T)
        s = torch.cuda.Stream(); s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            if graph:
                gr = torch.cuda.CUDAGraph()
                with torch.cuda.graph(gr, stream=s):
                    m.apply(x, scores, stream=s)
                gr.replay()
            else:
                m.apply(x, scores, stream=s)
        torch.cuda.synchronize()
        assert m.get_status() == 0
        m.destroy()
        return x, scores

    cuts = {c: t for _, gate in apps if gate is not None for c, _, t in [gate]}
    fresh = separate(torch.full((T, C), 9.0, device=DEV))[1]
    old = 9.0 - fresh
    for c, thr in cuts.items():
        old[:, c] = 2 * thr - fresh[:, c]
    want_x, want_s = separate(old)
    hooked = slots == 0
    if T > 2048:
        near = torch.zeros(T, dtype=torch.bool, device=DEV)
        for c, thr in cuts.items():
            near |= (want_s[:, c] - thr).abs() <= 2 * d * 2.0 ** -24 * 2 * h.float().norm(dim=1)
        assert int(near.sum()) < T // 8
        rows = ~near
    else:
        rows = torch.ones(T, dtype=torch.bool, device=DEV)
    for graph in (False, True):
        x, sc = chained(old, graph)
        if T > 2048:
            diff = (x.float() - want_x.float()).abs()[rows]
            assert bool((diff <= (want_x.float().abs()[rows] + 1.5 * v.float().abs()) * 2.0 ** -7 + 1e-6).all())
            assert bool(((sc - want_s).abs()[rows] <= SCORE_TOL).all())
        else:
            assert torch.equal(x, want_x) and torch.equal(sc, want_s)
        assert torch.equal(x[~hooked], h[~hooked]) and torch.equal(sc[~hooked], old[~hooked])


@pytest.mark.parametrize("T,classes", [(96, 1), (700, 3), (2200, 2)])
def test_an_sae_app_gated_on_a_score_of_its_own_chain(T, classes):
    """The routing kernel, which starts while the chain kernel in front of it still runs, decides the gate on the score that the chain
    has written, as separate calls do.  The buffer holds the opposite decisions; a row's scores share 32 bytes with its neighbours'."""
    mixlib = _mixlib()
    d, S = 256, 512
    g = torch.Generator(device=DEV); g.manual_seed(T)
    h = torch.randn((T, d), generator=g, device=DEV).to(torch.bfloat16)
    sign = torch.where(torch.arange(T, device=DEV) % 2 == 0, 1.0, -1.0)
    Wp = torch.zeros((classes, d), dtype=torch.bfloat16, device=DEV)
    Wp[:, 0] = 1.0
    h[:, 0] = (2.0 * sign).to(torch.bfloat16)                    # the logit: +-2, exactly, in every kernel
    sae = W.make_sae_weights(g, DEV, d, S, W.SAE_RELU)
    slots = torch.where(torch.arange(T, device=DEV) % 5 == 4, -1, 0).to(torch.int32)

    def context(n_slots, groups, flags):
        m = mixlib.Mix(d_model=d, T_max=T, n_slots_max=n_slots, n_groups_max=groups, C_max=classes, k_max=1, r_max=2, d_sae_max=S, flags=flags)
        if groups:
            m.register_sae_weights(0, S, sae.act, 0, sae.W_enc, sae.b_enc, sae.W_dec)
        return m

    def sae_app(m, slot, scores):
        m.register_sae_app(slot, 0, [3, 300], [2.0, -1.5], [0, 0], True)
        m.set_gate(slot, scores, column=classes - 1, threshold=0.0)

    def run(m, x, scores):
        m.set_slot_map(slots, T)
        s = torch.cuda.Stream(); s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            m.apply(x, scores, stream=s)
        torch.cuda.synchronize()
        assert m.get_status() == 0
        m.destroy()

    old = (-2.0 * sign)[:, None].repeat(1, classes)
    want, want_scores = h.clone(), old.clone()
    m = context(1, 0, 0)
    m.register_probe(0, Wp, None, mixlib.MIX_ACT_NONE)
    run(m, want, want_scores)
    m = context(1, 1, 0)
    sae_app(m, 0, want_scores)
    run(m, want, None)
    for _ in range(4):
        x, scores = h.clone(), old.clone()
        m = context(2, 1, mixlib.MIX_FLAG_SLOT_CHAINS)
        m.register_probe(0, Wp, None, mixlib.MIX_ACT_NONE)
        sae_app(m, 1, scores)
        m.set_chain(0, 1)
        run(m, x, scores)
        assert torch.equal(scores, want_scores) and torch.equal(x, want)
    changed = (want != h).any(dim=1)
    assert torch.equal(changed, (slots == 0) & (sign > 0))


@pytest.mark.parametrize("d,T", [(512, 2048), (8192, 700)])
def test_a_gate_on_another_rows_score_of_the_same_call_decides_the_whole_row(d, T):
    """Such a gate may see the score that was there or the one that the call writes, in another block at that moment; either way the
    row is written as a whole, and so are the scores behind the write."""
    mixlib = _mixlib()
    g = torch.Generator(device=DEV); g.manual_seed(d)
    rnd = lambda *shape: torch.randn(shape, generator=g, device=DEV)
    h = rnd(T, d).to(torch.bfloat16)
    w1, w5 = [(rnd(n, d) * d ** -0.5).to(torch.bfloat16) for n in (1, 5)]
    r = (rnd(d) * d ** -0.5).to(torch.bfloat16)
    slots = torch.zeros(T, dtype=torch.int32, device=DEV)
    flat = torch.zeros((T + 1) * 6, device=DEV)             # the call's scores, and the row behind them: row t is gated on row t + 1
    scores, ahead = flat[:T * 6].view(T, 6), flat[6:].view(T, 6)

    def run(old, threshold):
        flat.fill_(old)
        m = mixlib.Mix(d_model=d, T_max=T, n_slots_max=3, C_max=6, flags=mixlib.MIX_FLAG_SLOT_CHAINS)
        m.register_probe(0, w1, None, mixlib.MIX_ACT_NONE)
        m.register_project(1, r, 0.75)
        m.set_gate(1, ahead, column=0, threshold=threshold)
        m.register_probe(2, w5, None, mixlib.MIX_ACT_NONE)
        m.set_chain(0, 1)
        m.set_chain(1, 2)
        m.set_slot_map(slots, T)
        x = h.clone()
        m.apply(x, scores)
        torch.cuda.synchronize()
        assert m.get_status() == 0
        m.destroy()
        return x, scores.clone()

    opened, closed = run(9.0, -1e30), run(9.0, 1e30)
    for old in (-1e9, 1e9, -1e9, 1e9):
        x, sc = run(old, 0.0)
        is_open = (x == opened[0]).all(dim=1) & (sc == opened[1]).all(dim=1)
        is_closed = (x == closed[0]).all(dim=1) & (sc == closed[1]).all(dim=1)
        assert bool((is_open | is_closed).all()) and not bool((is_open & is_closed).any())
