"""Encode tiles narrower than 256 features, panel tiles with few rows, and rows rebuilt from their active features, at the
sizes where the splits change."""
import numpy as np
import pytest
import torch

import workloads as W

from parity import check_parity, run_gpu

pytestmark = pytest.mark.gpu


def _workload(d, S, T, act, add_error, k=24, fp8=None, n_sets=1, b_enc_mean=-0.1, seed=0, extra_topk=False):
    g = torch.Generator(device="cuda"); g.manual_seed(seed + S + T)
    rng = np.random.default_rng(seed)
    hidden = torch.randn((T, d), generator=g, device="cuda").to(torch.bfloat16)
    groups = {i: W.make_sae_weights(g, "cuda", d, S, act, k=k if act == W.SAE_TOPK else 0, theta_range=(0.05, 0.3), b_enc_mean=b_enc_mean,
                                    fp8=fp8 is not None) for i in range(n_sets)}
    if extra_topk:                                            # registered, no rows: the encode runs with eight epilogue warps
        groups[n_sets] = W.make_sae_weights(g, "cuda", d, 256, W.SAE_TOPK, k=4, fp8=fp8 is not None)
    apps = {i: W.SaeApp(i, rng.choice(S, 3, replace=False).astype(np.int32), np.array([4.0, 0.0, 2.0], np.float32),
                        np.array([0, 1, 0], np.uint8), add_error) for i in range(n_sets)}
    token_slot = (np.arange(T) * n_sets // T).astype(np.int32)
    return W.Workload("tiles", d, T, T, hidden, token_slot, apps, groups, n_slots_max=n_sets, n_groups_max=len(groups), C_max=1,
                      k_max=k, r_max=3, d_sae_max=S, fp8_act=fp8 == "input")


# features -> tiles of 256: 4 (width 64), 37 (64: 148 tiles), 38 (128), 74 (128), 75 (256); two sets halve the room
@pytest.mark.parametrize("S,n_sets", [(1024, 1), (37 * 256, 1), (38 * 256, 1), (74 * 256, 1), (75 * 256, 1), (18 * 256, 2), (19 * 256, 2)])
@pytest.mark.parametrize("act", [W.SAE_TOPK, W.SAE_JUMPRELU])
def test_tile_widths(S, n_sets, act):
    w = _workload(128, S, 50, act, True, n_sets=n_sets)
    check_parity(W.host(w), run_gpu(w))


@pytest.mark.parametrize("T", [1, 31, 32, 33, 64, 96, 97, 127, 128, 129, 193, 256, 300])
@pytest.mark.parametrize("fp8", [None, "weights", "input"])
def test_rows_of_a_tile(T, fp8):
    w = _workload(256, 2048, T, W.SAE_TOPK, False, fp8=fp8)
    flags = {None: 0, "weights": 32, "input": 96}[fp8]
    check_parity(W.host(w), run_gpu(w, flags=flags, graph=True, replays=2))


# widths: one vector pass, and a last pass of 32, 64, 96, 128 and 160 vectors
@pytest.mark.parametrize("d", [64, 2048, 2304, 2560, 2816, 3072, 3328])
@pytest.mark.parametrize("act", [W.SAE_RELU, W.SAE_JUMPRELU])
@pytest.mark.parametrize("extra_topk", [False, True])
def test_rebuilt_rows(d, act, extra_topk):
    w = _workload(d, 2048, 20, act, False, b_enc_mean=-1.8, extra_topk=extra_topk)
    check_parity(W.host(w), run_gpu(w))


def test_rebuilt_rows_with_more_active_features_than_a_list_holds():
    w = _workload(320, 4096, 9, W.SAE_RELU, False, b_enc_mean=0.1)
    out = run_gpu(w)
    assert out["n_active"].min() > 1100
    check_parity(W.host(w), out)


def test_rebuilt_rows_on_cta_pairs():
    w = _workload(320, 10240, 256, W.SAE_JUMPRELU, False, b_enc_mean=-2.0)
    check_parity(W.host(w), run_gpu(w))


@pytest.mark.parametrize("rows,d,S,act,k,add_error", [
    (1, 64, 256, W.SAE_TOPK, 1, True), (33, 320, 2304, W.SAE_TOPK, 24, False), (128, 4096, 8192, W.SAE_TOPK, 64, True),
    (7, 128, 8192, W.SAE_TOPK, 128, False), (128, 192, 4096, W.SAE_RELU, 0, True), (50, 2304, 1024, W.SAE_JUMPRELU, 0, False)])
@pytest.mark.parametrize("aligned", [True, False])
def test_allocation_free_call(rows, d, S, act, k, add_error, aligned):
    import paper_2607_22595_b200 as mixlib
    w = _workload(d, S, rows, act, add_error, k=max(k, 1), b_enc_mean=-0.1 if add_error or act == W.SAE_TOPK else -2.0)
    if act == W.SAE_TOPK and k > 64:                          # duplicated encoder rows: ties at the k-th value, the exact fallback
        w.groups[0].W_enc[1::2] = w.groups[0].W_enc[0::2]
        w.groups[0].b_enc[1::2] = w.groups[0].b_enc[0::2]
    if not aligned:
        b = torch.empty(S + 1, device="cuda")
        b[1:] = w.groups[0].b_enc
        w.groups[0].b_enc = b[1:]
    sw, app, h = w.groups[0], w.apps[0], w.hidden.clone()
    idx = torch.full((rows, max(k, 1)), -559038737, dtype=torch.int32, device="cuda")
    val = torch.from_numpy(np.full((rows, max(k, 1)), 0x7FC0DEAD, dtype=np.uint32).view(np.float32)).cuda()
    for _ in range(2):                                        # the second call finds the first one's scratch
        h.copy_(w.hidden)
        mixlib.sae_apply_static(h, S, act, k, sw.W_enc, sw.b_enc, sw.W_dec, app.edit_idx, app.edit_val, app.edit_mode, add_error,
                                theta=sw.theta, topk_idx=idx if k else None, topk_val=val if k else None)
    from oracle import mi_hook as O
    wh = W.host(w)
    ref = O.apply_hook(wh, list(range(rows)), keep_z=True)
    if k and k <= 64:
        for t in range(rows):
            z = ref.z[t]
            picked = idx[t].cpu().numpy()
            assert len(set(picked.tolist())) == k and z[picked].min() >= np.sort(z)[-k] - 1e-3
            assert np.abs(val[t].cpu().numpy() - z[picked]).max() <= 1e-3
    elif k:
        assert (idx.cpu().numpy()[:, 0] % 2 == 0).all()       # of two equal ones the lower id comes first
    hid, hmax = O.bf16_to_f64(W.bits(h)), np.abs(O.bf16_to_f64(wh.hidden)).max()
    assert max(np.abs(hid[t] - ref.y[t]).max() for t in range(rows)) <= 1e-2 * hmax


# rows of one CTA of the front kernel: 256; from 1025 rows on its CTAs exchange their counts
@pytest.mark.parametrize("T", [255, 257, 1023, 1024, 1025])
def test_rows_scattered_over_sets(T):
    w = _workload(64, 256, T, W.SAE_TOPK, True, k=4, n_sets=3)
    w.token_slot[:] = np.random.default_rng(T).integers(-1, 3, size=T)
    w.token_slot[: T // 2] = np.minimum(w.token_slot[: T // 2], 0)
    check_parity(W.host(w), run_gpu(w))


# pre-activations stored for the edited features alone (no read-out) against all of them: the same rows, bit for bit
@pytest.mark.parametrize("T", [1, 33, 130, 700])
@pytest.mark.parametrize("n_edit", [1, 9, 64])
@pytest.mark.parametrize("act", [W.SAE_RELU, W.SAE_JUMPRELU])
@pytest.mark.parametrize("fp8", [None, "weights", "input"])
def test_only_edited_features_stored(T, n_edit, act, fp8):
    S = 2048
    w = _workload(128, S, T, act, True, fp8=fp8, extra_topk=T == 33)
    rng = np.random.default_rng(T + n_edit)
    edges = np.array([0, 3, 4, 31, 32, 63, 64, 127, 128, 255, 256, S - 4, S - 1], np.int32)
    for slot in range(5):                                     # the last one replaces the residual
        idx = np.concatenate([rng.choice(edges, min(n_edit, 9)), rng.integers(0, S, max(n_edit - 9, 0))]).astype(np.int32)
        w.apps[slot] = W.SaeApp(0, idx, rng.normal(size=n_edit).astype(np.float32), rng.integers(0, 2, n_edit).astype(np.uint8), slot < 4)
    w.n_slots_max, w.r_max = 5, n_edit
    w.token_slot[:] = rng.integers(-1, 5, size=T) if T > 1 else 0
    flags = {None: 0, "weights": 32, "input": 96}[fp8]
    full = run_gpu(w, flags=flags)
    check_parity(W.host(w), full)
    sparse = run_gpu(w, flags=flags, feature_out=False, replays=2, graph=True)
    assert np.array_equal(full["hidden"], sparse["hidden"])
    assert sparse["status"] == 0


def test_an_edit_list_that_another_stream_replaces_between_encode_and_decode():
    """The call is captured, and a host function put between its encode and its tail: while that runs, another stream replaces
    the edit list.  What the encode did not know to store is left out of this call; the next one applies the whole list."""
    import ctypes
    import threading

    from cuda.bindings import runtime as rt

    import paper_2607_22595_b200 as mixlib

    def ok(result):
        assert int(result[0]) == 0, result
        return result[1:]

    S, T = 2048, 40
    w = _workload(128, S, T, W.SAE_RELU, True)
    w.apps[0] = W.SaeApp(0, np.array([8, 20], np.int32), np.array([5.0, 2.0], np.float32), np.array([0, 0], np.uint8), True)
    w.token_slot[:] = 0
    replaced = np.array([9, 700], np.int32), np.array([3.0, -4.0], np.float32), np.array([0, 0], np.uint8)

    def expected(idx, val, mode):
        w.apps[0] = W.SaeApp(0, idx, val, mode, True)
        return run_gpu(w, feature_out=False)["hidden"]

    old_mask = mixlib.set_pdl_mask(0)                         # (plain edges: a programmatic one cannot be cut)
    try:
        m = W.make_context(mixlib.Mix, w)
        h = w.hidden.clone()
        m.apply(h)
        h.copy_(w.hidden)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph):
            m.apply(h)
    finally:
        mixlib.set_pdl_mask(old_mask)
    raw = rt.cudaGraph_t(init_value=graph.raw_cuda_graph())
    n = ok(rt.cudaGraphGetEdges(raw))[-1]
    start, end = ok(rt.cudaGraphGetEdges(raw, n))[:2]
    after = {int(a): b for a, b in zip(start[:n], end[:n])}
    node = next(a for a in start[:n] if int(a) not in {int(b) for b in end[:n]})
    chain = [node]
    while int(chain[-1]) in after:
        chain.append(after[int(chain[-1])])
    assert len(chain) == 6                                    # hook, front, encode, tail and the two of the fallback
    encode, tail = chain[2], chain[3]
    reached, done = threading.Event(), threading.Event()

    @ctypes.CFUNCTYPE(None, ctypes.c_void_p)
    def pause(_):
        reached.set()
        done.wait(2.0)

    params = rt.cudaHostNodeParams()
    params.fn = rt.cudaHostFn_t(init_value=ctypes.cast(pause, ctypes.c_void_p).value)
    between = ok(rt.cudaGraphAddHostNode(raw, [encode], 1, params))[0]
    ok(rt.cudaGraphRemoveDependencies(raw, [encode], [tail], 1))
    ok(rt.cudaGraphAddDependencies(raw, [between], [tail], 1))
    graph.instantiate()

    other = torch.cuda.Stream()
    graph.replay()
    assert reached.wait(10.0)
    m.update_sae_edits(0, *replaced, stream=other)
    other.synchronize()
    assert not done.is_set()
    done.set()
    torch.cuda.synchronize()
    # feature 9 shares a group of four with the edited feature 8, so its value was stored; feature 700's was not
    during = W.bits(h)
    assert np.array_equal(during, expected(*[x[:1] for x in replaced]))
    assert not np.array_equal(during, expected(*replaced))
    h.copy_(w.hidden)
    m.apply(h)
    assert np.array_equal(W.bits(h), expected(*replaced))
    assert m.get_status() == 0
    torch.cuda.synchronize()
    del graph
    m.destroy()


def test_a_set_that_another_stream_is_about_to_remove():
    """The host's table has lost the TopK set, the device's has not: rows that need the exact fallback still get it."""
    import paper_2607_22595_b200 as mixlib
    w = _workload(128, 2048, 30, W.SAE_TOPK, False)
    w.groups[0].W_enc[256:512] = w.groups[0].W_enc[256].clone()          # 256 equal features: no tile's eight candidates can tell
    w.groups[0].b_enc[256:512] = 3.0
    want = run_gpu(w, feature_out=False)
    check_parity(W.host(w), want, check_features=False)
    assert not np.array_equal(want["hidden"], W.bits(w.hidden))
    m = W.make_context(mixlib.Mix, w)
    h = w.hidden.clone()
    late, now = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(late):
        torch.cuda._sleep(100_000_000)                        # 50 ms
    m.unregister_sae_weights(0, stream=late)
    m.apply(h, stream=now)
    now.synchronize()
    assert not late.query()                                   # the set is still there
    assert np.array_equal(W.bits(h), want["hidden"])
    torch.cuda.synchronize()
    m.destroy()


def test_padding_rows_of_a_tile_are_zero():
    """Rows of the panel behind a set's own are zeros, whatever a longer call before had there (seen through the CUDA-core
    encode, which writes the pre-activations of whole tiles)."""
    from cuda.bindings import runtime as rt

    import paper_2607_22595_b200 as mixlib
    S, T = 512, 200
    w = _workload(128, S, T, W.SAE_RELU, True)
    w.token_slot[:] = 0
    m = W.make_context(mixlib.Mix, w, flags=mixlib.MIX_FLAG_ENCODE_SIMT)
    h = w.hidden.clone()
    m.apply(h)
    m.set_slot_map(w.token_slot, 5)
    m.apply(h)
    torch.cuda.synchronize()
    _, z_ptr, ld, _ = m.debug_workspace()
    z = np.empty((128, ld), np.float32)
    assert int(rt.cudaMemcpy(z.ctypes.data, z_ptr, z.nbytes, rt.cudaMemcpyKind.cudaMemcpyDeviceToHost)[0]) == 0
    b = w.groups[0].b_enc.cpu().numpy()
    assert np.array_equal(z[5:, :S], np.broadcast_to(b, (123, S)))
    assert not np.array_equal(z[:5, :S], np.broadcast_to(b, (5, S)))
    m.destroy()


# k-blocks of a tile with every remainder of the producers' turns, several tiles a CTA (S / 256 = 300 tiles and more), on the rings
# of three to six stages that full tiles have: bf16 on single CTAs (100 rows) and pairs (200), and both 8-bit forms
@pytest.mark.parametrize("k_blocks", [1, 2, 3, 4, 5, 7, 8])
@pytest.mark.parametrize("T", [100, 200])
@pytest.mark.parametrize("fp8", [None, "weights", "input"])
def test_turns_of_the_producers(k_blocks, T, fp8):
    w = _workload(k_blocks * (64 if fp8 is None else 128), 300 * 256, T, W.SAE_TOPK, False, fp8=fp8)
    sample = np.random.default_rng(k_blocks).choice(T, 6, replace=False)
    out = run_gpu(w, flags={None: 0, "weights": 32, "input": 96}[fp8], graph=True, replays=2)
    check_parity(W.host(w), out, rows=np.sort(sample))


# rows for the panel boxes of 16 ... 128 rows, beside a set whose tiles have other rows
@pytest.mark.parametrize("T", [1, 15, 16, 17, 48, 65, 95, 98, 112])
@pytest.mark.parametrize("act", [W.SAE_TOPK, W.SAE_JUMPRELU])
def test_panel_boxes(T, act):
    w = _workload(320, 2048, T + 5, act, True, n_sets=2)
    w.token_slot[:] = np.minimum(np.arange(T + 5) // T, 1)
    check_parity(W.host(w), run_gpu(w, graph=True, replays=2))


@pytest.mark.parametrize("S", [1024, 128 * 256, 400 * 256])     # narrow tiles, one wave of full ones, waves with a bound in force
@pytest.mark.parametrize("kind", ["zeros", "steps", "clustered"])
def test_topk_of_values_that_tie_or_crowd(S, kind):
    """Pre-activations that equal one another at and around a tile's 8th value, many zeros among them, and winners that crowd
    in a few tiles (more than 8 of a tile, in one half of it or in both): ids and values must be the exact TopK, of equal values
    the lower id."""
    d, T, k = 64, 40, 24
    w = _workload(d, S, T, W.SAE_TOPK, False, k=k)
    g = torch.Generator(device="cuda"); g.manual_seed(S)
    sw = w.groups[0]
    sw.W_enc[:] = 0                                             # z[t, j] = hidden[t, j % 8] * level[j] + bias[j], all exact
    cols = torch.arange(S, device="cuda")
    if kind == "zeros":
        level = torch.where(torch.rand(S, generator=g, device="cuda") < 0.004, 1.0, 0.0)
        sw.b_enc[:] = 0
    elif kind == "steps":
        level = torch.randint(-2, 3, (S,), generator=g, device="cuda").float()
        sw.b_enc[:] = 0.5
    else:
        level = torch.where((cols % 256 >= 120) & (cols % 256 < 136) & (cols // 256 % 3 == 0), 1.0, -1.0)
        sw.b_enc[:] = (cols % 5).float() * 0.25
    sw.W_enc[cols, cols % 8] = level.to(torch.bfloat16)
    w.hidden[:] = torch.randint(1, 4, (T, d), generator=g, device="cuda").to(torch.bfloat16)
    out = run_gpu(w, graph=True, replays=2)
    z = (w.hidden.float() @ sw.W_enc.float().T + sw.b_enc).cpu().numpy()
    for t in range(T):
        want = np.lexsort((np.arange(S), -z[t]))[:k]
        assert np.array_equal(out["topk_idx"][t, :k], want), (t, out["topk_idx"][t, :k], want)
        assert np.array_equal(out["topk_val"][t, :k], z[t][want])
