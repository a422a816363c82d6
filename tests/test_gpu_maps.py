"""The slot map from every place it can come from, shrinking and growing from call to call: rows behind the live ones
pass through whatever the maps before had there."""
import ctypes

import numpy as np
import pytest
import torch

import workloads as W
from paper_2607_22595_b200 import Mix, MixError

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("with_sae", [False, True])
@pytest.mark.parametrize("source", ["device", "pinned", "pageable", "numpy", "requests_device", "requests_host"])
@pytest.mark.parametrize("T", [5, 896, 897, 3000])
def test_maps_of_changing_length(T, source, with_sae):
    d = 64
    m = Mix(d_model=d, T_max=T, n_slots_max=2, n_groups_max=int(with_sae), d_sae_max=256 if with_sae else 0)
    v = torch.ones(d, device="cuda", dtype=torch.bfloat16)
    m.register_steer(0, v, 1.0)
    m.register_steer(1, v, 2.0)
    rng = np.random.default_rng(T)
    for live in (T, T // 2, 0, 1, T - 1, T):
        token_slot = rng.integers(-1, 2, size=live).astype(np.int32)
        if source.startswith("requests"):
            req, slots = np.arange(live, dtype=np.int32), token_slot
            if source == "requests_device":
                m.set_request_map(torch.from_numpy(req).cuda(), torch.from_numpy(slots).cuda(), live)
            else:
                m.set_request_map(req, slots, live)
        else:
            src = {"device": lambda x: torch.from_numpy(x).cuda(), "pinned": lambda x: torch.from_numpy(x).pin_memory(),
                   "pageable": torch.from_numpy, "numpy": lambda x: x}[source](token_slot)
            m.set_slot_map(src, live)
        h = torch.zeros((T, d), device="cuda", dtype=torch.bfloat16)
        m.apply(h)
        m.apply(h)                                   # directly behind: the second call sees the same map
        want = np.zeros(T, dtype=np.float32)
        want[:live] = 2.0 * (token_slot + 1)
        assert np.array_equal(h.float().cpu().numpy(), np.repeat(want[:, None], d, 1)), live
    assert m.get_status() == 0
    m.destroy()


@pytest.mark.parametrize("live", [1, 256, 257, 896, 897])
@pytest.mark.parametrize("before", [0, 1000])
def test_pinned_maps_in_a_graph_and_in_eager_calls(live, before):
    d, T = 64, 1000
    ms, pins, hs = [], [], []
    for _ in range(2):
        m = Mix(d_model=d, T_max=T, n_slots_max=2)
        for slot in range(2):
            m.register_steer(slot, torch.ones(d, device="cuda", dtype=torch.bfloat16), slot + 1.0)
        m.set_slot_map(torch.zeros(before, dtype=torch.int32, device="cuda"), before)
        ms.append(m)
        pins.append(torch.full((live,), -1, dtype=torch.int32).pin_memory())
        hs.append(torch.zeros((T, d), device="cuda", dtype=torch.bfloat16))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for m, pin, h in zip(ms, pins, hs):
            m.set_slot_map(pin, live)
            m.apply(h)
    for replay in range(3):
        for i, (pin, h) in enumerate(zip(pins, hs)):
            pin.copy_(torch.from_numpy(np.random.default_rng(2 * replay + i).integers(-1, 2, size=live).astype(np.int32)))
            h.zero_()
        torch.cuda.synchronize()
        if replay < 2:
            graph.replay()
        else:
            for m, pin, h in zip(ms, pins, hs):
                m.set_slot_map(pin, live)
                m.apply(h)
        torch.cuda.synchronize()
        for pin, h in zip(pins, hs):
            want = np.zeros(T, dtype=np.float32)
            want[:live] = pin.numpy() + 1.0
            assert np.array_equal(h.float().cpu().numpy(), np.repeat(want[:, None], d, 1)), replay
    assert all(m.get_status() == 0 for m in ms)
    del graph
    for m in ms:
        m.destroy()


def _refused_install(m, src, n):
    """An install on the legacy stream while a blocking stream is being captured: CUDA refuses it, nothing is enqueued."""
    from cuda.bindings import runtime as rt

    err, blocking = rt.cudaStreamCreate()
    assert int(err) == 0
    assert int(rt.cudaStreamBeginCapture(blocking, rt.cudaStreamCaptureMode.cudaStreamCaptureModeThreadLocal)[0]) == 0
    with pytest.raises(MixError):
        m.set_slot_map(src, n, stream=0)
    err, graph = rt.cudaStreamEndCapture(blocking)   # (the failed call has invalidated it)
    if int(err) == 0:
        rt.cudaGraphDestroy(graph)
    rt.cudaStreamDestroy(blocking)
    rt.cudaGetLastError()


def test_an_error_that_a_call_returned_is_not_reported_again():
    m = Mix(d_model=64, T_max=3000, n_slots_max=1)
    src = torch.zeros(5, dtype=torch.int32, device="cuda")
    h = torch.ones((3000, 64), device="cuda", dtype=torch.bfloat16)
    _refused_install(m, src, 5)
    m.apply(h)                                       # (checks the runtime's record behind its launch)
    assert bool((h == 1).all())                      # (so does torch)
    m.destroy()


@pytest.mark.parametrize("with_sae", [False, True])
@pytest.mark.parametrize("source", ["device", "pinned", "pageable", "requests_device"])
def test_a_captured_map_among_eager_ones(source, with_sae):
    d, T = 64, 1000
    m = Mix(d_model=d, T_max=T, n_slots_max=2, n_groups_max=int(with_sae), d_sae_max=256 if with_sae else 0)
    for slot in range(2):
        m.register_steer(slot, torch.ones(d, device="cuda", dtype=torch.bfloat16), slot + 1.0)
    h = torch.zeros((T, d), device="cuda", dtype=torch.bfloat16)

    def make(slots):
        x = torch.from_numpy(np.ascontiguousarray(slots, dtype=np.int32))
        return {"device": lambda: x.cuda(), "pinned": x.pin_memory, "pageable": lambda: x, "requests_device": lambda: x.cuda()}[source]()

    def install(src, n):
        if source == "requests_device":
            m.set_request_map(every, src, n)
        else:
            m.set_slot_map(src, n)

    def check(slots, note):
        want = np.zeros(T, dtype=np.float32)
        want[:len(slots)] = np.asarray(slots) + 1.0
        assert np.array_equal(h.float().cpu().numpy(), np.repeat(want[:, None], d, 1)), note
        h.zero_()

    every = torch.arange(T, dtype=torch.int32, device="cuda")
    rng = np.random.default_rng(5)
    long, short, ten = rng.integers(-1, 2, T), rng.integers(-1, 2, 20), rng.integers(-1, 2, 10)
    src_long, src_short, src_ten = make(long), make(short), make(ten)
    install(src_long, T)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        install(src_ten, 10)
        m.apply(h)
    install(src_short, 20)                           # captured, not replayed: the long map is the one in front
    m.apply(h)
    check(short, "behind a capture")
    install(src_long, T)
    m.apply(h)
    check(long, "long")
    graph.replay()                                   # the captured map is shorter than the one installed meanwhile
    check(ten, "replayed behind a longer map")
    src_ten.copy_(torch.from_numpy(ten[::-1].copy().astype(np.int32)))
    torch.cuda.synchronize()
    graph.replay()
    check(ten[::-1], "replayed with another map in its source")
    install(src_long, T)
    install(src_short, 20)
    m.apply(h)
    check(short, "eager behind eager")
    assert m.get_status() == 0
    del graph
    m.destroy()


def test_an_install_that_fails_leaves_the_rows_of_the_map_before_to_the_next_one():
    d, T = 64, 500
    m = Mix(d_model=d, T_max=T, n_slots_max=1)
    m.register_steer(0, torch.ones(d, device="cuda", dtype=torch.bfloat16), 1.0)
    src = torch.zeros(T, dtype=torch.int32, device="cuda")
    m.set_slot_map(src, T)
    torch.cuda.synchronize()
    _refused_install(m, src, 5)
    h = torch.zeros((T, d), device="cuda", dtype=torch.bfloat16)
    m.set_slot_map(src, 20)
    m.apply(h)
    assert int((h[:, 0] != 0).sum()) == 20
    m.destroy()


# up to three hooks take a short pinned map by a copy, four by the kernel
@pytest.mark.parametrize("hooks", [1, 3, 4])
@pytest.mark.parametrize("live", [1, 255, 256, 257])
def test_pinned_maps_of_a_row_of_hooks(hooks, live):
    d, T = 64, 300
    ms, hs = [], []
    for _ in range(hooks):
        m = Mix(d_model=d, T_max=T, n_slots_max=2)
        for slot in range(2):
            m.register_steer(slot, torch.ones(d, device="cuda", dtype=torch.bfloat16), slot + 1.0)
        ms.append(m)
        hs.append(torch.zeros((T, d), device="cuda", dtype=torch.bfloat16))
    rng = np.random.default_rng(live)
    for n in (live, T, live, live // 2, live):               # longer, shorter, as long
        slots = [rng.integers(-1, 2, size=n).astype(np.int32) for _ in ms]
        pins = [torch.from_numpy(x).pin_memory() for x in slots]
        for m, pin, h in zip(ms, pins, hs):
            h.zero_()
            m.set_slot_map(pin, n)
            m.apply(h)
        for x, h in zip(slots, hs):
            want = np.zeros(T, dtype=np.float32)
            want[:n] = x + 1.0
            assert np.array_equal(h.float().cpu().numpy(), np.repeat(want[:, None], d, 1)), n
    for m in ms:
        m.destroy()


def _installs(m, T, live, ptr, src_is_device, slots):
    stream = torch.cuda.current_stream().cuda_stream
    assert m.lib.mix_set_slot_map(m.ctx, ptr, live, src_is_device, stream) == 0
    h = torch.zeros((T, 64), device="cuda", dtype=torch.bfloat16)
    m.apply(h)
    want = np.zeros(T, dtype=np.float32)
    want[:live] = slots + 1.0
    assert np.array_equal(h[:, 0].float().cpu().numpy(), want)


# sources that a copy takes and a kernel cannot read
@pytest.mark.parametrize("with_sae", [False, True])
@pytest.mark.parametrize("live", [3, 700, 1000])
def test_maps_that_do_not_lie_on_four_bytes(live, with_sae):
    T = 1000
    m = Mix(d_model=64, T_max=T, n_slots_max=2, n_groups_max=int(with_sae), d_sae_max=256 if with_sae else 0)
    for slot in range(2):
        m.register_steer(slot, torch.ones(64, device="cuda", dtype=torch.bfloat16), slot + 1.0)
    slots = np.random.default_rng(live).integers(-1, 2, live).astype(np.int32)
    raw = torch.zeros(4 * live + 4, dtype=torch.uint8)
    raw[1:4 * live + 1] = torch.from_numpy(slots.view(np.uint8))
    for where, src_is_device in ((raw.cuda(), 1), (raw.pin_memory(), 0), (raw, 0)):
        m.set_slot_map(torch.zeros(T, dtype=torch.int32, device="cuda"), T)
        _installs(m, T, live, where.data_ptr() + 1, src_is_device, slots)
    assert m.get_status() == 0
    m.destroy()


def test_a_map_in_memory_that_is_registered_in_part():
    T = live = 700
    m = Mix(d_model=64, T_max=T, n_slots_max=2)
    for slot in range(2):
        m.register_steer(slot, torch.ones(64, device="cuda", dtype=torch.bfloat16), slot + 1.0)
    slots = np.random.default_rng(1).integers(-1, 2, live).astype(np.int32)
    memory = np.zeros(4 * 4096, dtype=np.uint8)
    page = -memory.ctypes.data % 4096                # the first page in it is registered, the second is not
    start = page + 4096 - 4 * 100
    memory[start:start + 4 * live] = slots.view(np.uint8)
    cudart = torch.cuda.cudart()
    assert int(cudart.cudaHostRegister(memory.ctypes.data + page, 4096, 0)) == 0
    try:
        _installs(m, T, live, memory.ctypes.data + start, 0, slots)
        torch.cuda.synchronize()
    finally:
        cudart.cudaHostUnregister(memory.ctypes.data + page)
    m.destroy()


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("shift", [0, 1])
def test_long_pinned_maps_of_a_context_with_weight_sets(captured, shift):
    """Above 2048 live rows a kernel reads the map where it lies; at 2048 and below, and where it does not lie on four bytes, a
    copy takes it.  Lengths up and down across the line, each install followed by a call."""
    d, T = 64, 2200
    m = Mix(d_model=d, T_max=T, n_slots_max=2, n_groups_max=1, d_sae_max=256)
    for slot in range(2):
        m.register_steer(slot, torch.ones(d, device="cuda", dtype=torch.bfloat16), slot + 1.0)
    h = torch.zeros((T, d), device="cuda", dtype=torch.bfloat16)
    rng = np.random.default_rng(shift)
    for n in (2049, 2048, T, 1, 2100, 0, T):
        slots = rng.integers(-1, 2, size=n).astype(np.int32)
        pinned = torch.zeros(4 * n + 8, dtype=torch.uint8).pin_memory()
        address = pinned.data_ptr() + shift
        ctypes.memmove(address, slots.ctypes.data, 4 * n)
        install = lambda: m._check(m.lib.mix_set_slot_map(m.ctx, address, n, 0, torch.cuda.current_stream().cuda_stream))
        h.zero_()
        torch.cuda.synchronize()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                install()
                m.apply(h)
            graph.replay()
        else:
            install()
            m.apply(h)
        torch.cuda.synchronize()
        want = np.zeros(T, dtype=np.float32)
        want[:n] = slots + 1.0
        assert np.array_equal(h.float().cpu().numpy(), np.repeat(want[:, None], d, 1)), n
        if captured:
            del graph
    assert m.get_status() == 0
    m.destroy()
