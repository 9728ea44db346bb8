"""Calls that overlap: several streams, captured graphs, threads."""
import threading
import time

import pytest
import torch

from paper_2012_02030_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ap():
    from paper_2012_02030_b200 import binding

    assert torch.cuda.is_available()
    return binding


def _attention(ap, B, H, L, d, seed, keep=0.1, dtype=torch.bfloat16):
    """Inputs of a backward call, its output buffers and its workspace."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    q, k, v, d_o = (torch.randn((B, H, L, d), generator=gen, device="cuda").to(dtype) for _ in range(4))
    tiles = ap.Tiles(H, L, L)
    ap.ap_mask_to_tiles(inputs.random_mask(H, L, L, keep, seed=seed, causal=True).cuda(), tiles)
    out = ap.ap_sparse_attention_fwd(q, k, v, tiles)
    ws = torch.empty(ap.ap_sparse_attention_bwd_workspace_bytes(B, H, L, L), dtype=torch.uint8, device="cuda")
    return (q, k, v, out, d_o, tiles), [torch.empty_like(q) for _ in range(3)], ws


def test_backward_replayed_beside_eager_calls(ap):
    """A captured backward is replayed on one stream while an eager one runs on another, after enough calls in between that
    any state handed out in rotation has come round: both give the bits that they give alone."""
    side = torch.cuda.Stream()
    args, grads, ws = _attention(ap, 8, 8, 1024, 64, 1)
    args2, grads2, ws2 = _attention(ap, 8, 8, 1024, 64, 2)
    tiny, tiny_grads, tiny_ws = _attention(ap, 1, 1, 16, 64, 3)
    want = [t.clone() for t in ap.ap_sparse_attention_bwd(*args, *grads, workspace=ws)]
    want2 = [t.clone() for t in ap.ap_sparse_attention_bwd(*args2, *grads2, workspace=ws2)]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ap.ap_sparse_attention_bwd(*args, *grads, workspace=ws)
    for _ in range(8):
        for _ in range(1023):
            ap.ap_sparse_attention_bwd(*tiny, *tiny_grads, workspace=tiny_ws)
        for t in grads + grads2:
            t.fill_(float("nan"))
        torch.cuda.synchronize()
        graph.replay()
        with torch.cuda.stream(side):
            ap.ap_sparse_attention_bwd(*args2, *grads2, workspace=ws2)
        torch.cuda.synchronize()
        for got, ref in zip(grads + grads2, want + want2):
            assert torch.equal(got, ref)
    assert ap.ap_device_status() == ap.AP_OK


def _busy(stream, seconds=0.2):
    """Keeps `stream` busy for about that long (a bounded loop on the device)."""
    with torch.cuda.stream(stream):
        torch.cuda._sleep(int(seconds * 1.9e9))


def test_other_threads_run_while_a_launch_waits(ap):
    """A launch that waits for room in its stream's queue does not hold the interpreter lock."""
    args, _, _ = _attention(ap, 1, 1, 64, 64, 7)
    side = torch.cuda.Stream()
    out = torch.empty_like(args[0])
    torch.cuda.synchronize()
    done, errors = threading.Event(), []

    def launches():
        try:
            torch.zeros(1, device="cuda")  # the thread's first CUDA call
            for _ in range(4000):
                ap.ap_sparse_attention_fwd(*args[:3], args[5], out, stream=side)
        except Exception as e:  # noqa: BLE001
            errors.append(e)
        finally:
            done.set()

    _busy(side, 1.0)
    thread = threading.Thread(target=launches)
    began = last = time.perf_counter()
    gap = 0.0
    thread.start()
    while not done.wait(0.001) and last - began < 20.0:
        now = time.perf_counter()
        gap, last = max(gap, now - last), now
    thread.join(20.0)
    gap, took = max(gap, time.perf_counter() - last), time.perf_counter() - began
    torch.cuda.synchronize()
    assert done.is_set() and not errors, errors
    assert took < 0.5 or gap < 0.25  # (a queue without end would never make a launch wait)


def test_out_of_memory_is_raised_as_such(ap):
    H, L = 16, 1024
    acc = torch.zeros((H, L, L), device="cuda")
    mask = torch.empty((H, L, L), dtype=torch.uint8, device="cuda")
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.set_per_process_memory_fraction(torch.cuda.memory_reserved() / total)
    try:
        with pytest.raises(torch.cuda.OutOfMemoryError):
            ap.ap_build_mask(acc, 0.1, True, True, mask=mask)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)


def test_memory_of_calls_on_another_stream(ap):
    """Workspaces and outputs that the binding allocates for a call on a stream that is not the current one: the memory is not
    handed out to the current stream before the call has run."""
    side = torch.cuda.Stream()
    H, L = 4, 512
    acc = torch.rand((H, L, L), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    args, _, _ = _attention(ap, 2, H, L, 64, 6)
    mask = torch.empty((H, L, L), dtype=torch.uint8, device="cuda")
    tiles = ap.Tiles(H, L, L)

    def calls(stream):
        ap.ap_build_mask(acc, 0.1, True, True, mask=mask, tiles=tiles, stream=stream)
        ap.ap_mask_to_tiles(mask, tiles, stream=stream)
        out = ap.ap_sparse_attention_fwd(*args[:3], tiles, stream=stream)
        return (out,) + tuple(ap.ap_sparse_attention_bwd(*args[:3], out, args[4], tiles, stream=stream)) + (
            ap.ap_pool_scores(acc, 32, True, stream=stream),)

    want = [t.clone() for t in calls(None)] + [mask.clone()]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    _busy(side)
    got = calls(side)
    # the current stream, meanwhile: memory of every size that the calls used, overwritten at once
    junk = [torch.full((n,), 0x7f, dtype=torch.uint8, device="cuda") for n in [1 << k for k in range(9, 26)] * 4]
    torch.cuda.synchronize()
    del junk
    assert ap.ap_device_status() == ap.AP_OK
    for a, b in zip(list(got) + [mask], want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 64), (torch.float16, 64), (torch.bfloat16, 128), (torch.float32, 64)])
def test_calls_in_a_row_see_each_others_results(dtype, d):
    """Kernels may be set up on SMs that the one before has left: each call here reads what the one before has written and writes
    over what it has read, with and without waiting in between; bit for bit the same."""
    from paper_2012_02030_b200 import binding as ap

    B, H, L = 5, 7, 300
    gen = torch.Generator().manual_seed(4500 + d)
    q, k, v = (torch.randn((B, H, L, d), generator=gen).to(dtype).cuda() for _ in range(3))
    grads = [torch.empty_like(q) for _ in range(3)]
    acc = torch.zeros((H, L, L), device="cuda")
    tiles = ap.Tiles(H, L, L)
    mask = torch.zeros((H, L, L), dtype=torch.uint8, device="cuda")

    def chain(wait):
        done = torch.cuda.synchronize if wait else lambda: None
        x, y, z, a = q.clone(), torch.empty_like(q), torch.empty_like(q), acc.clone()
        out = []
        for step in range(12):  # (an output is never one of the same call's inputs)
            ap.ap_accumulate_attention(a, x, k, causal=True), done()
            ap.ap_build_mask(a, 0.2 + 0.05 * (step % 4), True, True, mask, tiles), done()
            ap.ap_sparse_attention_fwd(x, k, v, tiles, y), done()
            ap.ap_sparse_attention_entmax15_fwd(x, y, v, tiles, z), done()
            ap.ap_accumulate_attention_entmax15(a, z, y, causal=True), done()
            if dtype != torch.float32:
                ap.ap_sparse_attention_bwd(x, k, v, y, z, tiles, *grads), done()
                out += [t.clone() for t in grads]
                ap.ap_sparse_attention_fwd(grads[0], y, grads[2], tiles, x), done()
            ap.ap_sparse_attention_fwd(z, y, v, tiles, x), done()
            out += [x.clone(), y.clone(), z.clone(), mask.clone()]
        return out + [a]

    want = chain(True)
    for _ in range(3):
        got = chain(False)
        assert all(torch.equal(w, g) for w, g in zip(want, got))
    assert ap.ap_device_status() == ap.AP_OK


def _mask_chain(ap, shape, seed, dtype=torch.bfloat16):
    """The whole procedure a few times over, each call reading what the one before has written: averages, masks under both rules from
    the one workspace, both forwards and the backward.  Returns the function (which takes what to do between two calls) and its
    outputs' buffers."""
    H, Lq, Lk, causal = shape
    gen = torch.Generator(device="cuda").manual_seed(seed)
    q, d_o = (torch.randn((1, H, Lq, 64), generator=gen, device="cuda").to(dtype) for _ in range(2))
    k, v = (torch.randn((1, H, Lk, 64), generator=gen, device="cuda").to(dtype) for _ in range(2))
    acc = torch.zeros((H, Lq, Lk), device="cuda")
    ws = torch.empty(ap.ap_build_mask_workspace_bytes(H, Lq, Lk), dtype=torch.uint8, device="cuda")
    bwd_ws = torch.empty(ap.ap_sparse_attention_bwd_workspace_bytes(1, H, Lq, Lk), dtype=torch.uint8, device="cuda")
    tiles = ap.Tiles(H, Lq, Lk)
    rules = [(ap.ap_build_mask, 0.1), (ap.ap_build_mask_layer, 0.02), (ap.ap_build_mask, 0.4)]
    steps = []
    for _ in rules:
        steps.append(dict(x=torch.empty_like(q), y=torch.empty_like(q), grads=[torch.empty_like(t) for t in (q, k, v)],
                          mask=torch.empty((H, Lq, Lk), dtype=torch.uint8, device="cuda"),
                          nnz=torch.empty(H, dtype=torch.int64, device="cuda")))

    def run(between):
        acc.zero_()
        x = q
        for (build, keep), s in zip(rules, steps):
            ap.ap_accumulate_attention(acc, x, k, causal=causal), between()
            build(acc, keep, causal, causal, s["mask"], tiles, s["nnz"], workspace=ws), between()
            ap.ap_sparse_attention_fwd(x, k, v, tiles, s["x"]), between()
            ap.ap_sparse_attention_entmax15_fwd(s["x"], k, v, tiles, s["y"]), between()
            ap.ap_accumulate_attention_entmax15(acc, s["y"], k, causal=causal), between()
            ap.ap_sparse_attention_bwd(x, k, v, s["x"], d_o, tiles, *s["grads"], workspace=bwd_ws), between()
            x = s["y"]

    return run, [acc] + [t for s in steps for t in (s["x"], s["y"], s["mask"], s["nnz"], *s["grads"])]


# Entries held in shared memory; selected straight over the accumulator; pivots
CHAINS = [(3, 300, 300, True), (9, 1024, 1000, False), (4, 1792, 1800, False), (1, 5120, 5120, True), (16, 896, 896 + 448, True)]


@pytest.mark.parametrize("shape", CHAINS)
def test_masks_in_a_row_see_each_others_results(ap, shape):
    run, out = _mask_chain(ap, shape, 61)
    run(torch.cuda.synchronize)
    want = [t.clone() for t in out]
    for _ in range(3):
        for t in out[1:]:
            t.fill_(99)
        run(lambda: None)
        assert all(torch.equal(w, g) for w, g in zip(want, out))
    assert ap.ap_device_status() == ap.AP_OK


@pytest.mark.parametrize("shape", CHAINS)
def test_captured_procedure(ap, shape):
    """The same calls captured once and replayed, also beside other work on the device."""
    run, out = _mask_chain(ap, shape, 62)
    run(torch.cuda.synchronize)
    want = [t.clone() for t in out]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(lambda: None)
    side = torch.cuda.Stream()
    for beside in (False, True):
        for t in out[1:]:
            t.fill_(99)
        torch.cuda.synchronize()
        if beside:
            _busy(side, 0.01)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(w, g) for w, g in zip(want, out))
    assert ap.ap_device_status() == ap.AP_OK


# Entries held in the shared memory of every SM; of eight SMs; pivots
@pytest.mark.parametrize("shape", [(8, 1280, 1280, True), (2, 256, 256, False), (4, 1792, 1800, False)])
def test_masks_on_several_streams(ap, shape):
    """Selections wait for all of their thread blocks.  On several streams at once each finds room for all of them, behind averages
    that leave the SMs one by one, and gives the bits that it gives alone."""
    streams = [torch.cuda.Stream() for _ in range(3)]
    chains = [_mask_chain(ap, shape, 71 + x) for x in range(3)]
    want = []
    for run, out in chains:
        run(torch.cuda.synchronize)
        want.append([t.clone() for t in out])
    for _ in range(8):
        for _, out in chains:
            for t in out[1:]:
                t.fill_(99)
        torch.cuda.synchronize()
        for _ in range(5):
            for (run, _), stream in zip(chains, streams):
                with torch.cuda.stream(stream):
                    run(lambda: None)
        torch.cuda.synchronize()
        assert ap.ap_device_status() == ap.AP_OK
        for (_, out), ref in zip(chains, want):
            assert all(torch.equal(w, g) for w, g in zip(ref, out))


def _blocking_stream():
    """A stream that the default stream waits for and that waits for the default stream (torch's own do neither)."""
    from cuda.bindings import runtime

    err, handle = runtime.cudaStreamCreate()
    assert int(err) == 0
    return torch.cuda.ExternalStream(int(handle))


@pytest.mark.parametrize("how", ["event", "default stream"])
def test_calls_wait_for_what_other_streams_write(ap, how):
    """A kernel that may be set up early waits for all that its stream waits for, not only for the kernel before it."""
    args, grads, ws = _attention(ap, 2, 4, 384, 64, 8)
    q, k, v, _, d_o, tiles = args
    other = [torch.randn(q.shape, generator=torch.Generator(device="cuda").manual_seed(90 + x), device="cuda").to(q.dtype)
             for x in range(4)]
    out = torch.empty_like(q)
    x = q.clone()
    want = [ap.ap_sparse_attention_fwd(t, k, v, tiles) for t in other]
    side = torch.cuda.Stream() if how == "event" else _blocking_stream()
    torch.cuda.synchronize()
    here = torch.cuda.default_stream()
    for _ in range(3):
        got = []
        for t in other:
            ap.ap_sparse_attention_fwd(x, k, v, tiles, out)
            if how == "event":
                side.wait_stream(here)
            _busy(side, 0.005)
            with torch.cuda.stream(side):
                x.copy_(t)
            if how == "event":
                here.wait_stream(side)
            ap.ap_sparse_attention_fwd(x, k, v, tiles, out)
            got.append(out.clone())
        torch.cuda.synchronize()
        assert all(torch.equal(w, g) for w, g in zip(want, got))


def test_captured_fork_and_join(ap):
    """In a captured graph, too: the second call depends on the first one and on another stream's calls."""
    args, grads, ws = _attention(ap, 2, 4, 384, 64, 9)
    q, k, v, _, _, tiles = args
    x, y, z = (torch.empty_like(q) for _ in range(3))
    acc = torch.zeros((4, 384, 384), device="cuda")
    mask = torch.empty((4, 384, 384), dtype=torch.uint8, device="cuda")
    tiles2 = ap.Tiles(4, 384, 384)
    mask_ws = torch.empty(ap.ap_build_mask_workspace_bytes(4, 384, 384), dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()

    def calls(main):
        acc.zero_()
        ap.ap_sparse_attention_fwd(q, k, v, tiles, x)
        side.wait_stream(main)
        with torch.cuda.stream(side):
            ap.ap_accumulate_attention(acc, x, k, causal=True)
            ap.ap_build_mask(acc, 0.2, True, True, mask, tiles2, workspace=mask_ws)
            ap.ap_sparse_attention_fwd(x, k, v, tiles2, z)
        ap.ap_sparse_attention_fwd(x, k, v, tiles, y)
        main.wait_stream(side)
        ap.ap_sparse_attention_fwd(y, z, v, tiles2, x)

    out = [acc, mask, x, y, z]
    calls(torch.cuda.current_stream())
    torch.cuda.synchronize()
    want = [t.clone() for t in out]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls(torch.cuda.current_stream())
    for _ in range(3):
        for t in out[1:]:
            t.fill_(99)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(w, g) for w, g in zip(want, out))
    assert ap.ap_device_status() == ap.AP_OK
