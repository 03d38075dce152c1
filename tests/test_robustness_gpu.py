"""Failure handling and shared state of the tensor-core kernels, on the GPU, without faulting or hanging it.

* A bounded device-side wait that runs out: the kernel must return, raise the status word once, leave the work
  counters at zero, and the next ordinary call must be bit-exact.  The wait is made to run out by leaving out the
  product it waits for (tri_inv_selftest_wait_timeout) with a limit of microseconds; every wait stays bounded.
* Work-counter pairs are private to a launch: a captured graph replayed on one stream while more plain launches
  than there are pairs run on another stream must give every row right (compared with the fp64 oracle).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_21325_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bnd():
    import __graft_entry__ as entry
    entry.build()
    from paper_2605_21325_b200 import binding
    torch.cuda.set_device(0)
    return binding


def nan_outs(dev, inp):
    return (torch.full((inp.B, inp.T, inp.H, inp.C), float("nan"), dtype=torch.float32, device="cuda"),
            torch.full_like(dev["K"], float("nan")), torch.full_like(dev["V"], float("nan")))


@pytest.mark.parametrize("C", [64, 128])
def test_bounded_wait_gives_up_and_the_library_recovers(bnd, C):
    inp = wl.make("timeout", 2, 16 * C, 8, 128, 128, C, wl.BF16, seed=611)      # 256 matrices
    dev = bnd.to_device(inp)
    ref = bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], C)
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    out = nan_outs(dev, inp)
    idle = bnd.selftest_wait_timeout(dev["K"], dev["V"], dev["beta"], dev["g"], C, wait_limit_ns=20_000, out=out)
    assert idle, "a work-counter pair was left non-zero"
    assert bnd.last_device_status() == bnd.ERR_DEVICE_TIMEOUT     # raised ...
    assert bnd.last_device_status() == 0                          # ... and cleared by the read
    # every matrix but the one whose product was left out (thread block 0's first: chunk 0, head 0) is right
    for r, o in zip(ref, out):
        r2, o2 = r.clone(), o.clone()
        r2[0, :C, 0] = 0
        o2[0, :C, 0] = 0
        assert torch.equal(r2, o2)
    # the next ordinary call on the same stream is bit-exact
    again = bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], C, out=nan_outs(dev, inp))
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    for r, o in zip(ref, again):
        assert torch.equal(r, o)


def test_graph_replays_overlapping_many_plain_launches(bnd):
    a = wl.make("graph_side", 2, 16 * 64, 16, 128, 128, 64, wl.BF16, seed=621)    # 512 matrices: several items per CTA
    b = wl.make("plain_side", 2, 16 * 64, 16, 128, 128, 64, wl.BF16, seed=622)
    da, db = bnd.to_device(a), bnd.to_device(b)
    oa, ob = nan_outs(da, a), nan_outs(db, b)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    bnd.fused(da["K"], da["V"], da["beta"], da["g"], 64, out=oa, stream=s1)      # per-device set-up outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s1):
        with torch.cuda.graph(graph, stream=s1):
            bnd.fused(da["K"], da["V"], da["beta"], da["g"], 64, out=oa, stream=s1)
    for t in oa:
        t.fill_(float("nan"))
    torch.cuda.synchronize()
    for rep in range(8):
        with torch.cuda.stream(s1):
            graph.replay()
        for _ in range(20):                                                       # 160 plain launches in all, unsynchronised
            bnd.fused(db["K"], db["V"], db["beta"], db["g"], 64, out=ob, stream=s2)
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    for inp, out in ((a, oa), (b, ob)):
        A_ref = oracle.build_A(inp.K, inp.beta, inp.g, inp.C)
        W_ref, U_ref = oracle.wy(A_ref, inp.K, inp.V, inp.beta, inp.C)
        for o, r, tol in zip(out, (A_ref, W_ref, U_ref), (2e-3, 1e-2, 1e-2)):
            x = bnd.to_numpy_f64(o)
            assert not np.isnan(x).any(), "a row was not written: two launches shared a work counter"
            assert np.abs(x - r).max() <= tol * np.abs(r).max()


@pytest.mark.parametrize("B,H", [(1, 2), (4, 16)], ids=["narrow_slices", "wide_slices"])
def test_scan_waits_that_run_out(bnd, B, H):
    """The chunk-scan kernel's sixteen warps wait for one another through barriers only; with one product of the first thread
    block left out (tri_inv_selftest_scan_wait_timeout, limit 100 us) every one of that block's waits must give up in turn,
    the kernel must return with the status word raised once, the other blocks' output must be untouched by it, and the
    next ordinary call must give the bits of the call before."""
    inp = wl.make("scan_stall", B, 6 * 64, H, 128, 128, 64, wl.BF16, seed=631 + H)
    dev = bnd.to_device(inp)
    Q = bnd.kv_to_torch(wl.queries(inp, seed=632))
    _, W, U = bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], 64, method=bnd.W_DECAY, want_A=False)
    ref, _ = bnd.chunk_scan(Q, dev["K"], W, U, dev["g"], 64, scale=1.0, want_state=False)
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    O = torch.full_like(dev["V"], float("nan"))
    bnd.selftest_scan_wait_timeout(Q, dev["K"], W, U, dev["g"], 64, wait_limit_ns=100_000, out=O)
    assert bnd.last_device_status() == bnd.ERR_DEVICE_TIMEOUT     # raised ...
    assert bnd.last_device_status() == 0                          # ... and cleared by the read
    # the stalled block is (sequence 0, head 0, first slice of value columns); its first chunk was written
    # before the product was left out
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    width = 32 if B * H * 8 <= sms else 64 if B * H * 2 <= sms else 128
    r2, o2 = ref.clone(), O.clone()
    assert torch.equal(o2[0, :64, 0, :width].view(torch.int16), r2[0, :64, 0, :width].view(torch.int16))
    r2[0, 64:, 0, :width] = 0
    o2[0, 64:, 0, :width] = 0
    assert torch.equal(r2.view(torch.int16), o2.view(torch.int16))
    again, _ = bnd.chunk_scan(Q, dev["K"], W, U, dev["g"], 64, scale=1.0, want_state=False)
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    assert torch.equal(again.view(torch.int16), ref.view(torch.int16))


@pytest.mark.parametrize("d", [128, 64])
def test_inversions_on_a_second_stream_do_not_wait_for_a_scan(bnd, d):
    """A scan of few (sequence, head) pairs leaves most SMs free and takes all tensor memory of the others: inversions issued
    behind it on another stream must run on the free SMs and be done long before the scan (1024 chunks: about a
    millisecond; the inversions alone: some tens of microseconds)."""
    a = wl.make("long_scan", 1, 1024 * 64, 4, 128, 128, 64, wl.BF16, seed=651)
    b = wl.make("beside", 1, 64 * 64, 16, d, d, 64, wl.BF16, seed=652)
    da, db = bnd.to_device(a), bnd.to_device(b)
    Q = bnd.kv_to_torch(wl.queries(a, seed=653))
    _, W, U = bnd.fused(da["K"], da["V"], da["beta"], da["g"], 64, method=bnd.W_DECAY, want_A=False)
    O, A = torch.empty_like(da["V"]), torch.empty((b.B, b.T, b.H, 64), dtype=torch.float32, device="cuda")
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(2):   # the first pass sets the kernels up
        torch.cuda.synchronize()
        begin, scanned, built = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        begin.record(s1)
        s2.wait_event(begin)
        bnd.chunk_scan(Q, da["K"], W, U, da["g"], 64, out=O, want_state=False, stream=s1)
        bnd.build(db["K"], db["beta"], db["g"], 64, out=A, stream=s2)
        scanned.record(s1)
        built.record(s2)
        torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    assert begin.elapsed_time(built) < 0.8 * begin.elapsed_time(scanned)


@pytest.mark.parametrize("C,with_wy", [(64, True), (64, False), (128, True)], ids=["C64_one_kernel", "C64_build", "C128_two_launches"])
def test_per_channel_waits_that_run_out(bnd, C, with_wy):
    """The per-channel kernels' give-up path (tri_inv_selftest_kda_wait_timeout, limit 50 us): the first thread block leaves out
    the Gram product of its first matrix, its waits run out, it raises the status word, drains what it has in flight, frees
    its tensor memory and returns.  256 matrices, fewer than resident thread blocks, so every other matrix must come out
    bit for bit as in an ordinary call; the status word reads DEVICE_TIMEOUT once; the next ordinary call is exact."""
    inp = wl.make("kda_timeout", 2, 16 * C, 8, 128, 128, C, wl.BF16, seed=612)
    dev = bnd.to_device(inp)
    Gd = torch.from_numpy(wl.per_channel_gate(inp, seed=613)).cuda()

    def call(selftest):
        A = torch.full((inp.B, inp.T, inp.H, C), float("nan"), dtype=torch.float32, device="cuda")
        W, U = (torch.full_like(dev["K"], float("nan")), torch.full_like(dev["V"], float("nan"))) if with_wy else (None, None)
        if selftest:
            bnd.selftest_kda_wait_timeout(dev["K"], dev["V"] if with_wy else None, Gd, dev["beta"], C, wait_limit_ns=50_000, out=(A, W, U))
        elif with_wy:
            bnd.fused_kda(dev["K"], dev["V"], Gd, dev["beta"], C, out=(A, W, U))
        else:
            bnd.build_kda(dev["K"], Gd, dev["beta"], C, out=A)
        torch.cuda.synchronize()
        return [t for t in (A, W, U) if t is not None]

    ref = call(False)
    assert bnd.last_device_status() == 0
    out = call(True)
    assert bnd.last_device_status() == bnd.ERR_DEVICE_TIMEOUT     # raised ...
    assert bnd.last_device_status() == 0                          # ... and cleared by the read
    for r, o in zip(ref, out):
        r2, o2 = r.clone(), o.clone()
        r2[0, :C, 0] = 0
        o2[0, :C, 0] = 0
        assert torch.equal(r2.view(torch.int32 if r.dtype == torch.float32 else torch.int16),
                           o2.view(torch.int32 if o.dtype == torch.float32 else torch.int16))
    again = call(False)
    assert bnd.last_device_status() == 0
    for r, o in zip(ref, again):
        assert torch.equal(r.view(torch.int32 if r.dtype == torch.float32 else torch.int16),
                           o.view(torch.int32 if o.dtype == torch.float32 else torch.int16))


CHAINS = {  # name: B, T, H, d, dtype, cu_seqlens -- each layer route's kernels, one call's output the next one's input
    "tokens": (8, 1, 16, 128, wl.BF16, None), "tokens_fp32": (3, 5, 4, 64, wl.F32, None), "one_kernel": (1, 333, 16, 128, wl.BF16, None),
    "two_calls": (1, 4000, 24, 128, wl.BF16, list(range(0, 4001, 40))), "fp32": (2, 200, 3, 64, wl.F32, None), "fp32_one_chunk": (4, 50, 3, 64, wl.F32, None),
}


def same_chains(chain, times=3):
    """A chain of calls with nothing between them against the same with a synchronisation after each: same bits, all finite."""
    ref = chain(torch.cuda.synchronize)
    torch.cuda.synchronize()
    assert all(torch.isfinite(r).all() for r in ref)
    for _ in range(times):
        out = chain(lambda: None)
        torch.cuda.synchronize()
        assert len(out) == len(ref) and all(torch.equal(x, r) for x, r in zip(out, ref))
    return ref


@pytest.mark.parametrize("name", list(CHAINS))
def test_kernels_that_start_early_wait_for_their_predecessor(bnd, name):
    """Calls in a row with no other kernel between them -- layer behind layer, build behind layer, build behind build, layer behind build -- each on the last one's
    output and state and in buffers that it has just used, give the bits of calls with a synchronisation after each."""
    B, T, H, d, dt, cu = CHAINS[name]
    inp = wl.make(name, B, T, H, d, d, 64, dt, seed=900, cu_seqlens=None if cu is None else np.array(cu, np.int32))
    dev, Q = bnd.to_device(inp), bnd.kv_to_torch(wl.queries(inp, seed=901))

    def chain(between):
        shared, own = torch.empty(dev["K"].shape[:3] + (64,), device="cuda"), torch.empty((6,) + tuple(dev["K"].shape[:3]) + (64,), device="cuda")
        V, S, seen = dev["V"], None, []
        for step in range(6):
            for _ in range(2):
                V, S = bnd.gdn_forward(Q, dev["K"], V, dev["beta"], dev["g"], 64, scale=2.0, S0=S, cu_seqlens=cu)
                between()
            seen += [V, S]
            bnd.build(V, dev["beta"], dev["g"], 64, cu_seqlens=cu, out=shared)   # V as keys: reads what the call before has written, over what the last step's build has
            between()
            bnd.build(V, dev["beta"], dev["g"], 64, cu_seqlens=cu, out=own[step])
            between()
        return seen + [shared, own]

    same_chains(chain)
    assert bnd.last_device_status() == 0


FACTOR_CHAINS = {"C64": (9600, 16, 64), "C64_few": (640, 6, 64), "C128": (9600, 16, 128), "C128_few": (1280, 6, 128)}   # T, H, C; 2400, 60, 1200, 60 matrices: several a block, so that the counter is drawn, or one


@pytest.mark.parametrize("name", list(FACTOR_CHAINS))
def test_factor_calls_directly_behind_one_another(bnd, name):
    """build, wy, fused, fused_raw (and the scan at C = 64) in a row with no other kernel between them, on one pair of work counters, each reading what the
    one before has written and writing over what the step before has read; then captured in a graph and replayed on other values."""
    T, H, C = FACTOR_CHAINS[name]
    inp = wl.make(name, 1, T, H, 128, 128, C, wl.BF16, seed=930 + C)
    dev, Q = bnd.to_device(inp), bnd.kv_to_torch(wl.queries(inp, seed=931))
    gen = torch.Generator(device="cuda").manual_seed(932)
    logits = [torch.randn((1, T, H), device="cuda", generator=gen) for _ in range(2)]
    start = dev["V"].clone()

    def chain(between, steps=4):
        A, W, U, X, Y = torch.empty((1, T, H, C), device="cuda"), *(torch.empty_like(start) for _ in range(4))
        V, S, seen = start, None, []
        for step in range(steps):
            bnd.build(dev["K"], dev["beta"], dev["g"], C, out=A)
            between()
            bnd.wy(A, dev["K"], V, dev["beta"], out=(W, U))
            between()
            bnd.fused(dev["K"], U, dev["beta"], dev["g"], C, out=(A, X, Y))
            between()
            bnd.fused(dev["K"], Y, dev["beta"], dev["g"], C, method=bnd.W_DECAY, want_A=False, out=(None, W, U))
            between()
            bnd.fused_raw(dev["K"], U, *logits, C, want_A=False, out=(None, X, Y, None, None))
            between()
            if C == 64:
                V, S = bnd.chunk_scan(Q, dev["K"], W, Y, dev["g"], C, scale=2.0, S0=S)
                between()
                seen += [V, S]
            else:
                V, Y = Y, torch.empty_like(Y)
                seen.append(V)
        return seen + [A, W, X]

    ref = same_chains(chain)
    if C == 64:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            out = chain(lambda: None)
        for replay in range(2):   # flipped values, then the first ones again
            start.copy_(start.flip(1))
            other = chain(torch.cuda.synchronize)
            graph.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(x, r) for x, r in zip(out, other)) and torch.equal(other[0], ref[0]) == (replay == 1)
    assert bnd.last_device_status() == 0


def test_per_channel_kernels_that_start_early_wait_for_their_predecessor(bnd):
    inp = wl.make("kda chain", 2, 640, 8, 128, 128, 64, wl.BF16, seed=910)
    dev, Q, G = bnd.to_device(inp), bnd.kv_to_torch(wl.queries(inp, seed=911)), torch.from_numpy(wl.per_channel_gate(inp, seed=912)).cuda()

    def chain(between, C):
        V, S = dev["V"], None
        for _ in range(8):
            A, W, U = bnd.fused_kda(dev["K"], V, G, dev["beta"], C)
            between()
            if C == 64:
                V, S = bnd.chunk_scan_kda(Q, dev["K"], W, U, G, C, scale=2.0, S0=S)
            else:
                V, S = U, W
            between()
            bnd.build_kda(dev["K"], G, dev["beta"], C, out=A)
            between()
        return A, V, S

    for C in (64, 128):
        same_chains(lambda between: chain(between, C))
    assert bnd.last_device_status() == 0


SMALL = {  # B, T, H, C; thread blocks of a call: 148, 148, 128 -- several of which fit on an SM
    "build": (1, 2368, 4, 64), "fused_c128": (1, 4736, 4, 128), "decode": (4, 1, 8, 64),
}


@pytest.mark.parametrize("name", list(SMALL))
def test_small_calls_on_two_streams_run_beside_each_other(bnd, name):
    """Calls that leave most of each SM free do not keep another stream's calls waiting: a graph of calls on each of two streams takes at most 1.6 times
    what one of them takes alone (1.1 to 1.3 measured).  Calls that shut each other out take 1.6 to 1.9 times, calls one after the other 2."""
    B, T, H, C = SMALL[name]
    calls = 40
    streams, graphs, kept = [torch.cuda.Stream() for _ in range(2)], [], []
    for n, st in enumerate(streams):
        inp = wl.make(name, B, T, H, 128, 128, C, wl.BF16, seed=920 + n)
        dev, Q = bnd.to_device(inp), bnd.kv_to_torch(wl.queries(inp, seed=922))
        S0 = torch.from_numpy(wl.initial_state(inp, seed=923)).cuda()
        A, W, U = torch.empty((B, T, H, C), device="cuda"), torch.empty_like(dev["K"]), torch.empty_like(dev["V"])

        def call():
            if name == "build":
                return bnd.build(dev["K"], dev["beta"], dev["g"], C, out=A)
            if name == "decode":
                return bnd.gdn_forward(Q, dev["K"], dev["V"], dev["beta"], dev["g"], C, S0=S0)
            return bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], C, want_A=False, out=(None, W, U))

        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            call()
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            outs = [call() for _ in range(calls)]
        graphs.append(graph)
        kept.append((dev, Q, S0, A, W, U, outs))

    def microseconds(n):
        best = float("inf")
        for _ in range(20):
            torch.cuda.synchronize()
            begin, joined, end = (torch.cuda.Event(enable_timing=True) for _ in range(3))
            begin.record(streams[0])
            streams[1].wait_event(begin)
            for graph, st in list(zip(graphs, streams))[:n]:
                with torch.cuda.stream(st):
                    graph.replay()
            joined.record(streams[1])
            streams[0].wait_event(joined)
            end.record(streams[0])
            torch.cuda.synchronize()
            best = min(best, 1e3 * begin.elapsed_time(end) / calls)
        return best

    one, two = microseconds(1), microseconds(2)
    assert bnd.last_device_status() == 0
    assert two <= (1.5 if name == "decode" else 1.6) * one, (one, two)
