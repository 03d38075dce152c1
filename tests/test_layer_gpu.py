"""GPU tests of the layer forward's routes (tri_inv_gdn_forward).

One kernel (factors and scans side by side): the arithmetic is that of the two calls it replaces, so results are compared bit for
bit.  Token by token: fp32 arithmetic on the stored inputs, against the fp64 recurrence: fp32 storage 1e-5 of max|O| (at most 16
steps of sums of up to 128 terms, 2^-24 each), bf16 storage 2^-8 (the output's own rounding), the state 1e-5.
"""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2605_21325_b200 import workloads as wl
from parity_util import max_ratio

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bnd():
    import __graft_entry__ as entry
    entry.build()
    from paper_2605_21325_b200 import binding
    torch.cuda.set_device(0)
    return binding


def bits(t):
    return t.contiguous().view(torch.int16 if t.dtype == torch.bfloat16 else torch.int32)


def layer_inputs(bnd, name, B, T, H, d_k, d_v, dtype, cu, seed, with_s0=True):
    if cu is not None:
        B, T = 1, int(cu[-1])
    inp = wl.make(name, B, T, H, d_k, d_v, 64, dtype, seed=seed, cu_seqlens=cu)
    Q = wl.queries(inp, seed=seed + 1)
    S0 = wl.initial_state(inp, seed=seed + 2) if with_s0 else None
    dev = bnd.to_device(inp)
    return inp, Q, S0, dev, bnd.kv_to_torch(Q), None if S0 is None else torch.from_numpy(S0).cuda()


def two_calls(bnd, dev, Q, S0, cu, scale):
    _, W, U = bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], 64, method=bnd.W_DECAY, cu_seqlens=cu, want_A=False)
    return bnd.chunk_scan(Q, dev["K"], W, U, dev["g"], 64, scale=scale, S0=S0, cu_seqlens=cu)


# one chunk and one token over it, more chunks than tile stages, each slice width (few pairs: 32 columns, 32: 64, 75: 128), groups
# that build one matrix and several, packed sequences with empty ones, of one token, and more of them than walk at the same time
ONE_KERNEL = [
    ("one_chunk", 1, 64, 1, None),
    ("one_token_over", 1, 65, 2, None),
    ("partial", 2, 333, 3, None),
    ("slices_of_64", 2, 5 * 64 + 1, 16, None),
    ("slices_of_128", 1, 40 * 64, 75, None),
    ("many_matrices", 1, 96 * 64 + 7, 16, None),
    ("packed", 1, 0, 16, np.array([0, 64, 64, 65, 300, 531, 540], np.int32)),
    ("packed_many", 1, 0, 4, np.cumsum([0] + [1 + (37 * i) % 90 for i in range(24)]).astype(np.int32)),
]


@pytest.mark.parametrize("name,B,T,H,cu", ONE_KERNEL, ids=[c[0] for c in ONE_KERNEL])
def test_one_kernel_gives_the_bits_of_the_two_calls(bnd, name, B, T, H, cu):
    for with_s0 in (False, True):
        _, _, _, dev, Q, S0 = layer_inputs(bnd, name, B, T, H, 128, 128, wl.BF16, cu, 700 + H, with_s0)
        ref = two_calls(bnd, dev, Q, S0, cu, 0.25)
        n0 = bnd.launch_count()
        O, S = bnd.gdn_forward(Q, dev["K"], dev["V"], dev["beta"], dev["g"], 64, scale=0.25, S0=S0, cu_seqlens=cu)
        torch.cuda.synchronize()
        assert bnd.last_device_status() == 0
        assert bnd.launch_count() == n0 + 1, "not the one-kernel route"
        assert torch.equal(bits(O), bits(ref[0])) and torch.equal(bits(S), bits(ref[1]))


def test_one_kernel_on_two_streams_and_in_a_graph(bnd):
    """Two calls whose thread blocks share the chip (either may hold SMs that the other waits for), and a captured call replayed on
    new inputs in the same buffers: the bits of a call by itself."""
    args = [layer_inputs(bnd, "streams", 1, 20 * 64 + 5, 24, 128, 128, wl.BF16, None, 720 + 10 * i) for i in range(2)]
    run = lambda a, st=None: bnd.gdn_forward(a[4], a[3]["K"], a[3]["V"], a[3]["beta"], a[3]["g"], 64, scale=0.5, S0=a[5], stream=st)
    refs = [run(a) for a in args]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = []
    for _ in range(8):
        for a, st in zip(args, streams):
            with torch.cuda.stream(st):
                outs.append(run(a, st))
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    for i, o in enumerate(outs):
        assert torch.equal(bits(o[0]), bits(refs[i % 2][0])) and torch.equal(bits(o[1]), bits(refs[i % 2][1]))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        O, S = run(args[0])
    for x, y in ((args[0][4], args[1][4]), (args[0][5], args[1][5])):
        x.copy_(y)
    for k in ("K", "V", "beta", "g"):
        args[0][3][k].copy_(args[1][3][k])
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(bits(O), bits(refs[1][0])) and torch.equal(bits(S), bits(refs[1][1]))


def test_one_kernel_waits_that_run_out(bnd):
    """The give-up path: the scans of the first head wait for a chunk that is never announced (limit 2 ms, far above what the other
    scans ever wait here); the status word says so once, every other head is right, and so is the next call."""
    inp, _, _, dev, Q, _ = layer_inputs(bnd, "stall", 1, 6 * 64, 8, 128, 128, wl.BF16, None, 760, False)
    call = lambda: bnd.gdn_forward(Q, dev["K"], dev["V"], dev["beta"], dev["g"], 64, scale=1.0)[0]
    ref = call()
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    O = torch.full_like(dev["V"], float("nan"))
    bnd.selftest_layer_wait_timeout(Q, dev["K"], dev["V"], dev["beta"], dev["g"], 64, wait_limit_ns=2_000_000, out=O)
    assert bnd.last_device_status() == bnd.ERR_DEVICE_TIMEOUT
    assert bnd.last_device_status() == 0
    assert torch.equal(bits(O[:, :, 1:]), bits(ref[:, :, 1:]))
    again = call()
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    assert torch.equal(bits(again), bits(ref))


# few pairs (32 columns a slice), 32 (64), a last chunk of one token, packed sequences with an empty one
KDA_ONE_KERNEL = [
    ("few", 1, 130 * 64 + 1, 8, None),
    ("slices_of_64", 1, 80 * 64, 32, None),
    ("packed", 1, 0, 8, np.array([0, 9000, 9000, 9001, 13000], np.int32)),
]


@pytest.mark.parametrize("name,B,T,H,cu", KDA_ONE_KERNEL, ids=[c[0] for c in KDA_ONE_KERNEL])
def test_per_channel_scan_in_one_kernel_gives_the_bits_of_two(bnd, name, B, T, H, cu):
    """A head's result does not depend on how many there are: with many of them the preparation is a launch of its own."""
    many = 160 if cu is None else 40
    if cu is not None:
        T = int(cu[-1])
    inp = wl.make(name, B, T, H, 128, 128, 64, wl.BF16, seed=770 + H, cu_seqlens=cu)
    dev = bnd.to_device(inp)
    Q, G = bnd.kv_to_torch(wl.queries(inp, seed=771)), torch.from_numpy(wl.per_channel_gate(inp, seed=772)).cuda()
    S0 = torch.from_numpy(wl.initial_state(inp, seed=773)).cuda()
    _, W, U = bnd.fused_kda(dev["K"], dev["V"], G, dev["beta"], 64, cu_seqlens=cu)
    wide = lambda t, dim: t.repeat_interleave((many + H - 1) // H, dim).contiguous()
    n0 = bnd.launch_count()
    ref = bnd.chunk_scan_kda(*(wide(t, 2) for t in (Q, dev["K"], W, U, G)), 64, scale=0.5, S0=wide(S0, 1), cu_seqlens=cu)
    n1 = bnd.launch_count()
    O, S = bnd.chunk_scan_kda(Q, dev["K"], W, U, G, 64, scale=0.5, S0=S0, cu_seqlens=cu)
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    assert n1 == n0 + 2 and bnd.launch_count() == n1 + 1
    k = (many + H - 1) // H
    assert torch.equal(bits(O), bits(ref[0][:, :, ::k])) and torch.equal(bits(S), bits(ref[1][:, ::k]))


# partial last chunks in front of another sequence: packed, short ones beside long ones; a batch; all 128 columns in a block
KDA_NEIGHBOURS = [
    ("packed", 1, 8, np.array([0, 1, 8001, 8002, 8040, 16040], np.int32)),
    ("batch", 3, 4, 80 * 64 + 37),
    ("slices_of_128", 2, 26, 130 * 64 + 1),
]


@pytest.mark.parametrize("name,B,H,layout", KDA_NEIGHBOURS, ids=[c[0] for c in KDA_NEIGHBOURS])
def test_per_channel_scan_does_not_depend_on_what_its_scratch_held(bnd, name, B, H, layout):
    """A last chunk's tile reaches past its sequence, into rows of the scratch that another block prepares, maybe later.  The scratch is
    left full of NaN by a call of the same shape on NaN keys; the next call's bits are those of the form in two launches."""
    cu = layout if B == 1 else None
    T = int(cu[-1]) if B == 1 else layout
    gen = torch.Generator(device="cuda").manual_seed(790)
    normal = lambda *s: torch.randn(*s, device="cuda", generator=gen)
    unit = lambda x: (x / x.norm(dim=-1, keepdim=True)).to(torch.bfloat16)
    Q, K, V = unit(normal(B, T, H, 128)), unit(normal(B, T, H, 128)), normal(B, T, H, 128).to(torch.bfloat16)
    beta, G = torch.sigmoid(normal(B, T, H)), -0.05 * torch.rand(B, T, H, 128, device="cuda", generator=gen)
    edges = [T * b for b in range(B + 1)] if cu is None else list(cu)
    for a, b in zip(edges[:-1], edges[1:]):   # cumulative within the chunks of a sequence
        for c in range(a, b, 64):
            rows = G.reshape(B * T, H, 128)[c:min(c + 64, b)]
            rows.copy_(rows.cumsum(0))
    _, W, U = bnd.fused_kda(K, V, G, beta, 64, cu_seqlens=cu)
    k = (160 + H - 1) // H
    wide = [t.repeat_interleave(k, 2).contiguous() for t in (Q, K, W, U, G)]
    n0 = bnd.launch_count()
    ref = bnd.chunk_scan_kda(*wide, 64, scale=0.5, cu_seqlens=cu)
    n1 = bnd.launch_count()
    for _ in range(4):   # which block is late differs from run to run
        bnd.chunk_scan_kda(*(torch.full_like(t, float("nan")) for t in (Q, K)), W, U, torch.zeros_like(G), 64, cu_seqlens=cu)
        n2 = bnd.launch_count()
        O, S = bnd.chunk_scan_kda(Q, K, W, U, G, 64, scale=0.5, cu_seqlens=cu)
        torch.cuda.synchronize()
        assert bnd.last_device_status() == 0
        assert n1 == n0 + 2 and bnd.launch_count() == n2 + 1, "not one kernel against two"
        assert torch.isfinite(S).all()
        assert torch.equal(bits(O), bits(ref[0][:, :, ::k])) and torch.equal(bits(S), bits(ref[1][:, ::k]))


@pytest.mark.parametrize("H", [2, 16, 40], ids=["32_columns", "64_columns", "128_columns"])
def test_scan_does_not_multiply_a_neighbours_keys(bnd, H):
    """Keys that are not finite stay with their sequence: the one before it, whose last chunk's tile reaches into them, keeps its bits,
    in the scan by itself and in the layer."""
    cu = np.array([0, 70, 200], np.int32)
    _, _, _, dev, Q, S0 = layer_inputs(bnd, "neighbour", 1, 0, H, 128, 128, wl.BF16, cu, 795)
    _, W, U = bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], 64, method=bnd.W_DECAY, cu_seqlens=cu, want_A=False)
    for call in (lambda K: bnd.chunk_scan(Q, K, W, U, dev["g"], 64, scale=0.5, S0=S0, cu_seqlens=cu),
                 lambda K: bnd.gdn_forward(Q, K, dev["V"], dev["beta"], dev["g"], 64, scale=0.5, S0=S0, cu_seqlens=cu)):
        outs = []
        for value in (1.0, float("inf"), float("nan")):
            K = dev["K"].clone()
            K[0, 70:] *= value
            O, S = call(K)
            outs.append((bits(O[:, :70]), bits(S[0])))
        torch.cuda.synchronize()
        assert bnd.last_device_status() == 0
        assert torch.isfinite(S[0]).all()
        for o in outs[1:]:
            assert torch.equal(o[0], outs[0][0]) and torch.equal(o[1], outs[0][1])


def kda_operands(bnd, B, T, H, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    normal = lambda *s: torch.randn(*s, device="cuda", generator=gen)
    unit = lambda x: (x / x.norm(dim=-1, keepdim=True)).to(torch.bfloat16)
    Q, K, V, beta = unit(normal(B, T, H, 128)), unit(normal(B, T, H, 128)), normal(B, T, H, 128).to(torch.bfloat16), torch.sigmoid(normal(B, T, H))
    rate = -0.05 * torch.rand(B, 1, H, 128, device="cuda", generator=gen)
    G = rate * (1 + torch.arange(T, device="cuda") % 64)[None, :, None, None]   # cumulative within each chunk
    _, W, U = bnd.fused_kda(K, V, G.contiguous(), beta, 64)
    return Q, K, W, U, G.contiguous()


@pytest.mark.parametrize("B,T,H", [(1, 130 * 64, 8), (1, 80 * 64, 32), (2, 130 * 64, 26)], ids=["32_columns", "64_columns", "128_columns"])
def test_per_channel_one_kernel_waits_that_run_out(bnd, B, T, H):
    """As above: the first chunk's operands are never announced, so the scans of the first sequence's first head give up."""
    args = kda_operands(bnd, B, T, H, 796)
    n0 = bnd.launch_count()
    ref, S_ref = bnd.chunk_scan_kda(*args, 64)
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0 and bnd.launch_count() == n0 + 1
    O = torch.full_like(args[3], float("nan"))
    bnd.selftest_kda_scan_wait_timeout(*args, 64, wait_limit_ns=2_000_000, out=O)
    assert bnd.last_device_status() == bnd.ERR_DEVICE_TIMEOUT
    assert bnd.last_device_status() == 0
    assert torch.equal(bits(O[:, :, 1:]), bits(ref[:, :, 1:])) and torch.equal(bits(O[1:]), bits(ref[1:]))
    again, S = bnd.chunk_scan_kda(*args, 64)
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    assert torch.equal(bits(again), bits(ref)) and torch.equal(bits(S), bits(S_ref))


def test_per_channel_one_kernel_on_two_streams_and_in_a_graph(bnd):
    """As the layer's test of that name."""
    args = [kda_operands(bnd, 1, 80 * 64 + 5, 32, 797 + i) for i in range(2)]
    refs = [bnd.chunk_scan_kda(*a, 64) for a in args]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = []
    for _ in range(6):
        for a, st in zip(args, streams):
            with torch.cuda.stream(st):
                outs.append(bnd.chunk_scan_kda(*a, 64, stream=st))
    torch.cuda.synchronize()
    assert bnd.last_device_status() == 0
    for i, o in enumerate(outs):
        assert torch.equal(bits(o[0]), bits(refs[i % 2][0])) and torch.equal(bits(o[1]), bits(refs[i % 2][1]))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        O, S = bnd.chunk_scan_kda(*args[0], 64)
    for x, y in zip(*args):
        x.copy_(y)
    for _ in range(2):
        O.fill_(float("nan"))
        S.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(bits(O), bits(refs[1][0])) and torch.equal(bits(S), bits(refs[1][1]))


# one kernel (dense, packed with partial and empty sequences); two calls (bf16 with more pairs than walk at once; fp32 in one segment)
WORKSPACES = [
    ("one_kernel", 2, 333, 3, 128, wl.BF16, None),
    ("one_kernel_packed", 1, 0, 16, 128, wl.BF16, np.array([0, 64, 64, 65, 300, 531, 540], np.int32)),
    ("two_calls", 4, 70, 64, 128, wl.BF16, None),
    ("fp32", 2, 197, 3, 64, wl.F32, None),
    ("fp32_packed", 1, 0, 3, 72, wl.F32, np.array([0, 64, 64, 65, 300], np.int32)),
]


@pytest.mark.parametrize("name,B,T,H,d,dtype,cu", WORKSPACES, ids=[c[0] for c in WORKSPACES])
def test_workspace_contents_are_arbitrary(bnd, name, B, T, H, d, dtype, cu):
    """Zeros, all bits set (NaN in either type, counters far from zero) and what the call before left: the same bits."""
    inp, _, _, dev, Q, S0 = layer_inputs(bnd, name, B, T, H, d, d, dtype, cu, 860)
    desc, keep = bnd.make_desc(inp.B, inp.T, H, d, d, 64, dtype, cu)
    lib, need, results = bnd.load(), ctypes.c_size_t(0), []
    assert lib.tri_inv_gdn_forward_workspace(desc, 0, need) == bnd.OK and need.value > 0
    work = torch.zeros(need.value, dtype=torch.uint8, device="cuda")
    for fill in (None, 255, None):
        if fill is not None:
            work.fill_(fill)
        O, S = torch.full_like(dev["V"], float("nan")), torch.full_like(S0, float("nan"))
        assert lib.tri_inv_gdn_forward(*(bnd._p(t) for t in (Q, dev["K"], dev["V"], dev["beta"], dev["g"], S0, O, S)), 0.5, bnd._p(work), need, desc, 0,
                                       torch.cuda.current_stream().cuda_stream) == bnd.OK
        torch.cuda.synchronize()
        assert bnd.last_device_status() == 0
        results.append((O, S))
    for O, S in results[1:]:
        assert torch.equal(bits(O), bits(results[0][0])) and torch.equal(bits(S), bits(results[0][1]))
    assert torch.isfinite(results[0][0]).all() and torch.isfinite(results[0][1]).all()


# one token, the longest, features and columns on both sides of the kernel's instances and slices, an empty sequence
TOKENS = [
    ("decode", 4, 1, 3, 128, 128, None),
    ("longest", 1, 16, 2, 128, 128, None),
    ("narrow", 2, 5, 1, 8, 40, None),
    ("d72", 1, 3, 2, 72, 64, None),
    ("packed", 1, 0, 2, 64, 96, np.array([0, 1, 1, 17, 20], np.int32)),
]


@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
@pytest.mark.parametrize("name,B,T,H,d_k,d_v,cu", TOKENS, ids=[c[0] for c in TOKENS])
def test_token_by_token_against_the_recurrence(bnd, name, B, T, H, d_k, d_v, cu, dtype):
    inp, Q, S0, dev, Qd, S0d = layer_inputs(bnd, name, B, T, H, d_k, d_v, dtype, cu, 750 + d_k)
    O_ref, S_ref = oracle.gdn_recurrence(Q, inp.K, inp.V, inp.beta, inp.g, 64, scale=0.5, S0=S0, cu_seqlens=cu)
    O, S = bnd.gdn_forward(Qd, dev["K"], dev["V"], dev["beta"], dev["g"], 64, scale=0.5, S0=S0d, cu_seqlens=cu)
    torch.cuda.synchronize()
    assert max_ratio(bnd.to_numpy_f64(O), O_ref) <= (1e-5 if dtype == wl.F32 else 2.0 ** -8)
    assert max_ratio(bnd.to_numpy_f64(S), S_ref) <= 1e-5


# (pairs, chunks, launches that compute): points at which the slower form takes 5 to 25 % longer (figures beside choose_kda_split)
KDA_ROUTES = [(16, 32, 2), (32, 16, 2), (20, 32, 2), (16, 6, 2), (75, 64, 2), (64, 64, 2), (16, 128, 1), (32, 64, 1), (48, 128, 1), (8, 256, 1)]


def test_per_channel_scan_takes_the_form_that_was_measured_faster(bnd):
    x = torch.zeros((1, 64 * 256 * 8, 1, 128), dtype=torch.bfloat16, device="cuda")
    G = torch.zeros(x.shape, device="cuda")
    cut = lambda t, P, N: t.reshape(-1)[:64 * N * P * 128].reshape(1, 64 * N, P, 128)   # noqa: E731
    took = []
    for P, N, launches in KDA_ROUTES:
        if 64 * N * P > x.shape[1]:
            x = torch.zeros((1, 64 * N * P, 1, 128), dtype=torch.bfloat16, device="cuda")
            G = torch.zeros(x.shape, device="cuda")
        n0 = bnd.launch_count()
        t = cut(x, P, N)
        O, S = bnd.chunk_scan_kda(t, t, t, t, cut(G, P, N), 64)
        torch.cuda.synchronize()
        took.append((P, N, bnd.launch_count() - n0))
        assert not O.any() and not S.any()
    assert bnd.last_device_status() == 0
    assert took == KDA_ROUTES


def test_smoke_runs():
    """The entry that is run first on a machine, with its counts of launches and its comparisons."""
    import __graft_entry__ as entry
    entry.smoke()


def test_every_launch_that_computes_is_counted(bnd):
    """One token each for more sequences than a launch takes; the fp32 scan of one chunk (one kernel), of several (chain and output) and in
    segments of its scratch (as many pairs of launches); the per-channel scan in its two forms is counted above."""
    def counted(call):
        n0 = bnd.launch_count()
        call()
        torch.cuda.synchronize()
        assert bnd.last_device_status() == 0
        return bnd.launch_count() - n0

    for n_seqs, launches in ((960, 1), (961, 2), (2000, 3)):
        _, _, _, dev, Q, _ = layer_inputs(bnd, "count", 1, 0, 1, 16, 16, wl.F32, np.arange(n_seqs + 1, dtype=np.int32), 820, False)
        assert counted(lambda: bnd.gdn_forward(Q, dev["K"], dev["V"], dev["beta"], dev["g"], 64, cu_seqlens=np.arange(n_seqs + 1))) == launches
    slots = (128 << 20) // ((128 + 64) * 128 * 4)   # chunks whose state and U~ the scratch holds
    H = 40
    for chunks, launches in ((1, 1), (2, 2), (slots // H, 2), (slots // H + 1, 4)):
        x = torch.zeros((1, 64 * chunks, H, 128), device="cuda")
        g = torch.zeros((1, 64 * chunks, H), device="cuda")
        assert counted(lambda: bnd.chunk_scan(x, x, x, x, g, 64)) == launches


def graph_allocations(graph):
    """Memory nodes of a captured graph."""
    lib = ctypes.CDLL("libcuda.so.1")
    g, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert lib.cuGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert lib.cuGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    kind, count = ctypes.c_int(0), 0
    for x in nodes:
        assert lib.cuGraphNodeGetType(ctypes.c_void_p(x), ctypes.byref(kind)) == 0
        count += kind.value == 10   # CU_GRAPH_NODE_TYPE_MEM_ALLOC
    return count


@pytest.mark.parametrize("scan_only", [False, True])
def test_fp32_calls_in_a_graph(bnd, scan_only):
    """The layer's scratch is part of its workspace: a dense call takes nothing from the library's pool, so its graph has no memory
    nodes.  The scan by itself has them; either is replayed on new inputs in the same buffers, twice."""
    args = [layer_inputs(bnd, "graph32", 2, 3 * 64 + 5, 3, 64, 64, wl.F32, None, 850 + 10 * i) for i in range(2)]
    if scan_only:
        for a in args:
            a[3]["W"], a[3]["U"] = bnd.fused(a[3]["K"], a[3]["V"], a[3]["beta"], a[3]["g"], 64, method=bnd.W_DECAY, want_A=False)[1:]
        run = lambda a: bnd.chunk_scan(a[4], a[3]["K"], a[3]["W"], a[3]["U"], a[3]["g"], 64, scale=0.5, S0=a[5])
    else:
        run = lambda a: bnd.gdn_forward(a[4], a[3]["K"], a[3]["V"], a[3]["beta"], a[3]["g"], 64, scale=0.5, S0=a[5])
    refs = [[t.clone() for t in run(a)] for a in args]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        out = run(args[0])
    assert graph_allocations(graph) == (1 if scan_only else 0)
    graph.instantiate()
    for ref, src in ((refs[0], None), (refs[1], args[1]), (refs[1], None)):
        if src is not None:
            args[0][4].copy_(src[4])
            args[0][5].copy_(src[5])
            for k in args[0][3]:
                if torch.is_tensor(args[0][3][k]):
                    args[0][3][k].copy_(src[3][k])
        for t in out:
            t.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert bnd.last_device_status() == 0
        for x, r in zip(out, ref):
            assert torch.equal(x, r)


@pytest.mark.parametrize("case", ["decode", "decode_fp32", "short", "packed_list", "packed_tuple"])
def test_native_marshalling_gives_the_python_bodys_bits(bnd, case):
    """A call with a stream is marshalled in Python, one without in native code; other containers and number types take the Python body."""
    import importlib
    assert bnd.load_native() is importlib.import_module("paper_2605_21325_b200._native").gdn_forward
    cu = [0, 1, 1, 70, 200] if case.startswith("packed") else None
    B, T, dt, d = {"decode": (3, 1, wl.BF16, 128), "decode_fp32": (3, 2, wl.F32, 64), "short": (2, 130, wl.BF16, 128)}.get(case, (1, 200, wl.BF16, 128))
    inp = wl.make(case, B, T, 2, d, d, 64, dt, seed=880, cu_seqlens=None if cu is None else np.array(cu, np.int32))
    dev, Q = bnd.to_device(inp), bnd.kv_to_torch(wl.queries(inp, seed=881))
    S0 = torch.from_numpy(wl.initial_state(inp, seed=882)).cuda()
    args = (Q, dev["K"], dev["V"], dev["beta"], dev["g"], 64)
    cu = tuple(cu) if case == "packed_tuple" else cu
    for s0 in (None, S0):
        ref = bnd.gdn_forward(*args, scale=0.5, S0=s0, cu_seqlens=cu, stream=torch.cuda.current_stream())
        odd = bnd.gdn_forward(*args, scale=np.float32(0.5), S0=s0, cu_seqlens=None if cu is None else np.array(cu, np.int64))
        out = bnd.gdn_forward(*args, scale=0.5, S0=s0, cu_seqlens=cu)
        torch.cuda.synchronize()
        for r, x, y in zip(ref, odd, out):
            assert x.shape == r.shape and y.shape == r.shape and y.dtype == r.dtype and torch.equal(x, r) and torch.equal(y, r)
    assert bnd.last_device_status() == 0
    with pytest.raises(bnd.TriInvError):
        bnd.gdn_forward(Q, dev["K"], dev["V"], dev["beta"], dev["g"], 48)
    with pytest.raises(AssertionError):
        bnd.gdn_forward(Q.cpu(), dev["K"], dev["V"], dev["beta"], dev["g"], 64)
    with pytest.raises(AssertionError):
        bnd.gdn_forward(Q, dev["K"].repeat_interleave(2, -1)[..., ::2], dev["V"], dev["beta"], dev["g"], 64)
