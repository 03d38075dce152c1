"""C-ABI checks that need no GPU: the library loads, exports what the header declares,
and rejects bad arguments on the host before touching the device."""
import ctypes
import os
import re

import numpy as np
import pytest

import __graft_entry__ as entry

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    entry.build()
    from paper_2605_21325_b200 import binding
    return binding.load(), binding


def declared_functions():
    names = []
    for fn in sorted(os.listdir(os.path.join(ROOT, "include"))):
        if fn.endswith(".h"):
            src = open(os.path.join(ROOT, "include", fn)).read()
            src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
            names += re.findall(r"\b(tri_inv_[a-z_0-9]+)\s*\(", src)
    return sorted(set(names))


def test_every_declared_symbol_is_exported(lib):
    L, binding = lib
    names = declared_functions()
    assert len(names) >= 7
    for n in names:
        assert hasattr(L, n), "missing export %s" % n
    assert set(binding.EXPORTS) <= set(names)


def test_status_strings(lib):
    L, binding = lib
    assert binding.status_string(0) == "ok"
    assert len({binding.status_string(i) for i in range(5)}) == 5


def test_count_matrices_and_descriptor_validation(lib):
    L, binding = lib
    d, _ = binding.make_desc(4, 4096, 16, 128, 128, 64, binding.BF16)
    assert binding.count_matrices(d) == 4096
    d, _ = binding.make_desc(2, 100, 3, 64, 64, 64, binding.F32)         # partial last chunk
    assert binding.count_matrices(d) == 2 * 2 * 3
    cu = np.array([0, 1, 70, 134, 200], np.int32)
    d, keep = binding.make_desc(1, 200, 2, 64, 64, 64, binding.BF16, cu)
    assert binding.count_matrices(d) == (1 + 2 + 1 + 2) * 2
    for bad in (dict(C=48), dict(d_k=12), dict(H=0), dict(kv_dtype=7), dict(B=0)):
        kw = dict(B=1, T=64, H=1, d_k=64, d_v=64, C=64, kv_dtype=binding.F32)
        kw.update(bad)
        d, _ = binding.make_desc(**kw)
        with pytest.raises(binding.TriInvError) as e:
            binding.count_matrices(d)
        assert e.value.status == binding.ERR_INVALID_ARG
    for cu_bad in ([0, 10, 5, 200], [1, 200], [0, 100]):                 # decreasing, bad start, bad end
        d, keep = binding.make_desc(1, 200, 2, 64, 64, 64, binding.BF16, np.array(cu_bad, np.int32))
        with pytest.raises(binding.TriInvError):
            binding.count_matrices(d)


def test_null_and_misaligned_pointers_rejected_before_any_device_work(lib):
    L, binding = lib
    d, _ = binding.make_desc(1, 64, 1, 64, 64, 64, binding.F32)
    p = ctypes.byref(d)
    ok = ctypes.c_void_p(4096)
    assert L.tri_inv_build(None, ok, ok, ok, p, 0, None) == binding.ERR_INVALID_ARG
    assert L.tri_inv_build(ok, ok, ok, ctypes.c_void_p(4100), p, 0, None) == binding.ERR_INVALID_ARG
    assert L.tri_inv_build(ok, ok, ok, ok, None, 0, None) == binding.ERR_INVALID_ARG
    assert L.tri_inv_build(ok, ok, ok, ok, p, 7, None) == binding.ERR_UNSUPPORTED
    assert L.tri_inv_build(ok, ok, ok, ok, p, binding.PRODUCT_SERIES | binding.LEAF_SERIES, None) == binding.ERR_UNSUPPORTED
    assert L.tri_inv_wy(ok, ok, ok, ok, ok, None, p, None) == binding.ERR_INVALID_ARG   # V without U
    assert L.tri_inv_fused(ok, None, ok, ok, ok, ok, ok, p, 0, None) == binding.ERR_INVALID_ARG
    assert binding.launch_count() == 0 or binding.launch_count() > 0   # callable without a device


def test_newer_entry_points_validate_on_the_host(lib):
    L, binding = lib
    d, _ = binding.make_desc(1, 64, 1, 128, 128, 64, binding.BF16)
    p = ctypes.byref(d)
    ok = ctypes.c_void_p(4096)
    odd = ctypes.c_void_p(4100)
    # per-channel decay build
    assert L.tri_inv_build_kda(ok, None, ok, ok, p, 0, None) == binding.ERR_INVALID_ARG
    assert L.tri_inv_build_kda(ok, odd, ok, ok, p, 0, None) == binding.ERR_INVALID_ARG
    assert L.tri_inv_build_kda(ok, ok, ok, ok, p, binding.W_DECAY, None) == binding.ERR_UNSUPPORTED   # no W to weight
    # decay-weighted W is a fused-call option only
    assert L.tri_inv_build(ok, ok, ok, ok, p, binding.W_DECAY, None) == binding.ERR_UNSUPPORTED
    # chunk scan: Q, K, W, U, g, O are required; S0 and S_out are optional but must be aligned when given
    scale = ctypes.c_float(1.0)
    assert L.tri_inv_chunk_scan(None, ok, ok, ok, ok, None, ok, None, scale, p, None) == binding.ERR_INVALID_ARG
    assert L.tri_inv_chunk_scan(ok, ok, ok, ok, ok, None, None, None, scale, p, None) == binding.ERR_INVALID_ARG
    assert L.tri_inv_chunk_scan(ok, ok, ok, ok, ok, odd, ok, None, scale, p, None) == binding.ERR_INVALID_ARG
    assert L.tri_inv_chunk_scan(ok, ok, ok, ok, ok, None, ok, None, scale, None, None) == binding.ERR_INVALID_ARG
    wide, _ = binding.make_desc(1, 64, 1, 512, 64, 64, binding.F32)      # d_k beyond the CUDA-core scan's state slice
    assert L.tri_inv_chunk_scan(ok, ok, ok, ok, ok, None, ok, None, scale, ctypes.byref(wide), None) == binding.ERR_UNSUPPORTED


def test_layer_call_validates_on_the_host(lib):
    """Every call below is refused before any device work: one argument is wrong in each."""
    L, binding = lib
    ok, odd, scale = 4096, 4100, ctypes.c_float(1.0)
    for dims in ((1, 640, 2, 128, 128, 64, binding.BF16), (1, 640, 2, 64, 64, 64, binding.F32), (2, 3, 2, 64, 64, 64, binding.F32)):
        d, _ = binding.make_desc(*dims)
        p = ctypes.byref(d)
        need = ctypes.c_size_t(0)
        assert L.tri_inv_gdn_forward_workspace(p, 0, ctypes.byref(need)) == binding.OK
        assert L.tri_inv_gdn_forward_workspace(p, 0, None) == binding.ERR_INVALID_ARG
        assert L.tri_inv_gdn_forward_workspace(None, 0, ctypes.byref(need)) == binding.ERR_INVALID_ARG
        good = dict(Q=ok, K=ok, V=ok, beta=ok, g=ok, S0=ok, O=ok, S=ok, scale=scale, work=ok, bytes=need.value, desc=p, method=0, stream=None)
        call = lambda **kw: L.tri_inv_gdn_forward(*dict(good, **kw).values())
        for name in ("Q", "K", "V", "beta", "g", "O"):
            assert call(**{name: None}) == binding.ERR_INVALID_ARG
        for name in ("Q", "K", "V", "beta", "g", "S0", "O", "S", "work"):
            assert call(**{name: odd}) == binding.ERR_INVALID_ARG
        if need.value:
            assert call(work=None) == binding.ERR_INVALID_ARG and call(bytes=need.value - 1) == binding.ERR_INVALID_ARG
        assert call(desc=None) == binding.ERR_INVALID_ARG
        assert call(method=7) == binding.ERR_UNSUPPORTED and call(method=binding.LEAF_SERIES | binding.PRODUCT_SERIES) == binding.ERR_UNSUPPORTED


def test_layer_call_without_tokens(lib):
    """No token, no workspace: not an error, whatever the scheme (nothing is launched; without a device the status says so)."""
    L, binding = lib
    ok = 4096
    for method in (binding.BLOCK_RECURSIVE, binding.PRODUCT_SERIES):
        for d_k in (128, 192):
            d, _ = binding.make_desc(1, 0, 2, d_k, 128, 64, binding.BF16)
            need = ctypes.c_size_t(1)
            assert L.tri_inv_gdn_forward_workspace(ctypes.byref(d), method, ctypes.byref(need)) == binding.OK and need.value == 0
            rc = L.tri_inv_gdn_forward(ok, ok, ok, ok, ok, None, ok, None, ctypes.c_float(1.0), None, 0, ctypes.byref(d), method, None)
            assert rc in (binding.OK, binding.ERR_CUDA)


def test_scan_warps_wait_as_a_whole():
    """What follows a wait in the scan kernel's warp roles takes the full warp (tcgen05.ld / st, ldmatrix, __syncwarp), so no
    role may branch on the outcome of a wait lane by lane: each branches on wait(), whose lanes agree.  The per-lane
    waits that are left drain a warp that has given up and are not branched on."""
    src = open(os.path.join(ROOT, "paper_2605_21325_b200", "csrc", "scan_kernel.cu")).read()
    roles = src[src.index("if (warp == kControl) {"):src.index("constexpr int kSeqsPerLaunch")]
    assert not re.findall(r"if \([^;{]*mbar_(?:try_)?wait\w*\([^;{]*", roles)


@pytest.mark.parametrize("name", ["scan_kernel.cu", "scan_f32_kernel.cu"])
def test_a_block_that_gives_up_waits_for_the_last_copy_of_every_stage(name):
    """The loop behind a wait that has run out, as the source has it, against the copies that can be on their way: for every chunk at
    which the requests can end, each stage's last one is waited for with its own parity (another parity's wait returns at once)."""
    src = open(os.path.join(ROOT, "paper_2605_21325_b200", "csrc", name)).read()
    m = re.search(r"for \(int c = (requested[^;]*|n_chunks[^;]*); c (<=?) (\w+); \+\+c\)(?: *//[^\n]*)?\s*mbar_wait_bounded\(", src)
    cond, a, b = re.match(r"(.*) \? (.*) : (.*)", m.group(1).replace("cfg::", "")).groups()
    for stages in (2, 3):
        for n_chunks in (1, 2, 5, 32):
            for requested in range(n_chunks):
                env = dict(requested=requested, n_chunks=n_chunks, kStages=stages)
                first = eval(a, {}, env) if eval(cond, {}, env) else eval(b, {}, env)
                last = env[m.group(3)] if m.group(2) == "<=" else env[m.group(3)] - 1
                waited = {(c % stages, c // stages % 2) for c in range(first, last + 1)}
                for c in range(max(0, requested - stages + 1), requested + 1):
                    assert (c % stages, c // stages % 2) in waited, (stages, n_chunks, requested)


def test_scan_roles_that_copy_wait_for_their_copies_when_they_give_up():
    """The scan's roles that issue asynchronous copies and leave their loop where a wait has run out: the last statement of each waits for what it has
    on its way (the gate warp's cp.async groups, the copy warp's bulk loads), and the store warp waits inside the loop, ahead of its next wait."""
    src = open(os.path.join(ROOT, "paper_2605_21325_b200", "csrc", "scan_kernel.cu")).read()
    role = lambda a, b: re.sub(r"//[^\n]*", "", src[src.index("} else if (warp == %s) {" % a):src.index(b)]).strip()   # noqa: E731
    gate, copy = role("kGate", "} else if (warp == kCopy) {"), role("kCopy", "} else if (chain) {")
    assert gate.endswith("if (failed) fetched(Width<0>{});") and "fetch_g(" in gate and "fetch_e(" in gate
    assert copy.endswith("if (failed && lane == 0) drain_copies();") and "issue_copies(" in copy
    store = role("kStore", "if (failed) atomicMax(p.status")
    assert store.index("tma_store_2d(") < store.index("bulk_commit();") < store.index("bulk_wait_read();") < store.index("warp_arrive(bar_of, lane);")


def test_shared_arrays_that_are_read_as_vectors_are_aligned():
    """A static shared array that is read as float4 has its 16 bytes from its declaration, not from where the compiler happens to
    put it: every __shared__ float array is declared with an alignment, or is in a type that has one, where its file reads
    shared memory in fours."""
    import glob
    csrc = os.path.join(ROOT, "paper_2605_21325_b200", "csrc")
    for path in glob.glob(os.path.join(csrc, "*.cu")) + glob.glob(os.path.join(csrc, "*.cuh")):
        src = open(path).read()
        for line in re.findall(r"^.*__shared__.*;", src, flags=re.M):
            m = re.search(r"__shared__\s+(__align__\(16\)\s+)?float\s+(.*);", line)
            if not m or m.group(1) or "extern" in line:
                continue
            for name in re.findall(r"(\w+)(?:\[[^\]]*\])+", m.group(2)):
                assert not re.search(r"<(?:const )?float4\*>\(&?%s\b" % name, src), (os.path.basename(path), name)
