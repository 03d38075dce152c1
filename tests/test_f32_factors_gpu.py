"""GPU tests of the single-precision build / fused kernel (C = 64, head dimensions up to 128), against the fp64 oracle at the
1e-5 bound of fp32 storage and arithmetic, at the edges of its instances and tiles."""
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


# padded and full head dimensions on both sides of the two instances, a last column group that is cut, one token, one token
# over a chunk, packed sequences with an empty one, more matrices than blocks that fit on the chip
CASES = [
    ("d8_v8", 1, 70, 1, 8, 8, None),
    ("d64", 2, 65, 3, 64, 64, None),
    ("d64_v24_ragged", 1, 0, 3, 64, 24, np.array([0, 1, 65, 65, 192, 321], np.int32)),
    ("d72_v128", 2, 129, 2, 72, 128, None),
    ("d128_v40", 1, 63, 2, 128, 40, None),
    ("many", 5, 128, 64, 64, 64, None),
]


@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("name,B,T,H,d_k,d_v,cu", CASES, ids=[c[0] for c in CASES])
def test_f32_factors_against_the_oracle(bnd, name, B, T, H, d_k, d_v, cu, shifted):
    if cu is not None:
        T = int(cu[-1])
    inp = wl.make(name, B, T, H, d_k, d_v, 64, wl.F32, seed=800 + d_k + d_v, cu_seqlens=cu)
    A_ref = (oracle.build_A_shifted if shifted else oracle.build_A)(inp.K, inp.beta, inp.g, 64, cu_seqlens=cu)
    W_ref, U_ref = oracle.wy(A_ref, inp.K, inp.V, inp.beta, 64, cu_seqlens=cu)
    dev = bnd.to_device(inp)
    method = bnd.GATE_SHIFTED if shifted else bnd.BLOCK_RECURSIVE
    A = bnd.build(dev["K"], dev["beta"], dev["g"], 64, method=method, cu_seqlens=cu)
    out = tuple(torch.full_like(x, float("nan")) for x in (A, dev["K"], dev["V"]))
    bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], 64, method=method, cu_seqlens=cu, out=out)
    torch.cuda.synchronize()
    assert torch.equal(A.view(torch.int32), out[0].view(torch.int32))
    for x, ref in zip(out, (A_ref, W_ref, U_ref)):
        assert max_ratio(bnd.to_numpy_f64(x), ref) <= 1e-5
    if not shifted:   # the decay-weighted W
        Kg = inp.K.astype(np.float64) * np.exp(inp.g.astype(np.float64))[..., None]
        Wd_ref, _ = oracle.wy(A_ref, Kg, None, inp.beta, 64, cu_seqlens=cu)
        _, Wd, Ud = bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], 64, method=bnd.W_DECAY, cu_seqlens=cu, want_A=False)
        torch.cuda.synchronize()
        assert max_ratio(bnd.to_numpy_f64(Wd), Wd_ref) <= 1e-5 and torch.equal(Ud, out[2])


def test_f32_factors_keep_a_tokens_infinity_to_later_rows(bnd):
    """Rows before a token with a non-finite key or value are those of the chunk without it."""
    inp = wl.make("inf", 1, 64, 2, 64, 64, 64, wl.F32, seed=830)
    dev = bnd.to_device(inp)
    ref = bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], 64)
    for t in (5, 20, 40, 63):
        K, V = dev["K"].clone(), dev["V"].clone()
        K[0, t] = float("inf")
        V[0, t] = float("nan")
        out = bnd.fused(K, V, dev["beta"], dev["g"], 64)
        torch.cuda.synchronize()
        for x, r in zip(out, ref):
            assert torch.equal(x[:, :t], r[:, :t])


def test_static_packed_call_gives_the_ordinary_calls_bits_in_fp32(bnd):
    cu = np.array([0, 1, 65, 65, 192, 321], np.int32)
    for d_k, d_v in ((64, 64), (128, 40), (136, 64)):   # both instances, and a dimension that they do not take
        inp = wl.make("static", 1, 321, 3, d_k, d_v, 64, wl.F32, seed=840, cu_seqlens=cu)
        dev = bnd.to_device(inp)
        ref = bnd.fused(dev["K"], dev["V"], dev["beta"], dev["g"], 64, cu_seqlens=cu)
        got = bnd.fused_packed_static(dev["K"], dev["V"], dev["beta"], dev["g"], 64, cu)
        torch.cuda.synchronize()
        for x, r in zip(got, ref):
            assert torch.equal(x, r)
