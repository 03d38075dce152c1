"""GPU tests of the layer forward's routes (tri_inv_gdn_forward).

Token by token: fp32 arithmetic on the stored inputs, against the fp64 recurrence: fp32 storage 1e-5 of max|O| (at most 16
steps of sums of up to 128 terms, 2^-24 each), bf16 storage 2^-8 (the output's own rounding), the state 1e-5.
"""
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
