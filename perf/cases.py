"""Performance cases of the framework: what is timed, over which range, and what the results must be.

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same ranges.  A case says which public entry points
of ``paper_2605_21325_b200.binding`` a program calls (``call``), on what shape and with which options; ``prepare`` makes what
such a program holds before the call, ``run`` is one pass, ``exact`` the same results in 64-bit torch, written from the
definitions (unit lower triangular solve per chunk, chunk form of the recurrence) without this package's code.

Calls:
  layer   ``gdn_forward``: one Gated-DeltaNet layer (fused build + inversion + WY, then the chunk scan) -> O, final state
  fused   ``fused`` into buffers that the program keeps -> A, W, U
  raw     ``fused_raw`` (front end folded in) into kept buffers -> A, W, U, beta, g
  build   ``build`` into a kept buffer -> A
  kda     ``fused_kda`` + ``chunk_scan_kda``: one layer with a decay per key feature -> A, O, final state

Values: keys ~ N(0,1) normalised per token, values ~ N(0,1), beta = sigmoid(N(0,1)), g = within-chunk cumulative sum of
log sigmoid(N(2,1)); ``keys: "stress"`` un-normalised keys N(0,1)/sqrt(d), beta ~ U(0.9,1), g = 0.
"""
import math
import random

import torch

from paper_2605_21325_b200 import binding

_SIZES = {"float32": 4, "bfloat16": 2}


def _case(name, call, B, T, H, d=128, C=64, dtype="bfloat16", seqs=0, state=False, keys="gdn"):
    """``seqs`` > 0: that many packed sequences with lengths uniform in 1..T (B is 1 then); ``state``: a carried-in state."""
    c = {"call": call, "B": B, "T": T, "H": H, "d": d, "C": C, "dtype": dtype, "seqs": seqs, "state": state, "keys": keys}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one new token for each of eight sequences on their carried states: the smallest call of a serving loop
        _case("layer_decode", "layer", 8, 1, 16, state=True),
        # one short prompt of no round length: launches and latency
        _case("layer_short", "layer", 1, 333, 16),
        # the prefill batch of a GDN layer of Qwen-class size
        _case("layer_prefill", "layer", 4, 4096, 16),
        # one long document through a layer of 32 heads
        _case("layer_long", "layer", 1, 32768, 32),
        # a batch of prompts of mixed lengths, packed: partial last chunks, many more (sequence, head) pairs than SMs
        _case("layer_packed", "layer", 1, 2048, 16, seqs=64),
        # the layer in single precision, as it is run for checking and in small models (head dimension 64)
        _case("layer_fp32", "layer", 2, 2048, 8, d=64, dtype="float32"),
        # the fused call alone with A wanted too (what a training forward keeps), prefill size
        _case("fused_prefill", "fused", 4, 4096, 16),
        # the same with chunks of 128 tokens
        _case("fused_c128", "fused", 2, 8192, 16, C=128),
        # the fused call on what the projections hand over: logits and un-normalised keys
        _case("raw_prefill", "raw", 4, 4096, 16),
        # only the inverses, long context
        _case("build_long", "build", 1, 32768, 32),
        # only the inverses of a few chunks in single precision: the smallest configuration
        _case("build_fp32_small", "build", 1, 256, 2, d=64, dtype="float32"),
        # a layer with one decay per key feature, prefill size
        _case("kda_prefill", "kda", 4, 4096, 16),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    call = rng.choice(["layer", "layer", "layer", "fused", "fused", "raw", "build", "kda"])
    H = rng.choice([2, 3, 4, 6, 8, 12, 16, 20, 24, 32])
    fp32 = call in ("layer", "fused", "build") and rng.random() < 0.25
    d, C, most = 128, 64, 1 << 19
    if fp32:
        d, H, most = rng.choice([64, 128]), rng.choice([2, 3, 4, 6, 8]), 1 << 14   # at most 16,384 (token, head) rows
    elif call in ("fused", "build") and rng.random() < 0.4:
        d, C = rng.choice([(64, 64), (128, 128)])
    rows = _log_int(rng, 64, most)                                                  # (token, head) rows in all
    tokens = max(1, rows // H)
    stress = call in ("fused", "build") and rng.random() < 0.3
    keys = "stress" if stress else "gdn"
    dtype = "float32" if fp32 else "bfloat16"
    longest = 2048 if fp32 else 32768                                               # no sequence is longer than the listed ones
    if rng.random() < 0.3 and tokens >= 64:                                         # packed: 2..64 sequences
        seqs = _log_int(rng, 2, min(64, tokens // 16))
        return _case(None, call, 1, max(1, min(longest, 2 * tokens // seqs)), H, d, C, dtype, seqs, call in ("layer", "kda") and rng.random() < 0.5, keys)
    B = _log_int(rng, 1, min(32, tokens))
    return _case(None, call, B, max(1, min(longest, tokens // B)), H, d, C, dtype, 0, call in ("layer", "kda") and rng.random() < 0.5, keys)


def _lengths(case):
    """Tokens of each sequence: a matter of the case, not of the seed."""
    if not case["seqs"]:
        return [case["T"]] * case["B"]
    r = random.Random(1005 * case["seqs"] + case["T"])
    return [r.randint(1, case["T"]) for _ in range(case["seqs"])]


def _cu_seqlens(case):
    if not case["seqs"]:
        return None
    cu = [0]
    for n in _lengths(case):
        cu.append(cu[-1] + n)
    return cu


def _shape(case):
    """B, T of the tensors."""
    return (1, sum(_lengths(case))) if case["seqs"] else (case["B"], case["T"])


class _Chunks:
    """Between flat tokens [tokens, ...] and padded chunks [sequences, chunks, C, ...]."""

    def __init__(self, case, device):
        lens, C = _lengths(case), case["C"]
        n = (max(lens) + C - 1) // C
        beg = torch.tensor([sum(lens[:i]) for i in range(len(lens))] if case["seqs"] else [i * case["T"] for i in range(len(lens))], device=device)
        ln = torch.tensor(lens, device=device)
        at = torch.arange(n * C, device=device)
        self.real = (at[None] < ln[:, None]).reshape(len(lens), n, C)
        # the last real token before a padded place: of its own chunk wherever that chunk has one
        self.index = (beg[:, None] + torch.minimum(at[None], ln[:, None] - 1)).reshape(len(lens), n, C)
        self.tokens = sum(lens)

    def cut(self, x, fill="zero"):
        """x [tokens, ...] -> chunks; padded places hold zero, or (fill "last") the chunk's last real value, zero in an empty chunk."""
        y = x[self.index]
        keep = self.real if fill == "zero" else self.real.any(-1, keepdim=True).expand_as(self.real)
        return y * keep.reshape(keep.shape + (1,) * (y.dim() - 3)).to(y.dtype)

    def join(self, y):
        out = torch.zeros((self.tokens,) + y.shape[3:], dtype=y.dtype, device=y.device)
        out[self.index[self.real]] = y[self.real]
        return out


def _inputs(case, seed, device="cuda"):
    B, T = _shape(case)
    H, d, dt = case["H"], case["d"], getattr(torch, case["dtype"])
    gen = torch.Generator(device=device).manual_seed(1000003 * (int(seed) % (1 << 40)) + 17)
    normal = lambda *s: torch.randn(*s, device=device, generator=gen)   # noqa: E731
    unit = lambda x: x / x.square().sum(-1, keepdim=True).sqrt()        # noqa: E731
    K, V = normal(B, T, H, d), normal(B, T, H, d).to(dt)
    s = {"V": V}
    if case["call"] == "raw":
        return dict(s, K=K.to(dt), beta=normal(B, T, H), g=normal(B, T, H) + 2)
    gate = (B * T, H, d) if case["call"] == "kda" else (B * T, H)
    if case["keys"] == "stress":
        K, beta = K * d ** -0.5, 0.9 + 0.1 * torch.rand(B, T, H, device=device, generator=gen)
        g = torch.zeros(gate, device=device)
    else:
        K, beta = unit(K), torch.sigmoid(normal(B, T, H))
        ch = _Chunks(case, device)
        g = ch.join(ch.cut(torch.nn.functional.logsigmoid(normal(*gate) + 2)).cumsum(2))
    s.update(K=K.to(dt), beta=beta, g=g.reshape((B, T) + gate[1:]).contiguous())
    if case["call"] in ("layer", "kda"):
        s["Q"] = unit(normal(B, T, H, d)).to(dt)
        s["S0"] = normal(len(_lengths(case)), H, d, d) * d ** -0.5 if case["state"] else None
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s.update(call=case["call"], C=case["C"], cu=_cu_seqlens(case), scale=case["d"] ** -0.5)
    if case["call"] in ("fused", "raw", "build"):   # output buffers that the program keeps, as bench.py does
        A = torch.empty(s["K"].shape[:3] + (case["C"],), device="cuda")
        s["out"] = A
        if case["call"] != "build":
            s["out"] = (A, torch.empty_like(s["K"]), torch.empty_like(s["V"]))
        if case["call"] == "raw":
            s["out"] += (torch.empty_like(s["beta"]), torch.empty_like(s["g"]))
    return s


def run(s):
    C, cu = s["C"], s["cu"]
    if s["call"] == "layer":
        return binding.gdn_forward(s["Q"], s["K"], s["V"], s["beta"], s["g"], C, scale=s["scale"], S0=s["S0"], cu_seqlens=cu)
    if s["call"] == "fused":
        return binding.fused(s["K"], s["V"], s["beta"], s["g"], C, cu_seqlens=cu, out=s["out"])
    if s["call"] == "raw":
        return binding.fused_raw(s["K"], s["V"], s["beta"], s["g"], C, cu_seqlens=cu, out=s["out"])
    if s["call"] == "build":
        return binding.build(s["K"], s["beta"], s["g"], C, cu_seqlens=cu, out=s["out"])
    A, W, U = binding.fused_kda(s["K"], s["V"], s["g"], s["beta"], C, cu_seqlens=cu)
    O, S = binding.chunk_scan_kda(s["Q"], s["K"], W, U, s["g"], C, scale=s["scale"], S0=s["S0"], cu_seqlens=cu)
    return A, O, S


def work(case):
    """Each input read once, each output written once; products of the path, triangular ones by half."""
    lens, H, d, C, es = _lengths(case), case["H"], case["d"], case["C"], _SIZES[case["dtype"]]
    rows = sum(lens) * H                         # (token, head) rows
    call = case["call"]
    tensors = {"layer": 4, "fused": 4, "raw": 4, "build": 1, "kda": 4}[call]     # of d values in storage type (Q, K, V, O / K, V, W, U / K)
    b = rows * (tensors * d * es + 4 + (4 * d if call == "kda" else 4))          # beta and the gate
    if call in ("fused", "raw", "build", "kda"):
        b += rows * C * 4                        # A
    if call == "raw":
        b += rows * 8                            # beta and g out
    f = rows * (C * d + C * C / 3.0)             # N and the inverse
    if call != "build":
        f += rows * 2.0 * C * d                  # W and U
    if call in ("layer", "kda"):
        b += len(lens) * H * d * d * 4 * (2 if case["state"] else 1)
        f += rows * (2.0 * C * d + 6.0 * d * d)  # Q K^T and P U~; W S, Q S and the state increment
    return {"bytes": b, "flops": f}


def tolerance(case):
    # about four times the relative error against exact() that the sizes above show (the results of another correct
    # implementation at the same precision lie as far off, in another direction)
    if case["dtype"] == "float32":
        return {"rel": 2e-6}          # 32-bit sums throughout: 2e-8 .. 2.2e-7 seen, more where the chain is longer
    if case["call"] == "build":
        return {"rel": 1e-4}          # 11-bit significands in the products that join the blocks of A: 1e-5 .. 3e-5 seen
    return {"rel": 1e-2}              # bf16 results of products of bf16 operands: 2.3e-3 .. 4.2e-3 seen


def exact(case, seed):
    s = _inputs(case, seed)
    B, T = _shape(case)
    C, H, d, call = case["C"], case["H"], case["d"], case["call"]
    ch = _Chunks(case, "cuda")

    def cut(x, fill="zero"):                     # [B, T, H, ...] -> [sequences, H, chunks, C, ...] in 64 bits
        return ch.cut(x.reshape((B * T,) + x.shape[2:]).double(), fill).movedim(3, 1)

    def back(y):                                 # and back, to [B, T, H, ...]
        z = ch.join(y.movedim(1, 3))
        return z.reshape((B, T) + z.shape[1:])

    K, beta = cut(s["K"]), cut(s["beta"])[..., None]
    low = torch.ones(C, C, device="cuda", dtype=torch.bool).tril(-1)
    if call == "raw":
        norm = K.square().sum(-1, keepdim=True).sqrt()
        K = K / torch.where(norm > 0, norm, torch.ones_like(norm))
        beta_out = torch.sigmoid(s["beta"].double())
        beta = cut(beta_out)[..., None]
        g = cut(torch.nn.functional.logsigmoid(s["g"].double())).cumsum(3)
        g_out = back(g)
    else:
        g = cut(s["g"], "last")
    if call == "kda":
        mid = g[:, :, :, C // 2: C // 2 + 1]
        Kp, Km = K * torch.exp(g - mid), K * torch.exp(mid - g)
        N = torch.where(low, beta * (Kp @ Km.mT), 0.0)
        gamma = torch.exp(g)
    else:
        decay = torch.exp(torch.where(low, g[..., :, None] - g[..., None, :], 0.0))
        N = torch.where(low, beta * (K @ K.mT) * decay, 0.0)
        gamma = torch.exp(g)[..., None]
    eye = torch.eye(C, device="cuda", dtype=torch.float64)
    A = torch.linalg.solve_triangular(eye + N, eye.expand_as(N), upper=False, unitriangular=True)
    del N
    if call == "build":
        return back(A)
    U = A @ (beta * cut(s["V"]))
    if call in ("fused", "raw"):
        W = A @ (beta * K)
        return (back(A), back(W), back(U)) + ((beta_out, g_out) if call == "raw" else ())
    W = A @ (beta * gamma * K)
    Q, scale = cut(s["Q"]), d ** -0.5
    low = torch.ones(C, C, device="cuda", dtype=torch.bool).tril()
    if call == "kda":
        P = torch.where(low, (Q * torch.exp(g - mid)) @ Km.mT, 0.0)
    else:
        P = torch.where(low, (Q @ K.mT) * torch.exp(torch.where(low, g[..., :, None] - g[..., None, :], 0.0)), 0.0)
    S = s["S0"].double() if s["S0"] is not None else torch.zeros(K.shape[0], H, d, d, device="cuda", dtype=torch.float64)
    O = torch.empty_like(U)
    for c in range(K.shape[2]):
        u = U[:, :, c] - W[:, :, c] @ S
        O[:, :, c] = scale * ((Q[:, :, c] * gamma[:, :, c]) @ S + P[:, :, c] @ u)
        last = gamma[:, :, c, -1:]               # a padded place repeats the chunk's last decay
        if call == "kda":
            S = last.mT * S + (K[:, :, c] * torch.exp(g[:, :, c, -1:] - g[:, :, c])).mT @ u
        else:
            S = last * S + (K[:, :, c] * torch.exp(g[:, :, c, -1:] - g[:, :, c])[..., None]).mT @ u
    return (back(A), back(O), S) if call == "kda" else (back(O), S)
