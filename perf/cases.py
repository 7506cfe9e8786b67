"""What is timed: the calls that a program built on this package makes, over the sizes it makes them at.

Five kinds of case.

``block``    the linears of one transformer block (q/k/v, o, gate/up, down) as four grouped calls on prepared layers:
             what a serving engine runs once per layer and step.  ``tokens`` is 1 for a single sequence, tens for a
             decode batch, hundreds to thousands for prefill; 4, 6 or 8 bit codes, symmetric or asymmetric.
``a16``      the same linears at the weight-only operating point (bf16 rotated activations), one call per linear.
``linear``   one linear from raw tensors (no prepared handle): a custom-op slot, an evaluation script.
``binarize`` the last step of the offline pipeline: rows of a weight matrix to packed signs, scales and shifts.
``pack``     packing of already rotated weights.

Activations are heavy-tailed with a few outlier channels (Student-t, nu = 3), Kronecker factors are Haar-orthogonal,
signs are fair coin flips, scales log-normal, low-rank factors small Gaussians: the recipe of the parity tests.
"""
import math

import numpy as np
import torch

from paper_2605_00422_b200 import bwla

DEV = "cuda"

# (n1, n2) of a hidden width, and the attention widths that go with it; (n1, n2) of an MLP width
HIDDEN = [(32, 64), (48, 64), (64, 64), (64, 80), (64, 128)]
MLP = [(64, 88), (64, 128), (86, 128), (108, 128), (112, 128), (160, 160)]
# a single linear's input width
LINEAR = [(32, 32), (32, 64), (64, 64), (64, 80), (64, 128), (86, 128), (108, 128), (160, 160)]


def _block(name, kind, hidden, attn, kv, mlp, r, tokens, bits=6, asym=False, mu=False):
    return {"name": name, "kind": kind, "h1": hidden[0], "h2": hidden[1], "a1": attn[0], "a2": attn[1], "kv": kv,
            "f1": mlp[0], "f2": mlp[1], "r": r, "tokens": tokens, "bits": bits, "asym": asym, "mu": mu}


def listed():
    wide = ((64, 80), (64, 128), 1024, (160, 160), 64)      # Qwen3-32B's linears
    plain = ((64, 64), (64, 64), 4096, (86, 128), 32)       # LLaMA-2-7B's linears
    return [
        # one sequence being decoded: launches and latency
        _block("block_decode_1", "block", *wide, 1),
        # the batch that the benchmark quotes
        _block("block_decode_16", "block", *wide, 16),
        # a larger, ragged decode batch in the paper's stated quantiser (asymmetric, with the row shift), 4-bit codes
        _block("block_decode_50_asym", "block", *plain, 50, bits=4, asym=True, mu=True),
        # a short prompt, or a chunk of a chunked prefill: a ragged number of tokens, 8-bit codes
        _block("block_prefill_333", "block", *plain, 333, bits=8),
        # long prompts
        _block("block_prefill_4096", "block", *wide, 4096),
        # the weight-only operating point, decode and prefill
        _block("a16_decode_16", "a16", *wide, 16),
        _block("a16_prefill_1024", "a16", *plain, 1024, mu=True),
        # the smallest call: one linear, one token, from raw tensors
        {"name": "linear_1", "kind": "linear", "n1": 64, "n2": 64, "N": 4096, "r": 32, "tokens": 1, "bits": 6, "mu": False},
        # a raw call with an odd number of outputs and tokens, no low-rank branch
        {"name": "linear_129_ragged", "kind": "linear", "n1": 64, "n2": 80, "N": 8193, "r": 0, "tokens": 129, "bits": 6, "mu": True},
        # the widest down projection at low bit width
        {"name": "linear_2048_down", "kind": "linear", "n1": 160, "n2": 160, "N": 5120, "r": 64, "tokens": 2048, "bits": 4, "mu": False},
        # offline: one attention projection in fp32, and one MLP matrix of bf16 weights that are rotated already
        {"name": "binarize_5120", "kind": "binarize", "n1": 64, "n2": 80, "N": 5120, "dtype": "f32"},
        {"name": "pack_25600", "kind": "pack", "K": 5120, "N": 25600, "dtype": "bf16"},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["block", "block", "block", "a16", "linear", "linear", "binarize", "pack"])
    if kind in ("block", "a16"):
        h = rng.choice(HIDDEN)
        attn = (64, 128) if h == (64, 80) else h
        kv = rng.choice([512, 1024, attn[0] * attn[1]])
        f = rng.choice([m for m in MLP if m[0] * m[1] > h[0] * h[1]])
        c = _block("", kind, h, attn, kv, f, rng.choice([0, 16, 32, 64]), 1, mu=rng.random() < 0.3)
        del c["name"]
        # no more work than the longest listed prompt
        most = work(listed()[4])["flops"] // work(c)["flops"]
        c["tokens"] = _log_int(rng, 1, min(most, 4096 if kind == "block" else 1024))
        if kind == "block":
            c["bits"] = rng.choice([4, 6, 6, 8])
            c["asym"] = rng.random() < 0.3
        return c
    if kind == "linear":
        n1, n2 = rng.choice(LINEAR)
        return {"kind": kind, "n1": n1, "n2": n2, "N": _log_int(rng, 512, 12288), "r": rng.choice([0, 16, 32, 64]),
                "tokens": _log_int(rng, 1, 2048), "bits": rng.choice([4, 6, 6, 8]), "mu": rng.random() < 0.3}
    if kind == "binarize":
        n1, n2 = rng.choice(LINEAR[:6])
        return {"kind": kind, "n1": n1, "n2": n2, "N": _log_int(rng, 512, max(512, 5120 * 5120 // (n1 * n2))), "dtype": rng.choice(["f32", "bf16"])}
    K = rng.choice([2048, 4096, 5120, 8192, 11008])
    return {"kind": "pack", "K": K, "N": _log_int(rng, 512, 25600 * 5120 // K), "dtype": rng.choice(["f32", "bf16"])}


# ---- shapes ------------------------------------------------------------------------------------------------------
def _groups(c):
    """[((n1, n2) of the shared input, [output widths])] of a block, in the order they run."""
    h, a, f = (c["h1"], c["h2"]), (c["a1"], c["a2"]), (c["f1"], c["f2"])
    hidden, attn, mlp = h[0] * h[1], a[0] * a[1], f[0] * f[1]
    return [(h, [attn, c["kv"], c["kv"]]), (a, [hidden]), (h, [mlp, mlp]), (f, [hidden])]


def _linears(c):
    """[(n1, n2, N, reads an input of its own)]"""
    if c["kind"] == "linear":
        return [(c["n1"], c["n2"], c["N"], True)]
    return [(n[0], n[1], N, i == 0) for n, outs in _groups(c) for i, N in enumerate(outs)]


# ---- inputs ------------------------------------------------------------------------------------------------------
def _haar(n, rng):
    q, r = np.linalg.qr(rng.standard_normal((n, n)))
    return torch.from_numpy(np.ascontiguousarray(q * np.sign(np.diag(r))[None, :], dtype=np.float32)).to(DEV)


def _weights(n1, n2, N, r, mu, rng, g):
    """P1, P2, packed signs, alpha, U, V, mu of one linear."""
    K = n1 * n2
    packed = torch.randint(-2 ** 31, 2 ** 31, (N, K // 32), dtype=torch.int64, device=DEV, generator=g).to(torch.int32)
    alpha = torch.exp(-4.0 + 0.3 * torch.randn(N, device=DEV, generator=g))
    U = (0.01 * torch.randn(N, r, device=DEV, generator=g)).to(torch.bfloat16) if r else None
    V = (0.01 * torch.randn(r, K, device=DEV, generator=g)).to(torch.bfloat16) if r else None
    shift = 0.002 * torch.randn(N, device=DEV, generator=g) if mu else None
    return _haar(n1, rng), _haar(n2, rng), packed, alpha, U, V, shift


def _activations(M, K, g):
    x = torch.randn(M, K, device=DEV, generator=g)
    chi = torch.zeros(M, K, device=DEV)
    for _ in range(3):
        chi += torch.randn(M, K, device=DEV, generator=g).square_()
    x /= chi.div_(3.0).sqrt_()
    x[:, torch.randperm(K, device=DEV, generator=g)[:8]] *= 50.0
    return x.to(torch.bfloat16)


def prepare(case, seed):
    c = case
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    rng = np.random.default_rng(seed)
    if c["kind"] in ("binarize", "pack"):
        K = c["n1"] * c["n2"] if c["kind"] == "binarize" else c["K"]
        w = (0.02 * torch.randn(c["N"], K, device=DEV, generator=g)).to(torch.float32 if c["dtype"] == "f32" else torch.bfloat16)
        if c["kind"] == "pack":
            return {"kind": "pack", "w": w, "packed": torch.empty(c["N"], K // 32, dtype=torch.int32, device=DEV)}
        ws = torch.zeros(bwla.bwla_binarize_workspace_bytes(K), dtype=torch.uint8, device=DEV)
        return {"kind": "binarize", "w": w, "P1": _haar(c["n1"], rng), "P2": _haar(c["n2"], rng), "ws": ws}
    M = c["tokens"]
    if c["kind"] == "linear":
        K = c["n1"] * c["n2"]
        return {"kind": "linear", "bits": c["bits"], "x": _activations(M, K, g),
                "w": _weights(c["n1"], c["n2"], c["N"], c["r"], c["mu"], rng, g),
                "out": torch.empty(M, c["N"], dtype=torch.bfloat16, device=DEV),
                "ws": bwla.new_workspace(M, K, c["N"], c["r"], c["bits"], DEV)}
    # a block: every linear a prepared layer, one workspace for all of its calls
    groups, need = [], 256
    for (n1, n2), widths in _groups(c):
        layers = []
        for N in widths:
            P1, P2, packed, alpha, U, V, mu = _weights(n1, n2, N, c["r"], c["mu"], rng, g)
            layers.append(bwla.Layer(P1, P2, c["bits"], packed, alpha, U, V, mu, asymmetric=c["asym"]))
        outs = [torch.empty(M, N, dtype=torch.bfloat16, device=DEV) for N in widths]
        groups.append((layers, _activations(M, n1 * n2, g), outs))
        need = max([need] + ([bwla.bwla_group_workspace_bytes(layers, M)] if c["kind"] == "block"
                             else [bwla.bwla_w1a16_workspace_bytes(l, M) for l in layers]))
    return {"kind": c["kind"], "groups": groups, "ws": torch.zeros(need, dtype=torch.uint8, device=DEV)}


# ---- one pass ----------------------------------------------------------------------------------------------------
def run(state):
    s = state
    if s["kind"] == "block":
        for layers, x, outs in s["groups"]:
            bwla.bwla_w1ax_linear_group(layers, x, outs, s["ws"])
        return [o for _, _, outs in s["groups"] for o in outs]
    if s["kind"] == "a16":
        for layers, x, outs in s["groups"]:
            for layer, out in zip(layers, outs):
                bwla.bwla_layer_w1a16_linear(layer, x, out, s["ws"])
        return [o for _, _, outs in s["groups"] for o in outs]
    if s["kind"] == "linear":
        P1, P2, packed, alpha, U, V, mu = s["w"]
        return bwla.bwla_w1ax_linear(s["x"], P1, P2, s["bits"], packed, alpha, U, V, mu, s["out"], s["ws"])
    if s["kind"] == "binarize":
        return bwla.bwla_binarize_rows(s["w"], s["P1"], s["P2"], s["ws"])
    return bwla.bwla_pack_signs(s["w"], s["packed"])


# ---- what a pass cannot do without ---------------------------------------------------------------------------------
def work(case):
    c = case
    if c["kind"] == "pack":
        n = c["N"] * c["K"]
        return {"bytes": n * (4 if c["dtype"] == "f32" else 2) + n // 8, "flops": 0}
    if c["kind"] == "binarize":
        K = c["n1"] * c["n2"]
        n = c["N"] * K
        return {"bytes": n * (4 if c["dtype"] == "f32" else 2) + n // 8 + 8 * c["N"] + 4 * (c["n1"] ** 2 + c["n2"] ** 2),
                "flops": 2 * n * (c["n1"] + c["n2"])}
    M, r, nbytes, flops = c["tokens"], c["r"], 0, 0
    for n1, n2, N, own_input in _linears(c):
        K = n1 * n2
        nbytes += N * K // 8 + 2 * r * (N + K) + (8 if c["mu"] else 4) * N + 4 * (n1 * n1 + n2 * n2) + 2 * M * N
        nbytes += 2 * M * K if own_input else 0
        flops += 2 * M * K * N + 2 * M * r * (N + K) + 2 * M * K * (n1 + n2)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "pack":
        return "exact"
    if kind == "binarize":
        # fp32 statistics of rows that are rotated to about 1e-6 of their largest value: the mean is some K^-1/2 of that
        # value, so 1e-4 relative; a sign differs only where the rotated weight is within 1e-6 of the row's range of the mean
        return {"rel": 1e-4, "max": 1e-3, "differ": 1e-3}
    if kind == "a16":
        # bf16 activations and outputs
        return {"rel": 1e-2, "max": 0.1}
    # bf16 outputs; a rotated activation within 1e-6 of full scale of a rounding boundary may get the next code, which
    # moves every output of its token by one step of the scale
    return {"rel": 1e-2, "max": 0.25}
