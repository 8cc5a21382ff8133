"""The work this library is used for, as cases that can be timed.

A case is one pass of an encrypted layer: one or several products ct_out = Enc(W x), each with its rescale, on one context
with its rotation keys loaded.  The fields of a case:

  params   CKKS parameter set (workloads.PARAM_SETS)
  D, tau   tiling of the plan; every call's split has b * g = D / tau
  plan     variant of the evaluation: "plain", or letters of c (complex-slot packing), o (one division by P per output),
           h (double hoisting); "coh" is what the benchmark runs
  calls    the products, "d_in x d_out / b x g" each: "1024x4096/16x4 2048x1024/16x4"
  weights  how the weights are held: "cached" (encoded, 8-byte words), "compact" (narrow words), "coef32" (rounded 32-bit
           coefficients), "raw" (fp32, encoded inside the call)
  via      "device" (ciphertexts in device memory), "host" (pinned host buffers in and out), "fold" (device, with the
           partial sums folded inside the output ciphertexts before the rescale)

Ciphertexts and rotation keys are uniform residues, which is what fresh ones look like; weights are N(0, 0.02^2).
"""
import math

import torch

from paper_2606_17421_b200 import bifrost as bf
from paper_2606_17421_b200 import workloads as wl

_FLAG = {"c": bf.BF_PLAN_COMPLEX_PACK, "o": bf.BF_PLAN_MODDOWN_PER_OUTPUT, "h": bf.BF_PLAN_DOUBLE_HOIST}

_GPT2 = "768x2304/16x4 768x768/16x4 768x3072/16x4 3072x768/8x8"
_QWEN3 = "1024x4096/16x4 2048x1024/16x4 1024x6144/32x2 3072x1024/8x8"         # q+k+v, o, gate+up, down
_LLAMA3 = "4096x6144/8x4 4096x4096/8x4 4096x28672/16x2 14336x4096/4x8"        # the same, one layer of an 8B model


def _case(name, params, D, tau, plan, calls, weights="cached", via="device"):
    return dict(name=name, params=params, D=D, tau=tau, plan=plan, calls=calls, weights=weights, via=via)


def listed():
    return [
        # the smallest product: one 64 x 64 tile on a small ring, where latency and launches are everything
        _case("tiny_64x64", "n12", 64, 1, "plain", "64x64/8x8"),
        # the same ring with everything the benchmark's plan switches on, an odd shape, several tiles
        _case("small_ring_odd", "n12", 256, 8, "coh", "300x1000/8x4"),
        # one projection under the prototype's own parameters (60-bit base prime, 30-bit primes: the integer transforms)
        _case("qkv_n13_30bit", "paper_n13", 1024, 4, "plain", "768x2304/16x16"),
        # one projection of a 124M-parameter decoder under the plan a caller gets without flags
        _case("gpt2_qkv_plain", "n15", 1024, 16, "plain", "768x2304/16x4"),
        # one layer of a decode step of that model, weights cached: four products per layer
        _case("gpt2_layer", "n15", 1024, 16, "coh", _GPT2),
        # one layer of a decode step of a 0.6B model, weights cached: the benchmark's headline is 28 of these
        _case("qwen3_layer", "n15", 1024, 16, "coh", _QWEN3),
        # the same layer with the ciphertexts in host memory, as the trusted side hands them over
        _case("qwen3_layer_host", "n15", 1024, 16, "coh", _QWEN3, via="host"),
        # the same layer where the encoded weights do not fit: kept as 32-bit coefficients, transformed on every call
        _case("qwen3_layer_coef32", "n15", 1024, 16, "coh", _QWEN3, weights="coef32"),
        # a ragged projection in the compact cache format, folded inside the ciphertext for a thin client
        _case("ragged_compact_fold", "n15", 1024, 16, "coh", "1500x2500/16x4", weights="compact", via="fold"),
        # a projection beyond the cache budget: encoded inside the call
        _case("qwen3_gate_up_raw", "n15", 1024, 16, "coh", "1024x6144/16x4", weights="raw"),
        # one layer of an 8B model on the large ring, weights cached: the largest products
        _case("llama3_layer", "n16", 1024, 32, "coh", _LLAMA3),
        # attention output projection of that layer, encoded inside the call (a model's encoded form exceeds the card)
        _case("llama3_o_raw", "n16", 1024, 32, "coh", "4096x4096/8x4", weights="raw"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One product of the same ranges: ring, tiling, split, plan, shape, cache format and boundary at random."""
    params = rng.choice(["n12", "paper_n13", "n15", "n15", "n15", "n16"])
    D, tau, splits, most_in, most_out = {
        "n12": lambda: rng.choice([(64, 1, ["8x8", "16x4"], 512, 512), (256, 8, ["8x4", "4x8"], 1024, 2048),
                                   (128, 4, ["8x4", "16x2"], 512, 1024)]),
        "paper_n13": lambda: (1024, 4, ["16x16", "32x8"], 3072, 3072),
        "n15": lambda: rng.choice([(1024, 16, ["16x4", "16x4", "32x2", "8x8"], 4096, 8192)] * 3 + [(512, 32, ["4x4"], 2048, 4096)]),
        "n16": lambda: (1024, 32, ["8x4", "16x2", "4x8"], 8192, 16384),
    }[params]()
    d_in, d_out = _log_int(rng, D // 4, most_in), _log_int(rng, D // 4, most_out)
    if rng.random() < 0.4:                       # the multiples of 64 that real layers have
        d_in, d_out = max(64, d_in // 64 * 64), max(64, d_out // 64 * 64)
    plan = rng.choice(["coh", "coh", "coh", "coh", "plain", "plain", "oh", "co", "h"])
    via = rng.choice(["device", "device", "device", "device", "host", "fold"])
    # (32-bit coefficients do not hold the small rings' wider ones at this scale)
    held = ["cached", "cached", "cached", "cached", "raw"] + (["compact", "coef32"] if params in ("n15", "n16") else ["compact"])
    weights = rng.choice(held)
    if weights in ("raw", "coef32") and d_in * d_out > 4096 * 4096:
        d_out = max(64, 4096 * 4096 // d_in)
    case = _case(None, params, D, tau, plan, "%dx%d/%s" % (d_in, d_out, rng.choice(splits)), weights, via)
    del case["name"]
    return case


class _Call:
    def __init__(self, case, text):
        shape, split = text.split("/")
        self.d_in, self.d_out = (int(v) for v in shape.split("x"))
        self.b, self.g = (int(v) for v in split.split("x"))
        self.n_in = wl.ceil_div(self.d_in, case["D"])
        self.n_out = wl.ceil_div(self.d_out, case["D"] * (2 if "c" in _letters(case) else 1))


def _letters(case):
    return "" if case["plan"] == "plain" else case["plan"]


def _calls(case):
    return [_Call(case, t) for t in case["calls"].split()]


def _rotations(case, n):
    tau, steps = case["tau"], set()
    for c in _calls(case):
        steps |= {k * tau for k in range(1, c.b)} | {j * c.b * tau for j in range(1, c.g)}
    if case["via"] == "fold":
        steps |= {1 << i for i in range(tau.bit_length() - 1)}
    return sorted(s % n for s in steps if s % n)


def _residues(gen, moduli, lead, N):
    out = torch.empty((*lead, len(moduli), N), dtype=torch.int64, device="cuda")
    for m, q in enumerate(moduli):
        out[..., m, :] = torch.randint(0, q, (*lead, N), generator=gen, device="cuda", dtype=torch.int64)
    return out


_stream = None


def _the_stream():
    """A decode loop enqueues everything on one stream of its own."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


class _State:
    """What a program keeps between calls: context, keys, weights, ciphertext buffers."""
    ctx = None

    def __del__(self):
        if self.ctx is not None:
            bf.bf_ctx_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    ps = wl.PARAM_SETS[case["params"]]
    N, primes, P = ps["N"], list(ps["primes"]), ps["special"]
    r, calls = len(primes), _calls(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = _State()
    s.via, s.r, s.calls, s.W, s.handle, s.ct_in, s.ct_full, s.ct_low = case["via"], r, calls, [], [], [], [], []
    flags = sum(_FLAG[f] for f in _letters(case))
    s.ctx = bf.bf_ctx_create(N, primes + [P], r, ps["scale"], bf.bf_plan(case["D"], case["tau"], calls[0].b, calls[0].g, flags),
                             _the_stream().cuda_stream)
    if case["weights"] == "compact":
        bf.bf_set_compact_cache(s.ctx, True)
    if case["weights"] == "coef32":
        bf.bf_set_coefficient_cache(s.ctx, 32)
    steps = _rotations(case, N // 2)
    keys = _residues(gen, primes + [P], (len(steps), r, 2), N)
    torch.cuda.synchronize()
    bf.bf_load_eval_keys(s.ctx, steps, len(steps), keys)
    del keys
    host = case["via"] == "host"
    for c in calls:
        W = torch.randn((c.d_out, c.d_in), generator=gen, device="cuda", dtype=torch.float32) * 0.02
        ct = _residues(gen, primes, (c.n_in, 2), N)
        low = torch.empty((c.n_out, 2, r - 1, N), dtype=torch.int64, device="cpu" if host else "cuda", pin_memory=host)
        torch.cuda.synchronize()
        s.handle.append(None if case["weights"] == "raw" else bf.bf_encode_weights_split(s.ctx, W, c.d_out, c.d_in, c.b, c.g))
        s.W.append(W if case["weights"] == "raw" else None)
        s.ct_in.append(ct.cpu().pin_memory() if host else ct)
        s.ct_full.append(torch.empty((c.n_out, 2, r, N), dtype=torch.int64, device="cuda") if case["via"] == "fold" else None)
        s.ct_low.append(low)
    torch.cuda.synchronize()
    return s


def run(s):
    for c, W, handle, ct, full, low in zip(s.calls, s.W, s.handle, s.ct_in, s.ct_full, s.ct_low):
        if s.via == "host":
            bf.bf_linear_host(s.ctx, ct, c.n_in, handle, W, c.d_out, c.d_in, low, c.n_out)
        elif s.via == "fold":
            bf.bf_linear(s.ctx, ct, c.n_in, handle, W, c.d_out, c.d_in, full, c.n_out)
            bf.bf_fold(s.ctx, full, c.n_out)
            bf.bf_rescale(s.ctx, full, low, c.n_out, s.r)
        else:
            bf.bf_linear_rescaled(s.ctx, ct, c.n_in, handle, W, c.d_out, c.d_in, low, c.n_out)
    return s.ct_low


def work(case):
    """Bytes: ciphertexts in and out as 8-byte words, every rotation key of a call and the weights once, the resident
    ones at the bits their residues have.  Operations: two per multiply-accumulate (products with weights, key-switch
    inner products), three per butterfly of the transforms a call cannot do without, 5 n log2 n per encoded diagonal."""
    ps = wl.PARAM_SETS[case["params"]]
    N, r, letters = ps["N"], len(ps["primes"]), _letters(case)
    ct_bits = sum(q.bit_length() for q in ps["primes"])
    ext_bits = ct_bits + ps["special"].bit_length()
    held = r + 1 if "h" in letters else r                       # primes the weights are held in
    per_poly = 3 * (N // 2) * (N.bit_length() - 1)              # operations of one transform
    nbytes = ops = 0.0
    for c in _calls(case):
        diags, n_giant = c.n_in * c.n_out * c.b * c.g, c.n_out * (c.g - 1)
        n_keys, n_rot = (c.b - 1) + (c.g - 1), c.n_in * (c.b - 1) + n_giant
        polys = 2 * r * c.n_in + n_giant * r + 2 * r * c.n_out  # ciphertexts in, c1 of the giant steps, ciphertexts out
        polys += r * r * ((c.n_in if c.b > 1 else 0) + n_giant)  # digits in every other prime
        if case["via"] == "fold":
            rounds = case["tau"].bit_length() - 1
            n_keys, n_rot = n_keys + rounds, n_rot + rounds * c.n_out
            polys += rounds * c.n_out * (4 * r + r * r)
        nbytes += c.n_in * 2 * r * N * 8 + c.n_out * 2 * (r - 1) * N * 8 + n_keys * r * 2 * N * ext_bits / 8
        if case["weights"] in ("cached", "compact"):
            nbytes += diags * N * (ext_bits if "h" in letters else ct_bits) / 8
        else:
            nbytes += diags * N * 4 if case["weights"] == "coef32" else c.d_in * c.d_out * 4
            polys += diags * held
        if case["weights"] == "raw":
            ops += diags * 5 * (N // 2) * (N.bit_length() - 2)
        ops += 2 * 2 * diags * held * N + 2 * 2 * n_rot * r * (r + 1) * N + polys * per_poly
    return {"bytes": nbytes, "flops": ops}


def tolerance(case):
    return "exact"                                              # residues are whole numbers: one right answer per plan
