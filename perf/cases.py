"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one call (or one SPSA step) over a parameter set: the perturbation, the fused update of K
machines' pairs, the update from the weight backup, the replay of missed iterations, the checksum
and the perturbation of 4-bit weights. Parameter sets are shaped like OPT decoders or ragged, from a
thousand elements to billions, each tensor in an allocation of its own or packed without gaps.

``prepare`` makes parameters, table, seeds and byte codes from the seed alone; ``run`` makes the
calls; ``exact`` restates the method in 64-bit torch arithmetic without this library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2306_10015_gb300 as jb

EPS = 1e-3       # SPSA perturbation scale
QSCALE = 16.0    # scale S of the byte code
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}

# OPT decoder shapes: layers, d_model, ffn, vocabulary, learned positions.
OPT = {
    "opt-125m": (12, 768, 3072, 50272, 2050),
    "opt-1.3b": (24, 2048, 8192, 50272, 2050),
    "opt-6.7b": (32, 4096, 16384, 50272, 2050),
}

# Largest (elements x pairs) that exact() evaluates: a few seconds of 64-bit torch on the GPU.
EXACT_WORK = 1.2e10

# Lane operations that one Gaussian cannot do without: a quarter Philox4x32-10 block (10), half a
# Box-Muller pair (4) and the multiply-add that applies it (1).
OPS = 15


def listed():
    return [
        # One whole SPSA step of the toy quadratic: three perturbations, the byte, K = 4 machines.
        # Five calls on 4 MB: what a call costs counts as much as the kernels.
        dict(name="step-toy-f32-k4", op="step", dtype="f32", layout="ragged", packed=False,
             tensors=1, numel=1 << 20, sizes_seed=0, K=4, lr=1e-4),
        # The smallest call: a bias- and adapter-sized set of odd tensors, one perturbation.
        dict(name="perturb-small-bf16", op="perturb", dtype="bf16", layout="ragged", packed=False,
             tensors=40, numel=81_111, sizes_seed=1, K=1),
        # A checkpoint's tensors used in place, packed without gaps: odd sizes put most tensors
        # off the 16-byte grid of their flat offsets.
        dict(name="update-packed-bf16-k16", op="update", dtype="bf16", layout="ragged", packed=True,
             tensors=200, numel=20_000_003, sizes_seed=2, K=16, lr=1e-6),
        # The perturb/restore passes around the loss evaluations, fp32 and bf16 models.
        dict(name="perturb-125m-f32", op="perturb", dtype="f32", layout="opt-125m", K=1),
        dict(name="perturb-1.3b-bf16", op="perturb", dtype="bf16", layout="opt-1.3b", K=1),
        # The step update of a small fp32 model, K = 16 machines.
        dict(name="update-125m-f32-k16", op="update", dtype="f32", layout="opt-125m", K=16,
             lr=1e-6),
        # A single machine training alone: one pair to apply.
        dict(name="update-1.3b-bf16-k1", op="update", dtype="bf16", layout="opt-1.3b", K=1,
             lr=1e-4),
        # The headline: K = 64 machines on a large bf16 model. The largest case.
        dict(name="update-6.7b-bf16-k64", op="update", dtype="bf16", layout="opt-6.7b", K=64,
             lr=1e-6),
        # The update read from the weight backup, which is refreshed in the same pass.
        dict(name="restore-1.3b-bf16-k4", op="restore", dtype="bf16", layout="opt-1.3b", K=4,
             lr=1e-6, refresh=True),
        # A late joiner's catch-up: 24 missed iterations of one to eight pairs.
        dict(name="replay-125m-bf16", op="replay", dtype="bf16", layout="opt-125m", K=24 * 4,
             lr=1e-6, steps=24),
        # The model hash that peers compare.
        dict(name="checksum-1.3b-bf16", op="checksum", dtype="bf16", layout="opt-1.3b", K=0),
        # The perturbation of 4-bit weights.
        dict(name="perturb-q4-1.3b", op="q4", dtype="q4", layout="opt-1.3b", K=1),
    ]


def draw(rng):
    """One more case: every operation, type and layout, sizes and K spread over their logarithm."""
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["step", "perturb", "perturb", "update", "update", "update", "restore",
                     "replay", "checksum", "q4"])
    numel = log_uniform(1 << 10, 1 << 30) | 1
    case = dict(op=op, dtype="q4" if op == "q4" else rng.choice(["f32", "bf16"]), layout="ragged",
                packed=op != "q4" and rng.random() < 0.3,
                tensors=min(log_uniform(1, 1200), numel // 16), numel=numel,
                sizes_seed=rng.randrange(1 << 30), K=1)
    if op in ("step", "update", "restore", "replay"):
        case["K"] = min(log_uniform(1, 512), max(1, int(1e11 / numel)))
        case["lr"] = rng.choice([1e-6, 1e-4])
    if op == "restore":
        case["refresh"] = rng.random() < 0.5
    if op == "replay":
        case["steps"] = min(case["K"], log_uniform(1, 64))
    if op == "checksum":
        case["K"] = 0
    return case


# --- parameter sets -----------------------------------------------------------------

def _sizes(case):
    """(elements, kind) of each tensor, in order; kind: "w" weight, "1" gain, "0" bias."""
    if case["layout"] == "ragged":
        n, total = case["tensors"], case["numel"]
        if n == 1:
            return [(total, "w")]
        g = np.random.default_rng(case["sizes_seed"])
        w = np.exp(1.5 * g.standard_normal(n))
        return [(max(1, int(v)), "w") for v in w / w.sum() * total]
    L, d, F, V, P = OPT[case["layout"]]
    layer = [(d * d, "w"), (d, "0")] * 4 + [(d, "1"), (d, "0"), (F * d, "w"), (F, "0"),
                                            (d * F, "w"), (d, "0"), (d, "1"), (d, "0")]
    return [(V * d, "w"), (P * d, "w")] + layer * L + [(d, "1"), (d, "0")]


def _plan(case):
    """Tensor sizes, their flat offsets, and where each starts in the one buffer that holds them
    (in elements): on 512-byte boundaries as separate allocations are, or packed without gaps."""
    sizes = [n for n, _ in _sizes(case)]
    offsets = jb.default_flat_offsets(sizes)
    step = 1 if case.get("packed") else 512
    starts, at = [], 0
    for n in sizes:
        starts.append(at)
        at = -(-(at + n) // step) * step
    return sizes, offsets, starts, at


def _values(case, seed):
    """The parameters: weights N(0, 0.02) (N(0, 1) for the one-tensor toy set), gains 1, biases 0."""
    sizes, _, starts, total = _plan(case)
    dtype = DTYPES.get(case["dtype"], torch.float32)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    buf = torch.empty(total, dtype=dtype, device="cuda")
    buf.normal_(0.0, 1.0 if case["op"] == "step" else 0.02, generator=g)
    for (n, kind), at in zip(_sizes(case), starts):
        if kind != "w":
            buf[at:at + n] = float(kind)
    return buf


def _pairs(case, seed):
    """K distinct (machine, step, sample) seeds and uniform byte codes."""
    K = max(1, case["K"])
    g = np.random.default_rng([seed, 7])
    seeds = np.zeros(K, dtype=jb.SEED_DTYPE)
    seeds["machine_id"] = g.integers(0, 2**64, size=K, dtype=np.uint64)
    seeds["step"] = g.integers(0, 100_000)
    seeds["sample_id"] = np.arange(K) % 3
    return seeds, g.integers(-128, 128, size=K).astype(np.int8)


def _step_sizes(case, seed):
    """Pairs in each of a replay's iterations: about K in all, at least one each."""
    T, K = case["steps"], case["K"]
    cut = np.sort(np.random.default_rng([seed, 8]).choice(np.arange(1, K), T - 1, replace=False)) \
        if T > 1 else np.zeros(0, dtype=np.int64)
    return np.diff(np.concatenate([[0], cut, [K]])).astype(int)


def _q4_levels():
    """16 quantiles of N(0, 1) scaled to [-1, 1] (the levels of the 4-bit code), in 64 bits."""
    d = 1.0 / 32
    p = [d + (0.5 - d) * j / 7 for j in range(8)] + [0.5 + (0.5 - d) * j / 8 for j in range(1, 9)]
    x = torch.special.ndtri(torch.tensor(p, dtype=torch.float64))
    x[7] = 0.0
    return x / x.abs().max()


def _q4_parameters(case, seed):
    """Codes (two per byte) and fp32 scales of N(0, 0.02) weights, and where each tensor starts."""
    sizes, _, _, _ = _plan(case)
    code_at, scale_at, c, s = [], [], 0, 0
    for n in sizes:
        code_at.append(c)
        scale_at.append(s)
        c += -(-((n + 1) // 2) // 512) * 512
        s += -(-((n + 63) // 64) // 128) * 128
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    # absolute maxima of 64 draws lie around 2.5 standard deviations
    scale = (torch.rand(s, device="cuda", generator=g) * 0.04 + 0.035).float()
    mid = _q4_levels()
    mid = ((mid[1:] + mid[:-1]) / 2).float().cuda()
    codes = torch.empty(c, dtype=torch.uint8, device="cuda")
    for i in range(0, c, 1 << 26):
        n = min(1 << 26, c - i)
        w = torch.randn(2, n, device="cuda", generator=g) * 0.4
        k = torch.bucketize(w, mid, out_int32=True)
        codes[i:i + n] = (k[0] + 16 * k[1]).to(torch.uint8)
    return codes, scale, code_at, scale_at


def prepare(case, seed):
    sizes, offsets, starts, _ = _plan(case)
    seeds, codes = _pairs(case, seed)
    state = dict(case=case, seeds=seeds, codes=codes, seed=tuple(int(v) for v in seeds[0]))
    if case["op"] == "q4":
        packed, scale, ca, sa = _q4_parameters(case, seed)
        tensors = [(packed[a:a + (n + 1) // 2], scale[b:b + (n + 63) // 64], n)
                   for n, a, b in zip(sizes, ca, sa)]
        state.update(packed=packed, scale=scale, table=jb.Q4Table(tensors, offsets))
        return state
    theta = _values(case, seed)
    state["theta"] = theta
    state["table"] = jb.ParamTable([theta[a:a + n] for n, a in zip(sizes, starts)], offsets)
    if case["op"] == "restore":
        state["out"] = torch.zeros_like(theta)
        state["out_table"] = jb.ParamTable(
            [state["out"][a:a + n] for n, a in zip(sizes, starts)], offsets)
    elif case["op"] == "checksum":
        state["sum"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    elif case["op"] == "replay":
        steps, at = [], 0
        for k in _step_sizes(case, seed):
            steps.append((seeds[at:at + k], codes[at:at + k], case["lr"], 1.0))
            at += k
        state["steps"] = steps
    elif case["op"] == "step":
        state["loss"] = prepare_loss(seed)
    return state


def run(state):
    case, table = state["case"], state["table"]
    op = case["op"]
    if op == "perturb":
        jb.jb_perturb(table, state["seed"], EPS)
        return state["theta"]
    if op == "update":
        jb.jb_apply_updates(table, state["seeds"], state["codes"], case["lr"], 1.0, QSCALE)
        return state["theta"]
    if op == "step":
        jb.jb_perturb(table, state["seed"], EPS)
        jb.jb_perturb(table, state["seed"], -2 * EPS)
        jb.jb_perturb(table, state["seed"], EPS)
        state["codes"][0] = jb.jb_quantize_grad(state["loss"], QSCALE)
        jb.jb_apply_updates(table, state["seeds"], state["codes"], case["lr"], float(case["K"]),
                            QSCALE)
        return state["theta"]
    if op == "restore":
        jb.jb_apply_updates_from(table, state["out_table"], state["seeds"], state["codes"],
                                 case["lr"], 1.0, QSCALE, write_src=case["refresh"])
        return [state["out"], state["theta"]]
    if op == "replay":
        jb.jb_replay_updates(table, state["steps"], QSCALE)
        return state["theta"]
    if op == "checksum":
        jb.jb_checksum(table, state["sum"])
        return state["sum"]
    jb.jb_perturb_q4(table, state["seed"], EPS)
    return [state["packed"], state["scale"]]


def work(case):
    n, op = sum(_plan(case)[0]), case["op"]
    size = {"f32": 4.0, "bf16": 2.0, "q4": 0.5 + 4.0 / 64}[case["dtype"]]
    passes = {"perturb": 2, "update": 2, "step": 8, "replay": 2, "checksum": 1, "q4": 2,
              "restore": 3 if case.get("refresh") else 2}[op]
    draws = {"step": case["K"] + 3, "checksum": 0}.get(op, case["K"])
    # the checksum: four Philox rounds of four operations for each 16 bytes
    flops = n * size if op == "checksum" else float(OPS) * n * draws
    return {"bytes": n * size * passes, "flops": flops}


def tolerance(case):
    if case["op"] == "checksum":
        return "exact"
    if case["op"] == "q4":
        # the scale is one fp32 value of the block (2.7e-8 against 64 bits); a weight within fp32
        # error of the middle of two levels takes either (4e-8 of the bytes against 64 bits, and
        # a sample of four million bytes resolves 2.5e-7)
        return {"rel": 2e-7, "max": 1e-6, "differ": 1e-6}
    if case["dtype"] == "bf16":
        # one bf16 rounding of each element: 1.7e-3 against 64 bits; two correct results can lie
        # one step (2^-7 of the value) apart
        return {"rel": 7e-3, "max": 1.6e-2}
    # fp32: one or a few roundings of theta, and z to 1e-6 (K sums of it in an update): 3e-8 to
    # 5e-8 against 64 bits where theta dominates, more where a large sum does
    return {"rel": 1e-6, "max": 1e-5}


# --- the method in 64 bits ------------------------------------------------------------

_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al., SC 2011) of int64 tensors that hold 32-bit words."""
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # the product's 64 bits, whatever the sign
        c0, c1, c2, c3 = ((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, \
            ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _z(seed, e):
    """z of global elements e: Box-Muller of word pair (e & 2) of Philox block e >> 2."""
    mid = int(seed["machine_id"])
    b = e >> 2
    full = lambda v: torch.full_like(e, v)  # noqa: E731
    x0, x1, x2, x3 = _philox(b & _M32, b >> 32, full(int(seed["step"])),
                             full(int(seed["sample_id"])), mid & _M32, mid >> 32)
    second = (e & 2) != 0
    xa, xb = torch.where(second, x2, x0), torch.where(second, x3, x1)
    r = torch.sqrt(-2.0 * torch.log(((xa >> 9).double() + 0.5) * 2.0**-23))
    a = 2.0 * math.pi * (((xb >> 8).double() + 0.5) * 2.0**-24)
    return r * torch.where((e & 1) != 0, torch.sin(a), torch.cos(a))


def _coefficients(codes, lr, denom):
    m = np.minimum(np.abs(codes.astype(np.int64)), 127)
    c = -np.float64(np.float32(lr)) * np.sign(codes) * np.expm1(m / np.float64(QSCALE)) / denom
    return [float(np.float32(v)) for v in c]


def _byte(g):
    m = min(127.0, math.floor(QSCALE * math.log1p(abs(g)) + 0.5))
    return int(math.copysign(m, g))


def _chunks(sizes, offsets, starts, most=1 << 24):
    """(positions in the buffer, global indices) of all elements, `most` or a few more at a time."""
    at, e, held = [], [], 0
    for n, fo, start in zip(sizes, offsets, starts):
        for i in range(0, n, most):
            k = min(most, n - i)
            at.append(torch.arange(start + i, start + i + k, device="cuda"))
            e.append(torch.arange(fo + i, fo + i + k, device="cuda"))
            held += k
            if held >= most:
                yield torch.cat(at), torch.cat(e)
                at, e, held = [], [], 0
    if held:
        yield torch.cat(at), torch.cat(e)


def _exact_q4(case, seed):
    sizes, offsets, _, _ = _plan(case)
    codes, scale, code_at, scale_at = _q4_parameters(case, seed)
    s = _pairs(case, seed)[0][0]
    level = _q4_levels().float().double().cuda()
    out = scale.double()
    eps = float(np.float32(EPS))
    for n, fo, ca, sa in zip(sizes, offsets, code_at, scale_at):
        for i in range(0, n, 1 << 24):
            k = min(1 << 24, n - i)
            c = codes[ca + i // 2:ca + (i + k + 1) // 2].long()
            c = torch.stack([c & 15, c >> 4], 1).reshape(-1)[:k]
            blocks = (k + 63) // 64
            at = slice(sa + i // 64, sa + i // 64 + blocks)
            old = scale[at].double().repeat_interleave(64)[:k]
            w = level[c] * old + eps * _z(s, torch.arange(fo + i, fo + i + k, device="cuda"))
            w = torch.nn.functional.pad(w.abs(), (0, 64 * blocks - k))
            out[at] = w.reshape(blocks, 64).amax(1)
    return [None, out]


def exact(case, seed):
    op = case["op"]
    sizes, offsets, starts, _ = _plan(case)
    draws = {"step": case["K"] + 3}.get(op, case["K"])
    if op == "checksum" or sum(sizes) * draws > EXACT_WORK:
        return None
    if op == "q4":
        return _exact_q4(case, seed)
    theta = _values(case, seed)
    seeds, codes = _pairs(case, seed)
    dtype, out = theta.dtype, theta.double()
    store = lambda x: x.to(dtype).double()  # noqa: E731
    eps = float(np.float32(EPS))
    if op == "step":
        codes[0] = _byte(prepare_loss(seed))
    order = np.lexsort((seeds["sample_id"], seeds["step"], seeds["machine_id"]))
    coef = _coefficients(codes, case.get("lr", 0.0), float(case["K"]) if op == "step" else 1.0)
    groups = [order]
    if op == "replay":
        ends = np.cumsum(_step_sizes(case, seed))
        groups = [range(b - k, b) for b, k in zip(ends, _step_sizes(case, seed))]
    for at, e in _chunks(sizes, offsets, starts):
        x = out[at]
        if op in ("perturb", "step"):
            z = _z(seeds[0], e)
            if op == "perturb":
                out[at] = x + eps * z
                continue
            for scale in (eps, -2 * eps, eps):
                x = store(x + scale * z)
        for i, group in enumerate(groups):
            x = store(x) if i else x
            x = x + sum(coef[k] * _z(seeds[k], e) for k in group)
        out[at] = x
    if op == "restore":
        return [_placed(torch.zeros_like(out), out, sizes, starts),
                out if case["refresh"] else theta.double()]
    return out


def prepare_loss(seed):
    """The projected gradient of a step, as prepare() draws it."""
    return float(np.random.default_rng([seed, 9]).normal(0.0, 30.0))


def _placed(to, values, sizes, starts):
    """`values` at the tensors' places, `to` between them."""
    for n, at in zip(sizes, starts):
        to[at:at + n] = values[at:at + n]
    return to
