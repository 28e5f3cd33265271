"""The calls whose time matters to a user of this package, and how each is made, run and compared.

A case is one call of a public entry point of `paper_2505_18698_b200.binding` on one problem:

    entry   fwd | objective | bshd | padded | varlen | host    (monarch_attn_<entry>)
    dtype   f32 | f16 | bf16
    batch, heads, d, b, T                                      as the entry points take them
    n       rows of a sequence that count; the tensors have N = ceil(n / b) * b rows
    short   varlen only: the shortest sequence of the batch, in percent of n
    rank, s the shared low-rank component of Q and K (see `_qkv`): how peaked the attention is

The listed cases are the package's own configurations and the shapes of the experiments it names
(image classification, question answering, image generation, summarisation, graphs), from one head
to a full GPU.  `draw` spreads over the same kinds of call.
"""
import math

import torch

from paper_2505_18698_b200 import binding as ma

_DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


def _case(entry, dtype, batch, heads, n, b, T, d=64, rank=8, s=1.0, short=100):
    return {"entry": entry, "dtype": dtype, "batch": batch, "heads": heads, "n": n, "d": d, "b": b, "T": T,
            "short": short, "rank": rank, "s": s}


def listed():
    named = [
        # the smallest call: one fp32 head (configuration C1); latency and the host path are all there is
        ("one_head_f32", _case("fwd", "f32", 1, 1, 256, 16, 1, rank=0, s=0.0)),
        # one question with its context through one 12-head layer, 16 blocks of 24: an interactive request
        ("one_sentence", _case("fwd", "f16", 1, 12, 384, 24, 1)),
        # convergence diagnostic in full precision: output and objective of a batch after three rounds
        ("objective_f32", _case("objective", "f32", 8, 12, 256, 16, 3, s=0.5)),
        # image generation: 256 tokens, d = 72, three rounds, tensors as the QKV projection leaves them
        ("image_gen_bshd", _case("bshd", "f16", 8, 16, 256, 16, 3, d=72)),
        # encoder attention at a large batch, one round (configuration C2)
        ("encoder_256", _case("fwd", "f16", 64, 12, 256, 16, 1, s=2.0)),
        # image classification: 197 tokens padded to 15 blocks of 14, two rounds
        ("image_197", _case("padded", "f16", 64, 12, 197, 14, 2)),
        # question answering: a batch of sequences of different lengths up to 384, blocks of 24
        ("answers_varlen", _case("varlen", "f16", 32, 12, 384, 24, 1, short=25)),
        # the same model's batch from and to host memory: copies in, kernels, copy back
        ("host_384", _case("host", "f16", 16, 12, 384, 24, 1)),
        # N = 1024 at a large batch, two rounds (configuration C3)
        ("batch_1k", _case("fwd", "bf16", 16, 12, 1024, 32, 2, s=2.0)),
        # a graph of 7600 nodes, d = 48, blocks of 128 (60 of them, the last one ragged)
        ("graph_7600", _case("padded", "f16", 1, 8, 7600, 128, 2, d=48)),
        # medium sequences (configuration C4)
        ("medium_4k", _case("fwd", "bf16", 4, 16, 4096, 64, 2, rank=16, s=1.5)),
        # the long sequence (configuration C5): the most work of all
        ("long_16k", _case("fwd", "bf16", 1, 16, 16384, 128, 2, rank=16, s=1.5)),
    ]
    return [dict(c, name=name) for name, c in named]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["f32", "short", "short", "rounds", "ragged", "varlen", "host", "long", "long", "long"])
    if kind == "f32":
        # few to many heads in full precision, N up to what one launch holds
        b, m = rng.randint(8, 24), rng.randint(8, 16)
        return _case(rng.choice(["fwd", "objective"]), "f32", _log(rng, 1, 8), rng.choice([1, 4, 12]), b * m, b,
                     rng.randint(1, 3), s=0.5)
    dtype = rng.choice(["f16", "f16", "bf16"])
    if kind == "rounds":
        # three rounds: the hi + lo states of short sequences, either layout
        b, m = rng.randint(10, 16), rng.randint(10, 16)
        return _case(rng.choice(["bshd", "fwd"]), dtype, _log(rng, 1, 32), rng.choice([12, 16]), b * m, b, 3,
                     d=rng.choice([64, 72]))
    if kind in ("short", "ragged", "varlen", "host"):
        T = rng.choice([1, 2])
        b = rng.randint(10, 24)
        m = rng.randint(10, 24 if T == 1 else min(24, 432 // b))
        batch, n = _log(rng, 1, 64), b * m
        if kind == "short":
            return _case("fwd", dtype, batch, 12, n, b, T, s=rng.choice([1.0, 2.0]))
        if kind == "ragged":
            return _case("padded", dtype, batch, 12, n - rng.randint(1, b - 1), b, T)
        if kind == "varlen":
            return _case("varlen", dtype, batch, 12, n, b, T, short=rng.randint(10, 90))
        return _case("host", dtype, min(batch, 24), 12, n, b, T)
    # long: a power of two or any length, the block size near its square root, as many heads as
    # about a GPU's worth of rows allows
    n = rng.choice([1024, 2048, 4096, 8192, 16384]) if rng.random() < 0.5 else _log(rng, 900, 16384)
    b = 32 if n <= 2048 else (64 if n <= 8192 else 128)
    heads = rng.choice([8, 12, 16])
    most = max(1, (1 << 18) // (heads * n))
    return _case("padded" if n % b else rng.choice(["fwd", "fwd", "bshd"]), dtype, _log(rng, 1, most), heads, n, b,
                 rng.choice([1, 2]), d=rng.choice([64, 64, 48]), rank=16, s=1.5)


def _lengths(case):
    """Lengths of a varlen batch, spread evenly from the shortest to n."""
    lo, n, batch = max(1, case["n"] * case["short"] // 100), case["n"], case["batch"]
    return [n - (n - lo) * e // max(1, batch - 1) for e in range(batch)]


def _qkv(case, seed, device):
    """Q = GQ + s CQ W / sqrt(r), K = GK + s CK W / sqrt(r), V = GV with a rank-r basis W per head: the
    peaked attention of a trained encoder (rank 0: i.i.d. normal), rounded to the case's type."""
    g = torch.Generator(device=device).manual_seed(seed)
    batch, heads, n, d, b, r = (case[k] for k in ("batch", "heads", "n", "d", "b", "rank"))

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=device)

    basis = normal(heads, r, d) * (case["s"] / math.sqrt(r)) if r else None
    out = []
    for which in range(3):
        x = normal(batch, heads, n, d)
        if r and which < 2:
            x += torch.matmul(normal(batch, heads, n, r), basis)
        x = torch.nn.functional.pad(x, (0, 0, 0, -n % b)).to(_DTYPES[case["dtype"]])   # zero rows up to N
        if case["entry"] == "bshd":
            x = x.transpose(1, 2)
        out.append(x.contiguous())
    return out


def prepare(case, seed):
    state = {"case": case, "qkv": _qkv(case, seed, "cuda")}
    if case["entry"] == "varlen":
        g = torch.Generator().manual_seed(seed)
        lens = torch.tensor(_lengths(case), dtype=torch.int32)[torch.randperm(case["batch"], generator=g)]
        state["lens"] = lens.cuda()
        for x in state["qkv"]:                       # what a collating loader leaves behind a sequence's end
            for e, own in enumerate(lens.tolist()):
                x[e, :, own:] = 0
    if case["entry"] == "host":                      # pinned buffers, kept from call to call
        state["qkv"] = [x.cpu().pin_memory() for x in state["qkv"]]
        state["out"] = torch.empty_like(state["qkv"][0]).pin_memory()
    return state


def run(state):
    case = state["case"]
    Q, K, V = state["qkv"]
    entry, b, T = case["entry"], case["b"], case["T"]
    if entry == "fwd":
        return ma.monarch_attn_fwd(Q, K, V, b, T)
    if entry == "bshd":
        return ma.monarch_attn_fwd_bshd(Q, K, V, b, T)
    if entry == "objective":
        return ma.monarch_attn_fwd_objective(Q, K, V, b, T)
    if entry == "padded":
        return ma.monarch_attn_fwd_padded(Q, K, V, b, T, case["n"])
    if entry == "varlen":
        return ma.monarch_attn_fwd_varlen(Q, K, V, b, T, state["lens"])
    return ma.monarch_attn_fwd_host(Q, K, V, state["out"], b, T)


def work(case):
    """One read of Q, K, V and one write of Y (and of the row values of the objective) over the rows that
    count; two operations per multiply-add of the method: T (2 n d (b + m)) + n b d a head."""
    lens = _lengths(case) if case["entry"] == "varlen" else [case["n"]] * case["batch"]
    size = 4 if case["dtype"] == "f32" else 2
    nbytes = flops = 0
    for n in lens:
        m = -(-n // case["b"])
        nbytes += case["heads"] * n * (4 * case["d"] * size + (4 if case["entry"] == "objective" else 0))
        flops += 2 * case["heads"] * n * case["d"] * (2 * case["T"] * (case["b"] + m) + case["b"])
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """fp32 holds 1e-5 on these inputs.  The 16-bit types round the states that feed the logits round
    after round; a row whose two largest logits are close moves by more than the mean of all rows."""
    return {"f32": {"rel": 1e-5, "max": 1e-3}, "f16": {"rel": 2e-3, "max": 0.2}, "bf16": {"rel": 1e-2, "max": 0.4}}[case["dtype"]]
