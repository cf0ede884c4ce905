"""Performance cases: what programs that use causal Polysketch attention have it do.

Four kinds of work, all through the package's public calls:

* "train": one training step of an attention layer, forward then backward on one workspace with the
  forward's states kept (what a training loop does), for the random sketch (p = 4), its variant with exact
  same-block weights, the deeper sketch (p = 8), exact degree-2 attention (p = 2) and the learnable sketch
  with and without exact same-block weights;
* "prefill": the forward alone (evaluation, or reading a prompt), causal or not;
* "decode": one new token for every sequence of a batch on the running state;
* "lt": the block lower-triangular multiply on feature matrices that the caller has.

Shapes are GPT-2's attention layers (12 or 16 heads of 64) from one sequence to batches of a million
tokens, and smaller or ragged ones (odd numbers of heads, of batches and of blocks, blocks of 384 rows).
"""
import math

import torch

import paper_2310_01655_b200 as psk
from paper_2310_01655_b200 import binding
from paper_2310_01655_b200 import inputs as wl

H_DIM = 64
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def _attn(kind, variant, dtype, B, H, n, r, b, **more):
    return dict(more, kind=kind, variant=variant, dtype=dtype, B=B, H=H, n=n, r=r, b=b)


def _lt(dtype, batch, n, m, k, b, **more):
    return dict(more, kind="lt", dtype=dtype, batch=batch, n=n, m=m, k=k, b=b)


def _decode(dtype, B, H, r, **more):
    return dict(more, kind="decode", dtype=dtype, B=B, H=H, r=r)


def listed():
    return [
        # generating text for one user: one layer's step for one sequence, all latency
        _decode("bf16", 1, 12, 32, name="decode_one_sequence"),
        # a serving batch of 32 sequences, GPT-2 small
        _decode("bf16", 32, 12, 32, name="decode_batch_32"),
        # the fp32 parity configuration: one head, 1024 tokens
        _attn("prefill", "sketch", "f32", 1, 1, 1024, 16, 128, name="prefill_f32_one_head"),
        # fp32 training of a small model (debugging, fine-tuning where bf16 is not wanted)
        _attn("train", "sketch", "f32", 2, 12, 4096, 32, 256, name="train_f32_4k"),
        # reading one long prompt, GPT-2 small, an odd number of blocks of three row tiles
        _attn("prefill", "sketch", "bf16", 1, 12, 16512, 32, 384, name="prefill_one_sequence_16k"),
        # the headline configuration: GPT-2 small, 32k context, a batch of a million tokens
        _attn("train", "sketch", "bf16", 32, 12, 32768, 32, 256, name="train_32k_r32"),
        # the larger sketch (4096 features)
        _attn("train", "sketch", "bf16", 4, 12, 16384, 64, 512, name="train_16k_r64"),
        # exact weights inside each block, GPT-2 medium's heads, a short context and an odd batch
        _attn("train", "local", "bf16", 3, 16, 2688, 32, 384, name="train_local_2688"),
        # the paper's best variant: learnable sketch with exact same-block weights
        _attn("train", "learned_local", "bf16", 4, 12, 8192, 32, 256, name="train_learned_local_8k"),
        # degree 8
        _attn("train", "p8", "bf16", 8, 12, 8192, 32, 256, name="train_p8_8k"),
        # given features on the tensor cores (1024 features per token)
        _lt("bf16", 24, 8192, 1024, 64, 256, name="lt_bf16_1024_features"),
        # given fp32 features (a Performer's 256 positive features)
        _lt("f32", 12, 4096, 256, 64, 256, name="lt_f32_256_features"),
    ]


def _log_between(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _blocks(rng, tokens_lo, tokens_hi, b):
    """A sequence length of whole blocks, odd counts as likely as even ones."""
    return b * max(1, round(_log_between(rng, max(tokens_lo, b), max(tokens_hi, b)) / b))


def draw(rng):
    kind = rng.choice(["decode", "prefill", "train", "train", "train", "lt"])
    if kind == "decode":
        r = rng.choice([16, 32, 32, 64])
        top = {16: 256, 32: 64, 64: 16}[r]
        return _decode(rng.choice(["bf16", "bf16", "f32"]), round(_log_between(rng, 1, top)), rng.choice([8, 12, 16, 25]), r)
    if kind == "lt":
        b = rng.choice([128, 256])
        n = _blocks(rng, 512, 16384, b)
        if rng.random() < 0.6:
            m = 64 * rng.randint(2, 20)
            batch = max(1, min(48, round(_log_between(rng, 1, 2.0e8 / (n * m)))))
            return _lt("bf16", batch, n, m, 64, b)
        m, k = rng.choice([64, 100, 256, 384]), rng.choice([32, 64, 65, 96])
        batch = max(1, min(24, round(_log_between(rng, 1, 2.0e7 / (n * m)))))
        return _lt("f32", batch, n, m, k, b)
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    variants = {
        ("prefill", "bf16"): ["sketch", "sketch", "local", "noncausal", "p8", "learned_local"],
        ("prefill", "f32"): ["sketch", "local"],
        ("train", "bf16"): ["sketch", "sketch", "local", "local", "p8", "p2", "learned", "learned_local", "noncausal"],
        ("train", "f32"): ["sketch", "local"],
    }[(kind, dtype)]
    variant = rng.choice(variants)
    r = 64 if variant == "p2" else rng.choice([16, 32, 32, 32] if variant in ("p8", "learned", "learned_local") else [16, 32, 32, 64])
    b = rng.choice([128, 256, 256, 384, 512])
    H = rng.choice([5, 8, 12, 16])
    # head-tokens up to what keeps a step within tens of milliseconds
    most = {"f32": 1.0e5, "bf16": 3.0e6}[dtype]
    most /= {"learned": 8, "learned_local": 8, "p2": 4}.get(variant, 1) * (3 if r == 64 and variant != "p2" else 1)
    n = _blocks(rng, 512, min(32768, most / H), b)
    B = max(1, round(_log_between(rng, 1, max(1.0, most / (n * H)))))
    return _attn(kind, variant, dtype, B, H, n, r, b)


def _flags(variant):
    return {"local": psk.FLAG_LOCAL_EXACT, "learned_local": psk.FLAG_LOCAL_EXACT, "noncausal": psk.FLAG_NONCAUSAL}.get(variant, 0)


def _degree(variant):
    return {"p2": 2, "p8": 8}.get(variant, 4)


def _prepare_attn(c, seed):
    train = c["kind"] == "train"
    w = wl.Workload("case", c["B"], c["H"], c["n"], H_DIM, c["r"], 4, c["b"], c["dtype"], train, seed, seed + 1_000_003)
    s = dict(wl.make_inputs(w, "cuda", with_dO=train), c=c)
    variant, p = c["variant"], _degree(c["variant"])
    # keep the weights of the other degrees, and exact weights beside the bounded learnable sketch, on one scale
    shrink = {"p2": 0.5, "p8": 0.5, "learned_local": 0.35}.get(variant)
    if shrink is not None:
        s["Q"].mul_(shrink)
        s["K"].mul_(shrink)
    if p == 2:
        s["G1"] = s["G2"] = None
    if p == 8:
        gen = torch.Generator(device="cuda").manual_seed(seed + 1_000_003)
        for g in ("G1", "G2"):
            s[g] = torch.randn(c["H"], 2 * H_DIM + c["r"], c["r"], generator=gen, device="cuda").to(DTYPES[c["dtype"]])
    s["flags"] = _flags(variant) | (psk.FLAG_KEEP_STATES if train else 0)
    if variant.startswith("learned"):
        s["params"] = binding.pack_learned_params(*wl.learned_network_params(H_DIM, c["r"], seed))
        need = binding.learned_workspace_bytes(s["Q"], c["r"], c["b"], s["flags"], for_backward=train)
    else:
        shape = binding.make_shape(s["Q"], s["G1"], c["r"], c["b"], p, psk.PATH_AUTO, s["flags"])
        need = psk.workspace_bytes(shape, train)
    # the layer's workspace, which a program keeps for all of its steps
    s["workspace"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    return s


def _prepare_decode(c, seed):
    """Tokens of one step, and the running state after a short history: the sum of phi'(k) [v | 1]^T."""
    B, H, r, dt = c["B"], c["H"], c["r"], DTYPES[c["dtype"]]
    w = wl.Workload("case", B, H, 17, H_DIM, r, 4, 128, c["dtype"], False, seed, seed + 1_000_003)
    inp = wl.make_inputs(w, "cuda")
    G1, G2 = inp["G1"], inp["G2"]
    K = inp["K"][:, :, :16].float()
    M = torch.einsum("bhtx,hxr->bhtr", K, G1.float()) * torch.einsum("bhtx,hxr->bhtr", K, G2.float()) / math.sqrt(r)
    V1 = torch.cat([inp["V"][:, :, :16].float(), torch.ones(B, H, 16, 1, device="cuda")], dim=-1)
    state = psk.decode_state(B, H, r)
    for t in range(16):
        phi = (M[:, :, t, :, None] * M[:, :, t, None, :]).reshape(B, H, r * r, 1)
        state.addcmul_(phi, V1[:, :, t, None, :])
    q, k, v = (inp[x][:, :, 16].contiguous().to(dt) for x in ("Q", "K", "V"))
    return {"c": c, "q": q, "k": k, "v": v, "G1": G1, "G2": G2, "state": state}


def _prepare_lt(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = DTYPES[c["dtype"]]
    A, B = (torch.randn(c["batch"], c["n"], c["m"], generator=gen, device="cuda").div_(math.sqrt(c["m"])).to(dt) for _ in range(2))
    C = torch.randn(c["batch"], c["n"], c["k"], generator=gen, device="cuda").to(dt)
    if c["dtype"] == "f32":                     # positive features
        A, B = A.abs_(), B.abs_()
    args = (c["batch"], c["n"], c["m"], c["k"], c["b"])
    lib = psk.lib()
    need = (lib.psk_lt_multiply_bf16_workspace_bytes if c["dtype"] == "bf16" else lib.psk_lt_multiply_workspace_bytes)(*args)
    return {"c": c, "A": A, "B": B, "C": C, "workspace": torch.empty(need, dtype=torch.uint8, device="cuda")}


def prepare(case, seed):
    return {"decode": _prepare_decode, "lt": _prepare_lt}.get(case["kind"], _prepare_attn)(case, seed)


def run(s):
    c = s["c"]
    if c["kind"] == "decode":
        o, denom = psk.decode_step(s["q"], s["k"], s["v"], s["G1"], s["G2"], s["state"])
        return {"o": o, "denom": denom, "state": s["state"]}
    if c["kind"] == "lt":
        if c["dtype"] == "bf16":
            return psk.lt_multiply_bf16(s["A"], s["B"], s["C"], c["b"], s["workspace"])[0]
        return psk.lt_multiply(s["A"], s["B"], s["C"], c["b"], s["workspace"])
    Q, K, V, ws, flags, r, b = s["Q"], s["K"], s["V"], s["workspace"], s["flags"], c["r"], c["b"]
    if c["variant"].startswith("learned"):
        O, denom = binding.learned_attn_fwd(Q, K, V, s["params"], r, b, flags, ws)
        if c["kind"] == "prefill":
            return {"O": O, "denom": denom}
        dQ, dK, dV, dparams = binding.learned_attn_bwd(Q, K, V, s["params"], O, denom, s["dO"], r, b, flags, ws)
        return {"O": O, "denom": denom, "dQ": dQ, "dK": dK, "dV": dV, "dparams": dparams}
    G1, G2, p = s["G1"], s["G2"], _degree(c["variant"])
    O, denom = psk.causal_attn_fwd(Q, K, V, G1, G2, b, p, workspace=ws, flags=flags)
    if c["kind"] == "prefill":
        return {"O": O, "denom": denom}
    dQ, dK, dV = psk.causal_attn_bwd(Q, K, V, G1, G2, O, denom, s["dO"], b, p, workspace=ws, flags=flags)
    return {"O": O, "denom": denom, "dQ": dQ, "dK": dK, "dV": dV}


def _features(r):
    return r * (r + 1) // 2         # distinct entries of m (x) m


def work(case):
    """Inputs once, outputs once; operations of the block algorithm with the distinct features only."""
    size = 4 if case["dtype"] == "f32" else 2
    if case["kind"] == "decode":
        heads, r = case["B"] * case["H"], case["r"]
        state = heads * r * r * 65 * 4
        return {"bytes": 2 * state + heads * (4 * H_DIM * size + 4) + case["H"] * 2 * H_DIM * r * size,
                "flops": heads * (4 * _features(r) * 65 + 8 * H_DIM * r)}
    if case["kind"] == "lt":
        rows, m, k, b = case["batch"] * case["n"], case["m"], case["k"], case["b"]
        return {"bytes": rows * (2 * m * size + k * size + 4 * k), "flops": rows * (4 * m * k + (b + 1) * (m + k))}
    rows, r, b, v = case["B"] * case["H"] * case["n"], case["r"], case["b"], case["variant"]
    train = case["kind"] == "train"
    cols, F, half = H_DIM + 1, _features(r), (b + 1) / 2
    inner = H_DIM if v in ("local", "learned_local") else r         # what a same-block score contracts over
    pairs = 0.0 if v == "noncausal" else half
    sketch = 0 if v == "p2" else {"p8": 8 * H_DIM * r + 4 * r * r}.get(v, 4 * H_DIM * r)
    learned_weights = 2 * (H_DIM * 8 * r + 3 * 8 * r * r)
    if v.startswith("learned"):
        sketch = 2 * learned_weights
    fwd = 2 * sketch + 4 * F * cols + pairs * 2 * (inner + cols)
    # gradients of the half sketches, of V, and back through the sketch (learnable: through inputs and weights)
    bwd = 8 * F * cols + pairs * 2 * (2 * inner + 2 * cols) + 2 * sketch * (2 if v.startswith("learned") else 1)
    params = 2 * learned_weights // 2 * 4 * (2 if train else 1) if v.startswith("learned") else 2 * case["H"] * H_DIM * r * size
    # the forward reads Q, K, V and writes O and the normaliser; a training step also reads dO and writes dQ, dK, dV
    nbytes = rows * ((8 if train else 4) * H_DIM * size + 4) + params
    return {"bytes": nbytes, "flops": rows * (fwd + (bwd if train else 0))}


def tolerance(case):
    """fp32: sums of up to tens of thousands of terms, with the fourth power of cancelling scores;
    bf16: rounded operands."""
    if case["kind"] == "decode":
        # fp32 state and arithmetic; with bf16 tokens the output itself is rounded to bf16
        return {"rel": 4e-3 if case["dtype"] == "bf16" else 2e-5, "max": 0.05 if case["dtype"] == "bf16" else 1e-3}
    if case["kind"] == "lt":
        return {"rel": 4e-3 if case["dtype"] == "bf16" else 1e-5, "max": 0.1 if case["dtype"] == "bf16" else 1e-3}
    if case["dtype"] == "f32":
        return {"rel": 2e-5, "max": 0.02}
    # the parameter gradients of the learnable sketch sum bf16-rounded deltas
    return {"rel": 2e-2 if case["variant"].startswith("learned") else 1.5e-2, "max": 0.9}
