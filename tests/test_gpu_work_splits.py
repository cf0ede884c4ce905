"""Tensor-core path, degree-8 sketch and decode step where the division of the work changes: a head's states by one
CTA or several, in one run or several unequal ones; sketch CTAs with one tile or several; one CTA per decoded head or a
cluster."""
import pytest
import torch

import paper_2310_01655_b200 as psk
from paper_2310_01655_b200 import inputs as wl
from oracle import polysketch as orc
from parity_util import TOL, check, g_slice, oracle_backward, oracle_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,b,n,B,H", [
    (16, 128, 896, 1, 1), (16, 128, 1664, 2, 5), (16, 256, 512, 13, 12),                # seven blocks, 13 blocks, one run
    (32, 128, 1408, 1, 1), (32, 256, 2816, 2, 3), (32, 256, 1024, 6, 12), (32, 128, 256, 25, 12),
    (64, 128, 896, 1, 1), (64, 256, 1280, 4, 9), (64, 384, 1152, 8, 12),
])
def test_states_however_they_are_dealt(r, b, n, B, H):
    w = wl.small_workload(B=B, H=H, n=n, r=r, b=b, dtype="bf16", seed=900 + r + n)
    inp = wl.make_inputs(w, "cuda")
    Q, K, V, G1, G2, dO = (inp[k] for k in ("Q", "K", "V", "G1", "G2", "dO"))
    # The backward recomputes the forward's states.  (Kept ones come with O - c in bf16: row 0, one key and a normaliser
    # d, has v_0 - O_0 = v_0 / d, so the 2^-9 of that rounding becomes d 2^-9 of its gradient, which for d > 10 is
    # more than the tolerance of a tensor that this row dominates.)
    shp = psk.binding.make_shape(Q, G1, r, b)
    ws = torch.empty(max(psk.workspace_bytes(shp, False), psk.workspace_bytes(shp, True)), dtype=torch.uint8, device="cuda")
    O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, b, workspace=ws)
    assert psk.check(ws) == 0
    grads = psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b, workspace=ws)
    assert psk.check(ws) == 0
    for bi, hi in {(0, 0), (B - 1, H - 1)}:
        ref = tuple(oracle_forward(inp, bi, hi, b)) + tuple(oracle_backward(inp, bi, hi, b))
        for name, got, want in zip(("O", "denom", "dQ", "dK", "dV"), (O, den) + tuple(grads), ref):
            check(name, got[bi, hi], want, TOL["bf16"])


@pytest.mark.parametrize("r,n,B,H", [(16, 1152, 1, 1), (16, 1152, 9, 8), (32, 896, 12, 9)])
def test_degree8_with_several_tiles_per_cta(r, n, B, H):
    w = wl.small_workload(B=B, H=H, n=n, r=r, b=128, dtype="bf16", seed=930 + r)
    inp = wl.make_inputs(w, "cuda")
    Q, K, V, dO = (0.25 * inp["Q"], 0.25 * inp["K"], inp["V"], inp["dO"])
    g = torch.Generator(device="cpu").manual_seed(940 + r)
    G1, G2 = (torch.randn(H, 128 + r, r, generator=g).bfloat16().cuda() for _ in range(2))
    O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, 128, p=8)
    grads = psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, 128, p=8)
    for bi, hi in {(0, 0), (B - 1, H - 1)}:
        q, k, v, d = (x[bi, hi].double().cpu().numpy() for x in (Q, K, V, dO))
        a, c = G1[hi].double().cpu().numpy(), G2[hi].double().cpu().numpy()
        Gs = [a[:64], c[:64], a[64:128], c[64:128], a[128:], c[128:]]
        Mq, Mk = orc.half_sketch_degree4(q, Gs), orc.half_sketch_degree4(k, Gs)
        ref = tuple(orc.causal_attention_blocked_from_half_sketches(Mq, Mk, v, 128))
        ref += tuple(orc.causal_polysketch8_attention_backward(q, k, v, Gs, d))
        for name, got, want in zip(("O", "denom", "dQ", "dK", "dV"), (O, den) + tuple(grads), ref):
            check(name, got[bi, hi], want, TOL["bf16"])


@pytest.mark.parametrize("r", [16, 32, 64])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,H", [(1, 1), (3, 12), (13, 12), (40, 12)])
def test_decode_steps_for_few_and_many_heads(r, dtype, B, H):
    n = 3
    w = wl.small_workload(B=B, H=H, n=128, r=r, b=128, dtype=dtype, seed=950 + r + B)
    inp = wl.make_inputs(w, "cuda")
    G1, G2 = inp["G1"], inp["G2"]
    state = psk.decode_state(B, H, r)
    rows = []
    for t in range(n):
        q, k, v = (inp[x][:, :, t].contiguous() for x in "QKV")
        rows.append(psk.decode_step(q, k, v, G1, G2, state))
    for bi, hi in {(0, 0), (B // 2, H // 2), (B - 1, H - 1)}:
        q, k, v = (wl.head_slice_f64(inp[x], bi, hi)[:n] for x in "QKV")
        O_ref, d_ref = orc.causal_polysketch_attention(q, k, v, g_slice(G1, hi), g_slice(G2, hi))
        check("O", torch.stack([o[bi, hi] for o, _ in rows]), O_ref, TOL[dtype])
        check("denom", torch.stack([d[bi, hi] for _, d in rows]), d_ref, TOL[dtype])


@pytest.mark.parametrize("r,b,n,B,H", [
    (16, 128, 1664, 2, 5), (16, 256, 512, 13, 12), (32, 128, 1408, 1, 1), (32, 256, 2816, 2, 3), (32, 128, 256, 25, 12),
    (64, 128, 896, 1, 1), (64, 256, 1280, 4, 9), (64, 384, 1152, 8, 12),
])
def test_kept_states_however_they_are_dealt(r, b, n, B, H):
    # Weights of size one instead of 10^4: the first rows' normalisers stay below 10, and what the kept O - c loses in
    # bf16 stays below the tolerance (see above).
    w = wl.small_workload(B=B, H=H, n=n, r=r, b=b, dtype="bf16", seed=970 + r + n)
    inp = wl.make_inputs(w, "cuda")
    inp["Q"] = 0.3 * inp["Q"]
    inp["K"] = 0.3 * inp["K"]
    Q, K, V, G1, G2, dO = (inp[k] for k in ("Q", "K", "V", "G1", "G2", "dO"))
    shp = psk.binding.make_shape(Q, G1, r, b, flags=psk.FLAG_KEEP_STATES)
    ws = torch.empty(psk.workspace_bytes(shp, True), dtype=torch.uint8, device="cuda")
    O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, b, workspace=ws, flags=psk.FLAG_KEEP_STATES)
    grads = psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b, workspace=ws, flags=psk.FLAG_KEEP_STATES)
    assert psk.check(ws) == 0
    # dV is made of Q, K, dO and the normaliser alone
    assert torch.equal(grads[2], psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b)[2])
    for bi, hi in {(0, 0), (B - 1, H - 1)}:
        ref = tuple(oracle_forward(inp, bi, hi, b)) + tuple(oracle_backward(inp, bi, hi, b))
        for name, got, want in zip(("O", "denom", "dQ", "dK", "dV"), (O, den) + tuple(grads), ref):
            check(name, got[bi, hi], want, TOL["bf16"])
