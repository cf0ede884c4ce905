"""fp32 path at the edges of its 64-row tiles, feature chunks and dispatch: few and many CTAs (one or two
per SM), one block (no state), two blocks (no scan), kept states; the lt multiply at ragged m, k and b."""
import numpy as np
import pytest
import torch

import paper_2310_01655_b200 as psk
from paper_2310_01655_b200 import inputs as wl
from oracle import polysketch as orc
from parity_util import TOL, check, g_slice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,b,n,B,H", [
    (16, 128, 128, 1, 1), (32, 128, 256, 1, 3), (64, 384, 768, 1, 1),       # few CTAs
    (16, 128, 1408, 2, 7), (32, 384, 1920, 2, 5), (64, 256, 1024, 4, 5),    # more than two per SM
])
@pytest.mark.parametrize("local", [False, True])
def test_forward_and_kept_backward(r, b, n, B, H, local):
    w = wl.small_workload(B=B, H=H, n=n, r=r, b=b, dtype="f32", seed=40 + r + n)
    inp = wl.make_inputs(w, "cuda")
    Q, K, V, G1, G2, dO = (inp[k] for k in ("Q", "K", "V", "G1", "G2", "dO"))
    flags = psk.FLAG_KEEP_STATES | (psk.FLAG_LOCAL_EXACT if local else 0)
    shp = psk.binding.make_shape(Q, G1, r, b, flags=flags)
    ws = torch.empty(psk.workspace_bytes(shp, True), dtype=torch.uint8, device="cuda")
    O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, b, workspace=ws, flags=flags)
    kept = psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b, workspace=ws, flags=flags)
    again = psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b, flags=flags & ~psk.FLAG_KEEP_STATES)
    assert psk.check(ws) == 0
    for x, y in zip(kept, again):
        assert torch.equal(x, y)                      # the same kernels on the same states
    diag = "exact" if local else "LR"
    for bi, hi in {(0, 0), (B - 1, H - 1)}:
        f = lambda k: wl.head_slice_f64(inp[k], bi, hi)
        g1, g2 = g_slice(G1, hi), g_slice(G2, hi)
        ref = tuple(orc.causal_polysketch_attention_blocked(f("Q"), f("K"), f("V"), g1, g2, b, diagonal=diag))
        ref += tuple(orc.causal_polysketch_attention_backward_blocked(f("Q"), f("K"), f("V"), g1, g2, f("dO"), b, diagonal=diag))
        for name, got, want in zip(("O", "denom", "dQ", "dK", "dV"), (O, den) + tuple(kept), ref):
            check(name, got[bi, hi], want, TOL["f32"])


@pytest.mark.parametrize("batch,n,m,k,b", [
    (1, 32, 1, 1, 32), (2, 96, 33, 3, 96), (3, 160, 64, 128, 160), (1, 512, 100, 65, 32), (2, 384, 7, 97, 96),
    (1, 1024, 129, 96, 64), (2, 320, 130, 32, 64), (2, 448, 65, 64, 224),
])
def test_lt_multiply_ragged(batch, n, m, k, b):
    g = torch.Generator(device="cuda").manual_seed(n + m + k)
    A, B = (torch.randn(batch, n, m, generator=g, device="cuda") for _ in range(2))
    C = torch.randn(batch, n, k, generator=g, device="cuda")
    out = psk.lt_multiply(A, B, C, b)
    off = torch.empty(A.numel() + 1, device="cuda")[1:].view_as(A)       # rows that start off 16 bytes
    off.copy_(A)
    assert torch.equal(psk.lt_multiply(off, B, C, b), out)
    for i in range(batch):
        a, bb, c = (t[i].double().cpu().numpy() for t in (A, B, C))
        ref = np.tril(a @ bb.T) @ c
        # fp32 sums of at most n + m terms in a few partial sums: random rounding, about sqrt(terms) 2^-24
        assert orc.rel_l2(out[i].double().cpu().numpy(), ref) < 1e-5
