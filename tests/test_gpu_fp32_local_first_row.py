"""fp32, exact same-block weights: the gradient of a row with one key, where the forward's and the backward's errors
of the score have to be the same ones to cancel."""
import numpy as np
import pytest
import torch

import paper_2310_01655_b200 as psk
from paper_2310_01655_b200 import inputs as wl
from oracle import polysketch as orc
from parity_util import g_slice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [16, 32, 64])
def test_gradient_of_the_first_query(r):
    H, n, b = 24, 128, 128
    w = wl.small_workload(B=1, H=H, n=n, r=r, b=b, dtype="f32", seed=5 + r)
    inp = wl.make_inputs(w, "cuda")
    q, k = inp["Q"][0, :, 0].double(), inp["K"][0, :, 0].double()
    # x = q_0 . k_0 where x^3 / (1 + x^4)^2 is flat, as a sum of 64 terms of size one: the sum's error, 2^-24 times
    # partial sums of up to 8, is many times 2^-24 x
    x = 0.6 ** 0.25
    inp["K"][0, :, 0] = (k + ((x - (q * k).sum(-1)) / (q * q).sum(-1))[:, None] * q).float()
    Q, K, V, G1, G2, dO = (inp[t] for t in ("Q", "K", "V", "G1", "G2", "dO"))
    O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, b, flags=psk.FLAG_LOCAL_EXACT)
    dQ = psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b, flags=psk.FLAG_LOCAL_EXACT)[0]
    err = ref2 = 0.0
    for hi in range(H):
        f = lambda t: wl.head_slice_f64(inp[t], 0, hi)
        ref = orc.causal_polysketch_attention_backward_blocked(f("Q"), f("K"), f("V"), g_slice(G1, hi), g_slice(G2, hi), f("dO"), b,
                                                               diagonal="exact")[0][0]
        err += float(((dQ[0, hi, 0].double().cpu().numpy() - ref) ** 2).sum())
        ref2 += float((ref ** 2).sum())
    # What does not cancel: the 64-term sums dO . v and dO . O, about 16 roundings of 2^-24 beside sums of size 8 and
    # times d = 1.6, so 3 x 2^-24.  Two differently rounded scores: 3 / x times 2^-24 x 20, 70 x 2^-24.
    assert np.sqrt(err / ref2) < 12 * 2.0 ** -24, np.sqrt(err / ref2) * 2.0 ** 24
