"""Causality of the fp32 kernels with infinities and NaNs: a row that a pair does not count for is not touched by what
stands in the other row, not even where both lie in one 64-row tile."""
import pytest
import torch

import paper_2310_01655_b200 as psk
from paper_2310_01655_b200 import inputs as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("dtype,r,b", [("f32", 16, 128), ("f32", 32, 256), ("f32", 64, 128), ("bf16", 32, 128)])
@pytest.mark.parametrize("flags", [0, psk.FLAG_LOCAL_EXACT])
def test_attention(bad, dtype, r, b, flags):
    n, path = 512, psk.PATH_CUDA_CORES
    inp = wl.make_inputs(wl.small_workload(B=1, H=2, n=n, r=r, b=b, dtype=dtype, seed=17 + r), "cuda")
    Q, K, V, G1, G2, dO = (inp[k] for k in ("Q", "K", "V", "G1", "G2", "dO"))

    def run(Q, K, V, dO):
        O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, b, path=path, flags=flags)
        return (O, den) + psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b, path=path, flags=flags)

    def poisoned(x, rows):
        x = x.clone()
        x[:, :, rows] = bad
        return x

    clean = run(Q, K, V, dO)
    for s in (200, 331):                   # inside a tile and a block
        later, earlier = slice(s, None), slice(None, s)
        got = run(poisoned(Q, later), poisoned(K, later), poisoned(V, later), dO)
        for i in (0, 1, 2):                # O, denom, dQ: of later rows nothing counts
            assert torch.equal(got[i][:, :, earlier], clean[i][:, :, earlier]), ("O", "denom", "dQ")[i]
        got = run(poisoned(Q, earlier), K, V, poisoned(dO, earlier))
        for i in (3, 4):                   # dK, dV: of earlier queries nothing counts
            assert torch.equal(got[i][:, :, later], clean[i][:, :, later]), ("dK", "dV")[i - 3]


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("m,k,b,s", [(64, 64, 128, 96), (100, 65, 192, 160), (33, 128, 96, 32), (64, 32, 64, 40)])
def test_lt_multiply(bad, m, k, b, s):
    g = torch.Generator(device="cuda").manual_seed(m + k)
    A, B, C = (torch.randn(2, 2 * b, c, generator=g, device="cuda") for c in (m, m, k))
    clean = psk.lt_multiply(A, B, C, b)
    for base in (0, b):
        B2, C2 = B.clone(), C.clone()
        B2[:, base + s:] = bad
        C2[:, base + s:] = bad
        assert torch.equal(psk.lt_multiply(A, B2, C2, b)[:, :base + s], clean[:, :base + s])
