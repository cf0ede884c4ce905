"""Tensor-core path: nothing that an uninitialised workspace or the rows beyond a state's last feature hold may reach a result.

The last 128-feature tile of a state is partly empty (16 of 128 rows are features for r = 16, 32 for r = 32 and 64): the
kernels form no features for the empty rows, whose sums are then whatever shared memory held, and store zeros."""
import pytest
import torch

import paper_2310_01655_b200 as psk
from paper_2310_01655_b200 import inputs as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, psk.FLAG_LOCAL_EXACT, psk.FLAG_NONCAUSAL])
@pytest.mark.parametrize("r,b,n,B,H", [
    (16, 128, 384, 1, 3), (16, 128, 1664, 2, 5),       # one share, several runs
    (32, 256, 1024, 4, 12),                            # three shares of a head: two store warpgroups
    (32, 128, 384, 25, 12), (32, 128, 1408, 1, 1),     # one share of five tiles; runs
    (64, 128, 384, 1, 2), (64, 256, 1024, 8, 6),       # five to nine shares
])
def test_result_does_not_depend_on_what_the_workspace_held(r, b, n, B, H, flags):
    w = wl.small_workload(B=B, H=H, n=n, r=r, b=b, dtype="bf16", seed=700 + r + n)
    inp = wl.make_inputs(w, "cuda")
    Q, K, V, G1, G2, dO = (inp[k] for k in ("Q", "K", "V", "G1", "G2", "dO"))
    flags |= psk.FLAG_KEEP_STATES
    shp = psk.binding.make_shape(Q, G1, r, b, 4, psk.PATH_AUTO, flags)
    results = []
    for fill in (0, 0xFF):                             # 0xFFFF is a bf16 NaN, 0xFFFFFFFF an fp32 one
        ws = torch.full((psk.workspace_bytes(shp, True),), fill, dtype=torch.uint8, device="cuda")
        O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, b, workspace=ws, flags=flags)
        assert psk.check(ws) == 0
        grads = psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b, workspace=ws, flags=flags)
        assert psk.check(ws) == 0
        results.append((O, den) + tuple(grads))
    for name, x, y in zip(("O", "denom", "dQ", "dK", "dV"), *results):
        assert bool(torch.isfinite(y).all()), name
        assert torch.equal(x, y), name
