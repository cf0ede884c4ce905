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
    (16, 128, 384, 1, 3), (16, 128, 1664, 2, 5),       # two shares of a head (non-causal: several runs)
    (32, 256, 1024, 4, 12),                            # three shares: two store warpgroups
    (32, 128, 384, 25, 12), (32, 128, 1408, 1, 1),     # one share of five tiles; five shares
    (64, 128, 384, 1, 2), (64, 256, 1024, 8, 6),       # nine and six shares
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


FEATURES, STORED = {16: 144, 32: 544, 64: 2080}, {16: 256, 32: 640, 64: 2176}      # of a state: rows, and rows stored


@pytest.mark.parametrize("flags", [0, psk.FLAG_NONCAUSAL])
@pytest.mark.parametrize("r,b,n,B,H,runs", [
    (16, 128, 1024, 1, 3, 1), (16, 128, 1024, 1, 3, 4), (16, 128, 512, 13, 12, 2),
    (32, 128, 1024, 1, 2, 4), (32, 256, 1024, 4, 12, 1), (32, 256, 1024, 4, 12, 2), (32, 128, 256, 25, 12, 1),
    (64, 128, 512, 1, 2, 2), (64, 128, 512, 1, 2, 4), (64, 128, 256, 20, 12, 1),
])
def test_stored_rows_beyond_the_last_feature_are_zero(r, b, n, B, H, runs, flags):
    """The kept states themselves, in the workspace: rows beyond the last feature, columns beyond the last one and the first
    block's state are zero to the bit, also where the empty rows' sums (NaN here, from the workspace) go through the runs'
    totals, the scan over them and back into the accumulators."""
    w = wl.small_workload(B=B, H=H, n=n, r=r, b=b, dtype="bf16", seed=740 + r + n + runs)
    inp = wl.make_inputs(w, "cuda")
    Q, K, V, G1, G2 = (inp[k] for k in ("Q", "K", "V", "G1", "G2"))
    flags |= psk.FLAG_KEEP_STATES
    shp = psk.binding.make_shape(Q, G1, r, b, 4, psk.PATH_AUTO, flags, seq_segments=runs)
    ws = torch.full((psk.workspace_bytes(shp, True),), 0xFF, dtype=torch.uint8, device="cuda")
    psk.causal_attn_fwd(Q, K, V, G1, G2, b, workspace=ws, flags=flags, seq_segments=runs)
    assert psk.check(ws) == 0
    up = lambda x: (x + 255) // 256 * 256
    heads, F, FP, causal = B * H, FEATURES[r], STORED[r], not flags & psk.FLAG_NONCAUSAL
    blocks = n // b if causal else 1
    # status, value centres, the sketch matrices' image, the runs' totals, then the states
    totals = 0 if causal and runs == 1 else heads * runs * FP * 80 * 4
    at = 256 + up(heads * 64 * 4) + up(H * 2 * r * 128) + up(totals)
    Z = ws[at:at + heads * blocks * FP * 80 * 2].view(torch.int16).reshape(heads, blocks, FP, 80)
    assert bool((Z[:, -1, :F, :65] != 0).any(dim=2).all())         # (the right place: every feature's row is there)
    assert not Z[:, :, F:].any() and not Z[..., 65:].any()
    if causal:
        assert not Z[:, 0].any()
    assert bool(torch.isfinite(Z.view(torch.bfloat16).float()).all())
