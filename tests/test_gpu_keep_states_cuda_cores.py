"""PSK_FLAG_KEEP_STATES on the CUDA-core path: ignored there, so a backward call forms all it reads from its own
arguments, whatever workspace it is given."""
import pytest
import torch

import paper_2310_01655_b200 as psk
from paper_2310_01655_b200 import binding, inputs as wl

pytestmark = pytest.mark.gpu

KEEP = psk.FLAG_KEEP_STATES


def scratch(nbytes):
    """Memory that nobody has left anything useful in: every 16- and 32-bit float of it is a NaN."""
    return torch.full((nbytes,), 0xFF, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("dtype,p,r,path", [
    ("f32", 4, 16, psk.PATH_AUTO), ("f32", 4, 64, psk.PATH_AUTO), ("bf16", 4, 32, psk.PATH_CUDA_CORES),
    ("f32", 2, 64, psk.PATH_AUTO), ("f32", 8, 16, psk.PATH_AUTO), ("bf16", 8, 64, psk.PATH_AUTO),
])
@pytest.mark.parametrize("flags", [0, psk.FLAG_LOCAL_EXACT])
def test_backward_on_a_workspace_of_its_own(dtype, p, r, path, flags):
    if p == 8 and flags:
        pytest.skip("degree 8 has no exact same-block weights")
    B, H, n, b = 1, 2, 384, 128
    inp = wl.make_inputs(wl.small_workload(B=B, H=H, n=n, r=r, b=b, dtype=dtype, seed=7 + p + r), "cuda")
    Q, K, V, dO = (0.5 * inp["Q"], 0.5 * inp["K"], inp["V"], inp["dO"])
    G1, G2 = (None, None) if p == 2 else (inp["G1"], inp["G2"])
    if p == 8:
        g = torch.Generator(device="cuda").manual_seed(r)
        G1, G2 = (torch.randn(H, 128 + r, r, generator=g, device="cuda").to(Q.dtype) for _ in range(2))
    shp = psk.binding.make_shape(Q, G1, r, b, p, path, flags | KEEP)
    # each call on scratch of the size that the library states for that call
    O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, b, p, path, workspace=scratch(psk.workspace_bytes(shp, False)), flags=flags | KEEP)
    got = psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b, p, path, workspace=scratch(psk.workspace_bytes(shp, True)), flags=flags | KEEP)
    want = psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b, p, path, flags=flags)
    for x, y in zip(got, want):
        assert torch.equal(x, y)


@pytest.mark.parametrize("dtype,r", [("f32", 16), ("bf16", 64)])
def test_learnable_sketch_backward_on_a_workspace_of_its_own(dtype, r):
    b = 128
    inp = wl.make_inputs(wl.small_workload(B=1, H=2, n=384, r=r, b=b, dtype=dtype, seed=31 + r), "cuda")
    Q, K, V, dO = (inp[k] for k in ("Q", "K", "V", "dO"))
    params = binding.pack_learned_params(*wl.learned_network_params(64, r, 5))
    size = lambda bwd: binding.learned_workspace_bytes(Q, r, b, KEEP, for_backward=bwd)
    O, den = binding.learned_attn_fwd(Q, K, V, params, r, b, KEEP, scratch(size(False)))
    got = binding.learned_attn_bwd(Q, K, V, params, O, den, dO, r, b, KEEP, scratch(size(True)))
    want = binding.learned_attn_bwd(Q, K, V, params, O, den, dO, r, b, 0)
    for x, y in zip(got[:3], want[:3]):
        assert torch.equal(x, y)
    # the parameter gradients are summed by fp32 atomics over 2 * 768 rows, in an order of their own each time
    torch.testing.assert_close(got[3], want[3], rtol=0, atol=1536 * 2.0 ** -24 * float(want[3].abs().max()))
