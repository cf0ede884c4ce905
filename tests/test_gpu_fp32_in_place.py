"""CUDA-core forward with its output over its values."""
import pytest
import torch

import paper_2310_01655_b200 as psk
from paper_2310_01655_b200 import inputs as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,r,b", [("f32", 16, 128), ("f32", 32, 1024), ("f32", 64, 512), ("bf16", 32, 1024)])
@pytest.mark.parametrize("flags", [0, psk.FLAG_LOCAL_EXACT])
def test_output_over_the_values(dtype, r, b, flags):
    n, path = 2048, psk.PATH_CUDA_CORES
    inp = wl.make_inputs(wl.small_workload(B=2, H=9, n=n, r=r, b=b, dtype=dtype, seed=3 + r), "cuda")
    Q, K, V, G1, G2 = (inp[k] for k in ("Q", "K", "V", "G1", "G2"))
    O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, b, path=path, flags=flags)
    over = V.clone()
    O2, den2 = psk.causal_attn_fwd(Q, K, over, G1, G2, b, path=path, flags=flags, out=over)
    assert O2.data_ptr() == over.data_ptr()
    assert torch.equal(O2, O) and torch.equal(den2, den)
    # one row further on in the same memory
    if dtype == "f32" and not flags:
        mem = torch.empty(V.numel() + 64, dtype=V.dtype, device="cuda")
        values, out = mem[:-64].view_as(V), mem[64:].view_as(V)
        values.copy_(V)
        assert torch.equal(psk.causal_attn_fwd(Q, K, values, G1, G2, b, path=path, out=out)[0], O)
