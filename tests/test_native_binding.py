"""The native argument marshalling is an extra: where its module cannot be loaded, or was built for another Python or
torch, the same calls go through ctypes."""
import sys

import pytest
import torch

import paper_2310_01655_b200 as psk
from paper_2310_01655_b200 import binding, build
from paper_2310_01655_b200 import inputs as wl

MODULE = "paper_2310_01655_b200._psk_native"


@pytest.fixture
def unloaded(monkeypatch):
    build.build()
    monkeypatch.setattr(binding, "_fast", None)
    return monkeypatch


def refused(match):
    x, g = torch.zeros(1, 1, 128, 64), torch.zeros(1, 64, 16)
    with pytest.warns(RuntimeWarning, match=match):
        with pytest.raises(RuntimeError, match="CUDA"):        # the checks of the ctypes route
            psk.causal_attn_fwd(x, x, x, g, g, 128)
    with pytest.raises(RuntimeError, match="CUDA"):
        psk.causal_attn_fwd(x, x, x, g, g, 128)                # (said once)


def test_module_that_does_not_import(unloaded):
    unloaded.setitem(sys.modules, MODULE, None)
    refused("_psk_native")


def test_module_of_another_torch(unloaded):
    unloaded.setattr(binding, "native_tag", lambda: "another torch")
    refused("built for .*torch %s.*not another torch" % torch.__version__.replace("+", r"\+"))


def test_rebuilt_for_another_torch(unloaded):
    assert not build.native_stale()
    unloaded.setattr(binding, "native_tag", lambda: "another torch")
    assert build.native_stale()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_same_results_through_ctypes(monkeypatch, dtype):
    B, H, n, r, b = 2, 3, 256, 32, 128
    inp = wl.make_inputs(wl.small_workload(B=B, H=H, n=n, r=r, b=b, dtype=dtype, seed=21), "cuda")
    Q, K, V, G1, G2, dO = (inp[k] for k in ("Q", "K", "V", "G1", "G2", "dO"))
    params = binding.pack_learned_params(*wl.learned_network_params(64, r, 2))

    def run():
        O, den = psk.causal_attn_fwd(Q, K, V, G1, G2, b)
        out = [O, den, *psk.causal_attn_bwd(Q, K, V, G1, G2, O, den, dO, b)]
        O, den = binding.learned_attn_fwd(Q, K, V, params, r, b)
        out += [O, den, *binding.learned_attn_bwd(Q, K, V, params, O, den, dO, r, b)[:3]]
        A, X, C = (torch.cat([t[0], t[1]]) for t in (Q, K, V))
        out.append(psk.lt_multiply_bf16(A, X, C, b)[0] if dtype == "bf16" else psk.lt_multiply(A, X, C, b))
        state = psk.decode_state(B, H, r)
        for t in range(2):
            out += psk.decode_step(*(x[:, :, t].contiguous() for x in (Q, K, V)), G1, G2, state)
        return out + [state]

    native = run()
    assert not isinstance(binding._native(), binding._NoNative)
    monkeypatch.setattr(binding, "_fast", binding._NoNative())
    for x, y in zip(native, run()):
        assert torch.equal(x, y)
