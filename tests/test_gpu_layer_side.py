"""The layer's local calls run on the side stream that the layer has now, also
when the caller has given it another one."""
import pytest
import torch

from paper_2608_29539_gb300 import logo as L

pytestmark = pytest.mark.gpu


def test_layer_uses_the_side_stream_it_has(monkeypatch):
    from paper_2608_29539_gb300.layer import LayerConfig, LogoAttention
    layer = LogoAttention(LayerConfig(1, 64, 2, 2, 64, 32, ratio=0.5))
    g = torch.Generator(device="cuda").manual_seed(3)
    args = [torch.randn((1, 64, 2, 64), generator=g, device="cuda").bfloat16() for _ in range(6)]
    p = torch.rand((1, 64), generator=g, device="cuda")
    first = layer.forward(*args, p).clone()
    used, call = [], L.logo_local_attn_fwd
    monkeypatch.setattr(L, "logo_local_attn_fwd", lambda *a, **k: (used.append(k["stream"]), call(*a, **k))[1])
    layer.side = torch.cuda.Stream()
    again = layer.forward(*args, p)
    torch.cuda.synchronize()
    assert used == [layer.side.cuda_stream] and torch.equal(first, again)
