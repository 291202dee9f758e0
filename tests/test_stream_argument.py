"""stream= of the local calls: refused unless every buffer is given (a buffer made
by the call would go back to its pool while the other stream still uses it).  The
checks come before any CUDA work."""
import pytest
import torch

from paper_2608_29539_gb300 import logo as L

T = torch.zeros((1, 8, 1, 64), dtype=torch.bfloat16)


@pytest.mark.parametrize("kw", [{}, dict(o=T), dict(lse=T)])
def test_forward(kw):
    with pytest.raises(ValueError, match="stream="):
        L.logo_local_attn_fwd(T, T, T, 4, stream=1, **kw)


@pytest.mark.parametrize("missing", ["dq", "dk", "dv", "workspace"])
def test_backward(missing):
    kw = {n: T for n in ("dq", "dk", "dv", "workspace") if n != missing}
    with pytest.raises(ValueError, match="stream="):
        L.logo_local_attn_bwd(T, T, T, T, T, T, 4, stream=1, **kw)


def test_without_stream_nothing_changes():
    with pytest.raises(ValueError, match="CUDA tensor"):
        L.logo_local_attn_fwd(T, T, T, 4)
