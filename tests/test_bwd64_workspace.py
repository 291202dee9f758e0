"""What the d = 64 local backward holds of a query row beside dQ: two floats a
row and head, on an even number of rows a sequence, whatever the sequence's
length.  CPU only: nothing here launches a kernel."""
import pytest

from paper_2608_29539_gb300 import build


@pytest.mark.parametrize("B,T,H", [(1, 1, 1), (5000, 1, 4), (1000, 3, 2), (700, 100, 8), (3, 129, 12), (2, 4096, 16)])
def test_row_statistics(B, T, H):
    build.build()
    from paper_2608_29539_gb300 import logo as L
    got = L.lib().logo_local_attn_bwd_workspace_size(L.Dims(B, T, H, H, 64))
    dq = (B * T + 128) * H * 64 * 4
    stats = B * H * (T + T % 2) * 2 * 4
    assert dq + stats <= got <= dq + stats + 2048  # 1 KB of zeros, three parts on 256 bytes
