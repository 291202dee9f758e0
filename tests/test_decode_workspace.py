"""The decode workspace is no larger than what the call's own CTAs can leave in
it: two pieces of a KV head's group each, at most one CTA for two sub-tiles of 64
cache rows and two a multiprocessor.  CPU only: nothing here launches a kernel."""
import pytest

from paper_2608_29539_gb300 import build


@pytest.mark.parametrize("B,L,Hq,Hkv,D", [(1, 4096, 16, 1, 128), (1, 64, 1, 1, 64), (1, 500, 8, 8, 128), (32, 16384, 32, 8, 128),
                                          (2, 1 << 20, 16, 1, 64), (300, 1024, 16, 2, 64), (100000, 64, 1, 1, 64)])
def test_size(B, L, Hq, Hkv, D):
    build.build()
    from paper_2608_29539_gb300 import logo as G
    subs = B * Hkv * -(-L // 64)
    ctas = max(1, min(subs // 2, 2 * G.logo_num_sms()))
    need = 2 * ctas * (Hq // Hkv) * (D + 2) * 4 + B * Hkv * 4
    assert G.lib().logo_decode_workspace_size(G.Dims(B, L, Hq, Hkv, D)) <= need + 3 * 256
