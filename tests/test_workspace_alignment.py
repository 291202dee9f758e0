"""A workspace off a 16-byte boundary is refused before anything is launched by
the calls whose kernels read and write it 16 bytes at a time.  CPU only: nothing
here launches a kernel."""
import ctypes

import pytest

from paper_2608_29539_gb300 import build


@pytest.fixture(scope="module")
def L():
    build.build()
    from paper_2608_29539_gb300 import logo
    return logo.lib()


FAKE, OFF = ctypes.c_void_p(1 << 20), ctypes.c_void_p((1 << 20) + 4)  # never dereferenced: rejected before use


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("rows", [False, True])
def test_transform_bwd(L, D, rows):
    from paper_2608_29539_gb300 import logo
    d = logo.Dims(2, 300, 4, 4, D)
    r = (FAKE,) * 3 if rows else (None,) * 3
    assert L.logo_branch_transform_bwd(FAKE, FAKE, None, *r, FAKE, FAKE, 0, FAKE, None, None, d, OFF, 1 << 30,
                                       None) == logo.LOGO_ERR_WORKSPACE


@pytest.mark.parametrize("gain", [None, FAKE])
def test_combine_bwd_gains(L, gain):
    from paper_2608_29539_gb300 import logo
    d = logo.Dims(2, 300, 4, 4, 128)
    assert L.logo_combine_bwd_gains(FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, gain, gain, ctypes.c_float(1e-6), FAKE, FAKE, FAKE,
                                    FAKE, FAKE, d, OFF, 1 << 30, None) == logo.LOGO_ERR_WORKSPACE
