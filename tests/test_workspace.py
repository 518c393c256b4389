"""Workspace sizes against the buffers that the kernels use (no GPU needed)."""
import ctypes
import os

import pytest

from paper_2410_20501_gb300 import build, pm


@pytest.fixture(scope="module")
def lib():
    if not os.path.exists(pm.LIB_PATH):
        build.build()
    return pm.lib()


@pytest.mark.parametrize("n,partners", [(32, ()), (64, ()), (128, (128,)), (256, (256, 128))])
def test_scalaron_levels_with_a_ping_pong_partner(lib, n, partners):
    """Only the levels of marched sweeps (128^3 and larger) are smoothed out of place;
    every level below the first has three arrays, and the float64 partials come on top."""
    size = ctypes.c_size_t()
    assert lib.pm_workspace_size(n, 0, pm.PM_WS_FR, ctypes.byref(size)) == 0
    coarse = sum((n >> l) ** 3 for l in range(1, 11) if n >> l >= 4)
    partials = 16 * max((n // 4) ** 3, 152 * 64)
    need = 12 * coarse + 4 * sum(p ** 3 for p in partners) + partials
    assert need <= size.value < need + 64 * 256   # each of fewer than 64 pieces starts on 256 bytes
