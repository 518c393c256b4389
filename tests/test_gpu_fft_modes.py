"""The largest transforms, a mode at a time: columns along z in the first, a middle and
the last tile, on both sides of a tile's edge and at the Nyquist frequency."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os
    from paper_2410_20501_gb300 import build, pm as _pm
    if not os.path.exists(_pm.LIB_PATH):
        build.build()
    _pm.lib()
    return _pm


def symbol(n, m, kind):
    """lambda >= 0 of the mode m: phi_k = -f_k / lambda_k."""
    m = np.array(m, dtype=np.float64)
    if kind == 1:
        return 4.0 * n * n * np.sum(np.sin(np.pi * m / n) ** 2)
    return 4.0 * np.pi ** 2 * np.sum(m * m) * np.prod(np.sinc(m / n) ** 6)


@pytest.mark.parametrize("n,kind", [(512, 1), (512, 2), (1024, 1)])
@pytest.mark.parametrize("quarters,off", [(0, 1), (0, 7), (0, 8), (1, 3), (2, -1), (2, 0)])
def test_amplitude_of_a_mode(pm, n, kind, quarters, off):
    mode = (3, n - 5, quarters * n // 4 + off)
    k = torch.arange(n, device="cuda")
    phase = (mode[0] * k[:, None, None] + mode[1] * k[None, :, None] + mode[2] * k[None, None, :]) % n
    wave = torch.cos(phase.double() * (2.0 * np.pi / n))
    del phase
    phi = pm.poisson_fft(wave.float(), kind=kind).double()
    phi *= wave
    lam = symbol(n, (3, -5, mode[2]), kind)
    # Two transforms of n^3 points, each right to log2 n^3 roundings of the mode: 2 * 30 * 6e-8 at 1024,
    # and what they leave in other modes is orthogonal to this one.  Three times that.
    assert 2.0 * float(phi.mean()) * lam == pytest.approx(-1.0, abs=1.1e-5)
