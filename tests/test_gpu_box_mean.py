"""The mean density of a box (float64, the source of the Poisson equation is taken
from it) has the same bits alone and in every batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2410_20501_gb300 import inputs

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


def means(ws, count):
    """The `count` float64 means that a deposit left in its (zeroed) workspace: its
    pieces start on 256-byte boundaries, and only the means begin with a number as
    close to 1."""
    v = ws[: ws.numel() // 256 * 256].view(torch.float64).reshape(-1, 32)
    at = torch.nonzero((v[:, 0] - 1.0).abs() < 1e-6).flatten()
    assert at.numel() == (count + 31) // 32
    return v.flatten()[at[0] * 32:][:count].cpu().numpy()


@pytest.mark.parametrize("n,np_box,B", [(32, 20011, 3), (32, 40009, 40), (64, 300007, 2), (64, 100003, 40),
                                        (128, 1000003, 2), (256, 3000017, 2)])
def test_mean_alone_and_in_a_batch(pm, n, np_box, B):
    X = inputs.uniform_particles(B * np_box, 17)
    ws = pm.batch_workspace(n, B, np_box, "cuda").zero_()
    rho = pm.deposit_batch(pm.positions_to_device(X), n, B, ws=ws)
    batch = means(ws, B)
    for b in {0, 1, B - 1}:
        one = pm.workspace(n, np_box, pm.PM_WS_SORT, "cuda").zero_()
        alone = pm.deposit(pm.positions_to_device(np.ascontiguousarray(X[:, b * np_box:(b + 1) * np_box])), n, ws=one)
        assert torch.equal(rho[b], alone)
        assert means(one, 1)[0] == batch[b], b
        # compensated partial sums: the float64 sum's rounding (log2 n^3 bits deep, with room)
        assert batch[b] == pytest.approx(float(alone.double().mean()), rel=1e-14)
