"""The online tuner compares launches of equal work only: an entry of its own for
each stencil order of the force pass, and for the sweeps before and after the
coarse correction of a level."""
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


def entries(pm, site, n, B):
    torch.cuda.synchronize()
    return [r for r in pm.autotune_report() if (r["site"], r["n"], r["B"]) == (site, n, B)]


def test_force_chunks_are_tuned_by_stencil_order(pm):
    n, B = 64, 7
    X = inputs.uniform_particles(B * 4096, 3).reshape(3, B, 4096).transpose(1, 0, 2)
    for order, kinds in ((3, 1), (7, 2)):
        ens = pm.Ensemble(X, np.zeros(X.shape), n, np.full(B, 0.3), 64.0, grad_order=order)
        row = torch.zeros_like(ens.coef)
        row[3] = 1.0
        for _ in range(8):
            ens.step(row)
        got = entries(pm, "force_chunk", n, B)
        assert len(got) == kinds
        assert all(r["chosen"] in (16, 32, 64) and r["samples"] >= 6 for r in got), got


def test_smoother_forms_are_tuned_by_sweeps(pm):
    """The 64^3 level of a 128^3 batch starts from zeros before the coarse
    correction and from its values after it; one sweep more is another kind."""
    n, B = 128, 6
    f = torch.from_numpy(np.stack([inputs.random_field(n, 30 + b) for b in range(B)]).astype(np.float32)).cuda()
    for npost, kinds in ((2, 2), (3, 4)):
        pm.mg_solve_batch(f, fixed_cycles=8, npre=2 if npost == 2 else 1, npost=npost)
        torch.cuda.synchronize()
        pm.mg_solve_batch(f, fixed_cycles=1, npre=2 if npost == 2 else 1, npost=npost)
        got = entries(pm, "mg_smoother", 64, B)
        assert len(got) == kinds
        assert all(r["chosen"] in (0, 1) and r["samples"] >= 4 for r in got), got
