"""Forces at particles in any order: each way of looking the cells up gives the
sums of the one-thread-per-particle gather of batches bit for bit, near particles
are not sent through the packed field, and a call is one launch below the size from
which packing could pay."""
import ctypes

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


def particles(pm, n, N, order):
    """N particles: uniform in random order, uniform in cell order, or on the first
    sites of a lattice of n^3 (repeated), each displaced on its own by `order` cells rms."""
    X = inputs.uniform_particles(N, 6)
    if order == "cells":
        c = X >> np.uint32(32 - int(np.log2(n)))
        X = X[:, np.lexsort((c[2], c[1], c[0]))]
    elif order != "random":
        s = np.arange(N) % n ** 3
        q = (np.stack([s // n ** 2, s // n % n, s % n]) + 0.5) / n
        q += np.random.default_rng(5).standard_normal(q.shape) * order / n
        X = (q % 1.0 * 2.0 ** 32).astype(np.uint64).astype(np.uint32)
    return pm.positions_to_device(np.ascontiguousarray(X))


def field(n):
    return torch.from_numpy(np.stack([inputs.random_field(n, 40 + d) for d in range(3)]).astype(np.float32)).cuda()


@pytest.mark.parametrize("n,N,order", [(4, 1, "random"), (4, 257, "random"), (8, 33, "cells"), (8, 1000, "random"),
                                       (32, 255, 3.0), (64, 70001, "random"), (64, 70001, 1.0), (64, 70001, "cells"),
                                       (4, 2 ** 19, "random"), (16, 2 ** 19 + 3, "random"), (64, 2 ** 19, "random"),
                                       (64, 2 ** 19 + 31, "cells"), (64, 2 ** 19 + 1, 2.5), (128, 2 ** 19 - 1, "random"),
                                       (256, 2 ** 19 + 5, "random")])
def test_any_order_and_number_is_bitwise_the_batched_gather(pm, n, N, order):
    g, X = field(n), particles(pm, n, N, order)
    ref = pm.interp_batch(torch.stack([g, g]), X.repeat(1, 2))
    acc = pm.interp(g, X)
    assert torch.equal(acc, ref[:, :N]) and torch.equal(acc, ref[:, N:])


@pytest.mark.parametrize("n,order,scattered", [(64, "cells", 0), (128, 0.3, 0), (128, 1.0, 0), (128, 3.0, 1),
                                               (64, "random", 1), (16, "random", 1)])
def test_only_scattered_particles_are_packed(pm, n, order, scattered):
    """The sample's decision is the first word of the workspace.  A lattice displaced
    by up to a cell changes rows with nearly every particle and is near all the same."""
    N = 2 ** 20
    g, X = field(n), particles(pm, n, N, order)
    ws = torch.full((16 * n ** 3 + 256,), 255, dtype=torch.uint8, device="cuda")
    acc = torch.empty((3, N), dtype=torch.float32, device="cuda")
    assert pm.lib().pm_interp_packed(pm._p(g), pm._p(X), N, n, pm._p(acc), pm._p(ws), ctypes.c_size_t(ws.numel()),
                                     pm._stream()) == 0
    assert int(ws[:4].view(torch.int32)) == scattered


@pytest.mark.parametrize("n,N,launches", [(64, 2 ** 17, 1), (128, 2 ** 18, 1), (64, 2 ** 19 - 1, 1), (256, 2 ** 19, 1),
                                          (64, 2 ** 19, 2), (128, 2 ** 21, 2)])
@pytest.mark.parametrize("order", ["cells", "random"])
def test_launches_of_a_call(pm, n, N, launches, order):
    g, X = field(n), particles(pm, n, N, order)
    before = pm.launch_count()
    pm.interp(g, X)
    assert pm.launch_count() - before == launches
