"""The stages' batched entry points (the `batch` argument of the boundary):
every box of pm_deposit_batch, mg_solve_batch, pm_gradient_batch and
pm_interp_batch equals, bit for bit, the single-box call on that box."""
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


def boxes_of_particles(n, B, np_box, seed):
    """B boxes: a displaced lattice, uniform particles and a clumped box
    (cells above the one-thread limits), np_box particles each."""
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for b in range(B):
        if b % 3 == 0:
            pos = inputs.lattice(n)[:, :np_box] + rng.uniform(-0.4, 0.4, (3, np_box)) / n
        elif b % 3 == 1:
            pos = rng.uniform(0, 1, (3, np_box))
        else:
            pos = np.concatenate([rng.uniform(0, 1, (3, np_box - 3000)), 0.5 + 0.01 * rng.uniform(0, 1, (3, 3000))], 1)
        out.append(inputs.to_fixed_point(pos))
    return np.concatenate(out, axis=1)


@pytest.mark.parametrize("n,B", [(32, 3), (64, 2)])
def test_deposit_batch_equals_single_boxes(pm, n, B):
    np_box = n ** 3
    X = boxes_of_particles(n, B, np_box, 7 + n)
    rho = pm.deposit_batch(pm.positions_to_device(X), n, B).cpu().numpy()
    for b in range(B):
        one = pm.deposit(pm.positions_to_device(np.ascontiguousarray(X[:, b * np_box:(b + 1) * np_box])), n)
        assert np.array_equal(rho[b], one.cpu().numpy()), b


@pytest.mark.parametrize("n,B", [(32, 3), (64, 3)])
def test_mg_solve_batch_equals_single_boxes(pm, n, B):
    f = torch.from_numpy(np.stack([inputs.random_field(n, 40 + b) for b in range(B)]).astype(np.float32)).cuda()
    phi = pm.mg_solve_batch(f, fixed_cycles=2).cpu().numpy()
    for b in range(B):
        one, _ = pm.mg_solve(f[b].contiguous(), fixed_cycles=2, first_guess=pm.MG_GUESS_JACOBI)
        assert np.array_equal(phi[b], one.cpu().numpy()), b


def test_gradient_and_interp_batch_equal_single_boxes(pm):
    n, B, np_box = 32, 3, 5000
    phi = torch.from_numpy(np.stack([inputs.random_field(n, 60 + b) for b in range(B)]).astype(np.float32)).cuda()
    g = pm.gradient_batch(phi, order=5)
    X = inputs.uniform_particles(B * np_box, 61)
    acc = pm.interp_batch(g, pm.positions_to_device(X)).cpu().numpy()
    for b in range(B):
        gb = pm.gradient(phi[b].contiguous(), order=5)
        assert torch.equal(g[b], gb), b
        Xb = pm.positions_to_device(np.ascontiguousarray(X[:, b * np_box:(b + 1) * np_box]))
        assert np.array_equal(acc[:, b * np_box:(b + 1) * np_box], pm.interp(gb, Xb).cpu().numpy()), b


@pytest.mark.parametrize("n,N,order", [(64, 1 << 17, "random"), (64, (1 << 17) + 1, "cells"), (128, 300007, "random"),
                                       (4, 1 << 17, "random")])
def test_interp_of_many_particles_is_bitwise_the_plain_gather(pm, n, N, order):
    """Many particles take the packed field where their order is scattered
    (and the planes where it is not): bitwise pm_interp either way."""
    import ctypes
    g = torch.from_numpy(np.stack([inputs.random_field(n, 40 + d) for d in range(3)]).astype(np.float32)).cuda()
    X = inputs.uniform_particles(N, 6)
    if order == "cells":
        c = X >> np.uint32(32 - int(np.log2(n)))
        X = X[:, np.lexsort((c[2], c[1], c[0]))]
    Xd = pm.positions_to_device(X)
    plain = torch.empty((3, N), dtype=torch.float32, device="cuda")
    code = pm.lib().pm_interp(pm._p(g), pm._p(Xd), N, n, pm._p(plain), pm._stream())
    assert code == 0
    assert torch.equal(pm.interp(g, Xd), plain)
    small = torch.empty(16 * n ** 3, dtype=torch.uint8, device="cuda")
    assert pm.lib().pm_interp_packed(pm._p(g), pm._p(Xd), N, n, pm._p(plain), pm._p(small),
                                     ctypes.c_size_t(small.numel()), pm._stream()) == 2


@pytest.mark.parametrize("n,order", [(32, 5), (64, 3), (64, 7), (128, 5)])
def test_short_plane_chunks(pm, n, order):
    """Small grids are marched in few planes a block: the same forces as the
    gradient and the gather one after the other, and the same density as a batch
    whose blocks march longer."""
    X = inputs.uniform_particles(n ** 3, 5)
    V = np.zeros((3, n ** 3), dtype=np.float32)
    sim = pm.Simulation(X, V, n, Om=0.3, OL=0.7, boxsize=float(n), keep_acc=True, grad_order=order)
    sim.step(a=0.5, dt_kick=0.0, dt_drift=0.0)
    assert torch.equal(sim.acc, pm.interp(pm.gradient(sim.phi, order), sim.X))
    Xd, B = pm.positions_to_device(X), 2 if n == 128 else 16
    rho = pm.deposit(Xd, n)
    assert torch.equal(pm.deposit_batch(Xd.repeat(1, B), n, B)[B - 1], rho)


@pytest.mark.parametrize("B", [127, 128])
def test_cell_starts_on_both_sides_of_the_scan_rule(pm, B):
    """2033 chunks of cell counts (each block adds the totals before its own) and
    2049 (a scan of the totals): every box's density as if it were alone."""
    n, np_box = 64, 1537
    X = inputs.uniform_particles(B * np_box, 9)
    rho = pm.deposit_batch(pm.positions_to_device(X), n, B)
    for b in (0, 63, B - 1):
        one = pm.positions_to_device(np.ascontiguousarray(X[:, b * np_box:(b + 1) * np_box]))
        assert torch.equal(rho[b], pm.deposit(one, n)), b


def test_large_batch_is_bitwise_a_batch_of_one(pm):
    """40 boxes of 64^3 march more planes a block than one box does: neither the
    density nor its mean depends on that."""
    w = inputs.ensemble_workload(n=64, B=1, boxsize=128.0, steps=2)
    out = []
    for B in (1, 40):
        X, V = np.repeat(w["X"], B, axis=0), np.repeat(w["V"], B, axis=0)
        ens = pm.Ensemble(X, V, 64, np.repeat(w["Om"], B), w["boxsize"], cold_cycles=4)
        coef = ens.coefficients(w["a_steps"][:3])
        for i in range(2):
            ens.step(coef[i])
        out.append((ens.positions(), ens.velocities()))
    for b in (0, 17, 39):
        assert np.array_equal(out[1][0][b], out[0][0][0]) and np.array_equal(out[1][1][b], out[0][1][0]), b


@pytest.mark.parametrize("n,N,order", [(128, 1 << 22, "random"), (128, (1 << 22) + 3, "cells"), (16, 1 << 22, "random"),
                                       (64, (1 << 22) - 1, "random")])
def test_packed_positions_deposit_the_same(pm, n, N, order):
    """Many particles in random order are gathered from packed positions: the
    density (and the cotangents) of any order is that of the cell order."""
    X = inputs.uniform_particles(N, 8)
    c = X >> np.uint32(32 - int(np.log2(n)))
    by = np.lexsort((c[2], c[1], c[0]))
    Xd, Xc = pm.positions_to_device(X), pm.positions_to_device(X[:, by])
    if order == "cells":
        Xd, by = Xc, np.arange(N)
    assert torch.equal(pm.deposit(Xd, n), pm.deposit(Xc, n))
    g = torch.from_numpy(np.stack([inputs.random_field(n, 70 + d) for d in range(3)]).astype(np.float32)).cuda()
    bar = torch.from_numpy(np.random.default_rng(1).standard_normal((3, N)).astype(np.float32)).cuda()
    b = torch.from_numpy(by).cuda()
    one, two = pm.interp_adj(g, Xd, bar), pm.interp_adj(g, Xc, bar[:, b].contiguous())
    assert torch.equal(one[0], two[0]) and torch.equal(one[1][:, b], two[1])
