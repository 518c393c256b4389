"""The linear smoother's fused sweeps (one or two sweeps per pass over memory,
levels with n >= 64) against the colour passes, bitwise, over sweep counts,
factors, guesses and batches; the coarsest-level solve at each size it takes
against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import poisson
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


@pytest.mark.parametrize("n,npre,npost,omega,scale", [(64, 1, 0, 1.25, 1.0), (64, 2, 1, 1.25, 0.9), (128, 3, 2, 1.1, 1.3),
                                                      (64, 4, 4, 1.0, 1.1), (256, 2, 3, 1.25, 0.7)])
def test_fused_sweeps_are_bitwise_the_colour_passes(pm, n, npre, npost, omega, scale):
    f = torch.from_numpy(inputs.random_field(n, 11).astype(np.float32)).cuda()
    phi0 = torch.from_numpy(inputs.random_field(n, 12).astype(np.float32)).cuda()
    outs = []
    for smoother in (2, 0, 1):
        phi, _ = pm.mg_solve(f, phi=phi0.clone(), fixed_cycles=2, first_guess=pm.MG_GUESS_SCALED, guess_scale=scale,
                             npre=npre, npost=npost, omega=omega, smoother=smoother)
        outs.append(phi.cpu().numpy())
    assert np.array_equal(outs[0], outs[2]) and np.array_equal(outs[1], outs[2])


@pytest.mark.parametrize("n,B", [(64, 1), (64, 5), (128, 3)])
def test_fused_sweeps_of_a_batch(pm, n, B):
    f = torch.from_numpy(np.stack([inputs.random_field(n, 20 + b) for b in range(B)]).astype(np.float32)).cuda()
    phi = [pm.mg_solve_batch(f, fixed_cycles=2, smoother=s).cpu().numpy() for s in (2, 1)]
    assert np.array_equal(phi[0], phi[1])


@pytest.mark.parametrize("coarsest,sweeps", [(4, 200), (8, 200), (16, 200), (16, 0), (16, 3)])
def test_coarsest_sizes_match_the_oracle(pm, coarsest, sweeps):
    n = 32
    f = inputs.random_field(n, 5).astype(np.float32).astype(np.float64)
    phi, _ = pm.mg_solve(torch.from_numpy(f.astype(np.float32)).cuda(), fixed_cycles=2, coarsest=coarsest,
                         coarse_max_sweeps=sweeps, first_guess=pm.MG_GUESS_JACOBI)
    ref, _ = poisson.mg_solve(f, 1.0 / n, prm=poisson.MGParams(coarsest=coarsest, coarse_max_sweeps=sweeps), cycles=2)
    # the bar of the 16^3 case: float32 against float64 after the same steps
    assert np.linalg.norm(phi.cpu().numpy() - ref) < 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("nhs,a,n", [(1, 0.05, 128), (1, 1.0, 128), (2, 0.5, 128), (2, 1.0, 256)])
def test_fused_fr_sweeps_match_the_colour_passes(pm, nhs, a, n):
    """From the unscreened to the screened regime (eps towards -1), from a cold
    start: the pair root's second step and its fallback are taken."""
    rho = np.exp(1.2 * inputs.random_field(n, 31))
    rho = torch.from_numpy((rho / rho.mean()).astype(np.float32)).cuda()
    outs = [pm.fr_solve(rho, a=a, Om=0.3, OL=0.7, fR0=-1e-5, boxsize=float(n), cycles=1, nhs=nhs,
                        smoother=s)[0].cpu().numpy().astype(np.float64) for s in (2, 1)]
    assert np.all(np.isfinite(outs[0])) and outs[0].min() > -1.0
    # the same cell equations on the same neighbours, each root to float32 resolution
    assert np.linalg.norm(outs[0] - outs[1]) < 1e-6 * np.linalg.norm(outs[1])


@pytest.mark.parametrize("coarsest", [4, 8, 16])
def test_fr_coarsest_sizes_match_the_oracle(pm, coarsest):
    from oracle import fr as ofr
    n = 32
    rho = np.exp(0.8 * inputs.random_field(n, 8))
    rho = (rho / rho.mean()).astype(np.float32).astype(np.float64)
    model = ofr.FRModel(Om=0.3, OL=0.7, fR0=-1e-5, boxsize=float(n))
    eps, _ = pm.fr_solve(torch.from_numpy(rho.astype(np.float32)).cuda(), a=0.6, Om=0.3, OL=0.7, fR0=-1e-5,
                         boxsize=float(n), coarsest=coarsest, cycles=1)
    u, _ = ofr.fr_solve(rho, 0.6, model, prm=ofr.FASParams(coarsest=coarsest), cycles=1)
    # the bar of the 16^3 case
    assert np.linalg.norm(eps.cpu().numpy() - (u - 1.0)) < 1e-4 * np.linalg.norm(u - 1.0)


@pytest.mark.parametrize("n,coarsest", [(8, 4), (16, 4), (64, 16), (128, 16)])
def test_residual_norm_in_wide_loads(pm, n, coarsest):
    """The residual norm that ends a solve, from the smallest grid above the
    coarsest on, against float64 on the same iterate."""
    f = inputs.random_field(n, 12)
    f = (f - f.mean()).astype(np.float32)
    phi, st = pm.mg_solve(torch.from_numpy(f).cuda(), tol=0.9, coarsest=coarsest)
    u = phi.cpu().numpy().astype(np.float64)
    lap = sum(np.roll(u, s, d) for s in (1, -1) for d in range(3)) - 6.0 * u
    f = f.astype(np.float64)
    r = np.linalg.norm(f - lap * n * n)
    assert st["cycles"] == 1 and st["norm_f"] == pytest.approx(np.linalg.norm(f), rel=1e-6)
    # the residual is exact to a rounding of each cell's (and of the source less its float32 mean)
    assert st["res"] == pytest.approx(r, abs=2e-7 * st["norm_f"])


@pytest.mark.parametrize("n,B,npre,npost,coarsest", [(8, 1, 2, 2, 4), (16, 1, 1, 2, 4), (32, 1, 2, 2, 16),
                                                     (32, 2, 2, 1, 16), (32, 3, 2, 2, 8), (64, 5, 1, 1, 4)])
def test_small_levels_in_tiles_bitwise_equal_the_colour_passes(pm, n, B, npre, npost, coarsest):
    """Levels of up to 32^3 (tiles of 4 x 4 rows, of 8 x 8 in larger batches)
    against colour passes and transfers of their own."""
    f = np.stack([inputs.random_field(n, 60 + b) for b in range(B)]).astype(np.float32)
    f = torch.from_numpy(f).cuda()
    kw = dict(fixed_cycles=2, npre=npre, npost=npost, coarsest=coarsest, first_guess=pm.MG_GUESS_JACOBI)
    solve = (lambda s: pm.mg_solve(f[0], smoother=s, **kw)[0]) if B == 1 else (
        lambda s: pm.mg_solve_batch(f, smoother=s, **kw))
    assert torch.equal(solve(2), solve(1))
