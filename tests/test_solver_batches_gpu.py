"""The heat diffusion's sweeps in pairs and batches, and the velocity
extension's solver choice, at the sizes where they can go wrong."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_03477_gb300 import build
    build.build()
    import paper_2001_03477_gb300 as P
    return P


@pytest.mark.parametrize("shape", [(1, 1, 5), (3, 9, 33), (8, 8, 32), (5, 17, 40)])
@pytest.mark.parametrize("sweeps", [1, 2, 3, 4, 5, 8, 9, 13])
def test_capped_sweeps_are_jacobi_iterates(P, shape, sweeps):
    """Gas alone in a periodic box: after k sweeps (the budget, reported as not
    converged) the energy is that of k plain Jacobi sweeps.  The change is held
    in 48 bits: 2^-46 of its size per sweep."""
    import torch
    rng = np.random.default_rng(sweeps)
    nz, ny, nx = shape
    T0 = 300.0 + 10.0 * rng.random(shape)
    Cp, k, h, dt = 1200.0, 0.025, 1e-3, 0.03
    kq, cdt = k / h ** 2, Cp / dt
    T = T0.copy()
    for _ in range(sweeps):
        nb = sum(np.roll(T, s, a) for a in range(3) for s in (-1, 1))
        T = (cdt * T0 + kq * nb) / (cdt + 6 * kq)
    g = P.Grid(nx, ny, nz, (0, 0, 0), h, 4e6, Cp, 300.0)
    e = torch.from_numpy(Cp * T0).cuda()
    with pytest.raises(P.VofError) as err:
        P.vof_heat_diffusion(g, torch.zeros(shape, dtype=torch.float64, device="cuda"), e, 0.68, k, dt, tol=1e-300, max_iter=sweeps)
    assert err.value.status == P.VOF_ESOLVE
    d = np.abs(T - T0).max()
    ulps = 8 * np.finfo(float).eps * 320.0  # the plain form's own rounding of T, and of e
    assert np.abs(e.cpu().numpy() / Cp - T).max() <= sweeps * 2.0 ** -46 * d + sweeps * ulps


@pytest.mark.parametrize("power", [-300, -40, 60, 300])
def test_diffusion_scales_by_powers_of_two(P, power):
    """The change is held over the power of two of the largest temperature: a
    problem scaled by 2^power has the scaled solution, bit for bit."""
    import torch
    shape = (10, 12, 13)
    z, y, x = np.meshgrid(*[np.arange(n) + 0.5 for n in shape], indexing="ij")
    c = np.clip(3.5 - np.sqrt((x - 6) ** 2 + (y - 6) ** 2 + (z - 5) ** 2), 0.0, 1.0)
    T = 300.0 + 10.0 * np.random.default_rng(5).random(shape)
    e0 = (4e6 * c + 1200.0 * (1 - c)) * T
    out = []
    for s in (1.0, 2.0 ** power):
        g = P.Grid(shape[2], shape[1], shape[0], (0, 1, 0), 1e-3, 4e6, 1200.0, 303.0 * s)
        e = torch.from_numpy(e0 * s).cuda()
        r = P.vof_heat_diffusion(g, torch.from_numpy(c).cuda(), e, 0.68, 0.025, 0.03, tol=1e-9 * s,
                                 wall_T={(1, -1): 320.0 * s})
        out.append((e.cpu().numpy() / s, r))
    assert np.array_equal(out[0][0], out[1][0]) and np.isfinite(out[0][0]).all()


@pytest.mark.parametrize("shape,bc", [((7, 8, 9), (0, 0, 0)), ((6, 5, 12), (1, 0, 1)), ((24, 20, 22), (1, 1, 1))])
def test_extension_with_many_and_few_unknowns(P, shape, bc):
    """Tiny boxes whose unknowns outnumber the one-launch solver's records (the
    kernel-per-phase solver takes them) and a larger one, against the oracle's
    direct solve."""
    import torch
    import oracle as O
    from oracle.extension import velocity_extension
    nz, ny, nx = shape
    z, y, x = np.meshgrid(*[np.arange(n) + 0.5 for n in shape], indexing="ij")
    r = np.sqrt((x - 0.5 * nx) ** 2 + (y - 0.5 * ny) ** 2 + (z - 0.47 * nz) ** 2)
    c = np.clip(0.25 * min(shape) + 0.5 - r, 0.0, 1.0)  # a drop in gas
    mdot = np.where((c > 1e-12) & (c < 1 - 1e-12), 1e-3 * (1 + 0.1 * np.cos(x + y)), 0.0)
    og = O.Grid(nx, ny, nz, bc, 0.1, 1.0, 1.0, 0.0)
    ref = velocity_extension(og, c, mdot, 10.0, 1.0, 0.01)[:3]
    g = P.Grid(nx, ny, nz, bc, 0.1, 1.0, 1.0, 0.0)
    out = [torch.empty(g.face_shape(a), dtype=torch.float64, device="cuda") for a in range(3)]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    P.vof_velocity_extension(g, dev(c), dev(mdot), 10.0, 1.0, 0.01, ut=out[0], vt=out[1], wt=out[2])
    scale = max(np.abs(np.asarray(ref[a])).max() for a in range(3))
    for a in range(3):
        assert np.abs(out[a].cpu().numpy() - np.asarray(ref[a])).max() <= 1e-9 * scale
