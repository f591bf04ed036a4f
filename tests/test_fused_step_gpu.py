"""The fused sweeps of a time step (csrc/vof_fused.cu) against the stand-alone
calls, bit for bit, where the fused kernels can go wrong: edges of tiles (7, 8,
9, 15, 16, 17, 25 cells), axes shorter than a window, ragged halves of a tile,
periodic wraps and ghost donors, every form, quiet tiles next to active ones,
and grids large enough that tiles are walked in chains.  The stand-alone calls
are held to the oracle by their own tests.  Two steps, so both sweep orders
run and the second starts from the first's result."""
import math

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


def fields(shape, bc, seed, dense):
    """Drops of random size with graded interfaces, T varying in every cell or
    only in a layer, signed velocities within CFL 0.4."""
    import torch
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    z, y, x = torch.meshgrid(*[torch.arange(n, dtype=torch.float64, device="cuda") + 0.5 for n in shape], indexing="ij")
    c = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for _ in range(3):
        ctr, r = rng.uniform(0, 1, 3) * (nx, ny, nz), rng.uniform(0.15, 0.4) * max(min(shape), 6)
        d = ((x - ctr[0]) ** 2 + 1.3 * (y - ctr[1]) ** 2 + 0.8 * (z - ctr[2]) ** 2).sqrt()
        c = torch.maximum(c, (r - d + 0.5).clamp(0.0, 1.0))
    T = 1.0 + 0.3 * torch.sin(0.7 * x + 0.2) * torch.cos(0.9 * y) * torch.cos(0.5 * z)
    if not dense:
        T = torch.where((x < 0.3 * nx) & (y < 0.6 * ny + 2), T, torch.full_like(T, 1.0))
    e = (900.0 * c + 1.5 * (1.0 - c)) * T
    vel = []
    for a, sh in enumerate(((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx))):
        n = sh[0] * sh[1] * sh[2]
        i = torch.arange(n, dtype=torch.float64, device="cuda")
        u = 0.4 * torch.sin(i * 0.37 + a)
        u[:: 17] = 0.0
        vel.append(u.view(sh).contiguous())
    return c, e, vel


CASES = [
    # (nx, ny, nz), bc
    ((1, 1, 1), (0, 1, 0)), ((2, 3, 5), (0, 0, 0)), ((7, 9, 4), (1, 0, 1)), ((8, 8, 8), (0, 0, 0)), ((9, 7, 17), (1, 1, 1)),
    ((16, 15, 12), (0, 1, 0)), ((17, 16, 25), (1, 0, 0)), ((33, 20, 11), (0, 0, 1)), ((25, 41, 28), (0, 0, 0)), ((64, 40, 72), (1, 1, 0)),
]


def check(P, g, c, e, vel, dt, dd):
    import torch
    st = P.Stepper(g)
    c1, e1, c2, e2 = c.clone(), e.clone(), c.clone(), e.clone()
    for s in range(2):
        st.step(c1, e1, *vel, dt, s, dd_uniform=dd)
        state = torch.zeros(g.shape, dtype=torch.uint8, device="cuda")
        theta = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
        clip = torch.zeros(1, dtype=torch.float64, device="cuda")
        diag = torch.zeros(5, dtype=torch.float64, device="cuda")
        for axis in (0, 1, 2) if s % 2 == 0 else (2, 1, 0):
            P.SWEEPS[axis](g, c2, e2, c2, e2, vel[axis], dt, state, theta, None, clip)
        P.vof_phase_change_shift(g, c2, e2, c2, e2, None, dd, None, diag)
        assert torch.equal(c1, c2) and torch.equal(e1, e2)
        sums, d = st.sums.cpu().numpy(), diag.cpu().numpy()
        # c, e: n additions of values of one sign, each within half an ulp
        n = c.numel()
        tol = 4 * max(64, math.log2(n)) * 2.0 ** -53
        assert abs(sums[0] - float(c2.sum())) <= tol * float(c2.abs().sum()) + 1e-300
        assert abs(sums[1] - float(e2.sum())) <= tol * float(e2.abs().sum())
        for k in range(3):
            assert abs(sums[3 + k] - d[k]) <= 1e-11 * max(1.0, abs(d[k]))
    assert P.vof_get_device_status() in (0, P.VOF_ECFL)


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("form", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 2)], ids=["f64", "f32", "le", "youngs"])
def test_step_equals_standalone_calls(P, case, form):
    (nx, ny, nz), bc = CASES[case]
    c, e, vel = fields((nz, ny, nx), bc, 11 + case, dense=case % 2 == 0)
    g = P.Grid(nx, ny, nz, bc, 1.0, 900.0, 1.5, 1.0, precision=form[0], scheme=form[1], normal=form[2])
    check(P, g, c, e, vel, 1.0, -0.02 if case % 3 else 0.03)


@pytest.mark.parametrize("dense", [True, False])
def test_chains_equal_standalone_calls(P, dense):
    # 200^3: 15,625 tiles; all active (T varies): walked in chains; T uniform
    # away from a layer: the active tiles one by one
    n = 200
    c, e, vel = fields((n, n, n), (0, 1, 0), 5, dense)
    check(P, P.Grid(n, n, n, (0, 1, 0), 1.0, 900.0, 1.5, 1.0), c, e, vel, 1.0, -0.02)


@pytest.mark.parametrize("shape", [(41, 34, 26), (26, 41, 25), (33, 18, 50)])
@pytest.mark.parametrize("at", [0.0, 4.5, -2.5, -6.5, -10.5, 11.0])
def test_quiet_tiles_across_a_short_last_tile(P, shape, at):
    """Periodic axes whose last tile holds one or two cells: a small drop near
    the wrap leaves quiet tiles whose three-cell halo spans that tile."""
    import torch
    nx, ny, nz = shape
    z, y, x = torch.meshgrid(*[torch.arange(n, dtype=torch.float64, device="cuda") + 0.5 for n in (nz, ny, nx)], indexing="ij")
    d2 = 0.0
    for q, n, o in ((x, nx, at), (y, ny, 0.3 * at), (z, nz, -at)):
        d = (q - o) % n
        d2 = d2 + torch.minimum(d, n - d) ** 2
    c = (3.2 - d2.sqrt()).clamp(0.0, 1.0)
    vel = fields((nz, ny, nx), (0, 0, 0), 3, False)[2]
    g = P.Grid(nx, ny, nz, (0, 0, 0), 1.0, 900.0, 1.5, 1.0)
    check(P, g, c, 900.0 * c + 1.5 * (1.0 - c), vel, 1.0, 0.02)
