"""The shift of a time step (csrc/vof_shift.cu: marks, pairs, application per
tile) with a shift per cell -- both signs and exact zeros in one box -- and with
more (cell, neighbour) pairs than its list holds, against the stand-alone calls,
bit for bit, plain and grouped.  The stand-alone calls are held to the oracle by
their own tests."""
import numpy as np
import pytest

from test_fused_step_gpu import P, fields  # noqa: F401 -- P is a fixture

pytestmark = pytest.mark.gpu


def standalone(P, g, c, e, vel, dt, dd, steps):
    import torch
    c, e = c.clone(), e.clone()
    diag = torch.zeros(5, dtype=torch.float64, device="cuda")
    for s in range(steps):
        state = torch.zeros(g.shape, dtype=torch.uint8, device="cuda")
        theta = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
        diag.zero_()
        for axis in (0, 1, 2) if s % 2 == 0 else (2, 1, 0):
            P.SWEEPS[axis](g, c, e, c, e, vel[axis], dt, state, theta, None, None)
        P.vof_phase_change_shift(g, c, e, c, e, dd, 0.0, None, diag)
    return c, e, diag.cpu().numpy()


def check(P, g, c, e, vel, dt, dd, steps=2):
    import torch
    want_c, want_e, diag = standalone(P, g, c, e, vel, dt, dd, steps)
    st = P.Stepper(g)
    c1, e1 = c.clone(), e.clone()
    for s in range(steps):
        sums = st.step(c1, e1, *vel, dt, s, dd=dd).cpu().numpy()
    boxes = [P.Box(g, c.clone(), e.clone(), *vel, dt, dd) for _ in range(3)]
    grp = P.Group(boxes)
    for s in range(steps):
        grp.step(s)
    torch.cuda.synchronize()
    for cc, ee in [(c1, e1)] + [(b.c, b.e) for b in boxes]:
        assert torch.equal(cc, want_c) and torch.equal(ee, want_e)
    # sums of at most n changes of both signs, each at most 1 (c) or 900 (e)
    for k, size in ((0, 1.0), (1, 1.0), (2, 900.0)):
        assert abs(sums[3 + k] - diag[k]) <= c.numel() * 64 * 2.0 ** -53 * size
    grp.close()
    return float((want_c - c).abs().max())


@pytest.mark.parametrize("shape,bc", [((24, 17, 20), (0, 1, 0)), ((40, 33, 26), (1, 0, 1)), ((9, 10, 7), (0, 0, 0))])
@pytest.mark.parametrize("size", [0.03, 0.9])
@pytest.mark.parametrize("form", [(0, 0, 0), (1, 0, 0), (0, 1, 0)], ids=["f64", "f32", "le"])
def test_shift_per_cell(P, shape, bc, size, form):  # noqa: F811
    import torch
    nx, ny, nz = shape
    c, e, vel = fields((nz, ny, nx), bc, 21 + nx, dense=True)
    i = torch.arange(c.numel(), device="cuda")
    dd = size * torch.sin(0.61 * i.to(torch.float64)).view(c.shape)
    dd.view(-1)[i % 3 == 0] = 0.0  # cells that stay where they are
    dd.view(-1)[i % 9 == 1] = -0.0
    g = P.Grid(nx, ny, nz, bc, 1.0, 900.0, 1.5, 1.0, precision=form[0], scheme=form[1], normal=form[2])
    assert check(P, g, c, e, vel, 1.0, dd.contiguous()) > 0.0


@pytest.mark.parametrize("shape", [(4, 4, 4), (16, 8, 24), (34, 18, 22)])
@pytest.mark.parametrize("liquid", [False, True])
def test_more_pairs_than_the_list_holds(P, shape, liquid):  # noqa: F811
    """One mixed cell in eight, alone among pure ones, at rest: its normal is the
    degenerate (1, 0, 0) and its plane, moved by 0.6 .. 0.9, enters all 26
    neighbours (c + dd > 1 among gas, c + dd < 0 among liquid), so the pairs are
    26 / 8 of the list's one per cell and the walk over every neighbour runs.
    The edge cells (c within 1e-3 of the pure value) take the bisection."""
    import torch
    nx, ny, nz = shape
    rng = np.random.default_rng(nx)
    c = np.full((nz, ny, nx), 1.0 if liquid else 0.0)
    m = c[::2, ::2, ::2].shape
    v = rng.uniform(0.45, 0.55, m)
    v[rng.random(m) < 0.2] = 0.9995
    dd = np.zeros_like(c)
    dd[::2, ::2, ::2] = rng.uniform(0.6, 0.9, m)
    if liquid:
        v, dd = 1.0 - v, -dd
    c[::2, ::2, ::2] = v
    assert 26 * v.size > c.size
    T = 1.0 + 0.2 * rng.random(c.shape)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    g = P.Grid(nx, ny, nz, (0, 0, 0), 1.0, 900.0, 1.5, 1.0)
    vel = [torch.zeros(g.face_shape(a), dtype=torch.float64, device="cuda") for a in range(3)]
    moved = check(P, g, dev(c), dev((900.0 * c + 1.5 * (1 - c)) * T), vel, 1.0, dev(dd), steps=1)
    assert moved > 0.1
