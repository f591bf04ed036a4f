"""Accuracy of the heat diffusion where the change of T is as large as T itself
(a hot wall on cold gas, a jump from 300 to 600), small beside it, and on both
sides of the rule that chooses the sweeps' form, against the same sweeps in long
double.

Bound: the result may be no further off than plain FP64 sweeps of T.  Those are
made here in numpy; the library's differ in the order of roundings (fused
multiply-adds), for which three times their largest error and four ulps of the
largest T are allowed (pairs of FP32 numbers for the change, 48 bits of it, are 4
to 20 times as far off as FP64 on these)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CP, K_G, H = 1200.0, 0.025, 1e-3
SWEEPS = 3000


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_03477_gb300 import build
    build.build()
    import paper_2001_03477_gb300 as P
    return P


def sweeps(T0, Tw, fourier, real, count=SWEEPS):
    """T after `count` Jacobi sweeps of gas in a box of zero-gradient walls, the
    lower x wall at Tw (None: no heated wall), in the number type given."""
    f = lambda v: real(v)  # noqa: E731
    T0 = T0.astype(real)
    dt = fourier * H * H * CP / K_G
    kq, cdt = f(K_G) / (f(H) * f(H)), f(CP) / f(dt)
    off = []
    for axis in range(3):
        for s in (-1, 1):
            o = np.full(T0.shape, kq)
            edge = [slice(None)] * 3
            edge[axis] = 0 if s < 0 else -1
            o[tuple(edge)] = 0
            off.append(o)
    diag, rhs = np.full(T0.shape, cdt), cdt * T0
    if Tw is not None:  # x is the last axis: d = h / 2 to the wall, h beyond
        kd = kq / f(0.75)
        off[5][..., 0] = kd
        diag[..., 0] += 2 * kd
        rhs[..., 0] += 2 * kd * f(Tw)
    for o in off:
        diag = diag + o
    T = T0.copy()
    for _ in range(count):
        a = rhs
        for q, (axis, s) in enumerate((ax, s) for ax in range(3) for s in (-1, 1)):
            a = a + off[q] * np.roll(T, -s, axis)
        T = a / diag
    return T


def start(name, shape):
    rng = np.random.default_rng(3)
    if name == "cold gas, hot wall":
        return np.zeros(shape), 320.0
    if name == "a jump of the size of T":
        return np.where(np.arange(shape[2]) < shape[2] // 2, 600.0, 300.0) * np.ones(shape), None
    if name == "hot wall":
        return np.full(shape, 300.0), 600.0
    if name == "within the rule":  # for pairs: 16 times the range is at most the smallest T
        return np.full(shape, 320.0), 339.9
    if name == "beyond the rule":
        return np.full(shape, 320.0), 340.1
    if name == "below zero":
        return -300.0 - 10.0 * rng.random(shape), -310.0
    return 300.0 + 10.0 * rng.random(shape), 310.0  # a change small beside T


@pytest.mark.parametrize("fourier", [0.8, 5.0, 20.0])
@pytest.mark.parametrize("name", ["cold gas, hot wall", "a jump of the size of T", "hot wall", "small change",
                                  "within the rule", "beyond the rule", "below zero"])
def test_no_further_off_than_fp64_sweeps(P, name, fourier):
    import torch
    shape = (4, 5, 22)
    T0, Tw = start(name, shape)
    exact = sweeps(T0, Tw, fourier, np.longdouble)
    plain = float(np.abs(sweeps(T0, Tw, fourier, np.float64) - exact).max())
    g = P.Grid(shape[2], shape[1], shape[0], (1, 1, 1), H, 4e6, CP, 300.0)
    e = torch.from_numpy(CP * T0).cuda()
    try:
        P.vof_heat_diffusion(g, torch.zeros(shape, dtype=torch.float64, device="cuda"), e, 0.68, K_G,
                             fourier * H * H * CP / K_G, tol=1e-300, max_iter=SWEEPS,
                             wall_T=None if Tw is None else {(0, -1): Tw})
    except P.VofError as err:  # the budget, unless no T changes any more
        assert err.status == P.VOF_ESOLVE
    off = float(np.abs(e.cpu().numpy() / CP - exact).max())
    assert off <= 3 * plain + 4 * np.spacing(float(np.abs(exact).max()))


@pytest.mark.parametrize("budget,tol", [(1, 1e3), (2, 1e3), (3, 1e3), (1000, 1.0), (1000, 1e-2), (1000, 1e-4)])
@pytest.mark.parametrize("name", ["small change", "cold gas, hot wall"])
def test_reported_change_is_the_sweeps(P, name, budget, tol):
    """The change of the last sweep, to the rounding of FP64 temperatures: both
    iterates carry at most 16 ulps of the largest T each."""
    import torch
    shape = (3, 4, 9)
    T0, Tw = start(name, shape)
    g = P.Grid(shape[2], shape[1], shape[0], (1, 1, 1), H, 4e6, CP, 300.0)
    e = torch.from_numpy(CP * T0).cuda()
    it, change = P.vof_heat_diffusion(g, torch.zeros(shape, dtype=torch.float64, device="cuda"), e, 0.68, K_G,
                                      0.8 * H * H * CP / K_G, tol=tol, max_iter=budget, wall_T={(0, -1): Tw})
    last, before = (sweeps(T0, Tw, 0.8, np.longdouble, n) for n in (it, it - 1))
    want = float(np.abs(last - before).max())
    assert 1 <= it <= budget and change <= tol
    assert abs(change - want) <= 32 * np.spacing(float(np.abs(last).max()))
