"""The unfused energy update where its warps leave work out: patches of uniform
temperature and one phase, faces without flow, fluxes that are all liquid, all
gas or neither, at tile edges and remainders."""
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


def _weno5(v):
    q = [(2 * v[0] - 7 * v[1] + 11 * v[2]) / 6, (-v[1] + 5 * v[2] + 2 * v[3]) / 6, (2 * v[2] + 5 * v[3] - v[4]) / 6]
    b = [13 / 12 * (v[i] - 2 * v[i + 1] + v[i + 2]) ** 2 for i in range(3)]
    b[0] += (v[0] - 4 * v[1] + 3 * v[2]) ** 2 / 4
    b[1] += (v[1] - v[3]) ** 2 / 4
    b[2] += (3 * v[2] - 4 * v[3] + v[4]) ** 2 / 4
    w = [d / (1e-6 + x) ** 2 for d, x in zip((0.1, 0.6, 0.3), b)]
    return sum(x * y for x, y in zip(w, q)) / sum(w)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n,bc", [(8, 0), (9, 1), (37, 0), (64, 1)])
def test_energy_update_matches_plain_arithmetic(P, axis, n, bc):
    import torch
    rng = np.random.default_rng(100 * axis + n)
    shape = [5, 6, 34]  # z, y, x
    shape[2 - axis] = n
    Cl, Cg, lam = 1000.0, 1.5, 0.25
    c = rng.choice([0.0, 1.0, 0.3], size=shape)
    T = 1.0 + 0.5 * rng.random(shape)
    # along the axis as the last dimension
    L = lambda x: np.moveaxis(x, 2 - axis, -1)  # noqa: E731
    m = max(7, 3 * n // 4)  # lines that begin with uniform T and one phase
    L(c)[:3, :, :m], L(T)[:3, :, :m] = (np.arange(L(c).shape[1]) % 2.0)[None, :, None], 1.25
    e = (Cl * c + Cg * (1 - c)) * T
    idx = (lambda k: k % n) if bc == 0 else (lambda k: np.clip(k, 0, n - 1))
    a = 0.4 * (2 * rng.random(L(c).shape[:-1] + (n + 1,)) - 1)
    a[rng.random(a.shape) < 0.2] = 0.0
    if bc == 0:
        a[..., n] = a[..., 0]
    k = np.arange(n + 1)
    don = np.where(a > 0, np.take(L(c), idx(k - 1), -1), np.take(L(c), idx(k), -1))
    F = np.where(don == 0.3, a * (0.3 if n % 2 else 0.0) + 0.1 * a, don * a)
    c_after = L(c).copy()
    c_after[rng.random(c_after.shape) < 0.1] += 0.125
    # plain arithmetic
    Tl, Cp = L(e) / L(Cl * c + Cg * (1 - c)), L(Cl * (c > 0.5) + Cg * (c <= 0.5))
    st = [[np.take(Tl, idx(k + (r - 1 if s else -r)), -1) for r in range(-2, 3)] for s in (1, 0)]
    Tf = np.where(a > 0, _weno5(st[0]), _weno5(st[1]))
    G = np.where(a != 0, Tf * (Cl * F + Cg * (a - F)), 0.0)
    th = Cp * Tl
    ref = (L(e) + (G[..., :-1] - th * a[..., :-1])) - (G[..., 1:] - th * a[..., 1:])
    # the call
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(np.moveaxis(x, -1, 2 - axis))).cuda()  # noqa: E731
    g = P.Grid(shape[2], shape[1], shape[0], tuple(bc if i == axis else 0 for i in range(3)), 1.0, Cl, Cg, 1.0)
    out, state = torch.empty(shape, dtype=torch.float64, device="cuda"), torch.zeros(shape, dtype=torch.uint8, device="cuda")
    theta = torch.zeros(shape, dtype=torch.float64, device="cuda")
    P.energy_advect_consistent(g, axis, dev(L(c)), dev(c_after), dev(L(e)), out, dev(F), dev(a / lam), lam, state, theta)
    got, got_s, got_t = (L(x.cpu().numpy()) for x in (out, state, theta))
    # a rounding of T moves a WENO5 weight by at most 1e3 times as much
    # (the indicators' 1e-6), a handful of which meet in a face
    assert np.abs(got - ref).max() <= 1e-11 * Cl
    # uniform T, one phase across both donors: not a bit moves
    same = np.ones(ref.shape, bool)
    for r in range(-3, 4):
        same &= (np.take(L(c), idx(np.arange(n) + r), -1) == L(c)) & (np.take(L(T), idx(np.arange(n) + r), -1) == L(T))
    assert np.array_equal(got[same], L(e)[same]) and same.any()
    moved = (c_after != L(c)) | (got != L(e))
    assert np.array_equal(got_s, np.where(moved, 1 + 2 * (L(c) > 0.5), 0))
    assert np.abs(got_t - np.where(moved, th, 0.0)).max() <= 4 * np.finfo(float).eps * Cl * 1.5
