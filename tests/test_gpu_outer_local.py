"""Precision of the fused FP64 residual cell by cell: a cell's error is bounded by the size of its own taps, whatever
larger values the same tile holds elsewhere.  Narrow Gaussians (cells many widths away, before and after the
peak in the march along z), W components of very different size, values that jump by many orders from plane to
plane, regions that are exactly zero, noise whose size falls along the march.

Reference: the same discrete operator in extended precision (numpy longdouble: 64 bits of mantissa or more).
Bounds, with eps = 2^-53, T the largest |value| among a cell's axis taps, weights of total size 16/3 per axis of a
second difference, 18/12 of a first derivative.  A stored tap is within T eps (a cell with no tap of 2^53 units is
formed in FP64); shifts add at most one more unit, the conversion, the weight and the products 4 roundings of
the result.  FP64 itself takes at most 8 roundings of the weighted taps.
  Lap u           16/3 (8 + 1) sum_a 1/h_a^2              -> 48 eps T sum 1/h^2
  row A, own part 4/3 of that                              -> 64 eps T_A sum 1/h^2
  row A, mixed    (18/12)^2 / 3 (8 + 1) per pair           -> 8 eps X_B / (h_A h_B), X_B over the pair's 5 x 5 taps
  D_i W_j         18/12 (8 + 1)                            -> 14 eps T_j / h_i
and 32 eps of each term for the powers of psi.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2501_13046_gb300 import fields  # noqa: E402

EPS = 2.0 ** -53
L = np.longdouble


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_13046_gb300 import _build
    _build.build()
    from paper_2501_13046_gb300 import mg as m
    return m


def shifted(f, o):
    """f at the cells displaced by o = (x, y, z), periodic."""
    return np.roll(f, (-o[2], -o[1], -o[0]), axis=(0, 1, 2))


def along(a, s):
    return tuple(s if c == a else 0 for c in range(3))


def reference(order, h, u, W, src=None, K=0.0):
    """H, M of a state on a periodic box (src: rho0, rho2, S; None: vacuum), and their bounds."""
    F1 = {1: L(1) / 2, -1: -L(1) / 2} if order == 2 else {1: L(8) / 12, -1: -L(8) / 12, 2: -L(1) / 12, -2: L(1) / 12}
    F2 = ({0: L(-2), 1: L(1), -1: L(1)} if order == 2 else
          {0: -L(30) / 12, 1: L(16) / 12, -1: L(16) / 12, 2: -L(1) / 12, -2: -L(1) / 12})
    u, W, h = u.astype(L), W.astype(L), [L(x) for x in h]
    ih2 = sum(1 / x ** 2 for x in h)
    d1 = lambda f, a: sum(w * shifted(f, along(a, s)) for s, w in F1.items()) / h[a]
    d2 = lambda f, a: sum(w * shifted(f, along(a, s)) for s, w in F2.items()) / h[a] ** 2
    star = lambda f: np.maximum.reduce([np.abs(shifted(f, along(a, s))) for a in range(3) for s in F2])
    T = [star(f) for f in W]
    lap = sum(d2(u, a) for a in range(3))
    lap_err = 48 * EPS * ih2 * star(u)
    varies = lambda f, a: any((f != shifted(f, along(a, s))).any() for s in F1)   # (else its differences along a are exact zeros)
    mom, mom_err = [], []
    for A in range(3):
        m = sum(d2(W[A], a) for a in range(3)) + d2(W[A], A) / 3
        e = 64 * EPS * ih2 * T[A]
        for B in range(3):
            if B != A:
                m = m + d1(d1(W[B], B), A) / 3
                box = np.maximum.reduce([np.abs(shifted(shifted(W[B], along(A, s)), along(B, t))) for s in F2 for t in F2])
                e = e + (8 * EPS * box / (h[A] * h[B]) if varies(W[B], A) and varies(W[B], B) else 0)
        mom.append(m)
        mom_err.append(e)
    D = [[d1(W[b], a) for b in range(3)] for a in range(3)]
    third = (D[0][0] + D[1][1] + D[2][2]) / 3
    dD = [[14 * EPS * T[b] / h[a] if varies(W[b], a) else 0 for b in range(3)] for a in range(3)]
    aa = aa_err = 0
    for a in range(3):
        for b in range(3):
            at = D[a][b] + D[b][a] - (2 * third if a == b else 0)
            de = dD[a][b] + dD[b][a] + (2 * (dD[0][0] + dD[1][1] + dD[2][2]) / 3 if a == b else 0)
            aa, aa_err = aa + at * at, aa_err + 2 * np.abs(at) * de + de * de
    psi = 1 + u
    nl = aa / (8 * psi ** 7)
    F, terms = lap + nl, np.abs(lap) + nl
    mom, mom_err = np.stack(mom), np.stack(mom_err) + 32 * EPS * np.abs(np.stack(mom))
    if src is not None:
        pi = L("3.14159265358979323846264338327950288")
        rho0, rho2, S = (f.astype(L) for f in src)
        F = F + 2 * pi * (rho0 * psi ** 5 + rho2 * psi) - L(K) ** 2 / 12 * psi ** 5
        terms = terms + 2 * pi * (np.abs(rho0) * psi ** 5 + np.abs(rho2) * psi) + L(K) ** 2 / 12 * psi ** 5
        s = 8 * pi * psi ** 6 * S
        mean = s.mean(axis=(1, 2, 3), keepdims=True)
        mom = mom - s + mean
        # (a mean's sum rounds once per term at most)
        mom_err = mom_err + 32 * EPS * np.abs(s) + (s[0].size ** 0.5 + 64) * EPS * np.abs(s).mean(axis=(1, 2, 3), keepdims=True)
    H = -8 * F / psi ** 5
    tol_H = 8 / psi ** 5 * (lap_err + aa_err / (8 * psi ** 7) + 32 * EPS * terms)
    return H, mom / psi ** 6, tol_H, mom_err / psi ** 6


def gpu_fields(mg, n, h, order, u, W, src=None, K=0.0):
    p = dict(n=list(n), lo=[0.0] * 3, hi=[h[a] * n[a] for a in range(3)], order=order, bc=fields.PERIODIC,
             kmode=fields.K_FIXED, K=K, punctures=[])
    z = np.zeros_like(u)
    rho0, rho2, S = src if src is not None else (z, z, [z] * 3)
    ctx = mg.mg_create(mg.config_for(p, mg.MG_FP64), torch.cuda.current_stream().cuda_stream)
    try:
        mg.mg_set_sources(ctx, *[np.ascontiguousarray(f) for f in (rho0, rho2, *S)])
        mg.mg_set_initial_guess(ctx, np.ascontiguousarray(u), np.ascontiguousarray(W))
        H, M = np.empty_like(u), np.empty_like(W)
        mg.mg_constraint_fields(ctx, H, M)
    finally:
        mg.mg_destroy(ctx)
    return H, M


def check(mg, n, h, order, u, W, src=None, K=0.0):
    H, M = gpu_fields(mg, n, h, order, u, W, src, K)
    rH, rM, tol_H, tol_M = reference(order, h, u, W, src, K)
    l2 = lambda a, b: float(np.sqrt(((a - b) ** 2).sum() / np.maximum((b ** 2).sum(), L(1e-300))))
    print("order %d, spacings %s: relative L2 error of H %.2e, of M %.2e" % (order, h, l2(H, rH), l2(M, rM)))
    tiny = 1e-290   # (squares and products below the smallest normal number)
    assert (np.abs(H - rH) <= tol_H + tiny).all(), float(np.max(np.abs(H - rH) / (tol_H + tiny)))
    for a in range(3):
        assert (np.abs(M[a] - rM[a]) <= tol_M[a] + tiny).all(), (a, float(np.max(np.abs(M[a] - rM[a]) / (tol_M[a] + tiny))))
    return H, M


N = (40, 24, 48)
SPACINGS = [(1.0, 1.0, 1.0), (0.5, 0.75, 1.25)]


def gauss(centre, w, n=N):
    x, y, z = np.arange(n[0])[None, None, :], np.arange(n[1])[None, :, None], np.arange(n[2])[:, None, None]
    return np.exp(-((x - centre[0]) ** 2 + (y - centre[1]) ** 2 + (z - centre[2]) ** 2) / (2.0 * w * w))


@pytest.mark.parametrize("h", SPACINGS)
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("width", [1.2, 2.0, 3.0])
def test_narrow_gaussians(mg, width, order, h):
    u = 0.3 * gauss((13.3, 9.1, 21.4), width)
    W = np.stack([0.1 * gauss((11.0 + 9 * a, 10.5, 16.0 + 8 * a), width) for a in range(3)])
    check(mg, N, h, order, u, W)


@pytest.mark.parametrize("h", SPACINGS)
@pytest.mark.parametrize("order", [2, 4])
def test_components_of_unequal_size(mg, order, h):
    """W_y, ten orders larger than the others, varies along y only: rows x and z and AtAt's other entries see the
    small components alone."""
    x, y, z = np.arange(N[0])[None, None, :], np.arange(N[1])[None, :, None], np.arange(N[2])[:, None, None]
    one = np.ones(N[::-1])
    k = [2 * np.pi / m for m in N]
    small = np.cos(k[0] * x + 0.4) * np.cos(k[1] * y - 0.2) * np.cos(2 * k[2] * z + 1.0)
    W = np.stack([1e-11 * small, 0.1 * np.cos(k[1] * y + 0.3) * one, 1e-10 * np.roll(small, 5, axis=2)])
    check(mg, N, h, order, 0.01 * small, W)
    check(mg, N, h, order, 0 * small, np.stack([W[0], 0.1 * one, W[2]]))   # a constant component: H is AtAt alone


@pytest.mark.parametrize("order", [2, 4])
def test_jumps_between_planes(mg, order):
    """Noise of size 1e-30 with a few planes of size 0.01, and noise that falls fourfold per plane."""
    rng = np.random.default_rng(9)
    u = 1e-30 * rng.standard_normal(N[::-1])
    W = 1e-30 * rng.standard_normal((3,) + N[::-1])
    u[19:21] = 0.01 * rng.standard_normal(u[19:21].shape)
    W[1, 27:30] = 0.01 * rng.standard_normal(W[1, 27:30].shape)
    check(mg, N, SPACINGS[0], order, u, W)
    fall = 4.0 ** -np.arange(N[2])[:, None, None]
    check(mg, N, SPACINGS[1], order, 0.1 * fall * rng.standard_normal(u.shape), fall * rng.standard_normal(W.shape))


def test_zeros_stay_zero(mg):
    """Where every tap of a cell is zero, H and M are exactly zero, also beside non-zero values of the same tile."""
    rng = np.random.default_rng(4)
    u, W = np.zeros(N[::-1]), np.zeros((3,) + N[::-1])
    u[10:14, 4:8, 3:6] = 0.1 * rng.standard_normal((4, 4, 3))
    W[2, 10:14, 4:8, 3:6] = 0.1 * rng.standard_normal((4, 4, 3))
    for h in SPACINGS:
        H, M = check(mg, N, h, 4, u, W)
        near = np.zeros(u.shape, bool)
        near[8:16, 2:10, 1:8] = True
        assert (H[~near] == 0).all() and (M[:, ~near] == 0).all()


@pytest.mark.parametrize("h", SPACINGS)
@pytest.mark.parametrize("order", [2, 4])
def test_smooth_state_with_matter(mg, order, h):
    """A state on its way to the solution: smooth u and W, a nearly uniform scalar field's sources and the K of their mean."""
    rng = np.random.default_rng(2)
    x = [np.arange(N[a]).reshape([-1 if b == 2 - a else 1 for b in range(3)]) / N[a] for a in range(3)]

    def modes(amplitude):
        f = np.zeros(N[::-1])
        for _ in range(8):
            k = rng.integers(-3, 4, 3)
            f += amplitude / (1 + np.abs(k).sum()) * np.cos(2 * np.pi * sum(k[a] * x[a] for a in range(3)) + 2 * np.pi * rng.random())
        return f
    u, W = modes(0.01), np.stack([modes(1e-3) for _ in range(3)])
    rho0, rho2, S = 0.5 + modes(1e-3), modes(1e-4) ** 2, np.stack([modes(1e-5) for _ in range(3)])
    check(mg, N, h, order, u, W, (rho0, rho2, S), K=-np.sqrt(24 * np.pi * rho0.mean()))
