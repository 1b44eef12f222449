"""FP64 slice kernels in fixed point: every entry of the result, not only its norm, and the whole of
FP64's range.

Each pass applies an N x N operator A to lines whose table carries an absolute error (entries are
sums of N rounded terms, folded twice) and adds a few roundings of the line's largest entry; in
units of 2^-53 of it, e = 2 N + 16 covers both.  Three passes are therefore within
    ((|A| + e J) (x) (|A| + e J) (x) (|A| + e J)  -  |A| (x) |A| (x) |A|) |x|      (J: all ones)
of the exact result, entry by entry, whatever the sizes of x's entries: what FP64 multiply-adds
along each line satisfy.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

L = np.longdouble
EXTENTS = [(4, 9), (6, 7), (8, 6), (10, 5), (12, 4), (16, 3), (32, 3)]


@pytest.fixture(scope="module")
def ufg():
    from paper_1008_3647_gb300 import ufg as u
    u.load()
    return u


def _freq(nx):
    n = np.arange(nx)
    return 2 * np.arccos(L(-1)) * np.where(n <= nx // 2, n, n - nx) / L(nx)


def _kinetic(nx, tau, dispersion):
    k = _freq(nx)
    lam = np.exp(-L(tau) * (k * k / 2 if dispersion == 0 else 1 - np.cos(k)))
    T = np.array([np.sum(lam * np.cos(k * d)) / L(nx) for d in range(nx)], dtype=L)
    i = np.arange(nx)
    return T[(i[:, None] - i[None, :]) % nx]


def _fourier(nx):
    # rows: slots (constant, cosines, alternating, sines), columns: sites
    x, H = np.arange(nx), nx // 2
    F = np.zeros((nx, nx), dtype=L)
    a = 2 * np.arccos(L(-1)) / L(nx)
    F[0] = 1 / np.sqrt(L(nx))
    F[H] = np.where(x % 2, -1, 1) / np.sqrt(L(nx))
    for i in range(1, H):
        F[i] = np.sqrt(2 / L(nx)) * np.cos(a * i * x)
        F[H + i] = np.sqrt(2 / L(nx)) * np.sin(a * i * x)
    return F


def _axes(A, v):
    for axis in (1, 2, 3):
        v = np.moveaxis(np.tensordot(A, v, axes=(1, axis)), 0, axis)
    return v


def _bound(nx, A, x):
    e = L(2 * nx + 16) * L(2) ** -53
    return _axes(np.abs(A) + e, np.abs(x)) - _axes(np.abs(A), np.abs(x))


def _vector(nx, ntau, seed, kind):
    rng = np.random.default_rng(seed)
    shape = (ntau, nx, nx, nx)
    x = rng.standard_normal(shape)
    if kind == "point":  # one site per slice
        keep = np.zeros(shape)
        for t in range(ntau):
            keep[t, (5 * t) % nx, (3 * t + 1) % nx, (t + nx // 2) % nx] = 1.0
        return x * keep
    if kind == "lines":  # lines, rows and planes of very different size
        return x * 10.0 ** (rng.uniform(-6, 6, (ntau, nx, 1, 1)) + rng.uniform(-6, 6, (ntau, 1, nx, 1))
                            + rng.uniform(-6, 6, (ntau, 1, 1, nx)))
    return x * 10.0 ** rng.uniform(-8, 8, shape)  # "sites"


@pytest.mark.parametrize("kind", ["point", "lines", "sites"])
@pytest.mark.parametrize("tau,dispersion", [(0.05, 0), (0.05, 1), (20.0, 0)])
@pytest.mark.parametrize("nx,ntau", EXTENTS)
def test_every_entry_of_the_kinetic_factor(ufg, nx, ntau, tau, dispersion, kind):
    x = _vector(nx, ntau, 17 * nx + ntau, kind)
    lat = ufg.Lattice(nx, ntau, tau, 0.1, dispersion)
    field = ufg.Field(lat, torch.zeros(lat.shape, dtype=torch.float64, device="cuda"))
    y = ufg.ufg_apply_kinetic(field, torch.from_numpy(x).cuda()).cpu().numpy()
    A = _kinetic(nx, tau, dispersion)
    v = x.astype(L)
    err = np.abs(y - _axes(A, v))
    assert (err <= _bound(nx, A, v)).all(), float(np.max(err / _bound(nx, A, v)))


@pytest.mark.parametrize("kind", ["point", "lines", "sites"])
@pytest.mark.parametrize("nx,ntau", EXTENTS)
def test_every_entry_of_the_transforms(ufg, nx, ntau, kind):
    x = _vector(nx, ntau, 3 * nx + ntau, kind)
    lat = ufg.Lattice(nx, ntau)
    field = ufg.Field(lat, torch.zeros(lat.shape, dtype=torch.float64, device="cuda"))
    v = x.astype(L)
    for inverse in (False, True):
        y = ufg.ufg_fourier(field, torch.from_numpy(x).cuda(), inverse=inverse).cpu().numpy()
        A = _fourier(nx).T if inverse else _fourier(nx)
        err = np.abs(y - _axes(A, v))
        assert (err <= _bound(nx, A, v)).all(), (inverse, float(np.max(err / _bound(nx, A, v))))


@pytest.mark.parametrize("kind", ["point", "lines"])
@pytest.mark.parametrize("nx,ntau", EXTENTS)
def test_every_entry_of_M_and_its_transpose(ufg, nx, ntau, kind):
    x = _vector(nx, ntau, 29 * nx + ntau, kind)
    rng = np.random.default_rng(nx)
    sigma = rng.uniform(-np.pi, np.pi, x.shape)
    lat = ufg.Lattice(nx, ntau)
    field = ufg.Field(lat, torch.from_numpy(sigma).cuda())
    w = 1 + np.sqrt(L(2) * np.expm1(L(0.05) * L(5.0))) * np.sin(sigma.astype(L))
    A, v, u = _kinetic(nx, 0.05, 0), x.astype(L), L(2) ** -53
    for fn, shift in ((ufg.ufg_apply_M, 1), (ufg.ufg_apply_Mdag, -1)):
        y = fn(field, torch.from_numpy(x).cuda()).cpu().numpy()
        sgn = np.full((ntau, 1, 1, 1), -1)
        sgn[0 if shift == 1 else -1] = 1
        arg = w * v if shift == 1 else v
        # w = 1 + A sin(sigma) is off by a few units of 1 + A where it nearly vanishes; the sum and
        # the products round once each
        k, kb = _axes(A, arg), _bound(nx, A, arg) + 8 * u * _axes(np.abs(A), np.abs(v))
        k, kb, ka = (np.roll(q, shift, axis=0) for q in (k, kb, _axes(np.abs(A), np.abs(v))))
        if shift == -1:
            k, kb = w * k, np.abs(w) * kb + 8 * u * ka
        ref = v + sgn * k
        err = np.abs(y - ref)
        tol = kb + 4 * u * (np.abs(v) + np.abs(k))
        assert (err <= tol).all(), (shift, float(np.max(err / tol)))


@pytest.mark.parametrize("nx,ntau", EXTENTS)
def test_range_of_fp64(ufg, nx, ntau):
    x = torch.from_numpy(np.random.default_rng(nx).uniform(
        -1, 1, (ntau, nx, nx, nx))).cuda()
    lat = ufg.Lattice(nx, ntau)
    field = ufg.Field(lat, torch.zeros(lat.shape, dtype=torch.float64, device="cuda"))
    y = ufg.ufg_apply_kinetic(field, x)
    # a power of two scales every result exactly while none leaves the normal range, next to the
    # largest number (2^1023) included
    for k in (-960, 960, 1023):
        z = ufg.ufg_apply_kinetic(field, x * 2.0 ** (k // 2) * 2.0 ** (k - k // 2))
        assert torch.equal(z * 2.0 ** -(k // 2) * 2.0 ** -(k - k // 2), y), k
    # subnormal vectors: to the last unit of the range, rounded twice at most
    small = x * 2.0 ** -530 * 2.0 ** -530
    ref = ufg.ufg_apply_kinetic(field, small * 2.0 ** 530 * 2.0 ** 530) * 2.0 ** -530 * 2.0 ** -530
    assert float((ufg.ufg_apply_kinetic(field, small) - ref).abs().max() * 2.0 ** 1000) <= 2.0 ** -73


@pytest.mark.parametrize("nx,ntau", EXTENTS)
def test_range_of_the_operators(ufg, nx, ntau):
    # as above through every epilogue: the identity and the multipliers beside the line passes, and
    # the momentum-space operator, which leaves fixed point and comes back to it half way
    rng = np.random.default_rng(nx + 1)
    shape = (ntau, nx, nx, nx)
    sigma = torch.from_numpy(rng.uniform(-np.pi, np.pi, shape)).cuda()
    field = ufg.Field(ufg.Lattice(nx, ntau), sigma)
    x = torch.from_numpy(rng.uniform(-1, 1, shape)).cuda()
    fns = [ufg.ufg_apply_M, ufg.ufg_apply_M1, ufg.ufg_apply_M1T, ufg.ufg_fourier,
           lambda f, v: ufg.ufg_fourier(f, v, inverse=True)]
    if nx != 32:
        fns.append(ufg.ufg_apply_Mdag)
    if nx in (8, 16):
        fns += [ufg.ufg_apply_M_momentum, lambda f, v: ufg.ufg_apply_M_momentum(f, v, transpose=True)]
    for fn in fns:
        y = fn(field, x)
        # F sums up to N^(3/2) entries of x: 2^1015 leaves it and M finite
        for k in (-960, 1015):
            z = fn(field, x * 2.0 ** (k // 2) * 2.0 ** (k - k // 2))
            assert torch.equal(z * 2.0 ** -(k // 2) * 2.0 ** -(k - k // 2), y), (fn, k)
