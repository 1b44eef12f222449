"""FP64 slice kernels in 64-bit fixed point (integer pipe): precision against extended arithmetic,
exact behaviour under power-of-two scaling, and the ends of the exponent range.

Precision: the reference is M of the definition in numpy's long double.  Per axis the kernel's
table entries carry the rounding of sums of N FP64 terms (2 units of 2^-53 each at most, sqrt(N)
of them in the 2-norm of a line) and its pass a few roundings, so the 2-norm error stays below
3 (2 sqrt(N) + 4) 2^-53 for any vector, a single non-zero site included.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TAU, G = 0.05, 5.0
EXTENTS = [(4, 11), (6, 9), (8, 7), (10, 5), (12, 4), (16, 3), (32, 3)]


@pytest.fixture(scope="module")
def ufg():
    from paper_1008_3647_gb300 import ufg as u
    u.load()
    return u


def _inputs(nx, ntau, seed, kind):
    rng = np.random.default_rng(seed)
    shape = (ntau, nx, nx, nx)
    sigma = rng.uniform(-np.pi, np.pi, size=shape)
    x = rng.standard_normal(shape)
    if kind == "point":  # one site per slice
        keep = np.zeros(shape)
        for t in range(ntau):
            keep[t, t % nx, (3 * t + 1) % nx, nx - 1] = 1.0
        x = x * keep
    elif kind == "graded":  # slices, planes and sites of very different size
        x = x * 10.0 ** rng.uniform(-6, 6, size=(ntau, nx, 1, 1))
    return sigma, x


def _M_long(nx, sigma, x):
    L = np.longdouble
    n = np.arange(nx)
    k = 2 * np.arccos(L(-1)) * L(1) * np.where(n < nx // 2, n, n - nx) / L(nx)
    lam = np.exp(-L(TAU) * k * k / 2)
    T = np.array([[np.sum(lam * np.cos(k * (i - j))) / L(nx) for j in range(nx)]
                  for i in range(nx)], dtype=L)
    A = np.sqrt(L(2)) * np.sqrt(np.expm1(L(TAU) * L(G)))
    w = 1 + A * np.sin(sigma.astype(L))
    v = w * x.astype(L)
    for axis in (1, 2, 3):
        v = np.moveaxis(np.tensordot(T, v, axes=(1, axis)), 0, axis)
    up = -np.roll(v, 1, axis=0)
    up[0] = -up[0]
    return x.astype(L) + up


@pytest.mark.parametrize("kind", ["normal", "point", "graded"])
@pytest.mark.parametrize("nx,ntau", EXTENTS)
def test_precision_against_long_double(ufg, nx, ntau, kind):
    sigma, x = _inputs(nx, ntau, 31 * nx + ntau, kind)
    field = ufg.Field(ufg.Lattice(nx, ntau), torch.from_numpy(sigma).cuda())
    y = ufg.ufg_apply_M(field, torch.from_numpy(x).cuda()).cpu().numpy()
    ref = _M_long(nx, sigma, x)
    err = np.sqrt(((y - ref) ** 2).sum() / (ref ** 2).sum())
    assert err <= 3 * (2 * np.sqrt(nx) + 4) * 2.0 ** -53, float(err)


@pytest.mark.parametrize("nx,ntau", EXTENTS)
def test_power_of_two_scaling_is_exact(ufg, nx, ntau):
    sigma, x = _inputs(nx, ntau, nx + ntau, "normal")
    field = ufg.Field(ufg.Lattice(nx, ntau), torch.from_numpy(sigma).cuda())
    xd = torch.from_numpy(x).cuda()
    for fn in ("ufg_apply_M", "ufg_apply_Mdag", "ufg_apply_kinetic", "ufg_apply_M1T"):
        y = getattr(ufg, fn)(field, xd)
        for k in (-800, 300, 900):
            assert torch.equal(getattr(ufg, fn)(field, xd * 2.0 ** k), y * 2.0 ** k), (fn, k)


@pytest.mark.parametrize("nx,ntau", [(6, 9), (8, 7), (16, 5), (32, 4)])
def test_ends_of_the_exponent_range(ufg, nx, ntau):
    sigma, x = _inputs(nx, ntau, nx, "normal")
    field = ufg.Field(ufg.Lattice(nx, ntau), torch.from_numpy(sigma).cuda())
    xd = torch.from_numpy(x).cuda()
    clean = ufg.ufg_apply_M(field, xd)
    # the kinetic term of a slice around 2^-940 keeps 10 bits or more
    small = ufg.ufg_apply_kinetic(field, xd * 2.0 ** -940) * 2.0 ** 940
    ref = ufg.ufg_apply_kinetic(field, xd)
    assert float((small - ref).abs().max() / ref.abs().max()) < 2.0 ** -9
    # zeros in, zeros out
    assert float(ufg.ufg_apply_M(field, torch.zeros_like(xd)).abs().max()) == 0.0
    # a NaN or an infinity of slice 1 reaches slice 1 (its own site) and the whole of slice 2 only
    for bad in (float("nan"), float("inf"), -float("inf")):
        xb = xd.clone()
        xb[1, nx - 1, 0, nx // 2] = bad
        y = ufg.ufg_apply_M(field, xb)
        assert bool((~torch.isfinite(y[2])).all())
        y1 = y[1].clone()
        assert not bool(torch.isfinite(y1[nx - 1, 0, nx // 2]))
        y1[nx - 1, 0, nx // 2] = clean[1, nx - 1, 0, nx // 2]
        assert torch.equal(y1, clean[1])
        assert torch.equal(y[3:], clean[3:]) and torch.equal(y[0], clean[0])


@pytest.mark.parametrize("nx,ntau", [(8, 5), (16, 5)])
def test_momentum_operator_is_the_transformed_operator(ufg, nx, ntau):
    # F M F^T x against the separately applied F, M and F^T: each of the six passes within a few
    # roundings, 12 (2 sqrt(N) + 4) 2^-53 in all
    sigma, x = _inputs(nx, ntau, 5 + nx, "graded")
    field = ufg.Field(ufg.Lattice(nx, ntau), torch.from_numpy(sigma).cuda())
    xd = torch.from_numpy(x).cuda()
    for tr, fn in ((False, ufg.ufg_apply_M), (True, ufg.ufg_apply_Mdag)):
        a = ufg.ufg_apply_M_momentum(field, ufg.ufg_fourier(field, xd), transpose=tr)
        b = ufg.ufg_fourier(field, fn(field, xd))
        err = float((a - b).norm() / b.norm())
        assert err <= 12 * (2 * np.sqrt(nx) + 4) * 2.0 ** -53, (tr, err)
