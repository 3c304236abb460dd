"""The FP64 stencil in 64-bit fixed point against the oracle and against the
FP64 kernel.

Links 2 U at kappa / 2 give the same Wilson operator, bit for bit in its
products, but have no fixed-point copy (entries above 1), so their lattice
runs the FP64 kernel: the general path every form is compared with.

Tolerance 1e-15 (relative L2): a result of either side carries about sixteen
roundings of 1.1e-16 in a random walk (4.5e-16) and the two are independent.
"""

import numpy as np
import pytest

import synth
from oracle import dirac, evenodd
from oracle.lattice import Lattice

pytestmark = pytest.mark.gpu

TOL = 1e-15


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g

    g.build()
    from paper_2303_05883_gb300 import api

    return api


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def both(api, dims, bc, seed=3, eps=0.4, kappa=0.12):
    U = synth.gauge_field(dims, eps, seed)
    out = []
    for s in (1.0, 2.0):
        L = api.Lattice(dims)
        op = api.make_op("wilson", kappa / s, 0.0, bc)
        L.upload(s * U, op)
        out.append((L, op))
    return out


# half-lattice sites: 8, 64 (one block), 136, 720 (ragged warps and blocks), 4096
@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((4, 4, 4, 2), 2), ((2, 2, 2, 34), 3),
                                       ((6, 4, 10, 6), 2), ((8, 8, 8, 16), 1)])
@pytest.mark.parametrize("bc", [(1, 1, 1, -1), (-1, 1, -1, 1)])
def test_fixed_point_equals_the_fp64_kernel(api, dims, nrhs, bc):
    (L, op), (Lg, opg) = both(api, dims, bc)
    V = int(np.prod(dims))
    psi = synth.gaussian_spinor(dims, 5, nrhs=nrhs)
    # neighbouring sites of very different size, one site zero, one component only
    psi *= 10.0 ** np.random.default_rng(1).uniform(-12, 12, (nrhs, V, 1, 1))
    psi[:, V // 3] = 0
    psi[:, V // 2, 1:] = 0
    half = psi[:, : V // 2].copy()
    assert rel(L.D(op, psi), Lg.D(opg, psi)) < TOL
    for q in (0, 1):
        a, b = L.Deo(op, half, q), Lg.Deo(opg, half, q)
        assert rel(a, b) < TOL
        # site by site, against the largest neighbour that reaches the site
        scale = np.abs(b).max(axis=(2, 3))
        assert np.all(np.abs(a - b).max(axis=(2, 3)) <= 8e-15 * scale + 1e-300)
    assert rel(L.Dhat(op, half), Lg.Dhat(opg, half)) < TOL


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 10, 6)])
def test_fixed_point_clover_against_the_oracle(api, dims):
    lat = Lattice(dims)
    kappa, csw = 0.125, 1.2
    U = synth.gauge_field(dims, 0.4, 3)
    psi = synth.gaussian_spinor(dims, 5)
    L = api.Lattice(dims)
    op = api.make_op("clover", kappa, csw)
    L.upload(U, op)
    assert rel(L.D(op, psi), dirac.dirac(U, psi, lat, kappa, csw)) < TOL
    # the oracle inverts its 12x12 blocks: their condition number (about 3) on top
    assert rel(L.Dhat(op, psi[lat.even]), evenodd.EvenOdd(U, lat, kappa, csw).schur(psi[lat.even])) < 4 * TOL


def test_clover_blocks_out_of_range_stay_on_the_fp64_kernel(api):
    dims, kappa, csw = (4, 4, 4, 4), 0.4, 9.0
    lat = Lattice(dims)
    U = synth.gauge_field(dims, 2.0, 3)
    T = dirac.clover_term(U, lat, kappa, csw)
    assert max(np.abs(T.real).max(), np.abs(T.imag).max()) > 4
    psi = synth.gaussian_spinor(dims, 5)
    L = api.Lattice(dims)
    op = api.make_op("clover", kappa, csw)
    L.upload(U, op)
    assert rel(L.D(op, psi), dirac.dirac(U, psi, lat, kappa, csw)) < TOL


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 1e-305, 1e305])
def test_values_without_a_fixed_point_form(api, value):
    """Infinities and NaN reach the sites and components they reach in FP64;
    values at the ends of the FP64 range keep their accuracy."""
    dims = (6, 4, 10, 6)
    (L, op), (Lg, opg) = both(api, dims, (1, 1, 1, -1))
    psi = synth.gaussian_spinor(dims, 5)
    if np.isfinite(value):
        psi[100:300] *= value / 4
    else:
        psi[7, 2, 1] = value
        psi[500, 0, 0] = value * 1j
    with np.errstate(all="ignore"):
        a, b = L.D(op, psi), Lg.D(opg, psi)
        assert np.array_equal(np.isnan(a.real), np.isnan(b.real)) and np.array_equal(np.isnan(a.imag), np.isnan(b.imag))
        for x, y in ((a.real, b.real), (a.imag, b.imag)):
            assert np.array_equal(x[np.isinf(y)], y[np.isinf(y)])
            ok = np.isfinite(y)
            assert np.array_equal(ok, np.isfinite(x))
            big = np.abs(y[ok]).max()
            assert np.linalg.norm((x[ok] - y[ok]) / big) <= TOL * np.linalg.norm(y[ok] / big)
    if np.isfinite(value) and value < 1:
        # the small sites by themselves: inside the block every neighbour is small
        inner = [i for i in range(130, 270) if np.abs(b[i]).max() < 1e-300]
        for i in inner:
            assert np.abs(a[i] - b[i]).max() <= 8e-15 * np.abs(b[i]).max() + 1e-320


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((4, 4, 4, 4), 2), ((6, 4, 10, 6), 3)])
@pytest.mark.parametrize("bc", [(1, 1, 1, -1), (-1, 1, -1, 1)])
def test_staggered_fixed_point_equals_the_fp64_kernel(api, dims, nrhs, bc):
    """Links 2 U with mass 2 m give 2 D on the FP64 kernel (links above 1)."""
    U = synth.gauge_field(dims, 0.4, 3)
    V = int(np.prod(dims))
    chi = synth.gaussian_spinor(dims, 5, nrhs=nrhs)[:, :, 0].copy()
    chi *= 10.0 ** np.random.default_rng(1).uniform(-12, 12, (nrhs, V, 1))
    chi[:, V // 3] = 0
    chi[0, V // 2, 1] = 1e-303  # a site without a fixed-point form, finite
    chi[0, V // 2, [0, 2]] = 0
    got = []
    for s in (1.0, 2.0):
        L = api.Lattice(dims)
        op = api.make_staggered(0.1 * s, bc)
        L.upload(s * U, op)
        half = chi[:, : V // 2].copy()
        got.append([L.D(op, chi) / s, L.Deo(op, half, 0) / s, L.Deo(op, half, 1) / s, L.Dhat(op, half)])
    for a, b in zip(*got):
        assert rel(a, b) < TOL
        scale = np.abs(b).max(axis=2)
        assert np.all(np.abs(a - b).max(axis=2) <= 8e-15 * scale + 1e-318)


def test_staggered_nan_and_infinity(api):
    dims = (6, 4, 10, 6)
    U = synth.gauge_field(dims, 0.4, 3)
    chi = synth.gaussian_spinor(dims, 5)[:, 0].copy()
    chi[7, 1] = np.nan
    chi[500, 2] = np.inf
    got = []
    with np.errstate(all="ignore"):
        for s in (1.0, 2.0):
            L = api.Lattice(dims)
            op = api.make_staggered(0.1 * s)
            L.upload(s * U, op)
            got.append(L.D(op, chi) / s)
    a, b = (g.view(np.float64) for g in got)
    assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
    ok = np.isfinite(b)
    assert rel(a[ok], b[ok]) < TOL
