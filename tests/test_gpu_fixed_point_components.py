"""Every component of an FP64 result has the accuracy of its own size, where
components do not mix: unit links, links with a decoupled colour, nearly unit
links, real fields.  Component by component against the oracle, relative L2
over the sites.

Bar 4e-15: a component stays in fixed point where a hop reaches 2^-5 of the
largest neighbour component, whose typical error is then 2^-54 / 2^-5 = 1.8e-15
of the component; the oracle's sixteen FP64 roundings are 4.5e-16.
"""

import numpy as np
import pytest

import synth
from oracle import dirac, evenodd, staggered
from oracle.lattice import Lattice

pytestmark = pytest.mark.gpu

TOL = 4e-15
DIMS = (6, 4, 10, 6)
V = int(np.prod(DIMS))


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g

    g.build()
    from paper_2303_05883_gb300 import api

    return api


def links(kind):
    U = np.zeros((4, V, 3, 3), dtype=np.complex128)
    if kind == "unit":
        U[:] = np.eye(3)
    elif kind == "decoupled":  # SU(2) in the first two colours
        q = np.random.default_rng(4).standard_normal((4, V, 4))
        q /= np.linalg.norm(q, axis=2, keepdims=True)
        a, b = q[..., 0] + 1j * q[..., 1], q[..., 2] + 1j * q[..., 3]
        U[..., 0, 0], U[..., 0, 1], U[..., 1, 0], U[..., 1, 1] = a, b, -b.conj(), a.conj()
        U[..., 2, 2] = 1
    else:
        U = synth.gauge_field(DIMS, 1e-9, 3)
    return U


def spread(kind):
    psi = synth.gaussian_spinor(DIMS, 5)
    if kind == "unit":
        w = np.outer([1e-20, 1.0, 1e-16, 1e-7], [1.0, 1e-9, 1e-25])
    elif kind == "decoupled":
        w = np.outer([1.0, 1.0, 1.0, 1.0], [1.0, 1.0, 1e-18])
    else:
        w = np.outer([1.0, 1.0, 1.0, 1.0], [1.0, 0.0, 0.0])
    return psi * w


def same(got, want):
    """Real and imaginary part of every component, each relative to its own norm over the sites."""
    for a, b in ((got.real, want.real), (got.imag, want.imag)):
        n = np.sqrt((b**2).sum(axis=0))
        e = np.sqrt(((a - b) ** 2).sum(axis=0))
        assert np.all(e <= TOL * n), (e / np.maximum(n, 1e-300)).max()


# (near unit links have a clover term of rounding errors)
@pytest.mark.parametrize("kind,op,csw", [("unit", "wilson", 0.0), ("unit", "clover", 1.1), ("decoupled", "wilson", 0.0),
                                         ("decoupled", "clover", 1.1), ("near unit", "wilson", 0.0)])
def test_components_of_a_spinor(api, kind, op, csw):
    lat, U, psi, kappa = Lattice(DIMS), links(kind), spread(kind), 0.12
    L = api.Lattice(DIMS)
    o = api.make_op(op, kappa, csw)
    L.upload(U, o)
    same(L.D(o, psi), dirac.dirac(U, psi, lat, kappa, csw))
    eo = evenodd.EvenOdd(U, lat, kappa, csw)
    same(L.Deo(o, psi[lat.odd], 0), eo.D_hop(0, psi[lat.odd]))
    same(L.Deo(o, psi[lat.even], 1), eo.D_hop(1, psi[lat.even]))
    same(L.Dhat(o, psi[lat.even]), eo.schur(psi[lat.even]))


@pytest.mark.parametrize("kind", ["unit", "decoupled", "near unit"])
@pytest.mark.parametrize("real", [False, True])
def test_components_of_a_colour_vector(api, kind, real):
    lat, U, m = Lattice(DIMS), links(kind), 0.1
    chi = spread(kind)[:, 1].copy()
    if real and kind == "unit":
        chi.imag *= 1e-20
    L = api.Lattice(DIMS)
    o = api.make_staggered(m)
    L.upload(U, o)
    st = staggered.Staggered(U, lat, m)
    same(L.D(o, chi), st.full(chi))
    same(L.Deo(o, chi[lat.odd], 0), st.D_hop(0, chi[lat.odd]))
    same(L.Dhat(o, chi[lat.even]), st.schur(chi[lat.even]))


@pytest.mark.parametrize("value", [1e-305, 1e-290])
def test_small_sites_by_themselves(api, value):
    """Sites all of whose neighbours are near the lower end of the FP64 range, next to ordinary ones."""
    lat = Lattice(DIMS)
    U = synth.gauge_field(DIMS, 0.4, 3)
    psi = synth.gaussian_spinor(DIMS, 5)
    t = np.arange(V) // (V // DIMS[3])
    psi[(t >= 1) & (t <= 4)] *= value
    L = api.Lattice(DIMS)
    o = api.make_op("wilson", 0.12, 0.0)
    L.upload(U, o)
    inner = (t >= 2) & (t <= 3)
    got, want = L.D(o, psi)[inner], dirac.dirac(U, psi, lat, 0.12, 0.0)[inner]
    assert len(got) > 0 and np.abs(want).max() < 1e3 * value
    big = 2.0**900  # exact: the norms below stay in range
    assert np.linalg.norm((got - want) * big) <= TOL * np.linalg.norm(want * big)
    worst = np.abs(got - want).max(axis=(1, 2)) * big
    assert np.all(worst <= 8e-15 * np.abs(want * big).max(axis=(1, 2)))
