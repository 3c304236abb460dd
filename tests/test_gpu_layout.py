"""Canonical <-> GPU layout conversions at the edges of their tiles: every
value comes back from where it belongs (FP64 fields hold it exactly)."""

import numpy as np
import pytest

import synth
from oracle import staggered
from oracle.lattice import Lattice

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g

    g.build()
    from paper_2303_05883_gb300 import api

    return api


# volumes 16, 128 (one tile), 144 (one and a bit), 1440, odd half-extents along x
DIMS = [(2, 2, 2, 2), (4, 4, 4, 2), (6, 2, 2, 6), (6, 4, 10, 6)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec,tol", [("f64", 0.0), ("f32", 6e-8), ("f16", 2.0 ** -10), ("bf16", 2.0 ** -7)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_round_trip(api, dims, prec, tol, nrhs):
    """Import then export: the values rounded once to the storage type (16-bit
    storage: relative to the largest component of the site)."""
    V = int(np.prod(dims))
    L = api.Lattice(dims)
    for subset, n in ((2, V), (0, V // 2), (1, V // 2)):
        a = synth.gaussian_spinor(dims, 3, nrhs=nrhs)[:, :n].copy()
        out = np.empty_like(a)
        f = api.bridge_field_create(L.handle, prec, subset, nrhs)
        api.bridge_field_import(f, a)
        api.bridge_field_export(f, out)
        api.bridge_field_destroy(f)
        scale = np.abs(a.view(np.float64)).reshape(nrhs, n, -1).max(axis=2)[:, :, None, None]
        assert np.all(np.abs(out - a) <= np.sqrt(2) * tol * scale)


@pytest.mark.parametrize("dims", DIMS + [(8, 8, 4, 4)])
@pytest.mark.parametrize("prec,tol", [("f64", 1e-13), ("f32", 2e-6)])
def test_staggered_layout(api, dims, prec, tol):
    lat = Lattice(dims)
    U = synth.gauge_field(dims, 0.3, 2)
    L = api.Lattice(dims)
    op = api.make_staggered(0.1)
    L.upload(U, op)
    chi = synth.gaussian_spinor(dims, 3, nrhs=2)[:, :, 0].copy()
    st = staggered.Staggered(U, lat, 0.1)
    got, half = L.D(op, chi, prec), L.Deo(op, chi[:, lat.odd], 0, prec)
    for r in range(2):
        want = st.full(chi[r])
        assert np.abs(got[r] - want).max() <= 4 * tol * np.abs(want).max()
        want = st.D_hop(0, chi[r, lat.odd])
        assert np.abs(half[r] - want).max() <= 4 * tol * np.abs(want).max()
