"""The shared-link tile kernel in the operator applications, the even-odd
preparation and CG on the normal equations, and the launches it is the
default of.  Relative L2 bars of the build: FP32 2e-6, FP16/BF16 5e-3."""

import numpy as np
import pytest

import synth
from oracle import dirac, evenodd
from oracle.lattice import Lattice

pytestmark = pytest.mark.gpu

TOL = {"f32": 2e-6, "f16": 5e-3, "bf16": 5e-3}
PREC_ID = {"f32": 1, "f16": 2, "bf16": 3}


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g

    g.build()
    from paper_2303_05883_gb300 import api

    return api


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def pin(api, L, prec, dims, nrhs, variant):
    key = "x".join(str(d) for d in dims)
    for fl, rd in ((0, 0), (1, 0), (3, 0), (4, 0), (5, 0), (8, 0), (12, 0), (1, 1), (5, 1), (17, 0)):
        api.bridge_tune_set(L.handle, f"hop/{PREC_ID[prec]}/{fl}/{rd}/{key}/{nrhs}", 64, 3, variant)


# 8 sites (less than a tile), 720 (22 tiles and a half); one, uneven and two groups of right-hand sides
@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 2), ((6, 4, 10, 6), 5), ((6, 4, 10, 6), 13)])
@pytest.mark.parametrize("kind,csw", [("wilson", 0.0), ("clover", 1.0)])
@pytest.mark.parametrize("prec,variant", [("f32", 9), ("f32", 10), ("f16", 9), ("f16", 10), ("bf16", 10)])
def test_operators_on_the_tile_kernel(api, dims, nrhs, kind, csw, prec, variant):
    kappa = 0.12
    lat = Lattice(dims)
    U = synth.gauge_field(dims, 0.3, 2)
    psi = synth.gaussian_spinor(dims, 4, nrhs=nrhs)
    L = api.Lattice(dims)
    op = api.make_op(kind, kappa, csw)
    L.upload(U, op)
    pin(api, L, prec, dims, nrhs, variant)
    eo = evenodd.EvenOdd(U, lat, kappa, csw)
    T = dirac.clover_term(U, lat, kappa, csw)
    D, H = L.D(op, psi, prec), L.Dhat(op, psi[:, lat.even], prec)
    for r in range(nrhs):
        assert rel(D[r], dirac.dirac(U, psi[r], lat, kappa, csw, T=T)) < TOL[prec]
        assert rel(H[r], eo.schur(psi[r, lat.even])) < TOL[prec]


@pytest.mark.parametrize("kind,csw", [("wilson", 0.0), ("clover", 1.0)])
def test_cgnr_solve_on_the_tile_kernel(api, kind, csw):
    dims, nrhs, kappa = (6, 4, 10, 6), 5, 0.12
    lat = Lattice(dims)
    U = synth.gauge_field(dims, 0.3, 2)
    b = synth.gaussian_spinor(dims, 4, nrhs=nrhs)
    L = api.Lattice(dims)
    op = api.make_op(kind, kappa, csw)
    L.upload(U, op)
    pin(api, L, "f32", dims, nrhs, 9)
    x, info = L.solve(op, b, api.make_solver(tol=1e-10, method=2))
    for r in range(nrhs):
        assert info[r]["cgnr_passes"] > 0
        assert rel(dirac.dirac(U, x[r], lat, kappa, csw), b[r]) < 2e-10


@pytest.mark.parametrize("nrhs,prec", [(1, "f32"), (3, "f16"), (6, "f32"), (12, "f16")])
def test_default_shapes_agree_with_fp64(api, nrhs, prec):
    """The sizes at which the untuned launches change kernel."""
    dims = (16, 16, 16, 32) if nrhs >= 6 else (16, 16, 32, 32)
    U = synth.gauge_field(dims, 0.2, 2)
    half = int(np.prod(dims)) // 2
    psi = synth.gaussian_spinor(dims, 4, nrhs=nrhs)[:, :half].copy()
    L = api.Lattice(dims)
    op = api.make_op("clover", 0.12, 1.0)
    L.upload(U, op)
    got, want = L.Dhat(op, psi, prec), L.Dhat(op, psi, "f64")
    table = api.bridge_tune_table(L.handle)
    key = "x".join(str(d) for d in dims)
    variant = table[f"hop/{PREC_ID[prec]}/5/0/{key}/{nrhs}"][2]
    assert variant == {1: 4, 3: 4, 6: 9, 12: 10}[nrhs]
    for r in range(nrhs):
        assert rel(got[r], want[r]) < TOL[prec]
