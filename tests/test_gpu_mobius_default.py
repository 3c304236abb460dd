"""The untuned Moebius launches at sizes where their shape changes (2^17
five-dimensional sites of one parity; Ls below and above 10 and 16), against
FP64.  Bar: relative L2 2e-6."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g

    g.build()
    from paper_2303_05883_gb300 import api

    return api


@pytest.mark.parametrize("Ls,dims", [(4, (16, 16, 16, 16)), (5, (16, 16, 16, 14)), (10, (12, 12, 12, 16)), (16, (8, 8, 16, 16)),
                                     (17, (8, 8, 16, 16))])
def test_default_shapes_agree_with_fp64(api, Ls, dims):
    V = int(np.prod(dims))
    assert V // 2 * Ls >= 1 << 17
    L = api.Lattice(dims)
    op = api.make_mobius(Ls, 1.8, 1.5, 0.5, 0.05)
    L.upload(synth.gauge_field(dims, 0.2, 2), op)
    psi = synth.gaussian_spinor(dims, 4, nrhs=Ls)
    half = psi[:, : V // 2].copy()
    for f, v in ((L.D, psi), (L.Deo, half), (L.Dhat, half), (L.Dhat_dag, half)):
        a, b = f(op, v, prec="f32"), f(op, v, prec="f64")
        assert np.linalg.norm(a - b) < 2e-6 * np.linalg.norm(b)
    x, info = L.solve(op, psi, api.make_solver(tol=1e-10))
    assert info[0]["status"] == 0
    assert np.linalg.norm(L.D(op, x) - psi) < 2e-10 * np.linalg.norm(psi)
