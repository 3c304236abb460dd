"""Solves of sources near the end of the FP64 range."""

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


@pytest.mark.parametrize("norm2", [1e-155, 2e-155, 4e-155])
def test_denominators_whose_reciprocal_overflows(api, norm2):
    """BiCGStab in plain FP64 divides by |<rhat, v>|^2, about |b|^4: below 5.6e-309, finite, its
    reciprocal not.  One iteration (residual 0.05 at this kappa) takes the quotient."""
    dims = (4, 4, 4, 8)
    L = api.Lattice(dims)
    op = api.make_op("wilson", 0.05, 0.0)
    L.upload(synth.gauge_field(dims, 0.3, 2), op)
    b = synth.gaussian_spinor(dims, 4)
    b *= np.sqrt(2 * norm2) / np.linalg.norm(b)  # |b|^2 = norm2 on each parity
    x, info = L.solve(op, b, api.make_solver(tol=0.05, mixed=0, inner_tol=0.02))
    assert info[0]["status"] == 0 and np.all(np.isfinite(x))
    big = 2.0 ** 300  # exact, and within the range of a norm
    assert np.linalg.norm((b - L.D(op, x)) * big) <= 0.05 * np.linalg.norm(b * big)
