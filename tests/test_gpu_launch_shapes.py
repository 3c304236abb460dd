"""The launch table names kernels that exist: a recorded variant is one its
(flags, reduction) pair is instantiated for."""

import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g

    g.build()
    from paper_2303_05883_gb300 import api

    return api


def lattice(api, dims, kind="clover", csw=1.0):
    L = api.Lattice(dims)
    op = api.make_op(kind, 0.12, csw)
    L.upload(synth.gauge_field(dims, 0.2, 2), op)
    return L, op, "x".join(str(d) for d in dims)


@pytest.mark.parametrize("kind,first", [("wilson", 1), ("clover", 5)])
def test_untuned_normal_equations_record_their_kernel(api, kind, first):
    """D^ with |q|^2 and the gamma5 pass have no register-budget variants: 2^17 half-lattice sites record 0."""
    dims = (16, 16, 32, 32)
    L, op, key = lattice(api, dims, kind)
    L.solve(op, synth.gaussian_spinor(dims, 4), api.make_solver(tol=1e-3, method=2))
    table = api.bridge_tune_table(L.handle)
    assert table[f"hop/1/{first}/1/{key}/1"][2] == 0
    assert table[f"hop/1/17/0/{key}/1"][2] == 0


@pytest.mark.parametrize("nrhs", [1, 2])
def test_tuning_the_preparation_tries_its_own_kernels(api, nrhs):
    L, op, key = lattice(api, (8, 8, 8, 16))
    api.bridge_tune(L.handle, op, "f16", nrhs)
    assert api.bridge_tune_table(L.handle)[f"hop/2/12/0/{key}/{nrhs}"][2] in ((0,) if nrhs == 1 else (0, 9, 10))
