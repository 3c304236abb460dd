"""An untuned launch gives the same bits whichever kernel its working set
selects: the default shapes of 16^3 x 32 (the tile kernel from 6 right-hand
sides, one or two tiles a barrier) against the per-thread kernel."""

import numpy as np
import pytest

import synth
from oracle.lattice import Lattice

pytestmark = pytest.mark.gpu

DIMS = (16, 16, 16, 32)
PREC_ID = {"f32": 1, "f16": 2, "bf16": 3}


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g

    g.build()
    from paper_2303_05883_gb300 import api

    return api


@pytest.fixture(scope="module")
def links():
    return synth.gauge_field(DIMS, 0.3, 2)


def pin_per_thread(api, L, prec, nrhs):
    key = "x".join(str(d) for d in DIMS)
    for fl in (0, 1, 3, 4, 5):  # D_eo and pass 1, D, clover D, pass 1, pass 2
        api.bridge_tune_set(L.handle, f"hop/{PREC_ID[prec]}/{fl}/0/{key}/{nrhs}", 128, 512, 0)


@pytest.mark.parametrize("kind,csw", [("wilson", 0.0), ("clover", 1.0)])
@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nrhs", [6, 9])
def test_default_kernels_round_alike(api, links, kind, csw, prec, nrhs):
    even = Lattice(DIMS).even
    psi = synth.gaussian_spinor(DIMS, 4, nrhs=nrhs)
    got = []
    for pinned in (False, True):
        L = api.Lattice(DIMS)
        op = api.make_op(kind, 0.12, csw, (1, -1, 1, -1))
        L.upload(links, op)
        if pinned:
            pin_per_thread(api, L, prec, nrhs)
        half = psi[:, even]
        got.append((L.D(op, psi, prec), L.Deo(op, half, 0, prec), L.Deo(op, half, 1, prec), L.Dhat(op, half, prec)))
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec,nrhs", [("f16", 6), ("f16", 9), ("f32", 6)])
def test_the_printed_table_selects_the_same_kernels(api, links, prec, nrhs):
    """Every line of bridge_tune_table, set on another lattice, runs the kernel it was printed for."""
    half = synth.gaussian_spinor(DIMS, 4, nrhs=nrhs)[:, Lattice(DIMS).even]
    op = api.make_op("clover", 0.12, 1.0)
    got, table = [], {}
    for _ in range(2):
        L = api.Lattice(DIMS)
        L.upload(links, op)
        for key, shape in table.items():
            api.bridge_tune_set(L.handle, key, *shape)
        got.append(L.Dhat(op, half, prec))
        table = api.bridge_tune_table(L.handle)
        assert any(shape[2] in (9, 10) for shape in table.values())
    assert np.array_equal(*got)
