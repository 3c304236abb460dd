"""The launch table names kernels that exist: a recorded variant is one its
(flags, reduction) pair is instantiated for."""

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


def tuned(api, capfd, monkeypatch, scale):
    """The variants that tuning FP64 tries for D_eo on links scaled by `scale`."""
    dims = (4, 4, 4, 8)
    L = api.Lattice(dims)
    op = api.make_op("wilson", 0.12 / scale, 0.0)
    L.upload(scale * synth.gauge_field(dims, 0.2, 2), op)
    monkeypatch.setenv("BRIDGE_TUNE_VERBOSE", "1")
    capfd.readouterr()
    api.bridge_tune(L.handle, op, "f64", 1)
    lines = [x.split() for x in capfd.readouterr().err.splitlines() if x.startswith("tune hop/0/0/0/")]
    return {int(x[x.index("variant") + 1].rstrip(":")) for x in lines}


def test_tuning_fp64_arithmetic_tries_its_variants(api, capfd, monkeypatch):
    """Links above 1 run on the FP64 pipe, which has the register-budget variants; in fixed point there is one kernel."""
    assert tuned(api, capfd, monkeypatch, 2.0) == {0, 1, 2, 3, 4, 5}
    assert tuned(api, capfd, monkeypatch, 1.0) == {0}


@pytest.mark.parametrize("variant", [3, 5, 9])
@pytest.mark.parametrize("scale", [1.0, 2.0])
def test_fp64_entries_of_any_variant_run(api, variant, scale):
    """Table lines of FP64 keys, whether their hops run in fixed point or not."""
    dims = (4, 4, 4, 8)
    psi = synth.gaussian_spinor(dims, 4)
    got = []
    for pin in (False, True):
        L = api.Lattice(dims)
        op = api.make_op("wilson", 0.12 / scale, 0.0)
        L.upload(scale * synth.gauge_field(dims, 0.2, 2), op)
        for key in ("0/0", "1/0", "1/2", "1/3", "8/0", "9/1"):
            if pin:
                api.bridge_tune_set(L.handle, f"hop/0/{key}/4x4x4x8/1", 64, 2, variant)
        x, info = L.solve(op, psi, api.make_solver(tol=1e-10, mixed=0))
        assert info[0]["status"] == 0
        got.append((L.D(op, psi), L.Dhat(op, psi[:256])))
    assert all(np.array_equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("kind", ["wilson", "clover"])
@pytest.mark.parametrize("prec,nrhs", [("f64", 1), ("f32", 1), ("f16", 6)])
def test_the_call_without_allocations_gives_the_same_bits(api, kind, prec, nrhs):
    """bridge_mult_Dhat_noalloc against bridge_mult_Dhat, whichever came first."""
    import torch

    dims = (8, 8, 8, 16)
    L, op, _ = lattice(api, dims, kind)
    psi = torch.from_numpy(synth.gaussian_spinor(dims, 4, nrhs=nrhs)[:, :4096].copy()).cuda()
    L.Dhat(op, psi[:1], prec)  # builds the operands
    got = [torch.empty_like(psi) for _ in range(2)]
    for out in got:
        dhat_noalloc(api, L, op, prec, psi, out, nrhs)
        want = L.Dhat(op, psi, prec)
    assert torch.equal(got[0], want) and torch.equal(got[1], want)


def dhat_noalloc(api, L, op, prec, psi, out, nrhs):
    from ctypes import byref, c_void_p

    from paper_2303_05883_gb300 import _abi

    fn = _abi.load().bridge_mult_Dhat_noalloc
    _abi.check(fn(L.handle, byref(op), {"f64": 0, "f32": 1, "f16": 2}[prec], c_void_p(psi.data_ptr()),
                  c_void_p(out.data_ptr()), nrhs), "bridge_mult_Dhat_noalloc")
    api.bridge_sync(L.handle)
