"""Calls captured into a graph by the caller: what a replay reads must not move
with later calls on the lattice."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = (8, 8, 8, 8)


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g

    g.build()
    from paper_2303_05883_gb300 import api

    return api


@pytest.mark.parametrize("which", [0, 3])
def test_replay_after_the_scratch_has_grown(api, which):
    from paper_2303_05883_gb300 import _abi

    L = api.Lattice(DIMS)
    op = api.make_op("clover", 0.12, 1.0)
    L.upload(synth.gauge_field(DIMS, 0.3, 2), op)
    subset = _abi.BRIDGE_FULL if which == 0 else _abi.BRIDGE_EVEN
    n = 4096 if which == 0 else 2048
    f = [api.bridge_field_create(L.handle, "f64", subset, 1) for _ in range(2)]
    psi = synth.gaussian_spinor(DIMS, 4)[:n].copy()
    api.bridge_field_import(f[0], psi)
    api.bridge_apply(L.handle, op, which, f[1], f[0])  # everything built
    api.bridge_sync(L.handle)
    want = np.empty_like(psi)
    api.bridge_field_export(f[1], want)

    stream = torch.cuda.ExternalStream(_abi.load().bridge_lattice_stream(L.handle))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        g.capture_begin(capture_error_mode="thread_local")
        api.bridge_apply(L.handle, op, which, f[1], f[0])
        g.capture_end()
    many = synth.gaussian_spinor(DIMS, 5, nrhs=5)
    L.D(op, many), L.Dhat(op, many[:, :2048])  # grows the lattice's scratch
    got = np.zeros_like(psi)
    for _ in range(2):
        api.bridge_field_import(f[1], got)
        with torch.cuda.stream(stream):
            g.replay()
        api.bridge_sync(L.handle)
        api.bridge_field_export(f[1], got)
        assert np.array_equal(got, want)
        got[:] = 0
    for x in f:
        api.bridge_field_destroy(x)


def test_a_capture_survives_another_lattice_running_out_of_memory(api):
    """A call short of memory takes the copies of idle lattices; one whose stream is being captured is not idle."""
    import ctypes

    from paper_2303_05883_gb300 import _abi

    from .test_gpu_fixed_point_memory import DIMS as BIG
    from .test_gpu_fixed_point_memory import LINK_COPY, Scarce

    L = api.Lattice(DIMS)
    op = api.make_op("wilson", 0.12, 0.0)
    L.upload(synth.gauge_field(DIMS, 0.3, 2), op)
    f = [api.bridge_field_create(L.handle, "f64", _abi.BRIDGE_FULL, 1) for _ in range(2)]
    psi = synth.gaussian_spinor(DIMS, 4)
    api.bridge_field_import(f[0], psi)
    want = L.D(op, psi)  # the lattice has copies
    other, nrhs = api.Lattice(BIG), 24
    other.upload(synth.gauge_field(BIG, 0.3, 2), op)
    b = torch.randn((nrhs, int(np.prod(BIG)), 4, 3), dtype=torch.complex128, device="cuda")
    ref = torch.cat([other.D(op, b[k : k + 1]) for k in range(nrhs)])
    out = torch.empty_like(b)
    stream = torch.cuda.ExternalStream(_abi.load().bridge_lattice_stream(L.handle))
    g = torch.cuda.CUDAGraph()
    with Scarce(2 * b.numel() * 16 - LINK_COPY // 2):
        with torch.cuda.stream(stream):
            g.capture_begin(capture_error_mode="relaxed")
            api.bridge_apply(L.handle, op, 0, f[1], f[0])
            st = _abi.load().bridge_mult_D_dev(other.handle, ctypes.byref(op), 0, ctypes.c_void_p(b.data_ptr()),
                                               ctypes.c_void_p(out.data_ptr()), nrhs)
            g.capture_end()
        api.bridge_sync(other.handle)
    assert st == 0 and torch.equal(out, ref)
    with torch.cuda.stream(stream):
        g.replay()
    api.bridge_sync(L.handle)
    got = np.empty_like(psi)
    api.bridge_field_export(f[1], got)
    assert np.array_equal(got, want)
    for x in f:
        api.bridge_field_destroy(x)
