"""FP64 arithmetic is a matter of the operator's entries: the same bits
whatever memory is free, for the copies of the fixed-point stencil or not."""

import ctypes

import numpy as np
import pytest

import synth
from oracle.lattice import Lattice

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = (12, 12, 12, 24)
LINK_COPY = 8 * 144 * int(np.prod(DIMS)) // 2  # bytes; made where eight times as much is free


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g

    g.build()
    from paper_2303_05883_gb300 import api

    return api


class Scarce:
    """Leaves `left` bytes of device memory, the library's pool empty."""

    def __init__(self, left):
        self.left = left

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        cuda = ctypes.CDLL("libcuda.so.1")
        pool = ctypes.c_void_p()
        assert cuda.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
        assert cuda.cuMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0
        self.held = []
        while (more := torch.cuda.mem_get_info()[0] - self.left) > 1 << 21:
            self.held.append(torch.empty(more // 2 if more > 1 << 30 else more, dtype=torch.uint8, device="cuda"))
        return self

    def __exit__(self, *_):
        self.held = None
        torch.cuda.empty_cache()


def results(api, kind):
    lat, U = Lattice(DIMS), synth.gauge_field(DIMS, 0.3, 2)
    if kind == "staggered":
        op, f = api.make_staggered(0.2), synth.gaussian_spinor(DIMS, 4)[:, 0].copy()
    else:
        op, f = api.make_op(kind, 0.11, 1.0 if kind == "clover" else 0.0), synth.gaussian_spinor(DIMS, 4)
    calls = [lambda L: L.D(op, f), lambda L: L.Deo(op, f[lat.odd], 0), lambda L: L.Deo(op, f[lat.even], 1),
             lambda L: L.Dhat(op, f[lat.even]),
             lambda L: L.solve(op, f, api.make_solver(tol=1e-12, inner_prec="f32" if kind == "staggered" else "f16"))[0]]
    if kind != "clover":  # (its vectors beside the clover blocks are more than is left)
        calls.append(lambda L: L.solve(op, f, api.make_solver(tol=1e-10, mixed=0))[0])
    out = []
    for call in calls:  # a lattice each: little memory at a time
        L = api.Lattice(DIMS)
        L.upload(U, op)
        out.append(call(L))
        L.close()
    return out


@pytest.mark.parametrize("kind", ["wilson", "clover", "staggered"])
def test_the_same_bits_without_memory_for_copies(api, kind):
    want = results(api, kind)
    with Scarce(int(7.9 * LINK_COPY)):
        got = results(api, kind)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("spare", [8 << 20, -LINK_COPY // 2])
@pytest.mark.parametrize("kind", ["wilson", "staggered"])
def test_a_call_that_fits_without_copies_and_scratch_runs(api, kind, spare):
    """Room for the input and output fields of a call and little else, not for scratch; then not even for them,
    until the lattice gives back its link copy and the scratch of a smaller call."""
    from paper_2303_05883_gb300 import _abi

    U, nrhs = synth.gauge_field(DIMS, 0.3, 2), 24
    site = (6 if kind == "staggered" else 24) * 8
    op = api.make_staggered(0.2) if kind == "staggered" else api.make_op(kind, 0.11, 0.0)
    f = torch.randn((nrhs, U.shape[1]) + ((3,) if kind == "staggered" else (4, 3)), dtype=torch.complex128, device="cuda")
    L = api.Lattice(DIMS)
    L.upload(U, op)
    want = torch.cat([L.D(op, f[k : k + 1]) for k in range(nrhs)])
    got = torch.empty_like(f)
    with Scarce(2 * nrhs * U.shape[1] * site + spare):
        _abi.check(_abi.load().bridge_mult_D_dev(L.handle, ctypes.byref(op), 0, ctypes.c_void_p(f.data_ptr()),
                                                 ctypes.c_void_p(got.data_ptr()), nrhs), "bridge_mult_D_dev")
        api.bridge_sync(L.handle)
    assert torch.equal(got, want)
    L.close()
