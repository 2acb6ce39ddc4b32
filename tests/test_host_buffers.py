"""Result arrays of the solver on reused host memory: a mapping is handed out again only when
no array, view or tensor on it is left."""
import gc

import numpy as np
import pytest

solver = pytest.importorskip("paper_1001_3631_gb300.solver")

BIG = (4, 300, 700)   # 6.7 MB


def address(a):
    return a.__array_interface__["data"][0]


def test_memory_is_used_again_only_when_every_view_is_gone():
    h = solver._HostBuffers()
    a = h.empty(BIG)
    at = address(a)
    a[:] = 1.0
    view = a[1:, ::2]
    del a
    gc.collect()
    b = h.empty(BIG)
    assert address(b) != at and (view == 1.0).all()
    del view
    gc.collect()
    c = h.empty(BIG)
    assert address(c) == at
    torch = pytest.importorskip("torch")
    t = torch.from_numpy(c)[2:]
    del c
    gc.collect()
    assert address(h.empty(BIG)) not in (at, address(b))
    del t
    gc.collect()
    assert address(h.empty(BIG)) != address(b)


def test_shapes_types_and_sizes():
    h = solver._HostBuffers()
    for shape, dtype in ((BIG, np.float64), ((600, 700), np.complex128), ((3, 4), np.float64), ((0, 5, 2), np.float64)):
        a = h.empty(shape, dtype)
        assert a.shape == shape and a.dtype == dtype and a.flags["C_CONTIGUOUS"] and a.flags["WRITEABLE"]
        assert not np.shares_memory(a, h.empty(shape, dtype))
    with pytest.raises(ValueError):
        h.empty((-1, 4))


def test_idle_memory_is_bounded():
    h = solver._HostBuffers()
    h.KEEP = 20 << 20
    for k in range(8):
        h.empty((4, 300, 700 + 40 * k))
    gc.collect()
    assert sum(len(b[0]) for b in h._bufs) <= h.KEEP + (8 << 20)


def test_arrays_outlive_their_buffers_owner():
    h = solver._HostBuffers()
    a = h.empty(BIG)
    a[:] = 3.0
    del h
    gc.collect()
    assert (a == 3.0).all()
