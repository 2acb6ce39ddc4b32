"""Result arrays of the solver in host memory that is used again: what happens when memory is
not to be had."""
import mmap

import numpy as np
import pytest

solver = pytest.importorskip("paper_1001_3631_gb300.solver")

BIG = (4, 300, 700)   # 6.7 MB


@pytest.mark.parametrize("shape", [(1 << 40, 64, 64), (1 << 62, 4)])
def test_more_than_the_machine_has_is_a_memory_error_as_from_numpy(shape):
    with pytest.raises((MemoryError, ValueError)) as want:   # (ValueError: more than can be addressed)
        np.empty(shape)
    with pytest.raises(want.type):
        solver._HostBuffers().empty(shape)


def test_an_array_comes_from_numpy_where_no_mapping_is_to_be_had(monkeypatch):
    def refuse(*a, **k):
        raise OSError(12, "Cannot allocate memory")
    monkeypatch.setattr(solver.mmap, "mmap", refuse)
    a = solver._HostBuffers().empty(BIG)
    assert a.shape == BIG and a.dtype == np.float64 and a.flags["OWNDATA"]
    assert mmap.mmap is refuse
