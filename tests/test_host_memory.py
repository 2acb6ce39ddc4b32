"""Result arrays of the solver in host memory that is used again: what happens when memory is
not to be had, and how much of it stays."""
import gc
import mmap
import threading

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


def idle(h):
    return sum(len(b[0]) for b in h._bufs if b[1]() is None)


def test_what_is_kept_is_counted_when_arrays_are_dropped():
    h = solver._HostBuffers()
    h.KEEP = 20 << 20
    held = [h.empty(BIG) for _ in range(10)]
    assert len(h._bufs) == 10 and idle(h) == 0
    held.clear()
    assert 0 < idle(h) <= h.KEEP
    one = h.empty((8,) + BIG)   # larger than what may be kept
    del one
    assert idle(h) <= h.KEEP
    assert all(len(b[0]) < h.KEEP for b in h._bufs)


def test_nothing_stays_after_the_last_solver():
    h = solver._HostBuffers()
    h.open()
    h.open()
    a, b = h.empty(BIG), h.empty(BIG)
    a[:] = 2.0
    del b
    h.close()
    assert idle(h) > 0
    h.close()
    assert idle(h) == 0 and (a == 2.0).all()
    del a
    assert not h._bufs
    h.open()
    c = h.empty(BIG)
    del c
    assert idle(h) > 0


def test_growing_records_find_memory_again():
    h = solver._HostBuffers()
    made = set()
    for k in range(4000, 4100):
        a = h.empty((k, 128, 2))
        made.add(a.__array_interface__["data"][0])
        del a
    assert len(made) <= 3 and len(h._bufs) <= 3


def test_many_threads_drop_and_ask():
    h = solver._HostBuffers()
    h.KEEP = 30 << 20
    bad = []

    def work(seed):
        rng = np.random.default_rng(seed)
        kept = []
        for _ in range(60):
            a = h.empty((int(rng.integers(1, 4)),) + BIG[1:] + (4,))
            a[:] = seed
            kept.append(a)
            if len(kept) > 3:
                if not (kept.pop(0) == seed).all():
                    bad.append(seed)
        bad.extend(seed for a in kept if not (a == seed).all())

    ts = [threading.Thread(target=work, args=(k,)) for k in range(6)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    gc.collect()
    assert not bad and idle(h) <= h.KEEP and not h._lock.locked()


def test_a_finalizer_within_a_call_does_not_wait_for_it():
    # the collector may close a solver, drop an array or ask for one while this thread is in
    # empty(): the lock is then held by the thread itself
    h = solver._HostBuffers()
    h.open()
    a = h.empty(BIG)
    got = []

    def finalizer():
        with h._lock:
            h.close()
            got.append(h.empty(BIG))

    t = threading.Thread(target=finalizer, daemon=True)
    t.start()
    t.join(20)
    assert not t.is_alive() and got[0].flags["OWNDATA"]
    del a
    assert not h._bufs
