"""TeukSolver: a thin Python handle over the C ABI (include/teuk.h).

It marshals numpy arrays and torch streams into the C calls; the time loop, the
source and the extraction all run in the library's CUDA kernels."""
from __future__ import annotations

import ctypes
import json
import mmap
import os
import threading
import weakref

import numpy as np

from . import _lib
from ._lib import TEUK_FP32, TEUK_FP32_KAHAN, TEUK_FP64, TEUK_FP64_DF, check, ptr

PREC = {"fp64": TEUK_FP64, "fp32": TEUK_FP32, "fp32_kahan": TEUK_FP32_KAHAN, "fp64_df": TEUK_FP64_DF,
        TEUK_FP64: TEUK_FP64, TEUK_FP32: TEUK_FP32, TEUK_FP32_KAHAN: TEUK_FP32_KAHAN,
        TEUK_FP64_DF: TEUK_FP64_DF}

PARAM_DEFAULTS = dict(s=-2, m=2, M=1.0, a=0.9, rstar_min=-50.0, rstar_max=150.0, n_rstar=800,
                      n_theta=64, courant=0.5, dt_rule=1, dt=0.0, rstar_ext=140.0,
                      prec="fp64", wave_capacity=0, slab_col0=0, slab_ncols=0)


def make_params(**kw) -> _lib.teuk_params:
    d = dict(PARAM_DEFAULTS)
    for k, v in kw.items():
        if k not in d:
            raise KeyError("unknown parameter %r" % k)
        d[k] = v
    d["prec"] = PREC[d["prec"]]
    return _lib.teuk_params(**d)


_ALLOC_HOOKS = None   # the ctypes callbacks in force (kept alive while installed)


def set_allocator(alloc=None, free=None):
    """Route the device memory of contexts created from now on through Python callables
    alloc(bytes, stream_handle) -> device pointer (0 on failure) and free(ptr, stream_handle)
    (teuk_set_allocator); set_allocator() restores cudaMallocAsync.  Contexts keep the
    allocator they were created with."""
    global _ALLOC_HOOKS
    lib = _lib.load()
    if alloc is None and free is None:
        check(lib.teuk_set_allocator(None, None, None), None)
        _ALLOC_HOOKS = None
        return

    def _a(nbytes, stream, user):
        try:
            return int(alloc(int(nbytes), int(stream or 0))) or None
        except Exception:
            return None

    def _f(ptr, stream, user):
        try:
            free(int(ptr), int(stream or 0))
        except Exception:
            pass

    hooks = (_lib.ALLOC_FN(_a), _lib.FREE_FN(_f), alloc, free)
    check(lib.teuk_set_allocator(ctypes.cast(hooks[0], ctypes.c_void_p),
                                 ctypes.cast(hooks[1], ctypes.c_void_p), None), None)
    _ALLOC_HOOKS = hooks


def use_torch_allocator(enable=True):
    """Device memory of new contexts from torch's caching allocator (one pool with torch)."""
    if not enable:
        set_allocator()
        return
    import torch

    set_allocator(lambda n, st: torch.cuda.caching_allocator_alloc(n, stream=st),
                  lambda p, st: torch.cuda.caching_allocator_delete(p))


def _stream_handle(stream):
    if stream is None:
        import torch
        return torch.cuda.current_stream().cuda_stream
    if isinstance(stream, int):
        return stream
    return stream.cuda_stream


# of the rules that cut the columns automatically: tables tuned against other rules are not used
_CUT_VERSION = 2


class _HostBuffers:
    """Result arrays whose memory is used again once the caller has dropped them (every view
    included).  A fresh array of 134 MB (a 16384 x 256 state) costs 6 to 20 ms of page faults
    and unmapping a call, on GB300 with its fast host link the copy itself 0.9 ms.  Memory that
    the GPU alone goes on using is moved about by the driver, and every few copies then take
    15 to 35 ms; one access by the host to each page before the copy keeps it where it is
    (`_touch`, 0.05 ms).  Arrays below 4 MB come from numpy (its heap reuses them).  At most
    KEEP bytes are kept idle, counted whenever an array is dropped or asked for, the longest
    idle given back first, and none once the last solver is closed (any thread may drop an
    array or ask for one)."""
    MIN, KEEP = 4 << 20, 1 << 30

    def __init__(self):
        self._lock = threading.Lock()   # of _bufs
        self._count = threading.RLock()   # of _users and _closed
        self._bufs = []   # [mapping, weak reference to the object that its arrays hold], oldest first
        self._mapped = 0   # bytes of _bufs
        self._dropped = False   # an array died since the idle mappings were last counted
        pool = weakref.ref(self)

        def dropped(_):
            p = pool()
            if p is not None:
                p._dropped = True
                p._settle()
        self._watch = dropped
        self._users, self._closed = 0, False

    def open(self):
        """One more solver."""
        with self._count:
            self._users += 1
            self._closed = False

    def close(self):
        """One solver less; after the last nothing is kept idle.  (A solver's finalizer may run
        in a thread that is within empty(): the lock of _bufs is never waited for here.)"""
        with self._count:
            self._users -= 1
            self._closed = self._users <= 0
        self._dropped = True
        self._settle()

    def _settle(self):
        # runs in whatever thread drops an array, at any moment (within empty() too, by the
        # collector): it never waits; who holds the lock settles again after giving it back
        while self._dropped and (self._closed or self._mapped > self.KEEP) and self._lock.acquire(blocking=False):
            try:
                self._dropped = False
                idle = [b for b in self._bufs if b[1]() is None]
                kept = sum(len(b[0]) for b in idle)
                for b in idle:
                    if kept <= (0 if self._closed else self.KEEP):
                        break
                    self._bufs.remove(b)
                    kept -= len(b[0])
                    self._mapped -= len(b[0])
            finally:
                self._lock.release()

    def empty(self, shape, dtype=np.float64):
        dtype = np.dtype(dtype)
        count = 1
        for n in shape:
            count *= int(n)
        size = count * dtype.itemsize
        if size < self.MIN:
            return np.empty(shape, dtype)
        # mappings come in sixteen sizes an octave, so that records that grow from call to call
        # find one again
        step = 1 << (size.bit_length() - 5)
        whole = (size + step - 1) // step * step
        buf = None
        # (not waited for without end: a finalizer that asks for an array may have interrupted
        # this very thread's call)
        if self._lock.acquire(timeout=0.1):
            try:
                buf = next((b for b in self._bufs if len(b[0]) == whole and b[1]() is None), None)
                again = buf is not None
                if again:
                    self._bufs.remove(buf)
                else:
                    try:
                        buf = [mmap.mmap(-1, whole, flags=mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS), None]
                        # (as numpy does for its own arrays)
                        buf[0].madvise(mmap.MADV_HUGEPAGE)
                    except (AttributeError, OSError, OverflowError, ValueError):
                        pass
                    if buf is not None:
                        self._mapped += whole
                if buf is not None:
                    raw = (ctypes.c_char * size).from_buffer(buf[0])
                    buf[1] = weakref.ref(raw, self._watch)   # dead when the last array on the mapping is gone
                    self._bufs.append(buf)
            finally:
                self._lock.release()
        self._settle()
        if buf is None:   # no mapping to be had: numpy's own answer
            return np.empty(shape, dtype)
        if again:
            np.frombuffer(raw, np.uint8)[::mmap.PAGESIZE] = 0
        return np.frombuffer(raw, dtype, count).reshape(shape)


_HOST = _HostBuffers()   # of every solver of the process


def _touch(u):
    """Read one value of each page of a large contiguous host array before the GPU copies it:
    16384 x 256 states set in turn, 0.9 or 20 to 36 ms a call -> 0.95 ms every time."""
    if u.nbytes >= _HostBuffers.MIN:
        u.reshape(-1)[::mmap.PAGESIZE // u.itemsize].copy()


class TeukSolver:
    """One context of one or more instances (see teuk_create).

    Result arrays of 4 MB and more (get_state, extract, mode_sum) lie in host memory that is
    used again once every view of them is dropped; up to 1 GB of it stays idle while a solver
    of the process is open.  Such an array does not own its data: `ndarray.resize` refuses it
    (resize a copy)."""

    def __init__(self, params, stream=None):
        if isinstance(params, dict):
            params = [params]
        plist = [p if isinstance(p, _lib.teuk_params) else make_params(**p) for p in params]
        self.n = len(plist)
        arr = (_lib.teuk_params * self.n)(*plist)
        self.params = plist
        self._stream = stream
        h = ctypes.c_void_p()
        lib = _lib.load()
        st = lib.teuk_create(arr, self.n, ctypes.c_void_p(_stream_handle(stream)), ctypes.byref(h))
        check(st, None)
        self.ctx = h
        self._host = _HOST
        self._host.open()
        self._steps_per_launch = 1

    # -- lifetime
    def close(self):
        if getattr(self, "ctx", None):
            _lib.load().teuk_destroy(self.ctx)
            self.ctx = None
            self._host.close()

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass

    def __enter__(self):
        return self

    def __exit__(self, *a):
        self.close()

    # -- calls
    def set_source(self, r0, amps=None, instance=0, sigma_rstar_cells=4.0, sigma_theta_cells=4.0,
                   sigma_rstar_abs=0.0, sigma_theta_abs=0.0):
        orb = _lib.teuk_orbit(r0, sigma_rstar_cells, sigma_theta_cells, sigma_rstar_abs,
                              sigma_theta_abs)
        a = None if amps is None else np.ascontiguousarray(amps, dtype=np.float64)
        check(_lib.load().teuk_set_source(self.ctx, instance, ctypes.byref(orb), ptr(a),
                                          0 if a is None else a.size), self.ctx)

    def set_trajectory(self, traj, instance=0, sigma_rstar_cells=4.0, sigma_theta_cells=4.0,
                       sigma_rstar_abs=0.0, sigma_theta_abs=0.0):
        """Moving particle: traj [n_samples][4] = {r_p, theta_p, phi_p, A} at t = k dt/2
        (step n takes samples 2n and 2n + 1)."""
        orb = _lib.teuk_orbit(0.0, sigma_rstar_cells, sigma_theta_cells, sigma_rstar_abs,
                              sigma_theta_abs)
        t = np.ascontiguousarray(traj, dtype=np.float64).reshape(-1, 4)
        check(_lib.load().teuk_set_trajectory(self.ctx, instance, ctypes.byref(orb), ptr(t),
                                              t.shape[0]), self.ctx)

    def shape(self, instance=0):
        p = self.params[instance]
        return (4, p.n_theta, p.slab_ncols + 2 if p.slab_ncols > 0 else p.n_rstar)

    # -- slabs (teuk_params.slab_ncols > 0): halo columns, device to device
    def halo_bytes(self, instance=0):
        b = ctypes.c_int64(0)
        check(_lib.load().teuk_slab_halo_bytes(self.ctx, instance, ctypes.byref(b)), self.ctx)
        return b.value

    def slab_export(self, side, dev_ptr, instance=0):
        check(_lib.load().teuk_slab_export(self.ctx, instance, side, ctypes.c_void_p(dev_ptr)), self.ctx)

    def slab_import(self, side, dev_ptr, instance=0):
        check(_lib.load().teuk_slab_import(self.ctx, instance, side, ctypes.c_void_p(dev_ptr)), self.ctx)

    def set_state(self, u, step0=0, instance=0):
        u = np.ascontiguousarray(u, dtype=np.float64)
        assert u.shape == self.shape(instance)
        _touch(u)
        check(_lib.load().teuk_set_state(self.ctx, instance, ptr(u), step0), self.ctx)

    def get_state(self, instance=0):
        u = self._host.empty(self.shape(instance))
        check(_lib.load().teuk_get_state(self.ctx, instance, ptr(u)), self.ctx)
        return u

    def step(self, n):
        check(_lib.load().teuk_step_n(self.ctx, int(n)), self.ctx)

    def extract(self, cap=None, instance=0, scalar=False):
        """Returns (records [k][n_theta][2], first_step[, scalar [k][2]])."""
        p = self.params[instance]
        step, _ = self.time(instance)
        if cap is None:
            cap = step + 1
        out = self._host.empty((cap, p.n_theta, 2))
        sc = np.empty((cap, 2)) if scalar else None
        nw, first = ctypes.c_int64(0), ctypes.c_int64(0)
        check(_lib.load().teuk_extract(self.ctx, instance, ptr(out), ptr(sc), cap,
                                       ctypes.byref(nw), ctypes.byref(first)), self.ctx)
        k = nw.value
        if scalar:
            return out[:k], first.value, sc[:k]
        return out[:k], first.value

    def mode_sum(self, phi, first, n_records):
        """Psi = sum_m e^{i m phi~} r^3 Phi_m at the extraction radius over the instances
        (modes of one problem) for time levels first .. first + n_records - 1 and the
        azimuths phi: complex array [n_records][n_theta][len(phi)]."""
        ph = np.ascontiguousarray(np.atleast_1d(phi), dtype=np.float64)
        nth = self.params[0].n_theta
        out = self._host.empty((n_records, nth, ph.size), np.complex128)   # (re, im) pairs
        check(_lib.load().teuk_mode_sum(self.ctx, ptr(ph), ph.size, int(first), int(n_records),
                                        ptr(out)), self.ctx)
        return out

    def radiated_flux(self, first, n_records):
        """Energy, linear momentum and Jz carried off by the field of the instances (distinct
        modes of one problem), from the records first .. first + n_records - 1: array
        [n_records][10] = dE/dt, dPx/dt, dPy/dt, dPz/dt, dJz/dt, E, Px, Py, Pz, Jz (totals
        from `first`; the recoil velocity is -P / M_total)."""
        out = np.empty((int(n_records), 10))
        check(_lib.load().teuk_radiated_flux(self.ctx, int(first), int(n_records), ptr(out)),
              self.ctx)
        return out

    def adjoint(self, n, step0=0, grad_wave=None, ckpt_every=100, instance=0):
        """Returns (grad_amps [n], grad_r0, loss).  ckpt_every (built-in loss only): K > 0
        recomputes each K-step segment's records from a state checkpoint in the reverse
        sweep; 0 keeps every record's cotangent instead (no recomputation)."""
        gw = None if grad_wave is None else np.ascontiguousarray(grad_wave, dtype=np.float64)
        ga = np.zeros(n)
        gr, loss = ctypes.c_double(0.0), ctypes.c_double(0.0)
        check(_lib.load().teuk_adjoint_n(self.ctx, instance, step0, n, ckpt_every, ptr(gw),
                                         ptr(ga), ctypes.byref(gr), ctypes.byref(loss)), self.ctx)
        return ga, gr.value, loss.value

    def sync(self):
        check(_lib.load().teuk_sync(self.ctx), self.ctx)

    def save_state(self, path, instance=0):
        """Checkpoint: parameters, time level and the current level's planes, bit for bit."""
        check(_lib.load().teuk_save_state(self.ctx, instance, os.fsencode(path)), self.ctx)

    def load_state(self, path, instance=0):
        """Resume from save_state's file (the same problem; clears the waveform records)."""
        check(_lib.load().teuk_load_state(self.ctx, instance, os.fsencode(path)), self.ctx)

    def check_selftest(self):
        """Checked builds: make the next sync report TEUK_EBOUNDS (no memory is addressed)."""
        check(_lib.load().teuk_check_selftest(self.ctx), self.ctx)

    def time(self, instance=0):
        s, dt = ctypes.c_int64(0), ctypes.c_double(0.0)
        check(_lib.load().teuk_get_time(self.ctx, instance, ctypes.byref(s), ctypes.byref(dt)),
              self.ctx)
        return s.value, dt.value

    def geometry(self, instance=0):
        """dict(drs, dth, dt, rp, rm, r_ext, i_e, f_e) of one instance."""
        out = np.zeros(8)
        check(_lib.load().teuk_get_geometry(self.ctx, instance, ptr(out)), self.ctx)
        return dict(drs=out[0], dth=out[1], dt=out[2], rp=out[3], rm=out[4], r_ext=out[5],
                    i_e=int(out[6]), f_e=out[7])

    def set_tiling(self, strip=0, steps_per_launch=1):
        """strip: r* columns per thread block (0 = automatic); steps_per_launch 0 sends a
        single-instance context through the persistent batched kernel."""
        check(_lib.load().teuk_set_tiling(self.ctx, strip, steps_per_launch), self.ctx)
        self._steps_per_launch = steps_per_launch

    def tiling(self, instance=0):
        """The cut of an instance's columns in effect: dict(automatic, columns (of the longest
        piece), pieces, side_by_side (the block-size classes of a batch))."""
        out = (ctypes.c_int * 4)()
        check(_lib.load().teuk_get_tiling(self.ctx, instance, out), self.ctx)
        return dict(automatic=bool(out[0]), columns=out[1], pieces=out[2], side_by_side=bool(out[3]))

    def set_resident(self, halo=1, blocks_per_sm=1):
        """Resident launches (one cooperative launch per step() call, the grid held in
        shared memory, boundary columns exchanged every ``halo`` steps, the column runs cut
        for ``blocks_per_sm`` blocks per SM); halo 0 turns them off."""
        check(_lib.load().teuk_set_resident_shape(self.ctx, int(halo), int(blocks_per_sm)), self.ctx)

    def set_blocked(self, steps=2, blocks_per_sm=1):
        """Blocked launches (each launch advances ``steps`` steps of the grid held in shared
        memory, halos from the previous launch's output, no exchange); 0 turns them off."""
        check(_lib.load().teuk_set_blocked(self.ctx, int(steps), int(blocks_per_sm)), self.ctx)

    def kernel_launches(self):
        return _lib.load().teuk_kernel_launches(self.ctx)

    def set_instance_tiling(self, instance, strip):
        check(_lib.load().teuk_set_instance_tiling(self.ctx, instance, strip), self.ctx)

    def set_fill_fault(self, column=-1, instance=0):
        check(_lib.load().teuk_set_fill_fault(self.ctx, instance, column), self.ctx)

    def set_fault_injection(self, skip_release_item=-1, spin_limit=0):
        check(_lib.load().teuk_set_fault_injection(self.ctx, skip_release_item, spin_limit),
              self.ctx)

    def autotune(self, trial_steps=10, cache_path=None):
        """Strip length per instance from a cached table keyed by (GPU, launch mode, n_theta,
        precision, n_rstar bucket, version of the kernels' automatic cut); entries missing
        from the table are timed by teuk_autotune.  An entry 0 stands for no length of its own
        (the automatic cut: on another grid of the bucket, that grid's).  A negative entry -v
        (single instance stepped per call) selects resident launches with halo v % 16 and
        v // 16 + 1 blocks per SM.  The launch mode is "step" for one instance stepped one
        launch per step, and for contexts that run the persistent kernels a signature of the
        whole set of instances (their best strips depend on one another).  Returns the lengths
        in effect (of the longest piece for an automatic cut), or the negative entries."""
        import hashlib

        import torch
        path = cache_path or os.environ.get("TEUK_TUNE_CACHE") or os.path.join(
            os.path.expanduser("~"), ".cache", "teuk_gb300", "tune.json")
        gpu = torch.cuda.get_device_name()
        if self.n == 1 and self._steps_per_launch != 0:
            mode = "step"
        else:
            shapes = sorted((p.n_rstar, p.n_theta, p.prec) for p in self.params)
            mode = "batch:" + hashlib.sha1(repr(shapes).encode()).hexdigest()[:12]
        keys = ["%s|%s|%d|%d|%d|cut%d" % (gpu, mode, p.n_theta, p.prec, int(np.ceil(np.log2(p.n_rstar))),
                                          _CUT_VERSION) for p in self.params]
        table = {}
        if os.path.exists(path):
            try:
                with open(path) as f:
                    table = json.load(f)
            except (OSError, ValueError):
                table = {}
        if all(k in table for k in keys):
            for i, k in enumerate(keys):
                v = int(table[k])
                if v < 0:   # resident launches: halo (-v) % 16, (-v) // 16 + 1 blocks per SM
                    self.set_resident((-v) % 16, (-v) // 16 + 1)
                else:
                    self.set_instance_tiling(i, v)
                    if self.n == 1 and self._steps_per_launch != 0:
                        self.set_resident(0)
            return self._in_effect([int(table[k]) for k in keys])
        chosen = np.zeros(self.n, dtype=np.int32)
        check(_lib.load().teuk_autotune(self.ctx, trial_steps, chosen.ctypes.data_as(ctypes.c_void_p)),
              self.ctx)
        for k, c in zip(keys, chosen):
            table[k] = int(c)
        try:
            os.makedirs(os.path.dirname(path), exist_ok=True)
            tmp = path + ".tmp%d" % os.getpid()
            with open(tmp, "w") as f:
                json.dump(table, f, indent=1, sort_keys=True)
            os.replace(tmp, path)
        except OSError:
            pass
        return self._in_effect([int(c) for c in chosen])

    def _in_effect(self, chosen):
        return [c or self.tiling(i)["columns"] for i, c in enumerate(chosen)]
