"""Buffers sized by qla_query_buffer_sizes hold every context of their lattice and
precision."""
import ctypes

import numpy as np
import pytest

from paper_2301_13601_gb300.qla import Simulation
from test_gpu_march import medium

pytestmark = pytest.mark.gpu


def run(n, q, steps):
    with Simulation(*n, 0.2) as sim:
        sim.set_fields(q)
        sim.step(steps)
        return sim.get_fields()


def test_buffers_of_other_options_are_large_enough():
    """A context of both families inside buffers that were sized for one family and the
    persistent launch form: nothing is written past them."""
    import torch
    from paper_2301_13601_gb300 import qla

    Nx, Ny = 360, 101
    L = qla.load_library()
    opt, sizes = qla.Options(), qla.BufferSizes()
    L.qla_default_options(ctypes.byref(opt))
    opt.families, opt.launch = qla.FAMILY_TM, qla.LAUNCHES["persistent"]
    assert L.qla_query_buffer_sizes(Nx, Ny, ctypes.byref(opt), ctypes.byref(sizes)) == 0
    GUARD = 4 << 20  # more than both families' records
    names = ("state_bytes", "state_bytes", "coeff_bytes", "index_bytes", "scratch_bytes")
    bufs = [torch.full((getattr(sizes, k) + GUARD,), 0x5A, dtype=torch.uint8, device="cuda") for k in names]
    db = qla.DeviceBuffers()
    db.state[0], db.state[1], db.coeff, db.index, db.scratch = (b.data_ptr() for b in bufs)
    torch.cuda.synchronize()
    n, q = medium(Nx, Ny), np.random.default_rng(Nx + Ny).standard_normal((6, Ny, Nx)).astype(np.float32)
    ctx = ctypes.c_void_p()
    dp = lambda a: np.ascontiguousarray(a).ctypes.data_as(ctypes.POINTER(ctypes.c_double))  # noqa: E731
    planes = [np.ascontiguousarray(a) for a in n]
    assert L.qla_create(Nx, Ny, *(dp(a) for a in planes), 0.2, None, ctypes.byref(db), ctypes.byref(ctx)) == 0
    try:
        assert L.qla_set_fields_f32(ctx, q.ctypes.data_as(ctypes.POINTER(ctypes.c_float))) == 0
        assert L.qla_step(ctx, 6) == 0
        assert L.qla_synchronize(ctx) == 0
        out = np.empty_like(q)
        assert L.qla_get_fields_f32(ctx, out.ctypes.data_as(ctypes.POINTER(ctypes.c_float))) == 0
    finally:
        L.qla_destroy(ctx)
    assert np.array_equal(out, run(n, q, 6).astype(np.float32))
    for b, k in zip(bufs, names):
        assert torch.all(b[getattr(sizes, k):] == 0x5A), k
