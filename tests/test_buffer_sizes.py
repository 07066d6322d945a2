"""Device memory of a context (host arithmetic of the library, no GPU)."""
import ctypes
import itertools

import pytest


@pytest.fixture(scope="module")
def query():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2301_13601_gb300 import qla

    L = qla.load_library()

    def run(Nx, Ny, **kw):
        opt, sizes = qla.Options(), qla.BufferSizes()
        L.qla_default_options(ctypes.byref(opt))
        for k, v in kw.items():
            setattr(opt, k, v)
        assert L.qla_query_buffer_sizes(Nx, Ny, ctypes.byref(opt), ctypes.byref(sizes)) == 0
        return sizes

    return run


def total(s):
    return 2 * s.state_bytes + s.coeff_bytes + s.index_bytes + s.scratch_bytes


@pytest.mark.parametrize("Nx, Ny", [(1024, 512), (1001, 667), (8, 5), (4, 100000), (4, 1000000), (46340, 46340)])
@pytest.mark.parametrize("precision", [0, 1])
def test_sizes_depend_on_the_lattice_and_the_precision_only(query, Nx, Ny, precision):
    """Buffers that were sized for one set of options serve a context of any other."""
    ref = query(Nx, Ny, precision=precision)
    for families, launch, K, chunk, pot, seq in itertools.product((0, 1, 2), (0, 1, 2), (0, 1, 2), (0, 64), (0, 1), (0, 1)):
        s = query(Nx, Ny, precision=precision, families=families, launch=launch, steps_per_pass=K, chunk_rows=chunk,
                  potential=pot, sequence=seq)
        assert (s.state_bytes, s.coeff_bytes, s.index_bytes, s.scratch_bytes) == (
            ref.state_bytes, ref.coeff_bytes, ref.index_bytes, ref.scratch_bytes)
    assert ref.coeff_bytes >= 14 * Nx * Ny * (8 if precision else 4)  # pair planes


@pytest.mark.parametrize("Nx, Ny", [(46340, 46340), (45000, 47000), (2147483647 // 30000, 30000), (30000, 2147483647 // 30000)])
def test_the_largest_lattices_fit_the_device(query, Nx, Ny):
    """Of 284208 MiB: 128 bytes per FP32 site with pair planes, as ever."""
    assert total(query(Nx, Ny)) <= 128.1 * Nx * Ny + 1e6 < 284208 * 2 ** 20


def test_records_take_the_memory_that_is_there(query):
    s = query(8192, 8192)
    assert s.coeff_bytes > 70 * 8192 ** 2  # records
    assert query(4, 1000000).coeff_bytes < 60 * 4 * 1000000  # 8 KB of records per row of four sites
