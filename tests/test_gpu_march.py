"""The marching form of the sweep (one warp per strip and row range, state in
registers): edges of its strips and ranges, and the groups of rows whose
potentials are skipped.

Every site is computed by the same operations in the same order whichever warp
and row group computes it, so results do not depend on the row ranges, bit for
bit; against the oracle the bounds are those of test_gpu_parity.py (FP32: up to
13 steps of about 64 roundings of 2^-24 per component, 3e-6; FP64: 1e-12)."""
import numpy as np
import pytest

import oracle
from paper_2301_13601_gb300 import media
from paper_2301_13601_gb300.qla import Simulation

pytestmark = pytest.mark.gpu


def medium(Nx, Ny):
    """Two sharp-edged objects in vacuum, one across the y boundary: rows with
    and without potentials in every strip that they touch, groups that start on
    either side of the change."""
    n = np.ones((3, Ny, Nx))
    n[:, Ny // 3:Ny // 2, Nx // 4:Nx // 2] = np.array([1.5, 1.3, 2.0])[:, None, None]
    n[:, :max(1, Ny // 12), 2 * Nx // 3:] = np.array([1.2, 1.7, 1.4])[:, None, None]
    n[:, Ny - Ny // 9:, 2 * Nx // 3:] = np.array([1.2, 1.7, 1.4])[:, None, None]
    return tuple(n)


def run(n, q, steps, delta=0.2, **kw):
    with Simulation(*n, delta, **kw) as sim:
        sim.set_fields(q)
        sim.step(steps)
        return sim.get_fields()


# one strip exactly, one column more, a strip less than its halo, a narrow
# lattice under a wide strip, rows of every alignment, fewer rows than the halo
@pytest.mark.parametrize("Nx, Ny", [(112, 96), (113, 61), (228, 33), (116, 7), (18, 2), (4, 1), (339, 40), (450, 130)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("sequence, potential", [("interleaved", "paper"), ("plain", "unitary")])
def test_strip_and_range_edges(Nx, Ny, precision, sequence, potential):
    n = medium(Nx, Ny)
    q = np.random.default_rng(7).standard_normal((6, Ny, Nx))
    if precision == "fp32":
        q = q.astype(np.float32).astype(np.float64)
    kw = dict(precision=precision, sequence=sequence, potential=potential)
    steps = 7  # passes of two steps and a last one of one
    got = run(n, q, steps, **kw)
    theta, beta = oracle.angles(*n, 0.2)
    ref = q.copy()
    oracle.run(ref, theta, beta, steps, oracle.SEQ_INTERLEAVED if sequence == "interleaved" else oracle.SEQ_PLAIN,
               oracle.POT_PAPER if potential == "paper" else oracle.POT_UNITARY)
    assert np.linalg.norm(got - ref) < (3e-6 if precision == "fp32" else 1e-12) * np.linalg.norm(ref)
    for rows in (1, 5, Ny):
        assert np.array_equal(run(n, q, steps, chunk_rows=rows, **kw), got), rows


@pytest.mark.parametrize("family", ["TM", "TE"])
@pytest.mark.parametrize("K", [1, 2, 4])
def test_one_family_and_steps_per_pass_bit_exact(family, K):
    Nx, Ny = 360, 101
    n = medium(Nx, Ny)
    q = np.random.default_rng(9).standard_normal((6, Ny, Nx)).astype(np.float32)
    q[[0, 1, 5] if family == "TM" else [2, 3, 4]] = 0.0
    ref = run(n, q, 9)
    assert np.array_equal(run(n, q, 9, families=family, steps_per_pass=K), ref)
    # the shared-memory sweep that the persistent launch form keeps
    assert np.array_equal(run(n, q, 9, families=family, launch="persistent"), ref)


def test_single_operators_read_the_records():
    """qla_debug_apply finds a site's coefficients in the strip records: every
    operator agrees with the context that keeps pair planes."""
    Nx, Ny = 264, 30
    n = medium(Nx, Ny)
    q = np.random.default_rng(3).standard_normal((6, Ny, Nx)).astype(np.float32)
    for op in ("CX", "CY", "VX", "VY"):
        out = []
        for launch in ("auto", "persistent"):
            with Simulation(*n, 0.2, launch=launch) as sim:
                sim.set_fields(q)
                sim.debug_apply(op)
                out.append(sim.get_fields(np.float32))
        assert np.array_equal(*out), op


# one row range, several warps and CTAs, more CTAs than the device takes at once
@pytest.mark.parametrize("Nx, Ny, chunk_rows", [(64, 8, 0), (256, 256, 0), (301, 207, 0), (1024, 256, 1)])
def test_chained_passes_match_single_ones(Nx, Ny, chunk_rows):
    """Passes of one call are launched before the one before them has ended; a
    call of one step has nothing to overlap with. The same operations: the same
    bits, also when another context's passes run between them."""
    n = medium(Nx, Ny)
    q = np.random.default_rng(3).standard_normal((6, Ny, Nx))
    steps = 41
    kw = dict(chunk_rows=chunk_rows, steps_per_pass=1)
    with Simulation(*n, 0.2, **kw) as one, Simulation(*n, 0.2, **kw) as many, Simulation(*n, 0.2, **kw) as beside:
        for sim in (one, many, beside):
            sim.set_fields(q)
        for _ in range(steps):
            one.step(1)
        many.step(steps)
        beside.step(steps)
        ref = one.get_fields()
        assert np.array_equal(many.get_fields(), ref)
        assert np.array_equal(beside.get_fields(), ref)
