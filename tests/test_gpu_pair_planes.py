"""The shared-memory sweep (coefficients in pair planes), which serves lattices whose
strip records do not fit, against the marching sweep: the same operations per site in
the same order, so the same bits. And the marching sweep's two-step passes at the
edges of strips, row ranges and media, and on a lattice of many strips."""
import numpy as np
import pytest

import oracle
from paper_2301_13601_gb300 import media
from paper_2301_13601_gb300.qla import Simulation
from test_gpu_march import medium

pytestmark = pytest.mark.gpu


def run(n, q, steps, planes=False, delta=0.2, **kw):
    with Simulation(*n, delta, **kw) as sim:
        if planes:
            sim.use_pair_planes()
        sim.set_fields(q)
        sim.step(steps)
        return sim.get_fields()


def problem(Nx, Ny, precision):
    q = np.random.default_rng(Nx + Ny).standard_normal((6, Ny, Nx))
    return medium(Nx, Ny), q if precision == "fp64" else q.astype(np.float32)


# plain strips with a ragged one, odd rows, narrower than a strip; TMA strips, row
# blocks that straddle the wrap and the groups of the merged boxes; the seam layout
# with a clamped last strip; tiles and the balanced split
@pytest.mark.parametrize("Nx, Ny, chunk, K", [
    (500, 70, 24, 2), (500, 70, 0, 4), (37, 53, 0, 1), (8, 5, 0, 2), (64, 64, 16, 4), (1024, 96, 40, 2), (1024, 96, 0, 4),
    (1024, 100, 40, 4), (1024, 96, 37, 2), (1024, 98, 24, 4), (256, 40, 0, 2), (744, 50, 16, 2), (2048, 21, 0, 2),
    (496, 64, 24, 4), (1000, 777, 0, 2), (1, 9, 0, 1)])
@pytest.mark.parametrize("sequence, potential", [("interleaved", "paper"), ("plain", "unitary"),
                                                 ("interleaved", "unitary"), ("plain", "paper")])
def test_fp32_pair_planes_bit_identical(Nx, Ny, chunk, K, sequence, potential):
    n, q = problem(Nx, Ny, "fp32")
    kw = dict(sequence=sequence, potential=potential)
    ref = run(n, q, 3 * K + 1, **kw)
    assert np.array_equal(run(n, q, 3 * K + 1, planes=True, chunk_rows=chunk, steps_per_pass=K, **kw), ref)


@pytest.mark.parametrize("Nx, Ny, chunk, K", [(500, 70, 24, 2), (500, 70, 0, 1), (37, 53, 0, 2), (8, 5, 0, 1),
                                              (64, 64, 16, 2), (300, 41, 0, 2)])
@pytest.mark.parametrize("sequence, potential", [("interleaved", "paper"), ("plain", "unitary")])
def test_fp64_pair_planes_bit_identical(Nx, Ny, chunk, K, sequence, potential):
    n, q = problem(Nx, Ny, "fp64")
    kw = dict(sequence=sequence, potential=potential, precision="fp64")
    ref = run(n, q, 5, **kw)
    assert np.array_equal(run(n, q, 5, planes=True, chunk_rows=chunk, steps_per_pass=K, **kw), ref)


@pytest.mark.parametrize("family", ["TM", "TE"])
def test_one_family_on_pair_planes(family):
    n, q = problem(520, 40, "fp32")
    q[[0, 1, 5] if family == "TM" else [2, 3, 4]] = 0.0
    assert np.array_equal(run(n, q, 5, planes=True, families=family), run(n, q, 5, families=family))


@pytest.mark.parametrize("Nx, Ny", [(112, 96), (113, 61), (228, 33), (116, 7), (18, 2), (4, 1), (339, 40), (450, 130)])
@pytest.mark.parametrize("sequence, potential", [("interleaved", "paper"), ("plain", "unitary"),
                                                 ("interleaved", "unitary"), ("plain", "paper")])
def test_two_step_passes_at_the_edges(Nx, Ny, sequence, potential):
    """FP32, sharp-edged media (groups of rows without potentials, unchanged collision
    rows), rows in vectors and by elements, seven steps: three passes of two, one of
    one. Bounds as test_gpu_march.py; one-step passes and every row range give the
    same bits."""
    n, q = problem(Nx, Ny, "fp32")
    kw = dict(sequence=sequence, potential=potential)
    got = run(n, q, 7, steps_per_pass=2, **kw)
    theta, beta = oracle.angles(*n, 0.2)
    ref = q.astype(np.float64)
    oracle.run(ref, theta, beta, 7, oracle.SEQ_INTERLEAVED if sequence == "interleaved" else oracle.SEQ_PLAIN,
               oracle.POT_PAPER if potential == "paper" else oracle.POT_UNITARY)
    assert np.linalg.norm(got - ref) < 3e-6 * np.linalg.norm(ref)
    assert np.array_equal(run(n, q, 7, steps_per_pass=1, **kw), got)
    for rows in (1, 5, Ny):
        assert np.array_equal(run(n, q, 7, steps_per_pass=2, chunk_rows=rows, **kw), got), rows


@pytest.mark.parametrize("Nx, Ny", [(8192, 500), (5001, 801)])
def test_every_strip_and_range_of_a_wide_lattice(Nx, Ny):
    """74 (45) strips by many row ranges, every site against the oracle."""
    n = media.medium(Nx, Ny, [media.Ellipse(0.3 * Nx, 0.5 * Ny, 0.2 * Nx, 0.3 * Ny, 0.3, (1.6, 2.1, 2.7), 4.0)])
    q = np.random.default_rng(1).standard_normal((6, Ny, Nx)).astype(np.float32)
    got = run(n, q, 5)
    theta, beta = oracle.angles(*n, 0.2)
    ref = q.astype(np.float64)
    oracle.run(ref, theta, beta, 5, oracle.SEQ_INTERLEAVED, oracle.POT_PAPER)
    err = np.abs(got - ref)
    assert np.linalg.norm(err) < 3e-6 * np.linalg.norm(ref)
    # a wrong strip or range would be off by the size of the field (5 sigma) at single sites
    assert err.max() < 1e-4
