"""Edges of the diagnostics reductions: lattices smaller than a warp's columns, one
column or row past a tile, and states whose values leave the range in which
squares are kept as FP32 pairs (decaying tails, tiny, huge, mostly zero).

Tolerances as the diagnostics parity tests: sums 1e-14 (energy) and 1e-13 (the
squared divergence, whose terms lose a few bits to cancellation), maxima 1e-14 (one
FP64 evaluation of the winning site)."""
import numpy as np
import pytest

import oracle
from paper_2301_13601_gb300 import media
from paper_2301_13601_gb300.qla import Simulation

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (2, 3), (31, 7), (240, 33), (241, 64), (700, 129)]


def state(kind, shape, rng):
    q = rng.standard_normal((6,) + shape)
    if kind == "tails":
        q *= np.exp(-rng.uniform(0.0, 90.0, q.shape))
    elif kind == "tiny":
        q *= 1e-30
    elif kind == "huge":
        q *= 1e25
    elif kind == "sparse":
        q *= rng.random(q.shape) < 0.05
    elif kind == "uniform in y":  # every site of a column ties for the maxima
        q[:] = q[:, :1]
    return q


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["normal", "tails", "tiny", "huge", "sparse", "uniform in y"])
@pytest.mark.parametrize("Nx, Ny", SHAPES)
def test_diagnostics_and_divD_match_oracle(Nx, Ny, kind, precision):
    rng = np.random.default_rng(Nx + Ny)
    n = tuple(1.0 + rng.random((3, Ny, Nx)))
    q = state(kind, (Ny, Nx), rng)
    if precision == "fp32":
        q = q.astype(np.float32).astype(np.float64)
    with Simulation(*n, 0.1, precision=precision) as sim:
        sim.set_fields(q)
        d, D = sim.diagnostics(), sim.divD()
    assert d["nonfinite"] == 0
    close = lambda got, ref, tol: abs(got - ref) <= tol * abs(ref)  # noqa: E731
    s, m, b = oracle.divB(q)
    assert close(d["energy"], oracle.energy(q), 1e-14)
    assert close(d["div_l2_sq"], s, 1e-13) and close(d["div_max"], m, 1e-14) and close(d["b_max"], b, 1e-14)
    s, m, b = oracle.divD(q, *n)
    assert close(D[0], s, 1e-13) and close(D[1], m, 1e-13) and close(D[2], b, 1e-14)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_nonfinite_values_are_counted(precision):
    Nx, Ny = 70, 41
    q = np.random.default_rng(2).standard_normal((6, Ny, Nx))
    q.reshape(-1)[::97] = np.inf
    q.reshape(-1)[5::211] = np.nan
    with Simulation(*media.uniform_medium(Nx, Ny, (1.2, 1.3, 1.4)), 0.1, precision=precision) as sim:
        sim.set_fields(q)
        assert sim.diagnostics()["nonfinite"] == np.count_nonzero(~np.isfinite(q))
