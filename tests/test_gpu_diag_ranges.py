"""Diagnostics of states and media whose values are far from 1: products of indices and
fields, squares and differences that leave the range of FP32, and the accuracy of
the squared divergence. Maxima are one FP64 evaluation of the winning site (1e-14, as
test_gpu_diag_edges.py); the bounds of the sums are stated where they are used."""
import numpy as np
import pytest

import oracle
from paper_2301_13601_gb300.qla import Simulation

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("index, field", [(-40, -40), (-30, -45), (-20, -45), (0, -100), (30, 59), (-45, 40), (59, 40)])
def test_divD_maximum_of_one_component(index, field, precision):
    """max |D| where only D_z is nonzero: its square leaves FP32 although n_z and q_2 do not."""
    Nx, Ny = 70, 9
    rng = np.random.default_rng(5)
    n = tuple((1.0 + rng.random((3, Ny, Nx))) * 2.0 ** index)
    q = np.zeros((6, Ny, Nx))
    q[2] = np.float32(rng.standard_normal((Ny, Nx)) * 2.0 ** field)
    with Simulation(*n, 0.1, precision=precision) as sim:
        sim.set_fields(q)
        div, dmax, largest = sim.divD()
    assert div == 0.0 and dmax == 0.0
    ref = oracle.divD(q, *n)[2]
    assert abs(largest - ref) <= 1e-14 * ref


@pytest.mark.parametrize("Nx, Ny", [(200, 300), (513, 129)])
@pytest.mark.parametrize("kind", ["noise", "waves"])
def test_squared_divergence_to_the_last_bits(Nx, Ny, kind):
    """FP32 states, against exact integer arithmetic. A site's divergence and square round
    a few times in FP64 (unbiased, at most 3 units of 2^-53), and sums of at most 32
    sites round at most 32 times: over more than 6e4 sites both average to less than
    0.1 unit of the sum, whose compensated end rounds once or twice by half a unit."""
    rng = np.random.default_rng(8)
    if kind == "noise":
        q = rng.standard_normal((6, Ny, Nx))
    else:
        y, x = np.mgrid[0:Ny, 0:Nx]
        q = np.stack([0.2 * np.cos(2 * np.pi * ((k + 1) * x / Nx + 2 * y / Ny) + k) +
                      np.exp(-((x - Nx / 2) / (0.05 * Nx)) ** 2) for k in range(6)])
    q = q.astype(np.float32).astype(np.float64)
    with Simulation(*np.ones((3, Ny, Nx)), 0.1) as sim:
        sim.set_fields(q)
        got = sim.diagnostics()["div_l2_sq"]
    scaled = [int(v * 2.0 ** 64) for v in q[3:5].ravel()]
    bx, by = np.array(scaled[:Nx * Ny], dtype=object).reshape(Ny, Nx), np.array(scaled[Nx * Ny:], dtype=object).reshape(Ny, Nx)
    div = np.roll(bx, -1, 1) - np.roll(bx, 1, 1) + np.roll(by, -1, 0) - np.roll(by, 1, 0)
    ref = int((div * div).sum())  # times 4 * 2^128
    assert abs(int(got * 2.0 ** 130) - ref) <= 2 * ref >> 53


def field_of(kind, shape, rng):
    """States with small values: sites of one scale, of scales mixed site by site or within
    a site, and the tails of a pulse."""
    v = rng.standard_normal((6,) + shape)
    if kind == "edge -44" or kind == "edge -58" or kind == "edge -60":
        return v * 2.0 ** int(kind.split()[1])
    if kind == "subnormal":
        return v * 2.0 ** -140
    if kind == "mixed sites":
        return v * 2.0 ** rng.integers(-80, 3, shape)
    if kind == "mixed components":
        return v * 2.0 ** rng.integers(-80, 3, v.shape)
    x = np.arange(shape[1])
    g = np.exp(-(x - shape[1] / 8) ** 2 / (2 * (shape[1] / 40) ** 2))
    return np.stack([0 * v[0], 0 * v[0], g + 0 * v[0], 0 * v[0], -g + 0 * v[0], 0 * v[0]])


@pytest.mark.parametrize("Nx, Ny", [(1, 9), (300, 40), (1030, 300)])
@pytest.mark.parametrize("kind", ["edge -44", "edge -58", "edge -60", "subnormal", "mixed sites", "mixed components",
                                  "pulse"])
def test_small_values_fp32(Nx, Ny, kind):
    """A site's sum of squares is an FP32 pair (2^-46 of it, low parts rounded) or FP64:
    1e-14, as the other tests of the sums."""
    q = field_of(kind, (Ny, Nx), np.random.default_rng(Nx)).astype(np.float32).astype(np.float64)
    with Simulation(*np.ones((3, Ny, Nx)), 0.1) as sim:
        sim.set_fields(q)
        d = sim.diagnostics()
    s, m, b = oracle.divB(q)
    assert d["nonfinite"] == 0
    for got, ref, tol in ((d["energy"], oracle.energy(q), 1e-14), (d["div_l2_sq"], s, 1e-13), (d["div_max"], m, 1e-14),
                          (d["b_max"], b, 1e-14)):
        assert abs(got - ref) <= tol * abs(ref)
