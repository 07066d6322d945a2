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
