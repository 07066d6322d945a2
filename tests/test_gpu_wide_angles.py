"""Media with indices far below 1, whose rotation angles (Eq. 24, and Eq. 25 with the
unitary potentials) are not small: the half-angle forms of a rotation lose accuracy
towards angle pi, where tan(a / 2) is unbounded, so such a context rotates in the
form for any angle.

Bounds: a rotation of that form is within 1.2e-7 (FP32) or 2.2e-16 (FP64) of the
exact one, relative to its pair, at every angle (four roundings of the output's size,
two of the coefficients'). A step is 16 collisions and at most 8 potential
applications per family, and errors add up at most linearly: 5 steps stay below
120 * 1.2e-7 = 1.5e-5 and 120 * 2.2e-16 = 3e-14."""
import math

import numpy as np
import pytest

import oracle
from paper_2301_13601_gb300 import media
from paper_2301_13601_gb300.qla import Batch, Simulation

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1.5e-5, "fp64": 3e-14}
DELTA, STEPS = 0.5, 5


def medium(kind, Nx, Ny):
    """kind: a collision angle (a uniform medium, other indices beside it), or
    'jump': potential angles beyond pi beside collision angles of 0.4."""
    n = np.empty((3, Ny, Nx))
    if kind == "jump":
        n[:] = 0.32
        n[:, Ny // 4:Ny // 2, Nx // 3:2 * Nx // 3] = 4.0
        return tuple(n)
    for k, f in enumerate((1.0, 1.03, 0.98)):
        n[k] = DELTA / (4.0 * kind) * f
    n[2, :, :Nx // 2] = DELTA / (4.0 * kind)  # exactly that angle in half of the lattice
    return tuple(n)


def reference(n, q, sequence, potential="unitary", steps=STEPS):
    theta, beta = oracle.angles(*n, DELTA)
    ref = np.array(q, dtype=np.float64)
    oracle.run(ref, theta, beta, steps, oracle.SEQ_INTERLEAVED if sequence == "interleaved" else oracle.SEQ_PLAIN,
               oracle.POT_PAPER if potential == "paper" else oracle.POT_UNITARY)
    return ref


def state(Nx, Ny, seed=4):
    return np.random.default_rng(seed).standard_normal((6, Ny, Nx)).astype(np.float32)


def run(n, q, steps=STEPS, **kw):
    with Simulation(*n, DELTA, **kw) as sim:
        sim.set_fields(q)
        sim.step(steps)
        return sim.get_fields()


def check(got, ref, precision):
    assert np.linalg.norm(got - ref) < TOL[precision] * np.linalg.norm(ref)


@pytest.mark.parametrize("kind", [0.45, 0.55, 1.0, 3.0, 3.1415, math.pi, 4.0, "jump"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("sequence", ["interleaved", "plain"])
def test_unitary_steps_match_oracle(kind, precision, sequence):
    Nx, Ny = 260, 40
    n, q = medium(kind, Nx, Ny), state(Nx, Ny)
    ref = reference(n, q, sequence)
    for K in (1, 2):
        check(run(n, q, precision=precision, sequence=sequence, potential="unitary", steps_per_pass=K), ref, precision)


@pytest.mark.parametrize("kind", [3.0, 3.1415])
def test_other_forms(kind):
    """Rows that are copied element by element, one family, single operators, the
    shared-memory sweep (asked for by the persistent launch form), FP64 with the
    printed potentials."""
    n, q = medium(kind, 261, 37), state(261, 37)
    check(run(n, q, potential="unitary"), reference(n, q, "interleaved"), "fp32")
    n, q = medium(kind, 264, 37), state(264, 37)
    check(run(n, q, precision="fp64"), reference(n, q, "interleaved", "paper"), "fp64")
    both = run(n, q, potential="unitary")
    ref = reference(n, q, "interleaved")
    check(run(n, q, potential="unitary", launch="persistent"), ref, "fp32")
    for fam, mine in (("TM", [2, 3, 4]), ("TE", [0, 1, 5])):
        q1 = np.zeros_like(q)
        q1[mine] = q[mine]
        assert np.array_equal(run(n, q1, potential="unitary", families=fam)[mine], both[mine])
    with Simulation(*n, DELTA, potential="unitary") as sim:
        sim.set_fields(q)
        for op in ("CX", "CX_T", "CY", "CY_T"):
            sim.debug_apply(op)  # C followed by its transpose
        check(sim.get_fields(), q, "fp32")


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_narrow_lattice_on_pair_planes(precision):
    """So tall and narrow that its coefficients stay in pair planes."""
    Nx, Ny = 8, 132000
    n, q = medium(3.0, Nx, Ny), state(Nx, Ny)
    check(run(n, q, 3, precision=precision, potential="unitary"), reference(n, q, "interleaved", steps=3), precision)


@pytest.mark.parametrize("sequence", ["interleaved", "plain"])
def test_batch_of_both_kinds_is_bit_identical_to_single_runs(sequence):
    inst, single = [], []
    for k, kind in enumerate((3.0, None, math.pi, 0.45)):
        Nx, Ny = 128 + 36 * k, 50 + 7 * k
        n = media.smooth_periodic_medium(Nx, Ny, seed=k, amp=0.3) if kind is None else medium(kind, Nx, Ny)
        inst.append({"n": n, "delta": DELTA, "nsteps": 8, "pulse": ("Ez", Nx / 3, 9.0, 1.0)})
        with Simulation(*n, DELTA, potential="unitary", sequence=sequence) as sim:
            sim.init_pulse("Ez", Nx / 3, 9.0, 1.0)
            sim.step(8)
            single.append(sim.get_fields(np.float32))
    with Batch(inst, potential="unitary", sequence=sequence, steps_per_pass=2) as b:
        b.run()
        for k, ref in enumerate(single):
            assert np.array_equal(b.get_fields(k), ref), k
