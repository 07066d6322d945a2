"""Batches with lattices whose strip records are not worth their memory (tall, much
narrower than a strip): these keep pair planes and the shared-memory sweep, the
others the batch kernel."""
import numpy as np
import pytest
import torch

from paper_2301_13601_gb300 import media
from paper_2301_13601_gb300.qla import Batch, Simulation

pytestmark = pytest.mark.gpu

TALL = [(4, 140000), (8, 135000), (36, 150000)]


def instance(Nx, Ny, steps, k):
    n = media.smooth_periodic_medium(Nx, Ny, seed=k, amp=0.3)
    return {"n": n, "delta": 0.2, "nsteps": steps, "pulse": (("Ez", "Ey")[k % 2], Nx / 3, max(1.0, Nx / 9), 1.0)}


# an odd and an even number of passes of the tall ones; among others, and alone
@pytest.mark.parametrize("steps, with_others", [(6, True), (8, True), (6, False)])
@pytest.mark.parametrize("sequence, potential", [("interleaved", "paper"), ("plain", "unitary")])
def test_bit_identical_to_single_lattices(steps, with_others, sequence, potential):
    inst = [instance(Nx, Ny, steps, k) for k, (Nx, Ny) in enumerate(TALL)]
    if with_others:
        inst = inst[:1] + [instance(128, 100, 4, 5)] + inst[1:] + [instance(300, 64, 12, 6)]
    before = torch.cuda.mem_get_info()[0]
    with Batch(inst, steps_per_pass=2, sequence=sequence, potential=potential) as b:
        assert b.info()["site_updates"] == sum(i["n"][0].size * i["nsteps"] for i in inst)
        used = before - torch.cuda.mem_get_info()[0]
        b.run()
        b.run()  # graph replay
        got = [b.get_fields(i) for i in range(len(inst))]
        energy = [b.diagnostics(i)["energy"] for i in range(len(inst))]
    sites = sum(i["n"][0].size for i in inst)
    assert used < 300 * sites + (1 << 29)  # records: 1.1 to 1.2 GB for each tall lattice
    for k, ins in enumerate(inst):
        with Simulation(*ins["n"], 0.2, sequence=sequence, potential=potential) as sim:
            sim.init_pulse(*ins["pulse"])
            sim.step(2 * ins["nsteps"])
            assert np.array_equal(got[k], sim.get_fields(np.float32)), k
            assert energy[k] == sim.energy()
