"""Unitary-gauge passes over tiles of 2^13 amplitudes, where they save passes: 22 qubits (two
passes, a window of nine), 30 and 31 (three passes, a window that starts on qubits already
done), 32 (windows of ten, on 64-byte rows, and nine).  22 qubits against the oracle, the others
against the passes over 2^12 tiles, each within the complex64 tolerance 1e-5."""
import numpy as np
import pytest

import synth
from oracle import OracleLattice, Couplings
from oracle import core as O

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("Lx,Ly", [(4, 2), (7, 1)])
@pytest.mark.parametrize("order,steps,renorm", [(2, 3, 0), (1, 2, 0), (2, 4, 2)])
def test_22_qubits_match_the_oracle(Lx, Ly, order, steps, renorm):
    import torch
    from paper_2108_13410_gb300 import Simulator, QS_OPT_RENORM_EVERY
    lat = OracleLattice(Lx, Ly, False, "ug")
    s = O.schedule_linear(0.15 * steps, steps)
    psi0 = synth.random_state(22, seed=4)
    sim = Simulator(Lx, Ly, form="ug", dtype="c64", boundary="open")
    sim.upload(torch.from_numpy(psi0.reshape(1, -1)).to(torch.complex64))
    sim.set_option(QS_OPT_RENORM_EVERY, renorm)
    sim.launch_count()
    sim.evolve([(0.7, 0.4)], s, 0.15, order)
    sim.sync()
    groups = steps + 1 if order == 2 else steps
    if not renorm:
        assert sim.launch_count() == 2 + 2 * groups      # records, first H pass, two per group
    ref = O.evolve(lat, Couplings(0.7, 0.4), s, 0.15, order, psi0=psi0)
    got = sim.download()[0].numpy()
    assert np.linalg.norm(got - ref) <= 1e-5
    assert np.max(np.abs(got - ref)) <= 1e-5 * np.max(np.abs(ref))


@gpu
@pytest.mark.parametrize("Lx,Ly,boundary,n", [(5, 3, "periodic", 30), (4, 3, "open", 31), (4, 4, "periodic", 32)])
def test_large_lattices_agree_with_smaller_tiles(Lx, Ly, boundary, n):
    import torch
    from paper_2108_13410_gb300 import Simulator, QS_OPT_XPASS
    idx = torch.from_numpy(np.random.default_rng(6).integers(0, 1 << n, 4096)).cuda()
    amps = []
    for xpass in (0, 2):
        sim = Simulator(Lx, Ly, form="ug", dtype="c64", boundary=boundary)
        sim.set_option(QS_OPT_XPASS, xpass)
        sim.init_plus()
        sim.state[0, : 1 << 20] *= 1.5                    # not symmetric under the lattice
        sim.launch_count()
        sim.evolve([(0.5, 0.7)], [0.2, 0.5, 0.8], 0.1, 2)
        sim.sync()
        assert sim.launch_count() == 2 + (4 if xpass == 0 else 6) * 4
        amps.append(sim.state[0, idx].cpu().numpy().astype(np.complex128))
        del sim
        torch.cuda.empty_cache()
    assert np.max(np.abs(amps[0] - amps[1])) <= 1e-5 * np.max(np.abs(amps[1]))
