"""Simulators of different lattices side by side."""
import numpy as np
import pytest

import synth
from oracle import OracleLattice, Couplings
from oracle import core as O

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("xpass", [0, 1, 2])
def test_a_smaller_lattice_leaves_a_larger_one_working(dtype, xpass):
    """The 13-qubit lattice has a phase table of 24 entries, the 16-qubit one of 153: whatever the
    second one sets up, the first one's launches go through and match the oracle."""
    import torch
    from paper_2108_13410_gb300 import Simulator, QS_OPT_XPASS
    lat = OracleLattice(4, 2, True, "ug")
    big = Simulator(4, 2, form="ug", dtype=dtype)
    psi0 = synth.random_state(16, seed=12)
    big.upload(torch.from_numpy(psi0.reshape(1, -1)).to(torch.complex64 if dtype == "c64" else torch.complex128))
    small = Simulator(2, 1, form="gh", dtype=dtype, boundary="open")
    for sim in (big, small):
        sim.set_option(QS_OPT_XPASS, xpass)
    small.init_plus()
    small.evolve([(0.3, 0.3)], [0.5, 0.6], 0.1, 2)
    s = O.schedule_linear(0.5, 5)
    big.evolve([(0.6, 0.5)], s, 0.1, 2)
    ref = O.evolve(lat, Couplings(0.6, 0.5), s, 0.1, 2, psi0=psi0)
    tol = 1e-5 if dtype == "c64" else 1e-10
    assert np.linalg.norm(big.download()[0].numpy() - ref) <= tol
    e = big.energy([(0.6, 0.5)])[0]         # |H| <= 3 * 16 + 8 terms
    assert abs(e - O.energy(ref, lat, Couplings(0.6, 0.5))) <= 2 * 56 * tol


@gpu
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_gradients_with_a_smaller_lattice_beside(dtype):
    from paper_2108_13410_gb300 import Simulator
    s = O.schedule_linear(0.8, 8)
    out = []
    for beside in (False, True):
        big = Simulator(3, 2, form="gh", dtype=dtype, aux=True)
        if beside:
            small = Simulator(2, 1, form="gh", dtype=dtype, boundary="open")
            small.init_plus()
        big.init_plus()
        out.append(big.adjoint_grad([(0.7, 0.4)], s, 0.1, 2))
    for a, b in zip(*out):
        assert np.array_equal(np.asarray(a), np.asarray(b))
