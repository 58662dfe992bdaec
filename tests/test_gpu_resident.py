"""Resident evolution: a whole run of factor groups in one launch for small states.

The sizes sit at the edges of the tile choice: one tile smaller than, equal to and beyond
the smallest tile (4, 8, 10, 12 qubits; complex128 7 and 8), two tile sets with the widest
and the narrowest chunk (13 and 16 qubits), 2^11 and 2^12 tiles (18 and 19 qubits).
Tolerances are the ones of the tiled passes: 1e-5 of the state in complex64, 1e-10 in
complex128."""
import numpy as np
import pytest

import synth
from oracle import OracleLattice, Couplings
from oracle import core as O

gpu = pytest.mark.gpu

CASES = [  # form, Lx, Ly, periodic, dtype, batch
    ("ug", 1, 1, False, "c64", 3), ("ug", 2, 2, True, "c64", 1), ("gh", 1, 1, False, "c64", 2),
    ("ug", 3, 1, False, "c64", 1), ("gh", 2, 2, True, "c64", 5), ("ug", 3, 2, True, "c64", 2),
    ("ug", 4, 1, False, "c64", 2), ("gh", 2, 1, False, "c64", 1), ("ug", 4, 2, True, "c64", 3),
    ("ug", 3, 2, False, "c64", 1), ("gh", 3, 2, True, "c64", 2), ("ug", 3, 3, True, "c64", 1),
    ("ug", 6, 1, False, "c64", 1),
    ("ug", 2, 1, False, "c128", 2), ("ug", 2, 2, True, "c128", 1), ("gh", 1, 1, False, "c128", 1),
    ("gh", 2, 2, True, "c128", 3), ("ug", 3, 2, True, "c128", 1), ("gh", 2, 1, False, "c128", 2),
    ("ug", 4, 2, True, "c128", 2), ("gh", 3, 2, True, "c128", 1), ("ug", 3, 3, True, "c128", 1),
]


def _run(lat, form, Lx, Ly, periodic, dtype, batch, order, steps, seed, renorm=0):
    import torch
    from paper_2108_13410_gb300 import Simulator, QS_OPT_RENORM_EVERY
    sim = Simulator(Lx, Ly, form=form, dtype=dtype, boundary="periodic" if periodic else "open", batch=batch)
    psi0 = np.atleast_2d(synth.random_state(lat.n_qubits, seed=seed, batch=batch))
    tdt = torch.complex64 if dtype == "c64" else torch.complex128
    sim.upload(torch.from_numpy(psi0).to(tdt))
    if renorm:
        sim.set_option(QS_OPT_RENORM_EVERY, renorm)
    cpl = [(0.3 + 0.2 * b, 0.8 - 0.1 * b) for b in range(batch)]
    s = O.schedule_fourier(0.05 * steps, steps, synth.fourier_coeffs(4, seed=11, std=0.05))
    sim.launch_count()
    sim.evolve(cpl, s, 0.05, order)
    sim.sync()
    return psi0, cpl, s, sim


@gpu
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("form,Lx,Ly,periodic,dtype,batch", CASES)
def test_resident_run_matches_the_oracle(form, Lx, Ly, periodic, dtype, batch, order):
    lat = OracleLattice(Lx, Ly, periodic, form)
    steps = 13
    psi0, cpl, s, sim = _run(lat, form, Lx, Ly, periodic, dtype, batch, order, steps, seed=5)
    assert sim.launch_count() == 2                      # records, one launch
    got = sim.download().numpy()
    tol = 1e-5 if dtype == "c64" else 1e-10
    for b, (g, lam) in enumerate(cpl):
        ref = O.evolve(lat, Couplings(g, lam), s, 0.05, order, psi0=psi0[b])
        assert np.linalg.norm(got[b] - ref) <= tol
        assert np.max(np.abs(got[b] - ref)) <= tol * np.max(np.abs(ref))


@gpu
@pytest.mark.parametrize("form,Lx,Ly,periodic,dtype", [("gh", 3, 2, True, "c64"), ("ug", 3, 3, True, "c64"),
                                                       ("ug", 4, 2, True, "c128"), ("gh", 2, 2, True, "c64")])
def test_resident_pieces_between_renormalisations(form, Lx, Ly, periodic, dtype):
    """Renormalisation every 13 of 40 steps splits the run into pieces."""
    lat = OracleLattice(Lx, Ly, periodic, form)
    psi0, cpl, s, sim = _run(lat, form, Lx, Ly, periodic, dtype, 1, 2, 40, seed=7, renorm=13)
    ref = O.evolve(lat, Couplings(*cpl[0]), s, 0.05, 2, psi0=psi0[0])
    tol = 1e-5 if dtype == "c64" else 1e-10
    assert np.linalg.norm(sim.download()[0].numpy() - ref / np.linalg.norm(ref)) <= tol


@gpu
@pytest.mark.parametrize("form,Lx,Ly,dtype,batch", [("ug", 3, 2, "c64", 500), ("ug", 2, 2, "c128", 2100)])
def test_more_states_than_run_at_once(form, Lx, Ly, dtype, batch):
    """More states than fit the chip share the CTAs in turn (one tile each at 12 qubits, two
    tile sets on 2 CTAs at 8 qubits in complex128): the first and the last ones against the
    oracle, and equal states give equal bits wherever they ran."""
    import torch
    from paper_2108_13410_gb300 import Simulator
    lat = OracleLattice(Lx, Ly, True, form)
    sim = Simulator(Lx, Ly, form=form, dtype=dtype, batch=batch)
    psi0 = synth.random_state(lat.n_qubits, seed=3)
    sim.upload(torch.from_numpy(np.tile(psi0, (batch, 1))).to(torch.complex64 if dtype == "c64" else torch.complex128))
    s = O.schedule_linear(0.6, 12)
    sim.evolve([(0.4, 0.7)], s, 0.05, 2)
    got = sim.download().numpy()
    ref = O.evolve(lat, Couplings(0.4, 0.7), s, 0.05, 2, psi0=psi0)
    assert np.linalg.norm(got[0] - ref) <= (1e-5 if dtype == "c64" else 1e-10)
    assert all(np.array_equal(got[b], got[0]) for b in range(batch))


@gpu
@pytest.mark.parametrize("form,Lx,Ly,periodic,order", [("gh", 2, 2, True, 2), ("ug", 3, 2, True, 1), ("gh", 2, 1, False, 1),
                                                       ("gh", 3, 2, True, 2), ("ug", 6, 1, False, 2)])
def test_complex64_bits_equal_the_tiled_passes(form, Lx, Ly, periodic, order):
    """In 2^12 tiles (rotations from 12 qubits on; 12 and 19 qubits in the unitary gauge) the
    complex64 run applies the operations of the tiled passes in their order."""
    from paper_2108_13410_gb300 import Simulator, QS_OPT_XPASS
    s = O.schedule_linear(2.0, 20)
    out = []
    for xpass in (0, 2):
        sim = Simulator(Lx, Ly, form=form, dtype="c64", boundary="periodic" if periodic else "open")
        sim.set_option(QS_OPT_XPASS, xpass)
        sim.init_plus()
        sim.evolve([(0.6, 0.6)], s, 0.1, order)
        out.append(sim.download().numpy())
    assert np.array_equal(out[0], out[1])
