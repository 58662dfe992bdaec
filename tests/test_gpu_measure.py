"""Observables against the oracle and plain numpy at the edges of the reduction kernels: states
smaller than a tile (4 to 11 qubits), one tile, several tiles with one to three X passes, link
bits that straddle the register bits of a tile (8, 10 and 17 links), every X-string top bit.

Tolerances: complex64 observables of norm <= 1 3e-6, energies 1.2e-6 of the Hamiltonian norm
(the parity tests' ones); complex128 1e-12 of the same."""
import numpy as np
import pytest

import synth
from oracle import OracleLattice, Couplings
from oracle import core as O

gpu = pytest.mark.gpu

LATTICES = [("ug", 1, 1, False), ("ug", 2, 2, True), ("gh", 1, 1, False), ("ug", 3, 1, False), ("gh", 2, 2, True),
            ("gh", 2, 1, False), ("ug", 3, 2, False), ("gh", 3, 2, True), ("ug", 5, 2, True), ("gh", 2, 2, False)]


@gpu
@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("form,Lx,Ly,periodic", LATTICES)
def test_observables(form, Lx, Ly, periodic, dtype):
    import torch
    from paper_2108_13410_gb300 import Simulator, QS_NORM, QS_PLAQUETTE, QS_WILSON, QS_X
    lat = OracleLattice(Lx, Ly, periodic, form)
    n, B = lat.n_qubits, 2
    sim = Simulator(Lx, Ly, form=form, dtype=dtype, boundary="periodic" if periodic else "open", batch=B)
    tdt = torch.complex64 if dtype == "c64" else torch.complex128
    psi = synth.random_state(n, seed=9, batch=B) + 0.5 * 2.0 ** (-n / 2)
    psi /= np.linalg.norm(psi, axis=1, keepdims=True)
    host = torch.from_numpy(psi).to(tdt)
    sim.upload(host)
    psi = host.numpy().astype(np.complex128)
    tol = 3e-6 if dtype == "c64" else 1e-12
    cpl = [(0.7, 0.3), (0.2, 1.1)]
    hnorm = 3.0 * 2 * n
    e, es = sim.energy(cpl), sim.energy(cpl, s=0.4)
    norm, plaq = sim.expect(QS_NORM), sim.expect(QS_PLAQUETTE, 0)
    dos = sim.dos()
    other = synth.random_state(n, seed=10, batch=B)
    ref = torch.from_numpy(other).to(tdt).cuda()
    fid = sim.fidelity(ref)
    xs = [sim.expect(QS_X, q) for q in range(n)]
    zstr = sim.expect_pauli(0, (1 << n) - 1)
    z0, x0 = sim.expect_pauli(0, 0), sim.expect_pauli(1, 0)
    xstr = sim.expect_pauli(1, (1 << n) - 1)
    idx = np.arange(1 << n)
    pop = np.array([bin(i).count("1") for i in range(1 << n)]) if n <= 16 else np.bitwise_count(idx)
    for b, (g, lam) in enumerate(cpl):
        c = Couplings(g, lam)
        p = np.abs(psi[b]) ** 2
        assert abs(e[b] - O.energy(psi[b], lat, c)) <= (1.2e-6 if dtype == "c64" else 1e-12) * hnorm
        assert abs(es[b] - O.energy(psi[b], lat, c, 0.4)) <= (1.2e-6 if dtype == "c64" else 1e-12) * hnorm
        assert abs(norm[b] - p.sum()) <= tol and abs(z0[b] - p.sum()) <= tol and abs(x0[b] - p.sum()) <= tol
        assert abs(zstr[b] - np.sum(p * (1 - 2.0 * (pop & 1)))) <= tol
        assert abs(xstr[b] - np.vdot(psi[b], psi[b][::-1]).real) <= tol
        for q in range(n):
            assert abs(xs[q][b] - np.vdot(psi[b], psi[b][idx ^ (1 << q)]).real) <= tol
        links = (1 << (dos.shape[1] - 1)) - 1
        k = np.bitwise_count(idx & links)
        want = np.bincount(k, weights=p, minlength=dos.shape[1])
        assert np.max(np.abs(dos[b] - want)) <= 1e-12
        r = ref[b].cpu().numpy().astype(np.complex128)
        assert abs(fid[b] - abs(np.vdot(r, psi[b])) ** 2) <= tol
    if periodic:
        assert np.all(np.isfinite(sim.expect(QS_WILSON, 0))) and np.all(np.abs(plaq) <= 1 + tol)
