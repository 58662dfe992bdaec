"""complex64 observables against sums in 64 bits of the same amplitudes.

Products of floats and the sums of a thread's sixteen amplitudes are kept in two floats, sums beyond
that in FP64: at most 2^-48 per amplitude and thread, of which a thread takes fewer than 2^10 here,
so 2^-38 = 3.7e-12 of the sum of the terms' magnitudes (1 for a string, the number of terms for
their sum).  The single-qubit X terms of an energy beyond 20 qubits are chains of FP32 products
and not in here."""
import numpy as np
import pytest

import synth
from oracle import OracleLattice

gpu = pytest.mark.gpu
TOL = 2.0 ** -38


@gpu
@pytest.mark.parametrize("kind", ["random", "smooth", "evolved"])
@pytest.mark.parametrize("form,Lx,Ly,periodic", [("ug", 2, 2, True), ("gh", 1, 1, False), ("gh", 2, 2, True), ("gh", 2, 1, False),
                                                 ("ug", 4, 2, True), ("gh", 3, 2, True), ("ug", 5, 2, True)])
def test_sums_hold_more_than_single_precision(form, Lx, Ly, periodic, kind):
    import torch
    from paper_2108_13410_gb300 import Simulator, QS_NORM, QS_PLAQUETTE, QS_X
    lat = OracleLattice(Lx, Ly, periodic, form)
    n = lat.n_qubits
    sim = Simulator(Lx, Ly, form=form, dtype="c64", boundary="periodic" if periodic else "open")
    if kind == "evolved":
        sim.init_plus()
        sim.evolve([(0.7, 0.4)], [0.1, 0.2, 0.3, 0.4], 0.1, 2)
    else:
        psi = synth.random_state(n, seed=21)
        if kind == "smooth":
            psi = 0.1 * psi + 0.77 * 2.0 ** (-n / 2)
        sim.upload(torch.from_numpy(psi.reshape(1, -1)).to(torch.complex64))
    x = sim.download()[0].numpy().astype(np.complex128)
    p = x.real ** 2 + x.imag ** 2
    idx = np.arange(1 << n)
    sign = lambda m: 1.0 - 2.0 * (np.bitwise_count(idx & m) & 1)
    zsum = lambda ms: sum(float(np.sum(p * sign(int(m)))) for m in ms)
    xval = lambda m: float(np.sum((x.conj() * x[idx ^ m]).real))
    assert abs(sim.expect(QS_NORM)[0] - p.sum()) <= TOL
    for m in (1, 1 << (n - 1), 0b101, (1 << n) - 1):
        assert abs(sim.expect_pauli(0, m)[0] - zsum([m])) <= TOL
        assert abs(sim.expect_pauli(1, m)[0] - xval(m)) <= TOL
    assert abs(sim.expect(QS_X, n // 2)[0] - xval(1 << (n // 2))) <= TOL
    plaq, second = [int(m) for m in lat.z_plaquettes()], [int(m) for m in lat.z_second()]
    assert abs(sim.expect(QS_PLAQUETTE, -1)[0] - zsum(plaq) / len(plaq)) <= TOL
    assert abs(sim.energy([(0.0, 0.0, 0.0, 1.0)])[0] + zsum(plaq)) <= len(plaq) * TOL
    assert abs(sim.energy([(0.0, 1.0, 0.0, 0.0)])[0] + zsum(second)) <= len(second) * TOL
    xs = [q for q, kind in lat.x_single() if kind == "s"]
    assert abs(sim.energy([(1.0, 0.0, 0.0, 0.0)])[0] + sum(xval(1 << q) for q in xs)) <= len(xs) * TOL
    if form == "gh":
        xt = [q for q, kind in lat.x_single() if kind == "t"]
        assert abs(sim.energy([(0.0, 0.0, 1.0, 0.0)])[0] + sum(xval(1 << q) for q in xt)) <= len(xt) * TOL
    if form == "ug":
        stars = [int(m) for m in lat.x_strings()]
        assert abs(sim.energy([(0.0, 0.0, 1.0, 0.0)])[0] + sum(xval(m) for m in stars)) <= len(stars) * TOL
    other = torch.from_numpy(synth.random_state(n, seed=22).reshape(1, -1)).to(torch.complex64)
    want = abs(np.sum(other[0].numpy().astype(np.complex128).conj() * x)) ** 2
    assert abs(sim.fidelity(other.cuda())[0] - want) <= 4 * TOL
