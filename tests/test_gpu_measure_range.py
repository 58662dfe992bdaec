"""Observables of complex64 states that are not normalised: what the sums of FP32 products over
runs of eight amplitudes in FP64 can hold must come out finite and to rounding."""
import numpy as np
import pytest

gpu = pytest.mark.gpu

# a run of eight: two roundings a product, seven sums, 2^-24 each
RUN_TOL = 9 * 2.0 ** -24


@gpu
@pytest.mark.parametrize("form,Lx,Ly,periodic", [("ug", 2, 2, True), ("gh", 2, 2, True), ("gh", 2, 1, False),
                                                 ("gh", 3, 2, True)])
def test_large_amplitudes(form, Lx, Ly, periodic):
    """p = 2.5e37 per amplitude: eight of them are below the largest float, sixteen are not."""
    import torch
    from paper_2108_13410_gb300 import Simulator, QS_NORM, QS_WILSON, QS_X
    sim = Simulator(Lx, Ly, form=form, dtype="c64", boundary="periodic" if periodic else "open")
    a = np.float32(5e18)
    sim.upload(torch.full((1, 1 << sim.n), complex(a, 0.0), dtype=torch.complex64))
    want = float(a) ** 2 * 2.0 ** sim.n
    assert abs(sim.expect(QS_NORM)[0] / want - 1) <= RUN_TOL
    assert abs(sim.expect_pauli(0, 0)[0] / want - 1) <= RUN_TOL
    assert abs(sim.expect_pauli(0, 1)[0]) <= RUN_TOL * want
    assert abs(sim.expect(QS_X, sim.n - 1)[0] / want - 1) <= RUN_TOL
    assert abs(sim.expect_pauli(1, (1 << sim.n) - 1)[0] / want - 1) <= RUN_TOL
    if periodic:
        assert abs(sim.expect(QS_WILSON, 0)[0]) <= RUN_TOL * want
    assert abs(sim.fidelity(sim.state)[0] / want / want - 1) <= 3 * RUN_TOL


@gpu
@pytest.mark.parametrize("form,Lx,Ly,periodic", [("ug", 2, 2, True), ("gh", 2, 1, False), ("ug", 5, 1, False),
                                                 ("gh", 3, 2, True)])
def test_density_of_states_keeps_double_precision(form, Lx, Ly, periodic):
    """complex64 weights are exact FP64 products in FP64 sums, over the whole range of a float: bins
    of amplitudes near 1e-22, 1 and 1e20 in one state, subnormal ones among them.  2^18 sums at
    most in a bin, 2^-53 each in the worst order: 3e-11; in blocks and threads at most 2^10 in a
    row, 1.2e-13."""
    import torch
    from paper_2108_13410_gb300 import Simulator
    sim = Simulator(Lx, Ly, form=form, dtype="c64", boundary="periodic" if periodic else "open")
    n = sim.n
    rng = np.random.default_rng(8)
    sim.init_plus()
    nbins = sim.dos().shape[1]
    k = np.bitwise_count(np.arange(1 << n) & ((1 << (nbins - 1)) - 1))
    size = np.array([1e-22, 1.0, 1e20, 1e-42, 3e-4])[k % 5]
    psi = (size * (rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n))).astype(np.complex64)
    psi[rng.random(1 << n) < 0.1] = 0
    sim.upload(torch.from_numpy(psi).reshape(1, -1))
    got = sim.dos()[0]
    p = psi.real.astype(np.longdouble) ** 2 + psi.imag.astype(np.longdouble) ** 2
    for j in range(nbins):
        want = p[k == j].sum()
        assert abs(got[j] - want) <= 1.2e-13 * want
