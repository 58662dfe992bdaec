"""Long runs of small states on the passes over tiles (by default such runs are resident): graph
replay, renormalisation, both forms and precisions, against the oracle and against themselves."""
import numpy as np
import pytest

import synth
from oracle import OracleLattice, Couplings
from oracle import core as O

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("form,Lx,Ly,periodic", [("gh", 3, 2, True), ("ug", 3, 3, True), ("ug", 6, 1, False)])
@pytest.mark.parametrize("renorm", [0, 1, 7])
def test_graph_and_renormalisation(form, Lx, Ly, periodic, dtype, renorm):
    import torch
    from paper_2108_13410_gb300 import Simulator, QS_OPT_GRAPH, QS_OPT_RENORM_EVERY, QS_OPT_XPASS
    lat = OracleLattice(Lx, Ly, periodic, form)
    psi0 = synth.random_state(lat.n_qubits, seed=2)
    s = O.schedule_linear(0.8, 16)
    out = []
    for graph in (0, 1):
        sim = Simulator(Lx, Ly, form=form, dtype=dtype, boundary="periodic" if periodic else "open")
        sim.set_option(QS_OPT_XPASS, 2)
        sim.set_option(QS_OPT_GRAPH, graph)
        sim.set_option(QS_OPT_RENORM_EVERY, renorm)
        for _ in range(2):                      # the second run replays
            sim.upload(torch.from_numpy(psi0.reshape(1, -1)).to(sim.state.dtype))
            sim.evolve([(0.6, 0.4)], s, 0.05, 2)
            out.append(sim.download()[0].numpy().copy())
    assert all(np.array_equal(o, out[0]) for o in out)
    ref = O.evolve(lat, Couplings(0.6, 0.4), s, 0.05, 2, psi0=psi0)
    assert np.linalg.norm(out[0] - ref) <= (1e-5 if dtype == "c64" else 1e-10)
