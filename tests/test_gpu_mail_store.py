"""Mail boxes that a destroyed simulator leaves to the next one: cleared before use, bounded, and
given back with the last simulator."""
import gc

import numpy as np
import pytest

import synth
from oracle import OracleLattice, Couplings
from oracle import core as O

gpu = pytest.mark.gpu

CASES = [("gh", 3, 2, "c64"), ("ug", 3, 3, "c128"), ("ug", 3, 3, "c64"), ("gh", 3, 2, "c128")]


def _run(form, Lx, Ly, dtype, psi0, s):
    import torch
    from paper_2108_13410_gb300 import Simulator
    sim = Simulator(Lx, Ly, form=form, dtype=dtype)
    sim.upload(torch.from_numpy(psi0.reshape(1, -1)).to(sim.state.dtype))
    sim.launch_count()
    sim.evolve([(0.6, 0.4)], s, 0.05, 2)
    sim.sync()
    assert sim.launch_count() == 2
    return sim


@gpu
def test_boxes_of_gone_simulators_are_used_again():
    """18 qubits: 4 and 8 MiB.  The next simulator of that size finds a box that another form or
    precision, or a self test that gave up, has written to."""
    from paper_2108_13410_gb300.qsim import QsError, qs_selftest_wait
    psi0, s = synth.random_state(18, seed=8), O.schedule_linear(0.6, 12)
    ref = {f: O.evolve(OracleLattice(Lx, Ly, True, f), Couplings(0.6, 0.4), s, 0.05, 2, psi0=psi0)
           for f, Lx, Ly in (("gh", 3, 2), ("ug", 3, 3))}
    keep = _run(*CASES[0], psi0, s)               # the store stays while a simulator is there
    for k in range(8):
        form, Lx, Ly, dtype = CASES[k % 4]
        sim = _run(form, Lx, Ly, dtype, psi0, s)
        assert np.linalg.norm(sim.download()[0].numpy() - ref[form]) <= (1e-5 if dtype == "c64" else 1e-10)
        if k % 3 == 1:
            with pytest.raises(QsError):
                qs_selftest_wait(sim.h, 2.0)
        del sim
        gc.collect()
    assert np.linalg.norm(keep.download()[0].numpy() - ref["gh"]) <= 1e-5


def _outside_torch():
    """Device memory in use that PyTorch's allocator does not hold (its segments are larger than the
    states in them)."""
    import torch
    gc.collect()
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free - torch.cuda.memory_reserved()


@gpu
def test_the_store_is_bounded_and_given_back():
    from paper_2108_13410_gb300 import Simulator
    psi0, s = synth.random_state(18, seed=8), O.schedule_linear(0.6, 12)
    sims = [_run(*CASES[k % 4], psi0, s) for k in range(12)]      # 72 MiB of boxes
    first = sims.pop(0)                                           # the others: 68
    used = [_outside_torch()]
    del sims
    used.append(_outside_torch())
    assert used[0] - used[1] >= (68 - 32) << 20
    del first
    used.append(_outside_torch())
    if not [o for o in gc.get_objects() if isinstance(o, Simulator) and getattr(o, "h", None)]:
        assert used[0] - used[2] >= 72 << 20
