"""The resident form's mail boxes over states, launches, streams and failures, and its rounding over
many steps.

Tolerances: 1e-5 of the state in complex64, 1e-10 in complex128, as for the tiled passes."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

import synth
from oracle import OracleLattice, Couplings
from oracle import core as O

gpu = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@gpu
@pytest.mark.parametrize("groups", [1, 2, 3, 12, 13])
@pytest.mark.parametrize("form,Lx,Ly,periodic", [("gh", 1, 1, False), ("ug", 2, 2, True)])
def test_many_states_in_turn(form, Lx, Ly, periodic, groups):
    """2100 states of 8 qubits in complex128 share the CTAs, two tiles each: a group of rotations is
    one exchange, so with an odd number of groups successive states begin on alternating boxes
    and sets.  Equal states give equal bits."""
    import torch
    from paper_2108_13410_gb300 import Simulator
    lat = OracleLattice(Lx, Ly, periodic, form)
    B = 2100
    sim = Simulator(Lx, Ly, form=form, dtype="c128", boundary="periodic" if periodic else "open", batch=B)
    psi0 = synth.random_state(lat.n_qubits, seed=3)
    sim.upload(torch.from_numpy(np.tile(psi0, (B, 1))).to(torch.complex128))
    s = O.schedule_linear(0.6, groups)
    for _ in range(2):
        sim.evolve([(0.4, 0.7)], s, 0.05, 1)
    got = sim.download().numpy()
    ref = psi0
    for _ in range(2):
        ref = O.evolve(lat, Couplings(0.4, 0.7), s, 0.05, 1, psi0=ref)
    assert np.linalg.norm(got[0] - ref) <= 1e-10
    assert np.all(got == got[0])


@gpu
@pytest.mark.parametrize("steps,order", [(1, 1), (2, 1), (3, 1), (1, 2), (2, 2)])
@pytest.mark.parametrize("form,Lx,Ly,periodic", [("gh", 2, 1, False), ("ug", 4, 2, True), ("gh", 3, 2, True), ("ug", 3, 3, True),
                                                 ("ug", 6, 1, False)])
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_one_to_three_groups(form, Lx, Ly, periodic, dtype, steps, order):
    import torch
    from paper_2108_13410_gb300 import Simulator
    lat = OracleLattice(Lx, Ly, periodic, form)
    sim = Simulator(Lx, Ly, form=form, dtype=dtype, boundary="periodic" if periodic else "open")
    psi0 = synth.random_state(lat.n_qubits, seed=4)
    sim.upload(torch.from_numpy(psi0.reshape(1, -1)).to(torch.complex64 if dtype == "c64" else torch.complex128))
    s = O.schedule_linear(0.1 * steps, steps)
    sim.launch_count()
    sim.evolve([(0.8, 0.3)], s, 0.1, order)
    assert sim.launch_count() == 2
    ref = O.evolve(lat, Couplings(0.8, 0.3), s, 0.1, order, psi0=psi0)
    assert np.linalg.norm(sim.download()[0].numpy() - ref) <= (1e-5 if dtype == "c64" else 1e-10)


@gpu
@pytest.mark.parametrize("form,Lx,Ly", [("gh", 3, 2), ("ug", 3, 3), ("ug", 4, 2)])
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_a_poll_that_runs_out(form, Lx, Ly, dtype):
    """One CTA of a run alone: it gives up (bit 1 of the flag), leaves the state as it was and its
    tile in a mail box, which the next run clears."""
    import torch
    from paper_2108_13410_gb300 import Simulator
    from paper_2108_13410_gb300.qsim import QsError, qs_selftest_wait
    lat = OracleLattice(Lx, Ly, True, form)
    sim = Simulator(Lx, Ly, form=form, dtype=dtype)
    psi0 = synth.random_state(lat.n_qubits, seed=5)
    s = O.schedule_linear(0.6, 12)
    ref = O.evolve(lat, Couplings(0.4, 0.7), s, 0.05, 2, psi0=psi0)
    host = torch.from_numpy(psi0.reshape(1, -1)).to(sim.state.dtype)
    for _ in range(2):
        sim.upload(host)
        with pytest.raises(QsError) as e:
            qs_selftest_wait(sim.h, 5.0)
        assert e.value.status == 5 and "flag 3" in str(e.value)
        assert torch.equal(sim.download(), host)
        sim.launch_count()
        sim.evolve([(0.4, 0.7)], s, 0.05, 2)
        assert np.linalg.norm(sim.download()[0].numpy() - ref) <= (1e-5 if dtype == "c64" else 1e-10)
        assert sim.launch_count() == 2


@gpu
@pytest.mark.parametrize("form,Lx,Ly", [("gh", 3, 2), ("ug", 3, 3)])
def test_boxes_are_cleared_after_a_wait_that_ran_out(form, Lx, Ly):
    """A timeout leaves the boxes in doubt: the next run clears them."""
    import torch
    from paper_2108_13410_gb300 import Simulator
    from paper_2108_13410_gb300.qsim import QsError, qs_selftest_wait
    lat = OracleLattice(Lx, Ly, True, form)
    sim = Simulator(Lx, Ly, form=form, dtype="c64")
    psi0 = synth.random_state(lat.n_qubits, seed=5)
    s = O.schedule_linear(0.6, 12)
    ref = O.evolve(lat, Couplings(0.4, 0.7), s, 0.05, 2, psi0=psi0)
    for k in range(3):
        sim.upload(torch.from_numpy(psi0.reshape(1, -1)).to(torch.complex64))
        sim.evolve([(0.4, 0.7)], s, 0.05, 2)
        assert np.linalg.norm(sim.download()[0].numpy() - ref) <= 1e-5
        if k < 2:
            with pytest.raises(QsError) as e:
                qs_selftest_wait(sim.h, 5.0)
            assert e.value.status == 5


@gpu
def test_two_simulators_on_two_streams():
    """Two 18-qubit runs at once, each of more CTAs than half of the SMs, from two threads."""
    import torch
    from paper_2108_13410_gb300 import Simulator
    s = O.schedule_linear(2.0, 40)
    cpl = [(0.6, 0.5), (0.3, 0.9)]

    def one(k):
        sim = Simulator(3, 3, form="ug", dtype="c64")
        sim.init_plus()
        for _ in range(20):
            sim.evolve([cpl[k]], s, 0.05, 2)
        return sim.download()[0].numpy().copy()

    alone = [one(0), one(1)]
    got, errors = [None, None], []

    def worker(k):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                got[k] = one(k)
        except Exception as e:   # reported by the main thread
            errors.append(e)

    ts = [threading.Thread(target=worker, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors
    assert all(np.array_equal(got[k], alone[k]) for k in range(2))


@gpu
def test_small_rotations_round_no_more_than_the_factor_kernels():
    """8 qubits in complex64, 1000 steps: about 20 roundings of 2^-24 / sqrt(3) a step that add up
    like a random walk, 5e-6 of the state; three times that, and no more than the kernels that
    apply one factor at a time."""
    from paper_2108_13410_gb300 import Simulator, QS_OPT_XPASS
    s = 0.2 + 0.5 * np.arange(1000) / 1000
    psi = {}
    for dtype, xpass in (("c128", 0), ("c64", 0), ("c64", 2)):
        sim = Simulator(1, 1, form="gh", dtype=dtype, boundary="open")
        sim.set_option(QS_OPT_XPASS, xpass)
        sim.init_plus()
        sim.evolve([(0.9, 0.6)], s, 0.1, 2)
        psi[dtype, xpass] = sim.download()[0].numpy().astype(np.complex128)
    err = [np.linalg.norm(psi["c64", x] - psi["c128", 0]) for x in (0, 2)]
    assert err[0] <= 1.5e-5 and err[0] <= err[1]


SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static size_t refuse;
void refuse_size(size_t n) { refuse = n; }
int cudaMalloc(void **p, size_t n) {
    static int (*real)(void **, size_t);
    if (!real) real = (int (*)(void **, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
    return refuse && n == refuse ? 2 : real(p, n);
}
"""
CHILD = r"""
import ctypes, sys
import numpy as np
from paper_2108_13410_gb300 import Simulator, QS_OPT_XPASS
shim = ctypes.CDLL(sys.argv[1])
shim.refuse_size.argtypes = [ctypes.c_size_t]
s = np.linspace(0.1, 0.9, 12)
def run(xpass, refuse):
    sim = Simulator(3, 2, form="gh", dtype="c64")
    sim.set_option(QS_OPT_XPASS, xpass)
    sim.init_plus()
    sim.launch_count()
    shim.refuse_size(2 * 8 << 18 if refuse else 0)
    sim.evolve([(0.5, 0.6)], s, 0.1, 2)
    a, n = sim.download()[0].numpy().copy(), sim.launch_count()
    shim.refuse_size(0)
    sim.evolve([(0.5, 0.6)], s, 0.1, 2)
    sim.sync()
    return a, n, sim.launch_count()
want, n_passes, _ = run(2, False)
got, n, after = run(0, True)
assert n == n_passes and n > 12, (n, n_passes)
assert after == 2, after
assert np.array_equal(got, want)
print("fell back")
"""


@gpu
def test_without_memory_for_the_boxes_the_passes_run(tmp_path):
    """A cudaMalloc that refuses the mail boxes' size: the call takes the passes (the same bits for
    rotations), and the next one, with memory, the resident form."""
    src, lib = tmp_path / "refuse.c", tmp_path / "librefuse.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(lib), str(src), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, str(lib)], cwd=ROOT, env=env, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "fell back" in r.stdout, r.stdout + r.stderr
