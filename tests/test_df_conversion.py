"""Double-float passes of complex128 calls: the conversion from and to complex128 belongs to the
first and the last pass only.

On the CPU: the passes between, which a long call consists of, compile without registers spilled
for a conversion (at most the 8 bytes that the merged Walsh-Hadamard pass always spilled).  On
the GPU: calls whose first, last and only passes convert, in every combination, against the
oracle: runs cut at every step by renormalisation leave single passes that do both."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

import synth
from oracle import OracleLattice, Couplings
from oracle import core as O

gpu = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_inner_passes_do_not_pay_for_the_conversion(tmp_path):
    from paper_2108_13410_gb300.build import ARCH, CSRC, INCLUDE, nvcc
    if not (os.path.exists(nvcc()) or shutil.which(nvcc())):
        pytest.skip("no nvcc")
    src = tmp_path / "inner.cu"
    src.write_text('#include "xpass_df.cuh"\nvoid *inner[] = {%s};\n' % ", ".join(
        "(void *)qsim::k_xpass_df<%s, %s, 0>" % (m, r) for m in ("false", "true") for r in ("false", "true")))
    r = subprocess.run([nvcc(), "-O3", "-std=c++17", *ARCH, "-I" + INCLUDE, "-I" + CSRC, "--expt-relaxed-constexpr",
                        "-Xptxas", "-v", "-cubin", "-o", str(tmp_path / "inner.cubin"), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    spills = {(m, rot): int(n) for m, rot, n in
              re.findall(r"k_xpass_dfILb(\d)ELb(\d)ELi0E.*?(\d+) bytes spill stores", r.stdout + r.stderr, flags=re.S)}
    assert spills == {("0", "0"): 0, ("0", "1"): 0, ("1", "0"): spills[("1", "0")], ("1", "1"): 0}
    assert spills[("1", "0")] <= 8


@gpu
@pytest.mark.parametrize("order,steps,renorm", [(1, 1, 0), (2, 3, 0), (2, 3, 1), (1, 3, 1), (2, 4, 2)])
@pytest.mark.parametrize("form,Lx,Ly,periodic,batch", [("gh", 2, 1, False, 1), ("gh", 3, 2, True, 2),
                                                       ("ug", 4, 2, True, 1), ("ug", 7, 1, False, 1)])
def test_converting_passes_match_the_oracle(form, Lx, Ly, periodic, batch, order, steps, renorm):
    import torch
    from paper_2108_13410_gb300 import Simulator, QS_OPT_RENORM_EVERY, QS_OPT_XPASS
    lat = OracleLattice(Lx, Ly, periodic, form)
    sim = Simulator(Lx, Ly, form=form, dtype="c128", boundary="periodic" if periodic else "open", batch=batch)
    psi0 = np.atleast_2d(synth.random_state(lat.n_qubits, seed=6, batch=batch))
    sim.upload(torch.from_numpy(psi0).to(torch.complex128))
    sim.set_option(QS_OPT_XPASS, 2)
    sim.set_option(QS_OPT_RENORM_EVERY, renorm)
    s = O.schedule_linear(0.1 * steps, steps)
    cpl = [(0.4 + 0.3 * b, 0.7 - 0.2 * b) for b in range(batch)]
    sim.evolve(cpl, s, 0.1, order)
    got = sim.download().numpy()
    for b, (g, lam) in enumerate(cpl):
        ref = O.evolve(lat, Couplings(g, lam), s, 0.1, order, psi0=psi0[b])
        assert np.linalg.norm(got[b] - ref) <= 1e-10
        assert np.max(np.abs(got[b] - ref)) <= 1e-10 * np.max(np.abs(ref))
