"""The X-pass autotuner times the form that the default configuration takes in long calls."""
import pytest

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("n_steps", [3, 4, 10])
@pytest.mark.parametrize("form,Lx,Ly,periodic,dtype", [("ug", 3, 3, True, "c64"), ("gh", 3, 2, True, "c64"),
                                                       ("ug", 4, 2, True, "c128")])
def test_few_steps_do_not_switch_the_resident_form_off(form, Lx, Ly, periodic, dtype, n_steps):
    """3 to 10 steps are 4 to 11 factor groups, which run pass by pass beyond 12 qubits; the form
    of a long call (records and one launch; 0.5 to 0.8 of the time) has to win all the same."""
    from paper_2108_13410_gb300 import Simulator
    sim = Simulator(Lx, Ly, form=form, dtype=dtype, boundary="periodic" if periodic else "open")
    e = sim.autotune(n_steps=n_steps, cache=False)
    assert e["xpass"] == 0
    sim.init_plus()
    sim.launch_count()
    sim.evolve([(0.5, 0.4)], [0.4] * 20, 0.05, 2)
    sim.sync()
    assert sim.launch_count() == 2
