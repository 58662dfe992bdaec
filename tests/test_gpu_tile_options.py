"""Options that name a property of the passes over 2^12 tiles keep calls on those tiles."""
import pytest

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("option,value,passes", [(None, 0, 2), ("QS_OPT_TMA_BUFFERS", 2, 3), ("QS_OPT_TMA_BUFFERS", 3, 2),
                                                 ("QS_OPT_TMA_STORE", 0, 3), ("QS_OPT_SHARED_BUFFERS", 2, 3),
                                                 ("QS_OPT_SHARED_KERNEL", 1, 3), ("QS_OPT_XPASS", 2, 3)])
def test_tile_options_at_22_qubits(option, value, passes):
    """22 qubits in the unitary gauge: two passes over 2^13 tiles, three over 2^12; records, first H
    pass(es), then 2 (passes - 1) per factor group (shared passes)."""
    import paper_2108_13410_gb300.qsim as P
    from paper_2108_13410_gb300 import Simulator
    sim = Simulator(4, 2, form="ug", dtype="c64", boundary="open")
    if option:
        sim.set_option(getattr(P, option), value)
    sim.init_plus()
    sim.launch_count()
    sim.evolve([(0.5, 0.4)], [0.3, 0.5], 0.1, 2)
    sim.sync()
    assert sim.launch_count() == 2 + (2 * passes - 2) * 3
