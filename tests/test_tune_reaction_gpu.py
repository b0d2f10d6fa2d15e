"""The autotuner's cached choice belongs to the reaction it was timed with: a
handle starts from its own reaction's, a general handle never from another's where
the rule by size has a choice, and the other kernels from the last of their shape."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B
from paper_1007_3109_gb300 import inputs

pytestmark = pytest.mark.gpu

NX, NY = 524, 388  # a shape that no other test tunes


def _general(reaction, **kw):
    return B.Simulation("D2Q9", 4, NX, NY, [0.8, 0.65] * 2, reaction, precision="fp32", **kw)


def _variant(sim):
    return B.lb_rd_handle_variant_name(sim.h, B.lb_rd_get_variant(sim.h))


def test_network_handle_keeps_the_rule_by_size():
    net = inputs.coupled_gs_network()
    with _general("mass_action", network=net) as sim:
        untuned = _variant(sim)
    with _general("none") as sim:
        sim.init(np.full((4, NY, NX), 0.3))
        # a choice that the rule would not make
        other = next(v for v in range(B.lb_rd_handle_variant_count(sim.h)) if B.variant_steps(
            B.lb_rd_handle_variant_name(sim.h, v)) > 1 and B.lb_rd_handle_variant_name(sim.h, v) != untuned)
        sim.autotune(3)
        tuned = _variant(sim)
        sim.set_variant(other)
        sim.set_variant(-1)
        assert _variant(sim) == tuned
    for n in (10, 4):  # networks of three groups of four steps, and of one
        with _general("mass_action", network=tuple(x[:n] for x in net)) as sim:
            assert _variant(sim) == untuned
            sim.set_variant(0)
            sim.set_variant(-1)
            assert _variant(sim) == untuned
    with _general("none") as sim:
        assert _variant(sim) == tuned


def test_each_reaction_keeps_its_choice():
    nx, ny = 236, 124
    kw = dict(F=0.04, k=0.06)

    def make(reaction, **k):
        return B.Simulation("D2Q9", 2, nx, ny, [0.8, 0.65], reaction, precision="fp32", **k)

    with make("none") as sim:
        sim.init(np.full((2, ny, nx), 0.3))
        sim.autotune(3)
        first = _variant(sim)
    with make("gray_scott", **kw) as sim:  # not tuned itself: the last of the shape
        assert _variant(sim) == first
        sim.init(np.full((2, ny, nx), 0.3))
        sim.autotune(3)
        second = _variant(sim)
    with make("none") as a, make("gray_scott", **kw) as b, make("linear", kappa=0.1) as c:
        assert (_variant(a), _variant(b), _variant(c)) == (first, second, second)
