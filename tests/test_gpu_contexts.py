"""What calls on one context, and contexts in several threads, keep and share."""
import math

import numpy as np
import pytest

from tbpm_inputs import lattice, rng

pytestmark = pytest.mark.gpu
Z = math.pi / 2


def _run(p, theta, steps, precision):
    p.set_phase_states(theta)
    return p.propagate(Z, steps, precision), p.states(), p.norms()


# another number of states with the same number of steps: a fresh context's
# results, stepped in clusters (the default here) and term by term
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("variant", [None, 1])
def test_other_number_of_states_same_steps(precision, variant):
    import paper_2209_00806_gb300 as tb
    smp = lattice.graphene(12, 9, pbc=True, seed=6, onsite_w=1.0)
    theta = rng.phases(15, 16, smp.n_orb)

    def context():
        p = tb.Propagator()
        if variant is not None:
            p.launch_config(precision, 8, 64, variant)
        return p.build_sample(smp, 9.5)

    with context() as p:
        for S in (1, 16, 2, 5):
            got = _run(p, theta[:S], 9, precision)
            with context() as q:
                for a, b in zip(got, _run(q, theta[:S], 9, precision)):
                    assert np.array_equal(a, b)
