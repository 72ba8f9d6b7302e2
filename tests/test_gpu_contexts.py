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


# contexts of different sample sizes stepping at the same time in two threads:
# the single-thread results (cluster stepping in both precisions, row groups
# of the staged gathers)
@pytest.mark.parametrize("kind", ["cluster64", "cluster32", "groups"])
def test_two_threads_step_different_samples(kind):
    from concurrent.futures import ThreadPoolExecutor

    import paper_2209_00806_gb300 as tb
    from tbpm_inputs import tbg
    if kind == "groups":
        smps = [tbg.to_numpy_sample(tbg.twisted_bilayer(x)) for x in (4.0, 9.0)]
    else:
        sides = ((40, 41), (64, 64)) if kind == "cluster64" else ((70, 71), (128, 128))
        smps = [lattice.graphene(*s, pbc=True, seed=2, onsite_w=1.0, bond_sigma=0.05) for s in sides]
    precision = 0 if kind == "cluster64" else 1

    def work(smp, repeats):
        theta = rng.phases(3, 4, smp.n_orb)
        with tb.Propagator() as p:
            if kind == "groups":
                p.launch_config(precision, 8, 64, 4609)       # ZIGZAG | HALO | STAGED
            p.build_sample(smp, 13.0)
            return [_run(p, theta, 3, precision) for _ in range(repeats)]

    alone = [work(smp, 1)[0] for smp in smps]
    with ThreadPoolExecutor(2) as ex:
        both = list(ex.map(lambda smp: work(smp, 60), smps))
    for ref, runs in zip(alone, both):
        for got in runs:
            for a, b in zip(ref, got):
                assert np.array_equal(a, b)
