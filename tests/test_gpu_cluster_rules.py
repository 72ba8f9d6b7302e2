"""Cluster stepping: the norm carry inside the launch, and which samples take it
by default."""
import math

import numpy as np
import pytest

from tbpm_inputs import lattice, rng

pytestmark = pytest.mark.gpu
Z = math.pi / 2
PER_TERM = 8257            # ZIGZAG | WIDE | PREFETCH: the default's kernels, asked for by hand


# FP32 states whose norm drifts past the bound now and then (5e-7: 8e-9 a step)
# step on in the launch and equal the per-term kernels' bit for bit, C and the
# norms within the rounding of their sums (1e-12); one to eight rows a thread,
# a resumed run, the largest number of states
@pytest.mark.parametrize("S,sides,sigma", [(1, (20, 31), 0.0), (4, (64, 64), 0.05), (16, (40, 51), 0.0),
                                           (3, (128, 129), 0.05), (2, (180, 182), 0.0)])
def test_norm_carry_acts_in_the_launch(S, sides, sigma):
    import paper_2209_00806_gb300 as tb
    from paper_2209_00806_gb300 import _native as N
    smp = lattice.graphene(*sides, pbc=True, seed=6, onsite_w=1.0, bond_sigma=sigma)
    theta = rng.phases(15, S, smp.n_orb)
    out = []
    for variant in (PER_TERM, None):
        with tb.Propagator() as p:
            if variant is not None:
                p.launch_config(tb.TBPM_FP32, 16, 64, variant)
            N.tbpm_set_norm_policy(p.ctx, 5e-7)
            p.build_sample(smp, 9.5)
            p.set_phase_states(theta)
            C = p.propagate(Z, 260, tb.TBPM_FP32)
            a = p.stats()
            res = [C, p.norms(), p.states()]
            D = p.propagate(Z, 150, tb.TBPM_FP32, flags=N.TBPM_PROP_RESUME)
            b = p.stats()
            out.append((res + [D, p.norms(), p.states()], a, b))
    (ref, ra, rb), (got, ga, gb) = out
    assert ra["renormalisations"] == ga["renormalisations"] > 0
    assert rb["renormalisations"] == gb["renormalisations"]
    # one launch for the steps of each run, not the per-term kernels' 15 a step
    assert ra["kernel_launches"] > 260 * 15 and ga["kernel_launches"] < 60 > gb["kernel_launches"]
    for k in (2, 5):
        assert np.array_equal(ref[k], got[k])
    for k in (0, 1, 3, 4):
        assert np.abs(ref[k] - got[k]).max() < 1e-12


# the last step's drift, and the steps around it: runs that end before, at and
# after the step that drifts past the bound
def test_norm_carry_at_the_end_of_a_run():
    import paper_2209_00806_gb300 as tb
    from paper_2209_00806_gb300 import _native as N
    smp = lattice.graphene(20, 31, pbc=True, seed=6, onsite_w=1.0)
    theta = rng.phases(15, 1, smp.n_orb)

    def run(variant, steps):
        with tb.Propagator() as p:
            if variant is not None:
                p.launch_config(tb.TBPM_FP32, 16, 64, variant)
            N.tbpm_set_norm_policy(p.ctx, 5e-7)
            p.build_sample(smp, 9.5)
            p.set_phase_states(theta)
            p.propagate(Z, steps, tb.TBPM_FP32)
            return p.states(), p.norms(), p.stats()["renormalisations"]

    nn = run(PER_TERM, 260)[1][0, 0]
    first = int(np.argmax(np.abs(nn / nn[0] - 1) > 5e-7))
    assert first > 3
    for steps in (first - 1, first, first + 1, first + 2):
        (a, na, ca), (b, nb, cb) = run(PER_TERM, steps), run(None, steps)
        assert ca == cb == (steps >= first)
        assert np.array_equal(a, b) and np.abs(na - nb).max() < 1e-12


# which samples step in clusters by default: rows in lattice order do, the same
# lattice in an order that spreads every neighbour over the blocks does only
# where it is small; the states are the per-term kernels' either way
@pytest.mark.parametrize("precision,kind,S,cluster", [
    (0, (64, 64), 1, True), (0, (64, 64), 8, True), (0, "shuffled 64", 1, False),
    (0, "shuffled 22", 1, True), (0, "ragged", 1, False), (0, "ragged", 3, True),
    (1, (64, 64), 16, True), (1, (180, 180), 7, True), (1, "shuffled 180", 1, False),
    (1, "shuffled 64", 8, False), (1, "shuffled 22", 4, True), (1, "ragged", 16, False)])
def test_cluster_default_by_row_order(precision, kind, S, cluster):
    import paper_2209_00806_gb300 as tb
    if kind == "ragged":
        smp = lattice.random_graph(8000, 12000, seed=9, onsite_w=1.0, t_scale=0.8)
    elif isinstance(kind, str):
        L = int(kind.split()[1])
        smp = lattice.graphene(L, L, pbc=True, seed=6, onsite_w=1.0)
        smp = lattice.permute(smp, np.random.default_rng(3).permutation(smp.n_orb))
    else:
        smp = lattice.graphene(*kind, pbc=True, seed=6, onsite_w=1.0)
    theta = rng.phases(4, S, smp.n_orb)
    out = []
    for variant in (1, None):
        with tb.Propagator() as p:
            if variant is not None:
                p.launch_config(precision, 8, 64, variant)
            p.build_sample(smp, 12.0)
            C = _run_states(p, theta, precision)
            out.append((C, p.states(), p.stats()["kernel_launches"]))
    (Ca, a, la), (Cb, b, lb) = out
    assert np.array_equal(a, b) and np.abs(Ca - Cb).max() < 1e-12
    assert la > 6 * 15 and (lb < 6 * 15) == cluster


def _run_states(p, theta, precision):
    p.set_phase_states(theta)
    return p.propagate(Z, 6, precision)
