"""The autotuner's shape, set by hand in another context, runs the kernels it timed."""
import math

import pytest

from tbpm_inputs import lattice, rng, tbg

pytestmark = pytest.mark.gpu
Z = math.pi / 2


# long rows, whose register-pipelined candidates are the staged gathers once the
# lists are there, on a rebuilt matrix and in a fresh context, where they are not
# yet (the bytes of a term tell the kernels apart); small FP64 samples in clusters
# (the launches of a run)
@pytest.mark.parametrize("precision,kind,S", [(0, (30, 31), 3), (1, 20.0, 8), (1, 12.0, 5), (1, 12.0, 16),
                                              (1, 9.0, 2)])
def test_returned_shape_runs_what_was_timed(precision, kind, S):
    import paper_2209_00806_gb300 as tb
    if isinstance(kind, float):
        smp = tbg.to_numpy_sample(tbg.twisted_bilayer(kind))
    else:
        smp = lattice.graphene(*kind, pbc=True, seed=6, onsite_w=1.0)
    theta = rng.phases(4, S, smp.n_orb)

    def ran(p):
        p.propagate(Z, 2, precision)
        st = p.stats()
        return st["kernel_launches"], st["bytes_term"], st["group_width"]

    with tb.Propagator() as p:
        p.build_sample(smp, 13.0)
        p.set_phase_states(theta)
        best = p.autotune(Z, precision=precision, probe_steps=3)
        tuned = ran(p)
        p.build_sample(smp, 13.0)            # a rebuilt matrix, the shape kept
        p.set_phase_states(theta)
        again = ran(p)
    with tb.Propagator() as q:
        q.launch_config(precision, best["group"], best["threads"], best["variant"])
        q.build_sample(smp, 13.0)
        q.set_phase_states(theta)
        assert ran(q) == tuned == again
