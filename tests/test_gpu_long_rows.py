"""Long rows of real FP32 values: which kernel a group's width takes by default."""
import math

import pytest

from tbpm_inputs import lattice, rng, tbg

pytestmark = pytest.mark.gpu
Z = math.pi / 2


# the default shape before and after the steps that pay for the lists, against
# one row a thread: every width it splits into, and rows too long for the
# one-stage staged gathers (340 entries)
@pytest.mark.parametrize("S", [1, 2, 3, 7, 16, 20, 29])
@pytest.mark.parametrize("kind", ["flake", "wide"])
def test_default_widths_are_bit_identical(S, kind):
    import torch
    import paper_2209_00806_gb300 as tb
    from paper_2209_00806_gb300 import _native as N
    if kind == "flake":
        smp, s = tbg.to_numpy_sample(tbg.twisted_bilayer(6.0, order="morton")), 13.0
    else:
        smp, s = lattice.random_graph(1500, 1500 * 170, seed=1, onsite_w=1.0, t_scale=0.05), 40.0
    theta = rng.phases(9, S, smp.n_orb)
    out = []
    for variant in (65, None):
        with tb.Propagator() as p:
            if variant is not None:
                p.launch_config(tb.TBPM_FP32, 16, 64, variant)
            p.build_sample(smp, s)
            p.set_phase_states(theta)
            for k, steps in enumerate((2, 130, 3)):
                p.propagate(Z, steps, tb.TBPM_FP32, flags=N.TBPM_PROP_RESUME if k else 0)
                phi = torch.empty((S, smp.n_orb), dtype=torch.complex128, device="cuda")
                N.tbpm_get_states(p.ctx, phi)
                out.append(phi)
    for a, b in zip(out[:3], out[3:]):
        assert (a == b).all()


# rows too long for a stage of any width (340 entries): the default keeps no lists
def test_lists_without_a_stage_are_given_back():
    import numpy as np
    import torch
    import paper_2209_00806_gb300 as tb
    n, w = 20000, 170
    i = np.repeat(np.arange(n, dtype=np.int64), w)
    j = (i + np.tile(np.arange(1, w + 1), n)) % n
    v = np.random.default_rng(1).uniform(-0.05, 0.05, n * w)
    theta = rng.phases(9, 4, n)
    with tb.Propagator() as p:
        p.build(n, None, i, j, v, 20.0)
        p.set_phase_states(theta)
        p.propagate(Z, 2, tb.TBPM_FP32)
        before = torch.cuda.mem_get_info()[0]
        p.propagate(Z, 40, tb.TBPM_FP32)
        p.propagate(Z, 40, tb.TBPM_FP32)         # 168 states x steps and 328, of 128
        # the lists and the values alone would be 41 MB
        assert before - torch.cuda.mem_get_info()[0] < 8e6
