"""Launch rules of the register-pipelined variant (TBPM_VARIANT_PREFETCH): the
states equal the plain kernel's bit for bit on both sides of every rule."""
import math

import numpy as np
import pytest

from tbpm_inputs import lattice, rng

pytestmark = pytest.mark.gpu
Z = math.pi / 2
PLAIN, PREFETCH = 1, 8257          # ZIGZAG; ZIGZAG | WIDE | PREFETCH


def _states(tb, smp, theta, precision, B, variant, steps):
    import torch
    from paper_2209_00806_gb300 import _native as N
    with tb.Propagator() as p:
        p.launch_config(precision, B, 64, variant)
        p.build_sample(smp, 9.5)
        p.set_phase_states(theta)
        C = p.propagate(Z, steps, precision)
        out = torch.empty((theta.shape[0], smp.n_orb), dtype=torch.complex128, device="cuda")
        N.tbpm_get_states(p.ctx, out)
        return C, out


# rows a multiple of 1024: 2^20 lanes of 16 bytes are 2^20 / max(1, B / 2) rows
@pytest.mark.parametrize("values", ["one", "real"])
@pytest.mark.parametrize("B", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("over", [0, 1])
def test_lane_rule_is_bit_identical(B, over, values):
    import paper_2209_00806_gb300 as tb
    rows = (1 << 20) // max(1, B // 2) + 1024 * over
    smp = lattice.graphene(rows // 1024, 512, pbc=True, seed=3, onsite_w=1.0,
                           vacancy_frac=0.0 if over else 0.0003,
                           bond_sigma=0.05 if values == "real" else 0.0)
    theta = rng.phases(5, B, smp.n_orb)
    C0, a = _states(tb, smp, theta, tb.TBPM_FP32, B, PLAIN, 2)
    C1, b = _states(tb, smp, theta, tb.TBPM_FP32, B, PREFETCH, 2)
    assert (a == b).all()
    # the sums of float pairs differ in order only: 1e-12 as for the other variants
    assert np.abs(C0 - C1).max() < 1e-12


@pytest.mark.parametrize("sides", [(2048, 1024), (2049, 1024)])   # one vector of 128 MB, and above
def test_wide_lane_rule_is_bit_identical(sides):
    import paper_2209_00806_gb300 as tb
    smp = lattice.graphene(*sides, pbc=True, seed=4, onsite_w=1.0)
    theta = rng.phases(6, 4, smp.n_orb)
    C0, a = _states(tb, smp, theta, tb.TBPM_FP32, 4, PLAIN, 2)
    C1, b = _states(tb, smp, theta, tb.TBPM_FP32, 4, PREFETCH, 2)
    assert (a == b).all()
    assert np.abs(C0 - C1).max() < 1e-12


# three-slot rows (fixed slice width 3) against the TMA kernel, which reads the
# widths at run time: every matrix form, FP32 and FP64
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("B", [1, 2, 8])
@pytest.mark.parametrize("onsite_w,sigma", [(0.0, 0.0), (1.0, 0.0), (0.0, 0.05), (1.0, 0.05)])
def test_three_slot_forms_are_bit_identical(precision, B, onsite_w, sigma):
    import paper_2209_00806_gb300 as tb
    smp = lattice.graphene(23, 31, pbc=True, seed=8, onsite_w=onsite_w, bond_sigma=sigma,
                           vacancy_frac=0.01)
    theta = rng.phases(9, B, smp.n_orb)
    C0, a = _states(tb, smp, theta, precision, B, 5, 3)       # ZIGZAG | TMA
    C1, b = _states(tb, smp, theta, precision, B, PLAIN, 3)
    assert (a == b).all()
    assert np.abs(C0 - C1).max() < 1e-12


# the Fermi preparation's one-value forms against the entry-by-entry form of
# the same matrix (rounding of the FP64 preparation: 1e-10 of the largest
# value, as against the oracle), uneven samples and several quads a group
@pytest.mark.parametrize("onsite_w,mu", [(0.0, 0.0), (0.8, 0.0), (0.8, 0.3)])
def test_fermi_preparation_forms_agree(onsite_w, mu):
    import paper_2209_00806_gb300 as tb
    from paper_2209_00806_gb300 import _native as N
    parts = [lattice.graphene(L, L, pbc=True, seed=L, onsite_w=onsite_w, with_pos=True)
             for L in (8, 33)]
    smp, offs = lattice.concat(parts)
    if not onsite_w:
        smp.onsite = None
    out = []
    for flags in (0, N.TBPM_BUILD_NO_UNIFORM):
        with tb.Propagator() as p:
            p.build_sample(smp, 9.5, offs, flags=flags)
            p.set_bond_vectors(lattice.bond_vectors(smp))
            p.set_phase_states(rng.phases(11, 3, smp.n_orb))
            out.append(p.ac_correlation(Z, 6, 20.0, mu, tb.TBPM_FP64))
    assert np.abs(out[0] - out[1]).max() < 1e-10 * np.abs(out[1]).max()


# gradient kernels per group width and row form against the oracle's reverse
# mode (1e-11 of the largest, the tolerance of the adjoint tests): widths 1,
# 2 + 1, 4 and 8, three-slot rows and ragged ones, one step to several segments
@pytest.mark.parametrize("S", [1, 3, 4, 8])
@pytest.mark.parametrize("kind", ["graphene", "ragged"])
@pytest.mark.parametrize("steps,K", [(1, 1), (5, 2)])
def test_adjoint_forms(S, kind, steps, K):
    import oracle
    import paper_2209_00806_gb300 as tb
    if kind == "graphene":
        smp = lattice.graphene(9, 7, pbc=True, seed=2, onsite_w=0.5, bond_sigma=0.1)
    else:
        smp = lattice.random_graph(130, 400, seed=3, onsite_w=0.5, t_scale=0.7)
    theta = rng.phases(4, S, smp.n_orb)
    g = np.random.default_rng(5).normal(size=(1, S, steps + 1, 2)) @ np.array([1, 1j])
    with tb.Propagator() as p:
        p.build_sample(smp, 12.0)
        p.set_phase_states(theta)
        gh, go = p.adjoint(Z, steps, g, K)
    rh, ro = oracle.gradient(smp, 12.0, Z, steps, oracle.phase_states(theta), g[0])
    scale = max(np.abs(rh).max(), np.abs(ro).max())
    assert np.abs(gh - rh).max() < 1e-11 * scale
    assert np.abs(go - ro).max() < 1e-11 * scale


# quasi-eigenstate accumulation one or two lanes a thread, norms from chunk
# partials: group splits 1, 2 + 1, 4 + 2, 16 + 1, uneven samples, FP32 against
# FP64 (2e-5 of the unit norm, the tolerance of the FP32 form)
@pytest.mark.parametrize("S", [1, 3, 6, 17])
def test_quasi_lanes_and_norms(S):
    import paper_2209_00806_gb300 as tb
    parts = [lattice.graphene(L, L + 2, pbc=True, seed=L, onsite_w=1.0) for L in (5, 30)]
    smp, offs = lattice.concat(parts)
    out = []
    for precision in (tb.TBPM_FP64, tb.TBPM_FP32):
        with tb.Propagator() as p:
            p.build_sample(smp, 9.5, offs)
            p.set_phase_states(rng.phases(12, S, smp.n_orb))
            out.append(p.quasi_eigenstates(Z, 12, [0.3, -1.1], precision))
    (a, na), (b, nb) = out
    for lo, hi in zip(offs, offs[1:]):
        assert np.abs((np.abs(a[:, :, lo:hi]) ** 2).sum(-1) - 1).max() < 1e-12
        assert np.linalg.norm(a[:, :, lo:hi] - b[:, :, lo:hi], axis=-1).max() < 2e-5
    assert np.abs(nb / na - 1).max() < 2e-5


# rows in groups of four (one-stage staged gathers, FP32 values per entry)
# against the plain kernel: flakes with ragged edges, pairs listed twice, two
# uneven samples, both group widths the kernel takes, and lists too long for it
@pytest.mark.parametrize("S", [4, 8, 13])
@pytest.mark.parametrize("kind", ["flake", "layers", "twice", "batch", "random"])
def test_grouped_rows_are_bit_identical(S, kind):
    import torch
    import paper_2209_00806_gb300 as tb
    from paper_2209_00806_gb300 import _native as N
    from tbpm_inputs import tbg
    offs = None
    if kind == "random":
        smp = lattice.random_graph(700, 9000, seed=1, onsite_w=1.0, t_scale=0.2)
    else:
        smp = tbg.to_numpy_sample(tbg.twisted_bilayer(7.3, order="layers" if kind == "layers" else
                                                      "morton"))
        smp.onsite = rng.uniform_range(5, rng.ONSITE, smp.n_orb, -0.2, 0.2)
    if kind == "twice":
        again = np.arange(0, smp.n_hop, 7)
        for f in ("hop_i", "hop_j"):
            setattr(smp, f, np.concatenate([getattr(smp, f), getattr(smp, f)[again]]))
        smp.hop_v = np.concatenate([smp.hop_v, 0.01 * smp.hop_v[again]])
    if kind == "batch":
        smp, offs = lattice.concat([smp, tbg.to_numpy_sample(tbg.twisted_bilayer(4.0))])
    theta = rng.phases(7, S, smp.n_orb)
    out = []
    # ZIGZAG | WIDE; ZIGZAG | HALO | STAGED; the default
    for variant in (65, 4609, 8257):
        with tb.Propagator() as p:
            p.launch_config(tb.TBPM_FP32, 8, 64, variant)
            p.build_sample(smp, 13.0, offs)
            p.set_phase_states(theta)
            p.propagate(Z, 3, tb.TBPM_FP32)
            phi = torch.empty((S, smp.n_orb), dtype=torch.complex128, device="cuda")
            N.tbpm_get_states(p.ctx, phi)
            out.append(phi)
    assert (out[0] == out[1]).all() and (out[0] == out[2]).all()


@pytest.mark.parametrize("S,steps", [(1, (100, 27, 1, 2)), (4, (31, 1, 3)), (8, (15, 1, 2)), (3, (42, 2))])
def test_default_takes_the_lists_between_calls(S, steps):
    """Long rows: resumed runs on both sides of the step from which the default
    builds the staged gathers' lists give the plain kernel's states."""
    import torch
    import paper_2209_00806_gb300 as tb
    from paper_2209_00806_gb300 import _native as N
    from tbpm_inputs import tbg
    smp = tbg.to_numpy_sample(tbg.twisted_bilayer(6.0, order="morton"))
    theta = rng.phases(9, S, smp.n_orb)
    out = []
    for variant in (65, 8257):
        with tb.Propagator() as p:
            p.launch_config(tb.TBPM_FP32, 8, 64, variant)
            p.build_sample(smp, 13.0)
            p.set_phase_states(theta)
            for k, n in enumerate(steps):
                p.propagate(Z, n, tb.TBPM_FP32, flags=N.TBPM_PROP_RESUME if k else 0)
                phi = torch.empty((S, smp.n_orb), dtype=torch.complex128, device="cuda")
                N.tbpm_get_states(p.ctx, phi)
                out.append(phi)
    for a, b in zip(out[:len(steps)], out[len(steps):]):
        assert (a == b).all()


# cluster stepping of several states at once, and as the default up to 8192
# rows, against the per-term launches: states bit for bit, C within the
# rounding of its sums (1e-13, as the one-state test), with a resumed run
@pytest.mark.parametrize("S", [1, 3, 9])
@pytest.mark.parametrize("onsite_w,sigma,sides", [(0.0, 0.0, (64, 64)), (1.0, 0.0, (13, 17)),
                                                  (1.0, 0.05, (40, 51)), (1.0, 0.0, (64, 65))])
def test_cluster_states_are_bit_identical(S, onsite_w, sigma, sides):
    import paper_2209_00806_gb300 as tb
    from paper_2209_00806_gb300 import _native as N
    smp = lattice.graphene(*sides, pbc=True, seed=6, onsite_w=onsite_w, bond_sigma=sigma)
    theta = rng.phases(13, S, smp.n_orb)
    out = []
    for variant in (1, 2049, None):
        with tb.Propagator() as p:
            if variant is not None:
                p.launch_config(tb.TBPM_FP64, 8, 64, variant)
            p.build_sample(smp, 9.5)
            p.set_phase_states(theta)
            C = p.propagate(Z, 7, tb.TBPM_FP64)
            D = p.propagate(Z, 4, tb.TBPM_FP64, flags=N.TBPM_PROP_RESUME)
            out.append((C, D, p.states(), p.norms()))
    for o in out[1:]:
        assert np.array_equal(out[0][2], o[2])
        for a, b in zip((out[0][0], out[0][1], out[0][3]), (o[0], o[1], o[3])):
            assert np.abs(a - b).max() < 1e-13


# FP32 cluster stepping against the per-term kernels: one to eight rows a
# thread and their edges, one value and values per entry, ragged rows; and
# the repeat by the per-term kernels when the norm carry has to act, from a
# fresh start and a resumed one
def _f32(tb, smp, theta, variant, norm=None):
    from paper_2209_00806_gb300 import _native as N
    with tb.Propagator() as p:
        if variant is not None:
            p.launch_config(tb.TBPM_FP32, 16, 64, variant)
        p.build_sample(smp, 9.5)
        p.set_phase_states(theta)
        C = p.propagate(Z, 6, tb.TBPM_FP32)
        if norm:
            N.tbpm_set_norm_policy(p.ctx, norm)
        D = p.propagate(Z, 5, tb.TBPM_FP32, flags=N.TBPM_PROP_RESUME)
        st = p.stats()["renormalisations"]
        if norm:
            p.set_phase_states(theta)
            p.propagate(Z, 5, tb.TBPM_FP32)
            st += p.stats()["renormalisations"]
        return C, D, p.states(), p.norms(), st


@pytest.mark.parametrize("S", [1, 3, 9])
@pytest.mark.parametrize("kind", [(9, 11), (64, 64), (64, 65), (90, 91), (91, 180), (128, 128),
                                  (128, 129), (180, 182), "ragged"])
def test_fp32_cluster_is_bit_identical(S, kind):
    import paper_2209_00806_gb300 as tb
    if kind == "ragged":
        smp = lattice.random_graph(9000, 13000, seed=9, onsite_w=1.0, t_scale=0.8)
    else:
        smp = lattice.graphene(*kind, pbc=kind[0] != 90, seed=6, onsite_w=1.0,
                               bond_sigma=0.05 if kind[0] in (91, 180) else 0.0, vacancy_frac=0.004)
    theta = rng.phases(14, S, smp.n_orb)
    out = [_f32(tb, smp, theta, v) for v in (1, 2049, None)]
    for o in out[1:]:
        assert np.array_equal(out[0][2], o[2])
        for a, b in zip(out[0][:2] + out[0][3:4], o[:2] + o[3:4]):
            assert np.abs(a - b).max() < 1e-12


@pytest.mark.parametrize("S", [1, 4])
def test_fp32_cluster_repeats_for_the_norm_carry(S):
    import paper_2209_00806_gb300 as tb
    smp = lattice.graphene(20, 31, pbc=True, seed=6, onsite_w=1.0)
    theta = rng.phases(15, S, smp.n_orb)
    # 8257: the default's launch shape set by hand, per-term kernels with the same sums
    a, b = (_f32(tb, smp, theta, v, norm=1e-12) for v in (8257, None))
    assert a[4] > 0 and a[4] == b[4]
    assert np.array_equal(a[2], b[2]) and np.array_equal(a[1], b[1])
# buffers kept between calls: new states of the same number after a run (one of
# them not finite), of another number, in both precisions, C over and under
# the size of the page-locked result buffer (64 KB)
def test_states_set_again_start_afresh():
    import paper_2209_00806_gb300 as tb
    smp = lattice.graphene(12, 9, pbc=True, seed=6, onsite_w=1.0)
    th = rng.phases(15, 6, smp.n_orb)
    def fresh(t, steps, precision):
        with tb.Propagator() as q:
            q.build_sample(smp, 9.5)
            q.set_phase_states(t)
            return q.propagate(Z, steps, precision), q.states(), q.norms()
    with tb.Propagator() as p:
        p.build_sample(smp, 9.5)
        for t, steps, precision in ((th[:3], 5, 1), (th[3:], 5, 1), (th[:3], 5, 0), (th[1:4], 2000, 0),
                                    (th[:2], 1500, 1), (th, 3, 1)):
            bad = np.full((t.shape[0], smp.n_orb), np.nan, dtype=np.complex128)
            p.set_states(bad)
            with pytest.raises(tb.TbpmError):
                p.propagate(Z, 3, precision)
            p.set_phase_states(t)
            with pytest.raises(tb.TbpmError):       # nothing to resume after new states
                p.propagate(Z, 3, precision, flags=4)
            got = (p.propagate(Z, steps, precision), p.states(), p.norms())
            for a, b in zip(got, fresh(t, steps, precision)):
                assert np.array_equal(a, b)


# a segment's polynomials kept (50 steps, 11.7 GB) and recomputed per step (above
# 24 GB): the same gradients to the rounding of another summation order
def test_adjoint_segments_kept_and_recomputed():
    import paper_2209_00806_gb300 as tb
    smp = lattice.graphene(512, 512, pbc=True, seed=2, onsite_w=0.4, bond_sigma=0.05)
    theta = rng.phases(4, 2, smp.n_orb)
    g = np.random.default_rng(5).normal(size=(1, 2, 121, 2)) @ np.array([1, 1j])
    with tb.Propagator() as p:
        p.build_sample(smp, 9.5)
        p.set_phase_states(theta)
        (ah, ao), (bh, bo) = (p.adjoint(Z, 120, g, K) for K in (50, 120))
    scale = max(np.abs(ah).max(), np.abs(ao).max())
    assert np.abs(ah - bh).max() < 1e-11 * scale and np.abs(ao - bo).max() < 1e-11 * scale
