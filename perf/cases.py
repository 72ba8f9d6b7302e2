"""The calls that users of the library make, as measurable cases.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (lattice and random phases from the seed, the propagation
context with its Hamiltonian and states), ``run`` makes one pass through the
public entry points, ``exact`` gives the same outputs in plain 64-bit torch.
Lattices are the graphene family of the repository's workloads: periodic
disordered graphene, batches of uneven samples, open flakes in a magnetic
field, twisted bilayer graphene.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

import paper_2209_00806_gb300 as tb
from paper_2209_00806_gb300 import _native as N
from paper_2209_00806_gb300.autograd import TbpmDos
from tbpm_inputs import tbg

Z = math.pi / 2                 # s tau of every workload: 15 products a time step
T_NN = -2.7
A1 = (0.246, 0.0)
A2 = (0.123, 0.21304)
BETA = 38.68                    # 1/eV, 300 K
FLUX_QUANTUM = 4135.667696      # T nm^2
PREC = {"fp32": tb.TBPM_FP32, "fp64": tb.TBPM_FP64}
# launch shapes that the documentation recommends by hand; "default" sets none
CONFIG = {
    "cluster": (tb.TBPM_FP64, 8, 64, N.TBPM_VARIANT_ZIGZAG | N.TBPM_VARIANT_CLUSTER),
    "staged": (tb.TBPM_FP32, 8, 64, N.TBPM_VARIANT_ZIGZAG | N.TBPM_VARIANT_HALO
               | N.TBPM_VARIANT_STAGED),
}


def _case(name, kind, L1, L2, **kw):
    c = dict(name=name, kind=kind, L1=L1, L2=L2, pbc=True, disorder=0.0, vacancies=0.0,
             sigma=0.0, field=0.0, sides="", s=9.5, precision="fp32", states=4, steps=64,
             config="default")
    c.update(kw)
    return c


def listed():
    return [
        # density of states of the smallest stated workload: 64 x 64 pristine graphene, one
        # FP64 state, all 1024 time steps, the one-launch stepping meant for small samples
        _case("dos_64_cluster_fp64", "dos", 64, 64, s=9.0, precision="fp64", states=1, steps=1024,
              config="cluster"),
        # a small ragged sample without any launch setting: three states are two state groups,
        # and the pass is a long chain of short launches
        _case("dos_small_fp64", "dos", 45, 51, disorder=1.0, vacancies=0.01, precision="fp64",
              states=3, steps=128),
        # snapshots of a wave packet: one state, a few steps, the state itself is the result
        _case("wave_packet_fp32", "packet", 129, 97, pbc=False, states=1, steps=4),
        # the benchmark's sample: 2048 x 2048 disordered graphene with vacancies, four states
        _case("dos_2048_fp32", "dos", 2048, 2048, disorder=1.0, vacancies=0.01),
        # the same kind of sample in the FP64 form
        _case("dos_1024_fp64", "dos", 1024, 1024, disorder=1.0, vacancies=0.01, precision="fp64",
              steps=24),
        # one disordered sample per entry, sixteen states each, in one context
        _case("batch_fp32", "dos", 0, 0, sides="256,512,384,768,256,512", disorder=1.3, states=16,
              steps=24),
        # loss gradient with respect to every hopping and onsite energy (forward and backward)
        _case("gradient_512_fp64", "gradient", 512, 512, disorder=0.4, sigma=0.05,
              precision="fp64", states=3, steps=48),
        # optical conductivity: Fermi operator, then four propagated lanes with the current
        _case("optical_512_fp32", "optical", 512, 512, s=9.0, states=1, steps=192),
        # quasi-eigenstates at four energies: a forward and a backward run
        _case("quasi_640_fp32", "quasi", 640, 640, disorder=1.0, vacancies=0.01, steps=32),
        # twisted bilayer flake, 68 entries a row, eight states, the staged-gather kernel
        _case("bilayer_120nm_fp32", "bilayer", 120, 0, s=12.0, states=8, steps=16,
              config="staged"),
        # open flake in a magnetic field (complex hoppings), density of states in FP64
        _case("field_flake_fp64", "dos", 385, 333, pbc=False, disorder=0.6, vacancies=0.02,
              field=200.0, precision="fp64", states=2, steps=24),
        # everything of one evaluation from host arrays: build, states, propagation, DOS
        _case("whole_from_host_fp32", "whole", 700, 512, disorder=1.0, vacancies=0.01, steps=32),
    ]


def draw(rng):
    """One more case: the family by its share in use, sizes log-uniform."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["dos"] * 5 + ["batch", "packet", "gradient", "optical", "quasi", "bilayer",
                                     "field", "whole"])
    prec = rng.choice(["fp32", "fp64"])
    wide = dict(disorder=rng.choice([0.0, rng.uniform(0.1, 2.0)]),
                vacancies=rng.choice([0.0, rng.uniform(0.002, 0.03)]))
    if kind == "dos":
        L1 = size(24, 2048 if prec == "fp32" else 1024)
        L2 = max(8, min(2048, int(L1 * rng.uniform(0.6, 1.3))))
        c = _case("", "dos", L1, L2, precision=prec, states=rng.choice([1, 2, 3, 4, 5, 7, 8, 16]),
                  sigma=rng.choice([0.0, 0.0, 0.05]), pbc=rng.random() < 0.7, **wide)
        if c["sigma"]:
            c["disorder"] = min(c["disorder"], 1.0)     # the spectrum stays inside s
    elif kind == "batch":
        sides = [rng.choice([size(40, 700), 256, 384]) for _ in range(rng.randint(2, 6))]
        c = _case("", "dos", 0, 0, sides=",".join(map(str, sides)), precision=prec,
                  states=rng.choice([4, 8, 16]), **wide)
    elif kind == "packet":
        c = _case("", "packet", size(24, 600), size(24, 600), pbc=False, precision=prec,
                  states=rng.choice([1, 2]), **wide)
    elif kind == "gradient":
        c = _case("", "gradient", size(48, 512), size(48, 512), precision="fp64", sigma=0.05,
                  disorder=0.4, states=rng.choice([1, 2, 3, 4]))
    elif kind == "optical":
        c = _case("", "optical", size(96, 640), size(96, 640), s=9.5, precision=prec,
                  states=rng.choice([1, 2]), disorder=wide["disorder"])
    elif kind == "quasi":
        c = _case("", "quasi", size(64, 800), size(64, 800), precision=prec,
                  states=rng.choice([1, 2, 4]), **wide)
    elif kind == "bilayer":
        c = _case("", "bilayer", size(12, 130), 0, s=12.0, precision="fp32",
                  states=rng.choice([4, 8]), config=rng.choice(["staged", "default"]))
    elif kind == "field":
        c = _case("", "dos", size(40, 700), size(40, 500), pbc=False, precision=prec,
                  field=rng.uniform(50.0, 300.0), states=rng.choice([1, 2, 4]), **wide)
    else:
        c = _case("", "whole", size(64, 900), size(64, 900), precision=prec, **wide)
    # time steps: what keeps the pass below the largest listed one
    cells = sum(int(x) ** 2 for x in c["sides"].split(",")) if c["sides"] else c["L1"] * c["L2"]
    rows = 2 * cells if kind != "bilayer" else 1300 * c["L1"] ** 2   # about 17 graphene rows each
    per_step = rows * c["states"] * (4 if c["precision"] == "fp64" else 1)
    per_step *= {"gradient": 12, "optical": 8, "quasi": 3}.get(kind, 1)
    most = 1.5e9 / per_step
    c["steps"] = max(2, min(int(most), rng.choice([1, 3, 10]) if kind == "packet"
                            else rng.randint(12, 160)))
    del c["name"]
    return c


# ---- inputs --------------------------------------------------------------------


def _graphene(c, L1, L2, gen):
    """Bonds of a graphene supercell on the GPU: onsite, i, j, v, dr, number of orbitals."""
    dev = gen.device
    cell = torch.arange(L1 * L2, device=dev)
    n1, n2 = cell // L2, cell % L2
    i = torch.stack([2 * cell, 2 * cell + 1, 2 * cell + 1], 1).reshape(-1)
    j = torch.stack([2 * cell + 1, 2 * (((n1 + 1) % L1) * L2 + n2),
                     2 * (n1 * L2 + (n2 + 1) % L2)], 1).reshape(-1)
    b = torch.tensor([(A1[0] + A2[0]) / 3, (A1[1] + A2[1]) / 3], dtype=torch.float64, device=dev)
    a1 = torch.tensor(A1, dtype=torch.float64, device=dev)
    a2 = torch.tensor(A2, dtype=torch.float64, device=dev)
    dr = torch.stack([b, a1 - b, a2 - b]).repeat(L1 * L2, 1)
    keep = torch.ones(3 * L1 * L2, dtype=torch.bool, device=dev)
    if not c["pbc"]:
        keep.view(-1, 3)[:, 1] = n1 + 1 < L1
        keep.view(-1, 3)[:, 2] = n2 + 1 < L2
    v = torch.full((3 * L1 * L2,), T_NN, dtype=torch.float64, device=dev)
    if c["sigma"]:
        v = v * (1 + c["sigma"] * torch.randn(v.shape, generator=gen, dtype=torch.float64,
                                              device=dev))
    n = 2 * L1 * L2
    onsite = None
    if c["disorder"]:
        onsite = c["disorder"] * (torch.rand(n, generator=gen, dtype=torch.float64, device=dev) - 0.5)
    origin = n1[:, None] * a1 + n2[:, None] * a2
    pos = torch.stack([origin, origin + b], 1).reshape(-1, 2)
    if c["vacancies"]:
        gone = torch.randperm(n, generator=gen, device=dev)[:round(c["vacancies"] * n)]
        alive = torch.ones(n, dtype=torch.bool, device=dev)
        alive[gone] = False
        new = torch.cumsum(alive, 0) - 1
        keep &= alive[i] & alive[j]
        i, j = new[i], new[j]
        onsite = None if onsite is None else onsite[alive]
        pos = pos[alive]
        n = int(alive.sum())
    i, j, v, dr = i[keep].contiguous(), j[keep].contiguous(), v[keep].contiguous(), dr[keep]
    if c["field"]:              # Peierls phases, Landau gauge A = (B y, 0, 0)
        ph = math.pi * c["field"] / FLUX_QUANTUM * (pos[j, 0] - pos[i, 0]) * (pos[j, 1] + pos[i, 1])
        v = v * torch.exp(1j * ph)
    return n, onsite, i, j, v, dr.contiguous(), pos


def _inputs(c, seed):
    """Everything a pass is computed from, as tensors on the GPU."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = dict(offsets=None)
    if c["kind"] == "bilayer":
        d = tbg.twisted_bilayer(float(c["L1"]), device="cuda")
        x.update(n=d.n_orb, onsite=None, i=d.hop_i, j=d.hop_j, v=d.hop_v)
    elif c["sides"]:
        parts = [_graphene(c, int(L), int(L), gen) for L in c["sides"].split(",")]
        off = np.concatenate([[0], np.cumsum([p[0] for p in parts])]).astype(np.int64)
        x.update(n=int(off[-1]), offsets=off,
                 onsite=torch.cat([p[1] for p in parts]) if c["disorder"] else None,
                 i=torch.cat([p[2] + int(o) for p, o in zip(parts, off)]),
                 j=torch.cat([p[3] + int(o) for p, o in zip(parts, off)]),
                 v=torch.cat([p[4] for p in parts]))
    else:
        n, on, i, j, v, dr, pos = _graphene(c, c["L1"], c["L2"], gen)
        x.update(n=n, onsite=on, i=i, j=j, v=v, dr=dr, pos=pos)
    if c["kind"] == "packet":   # Gaussian packets with a momentum, inside the flake
        p = x["pos"] - x["pos"].mean(0)
        r = 0.15 * float(p.abs().max())
        k = 8 * torch.rand((c["states"], 2), generator=gen, dtype=torch.float64, device="cuda") - 4
        at = r * torch.rand((c["states"], 1, 2), generator=gen, dtype=torch.float64, device="cuda")
        psi = torch.exp(-((p[None] - at) ** 2).sum(-1) / (2 * r * r)) * torch.exp(1j * (k @ p.T))
        x["psi0"] = (psi / torch.linalg.vector_norm(psi, dim=1, keepdim=True)).contiguous()
    else:
        x["theta"] = 2 * math.pi * torch.rand((c["states"], x["n"]), generator=gen,
                                              dtype=torch.float64, device="cuda")
    if c["kind"] == "gradient":     # weights of the loss, dL/dD
        x["weight"] = torch.randn(512, generator=gen, dtype=torch.float64, device="cuda")
    x["energies"] = [-2.7, -1.0, 0.4, 2.0]
    return x


def _n_e(c):
    return 512 if c["kind"] == "gradient" else 2048


def prepare(case, seed):
    c, x = case, _inputs(case, seed)
    st = dict(c=c, x=x)
    if c["kind"] == "gradient":
        st["dos"] = TbpmDos(x["n"], x["i"], x["j"], x["theta"], c["s"], Z, c["steps"],
                            (-c["s"], c["s"]), _n_e(c), K=16)
        st["v"] = x["v"].clone().requires_grad_(True)
        st["onsite"] = x["onsite"].clone().requires_grad_(True)
        return st
    if c["kind"] == "whole":        # host arrays in the form a bond-list builder leaves them
        st["host"] = [None if x[k] is None else x[k].cpu().numpy()
                      for k in ("onsite", "i", "j", "v", "theta")]
        st["p"] = tb.Propagator()
        return st
    p = st["p"] = tb.Propagator()
    if c["config"] != "default":
        p.launch_config(*CONFIG[c["config"]])
    p.build(x["n"], x["onsite"], x["i"], x["j"], x["v"], c["s"], x["offsets"],
            flags=N.TBPM_BUILD_COMPLEX_HOPS if c["field"] else 0)
    if c["kind"] == "packet":
        p.set_states(x["psi0"])
    else:
        p.set_phase_states(x["theta"])
    if c["kind"] == "optical":
        p.set_bond_vectors(x["dr"].cpu().numpy())
    return st


def run(state):
    c, x = state["c"], state["x"]
    prec, steps, tau = PREC[c["precision"]], c["steps"], Z / c["s"]
    if c["kind"] == "gradient":
        v, onsite = state["v"], state["onsite"]
        v.grad = onsite.grad = None
        D = state["dos"](v, onsite)
        (D * x["weight"]).sum().backward()
        return dict(D=D.detach(), grad_hop=v.grad, grad_onsite=onsite.grad)
    p = state["p"]
    if c["kind"] == "whole":
        onsite, i, j, v, theta = state["host"]
        p.build(x["n"], onsite, i, j, v, c["s"])
        p.set_phase_states(theta)
    if c["kind"] == "packet":
        p.set_states(x["psi0"])
        C = p.propagate(Z, steps, prec)
        psi = torch.empty_like(x["psi0"])
        N.tbpm_get_states(p.ctx, psi)
        return dict(C=C, psi=psi)
    if c["kind"] == "optical":
        C = p.ac_correlation(Z, steps, BETA, 0.0, prec)
        return dict(C=C)
    if c["kind"] == "quasi":
        K, S = len(x["energies"]), c["states"]
        psi = torch.empty((K, S, x["n"]), dtype=torch.complex128, device="cuda")
        norms = np.empty((K, S, 1))
        N.tbpm_quasi_eigenstates(p.ctx, Z, steps, np.array(x["energies"]), prec, psi, norms)
        return dict(psi=psi, norms=norms)
    C = p.propagate(Z, steps, prec)
    avg = p.correlation()
    D = np.stack([tb.dos(a, tau, -c["s"], c["s"], _n_e(c))[1] for a in avg])
    out = dict(C=C, norms=p.norms(), D=D)
    if c["kind"] != "whole":        # the states of the last step, to go on from later
        out["psi"] = torch.empty((c["states"], x["n"]), dtype=torch.complex128, device="cuda")
        N.tbpm_get_states(p.ctx, out["psi"])
    return out


# ---- work ----------------------------------------------------------------------


def work(case):
    """Each input and each output once; the operations of the sparse products."""
    c = case
    if c["sides"]:
        n = sum(2 * int(L) ** 2 for L in c["sides"].split(","))
    elif c["kind"] == "bilayer":
        n = 2 * 38.2 * c["L1"] ** 2
    else:
        n = 2 * c["L1"] * c["L2"] * (1 - c["vacancies"])
    deg = 68.5 if c["kind"] == "bilayer" else 3 * (1 - c["vacancies"])
    S, steps = c["states"], c["steps"]
    cb = 8 if c["precision"] == "fp32" else 16
    vb = 0 if not c["sigma"] and not c["field"] and c["kind"] != "bilayer" else cb // 2
    vb *= 2 if c["field"] else 1
    matrix = n * (deg * (4 + vb) + (cb // 2 if c["disorder"] else 0))
    state = n * S * cb
    mul = 8 if c["field"] else 4                          # operations of one entry times one state
    term = n * S * (mul * deg + (4 if c["disorder"] else 0) + 8)
    if c["kind"] == "gradient":
        # forward, its polynomials once more, the adjoint with two products a stored entry
        return dict(bytes=2 * matrix + state, flops=15 * steps * (3 * term + n * S * 4 * (deg + 1)))
    if c["kind"] == "optical":
        fermi = len(tb.fermi_coefficients(BETA * c["s"], 0.0))
        prep = n * S * 3 * (4 * deg + 8) * fermi
        return dict(bytes=matrix + state + 16 * n * deg, flops=15 * steps * 4 * term + prep)
    if c["kind"] == "quasi":
        return dict(bytes=matrix + state + 4 * 16 * n * S,
                    flops=2 * steps * (15 * term + 4 * 8 * n * S))
    extra = 16 * n * S if c["kind"] != "whole" else 0
    extra += n * (24 * deg / 2 + 8 + 8 * S) if c["kind"] == "whole" else 0
    return dict(bytes=matrix + state + extra, flops=steps * (15 * term + 12 * n * S))


# ---- the same results in plain 64-bit torch ---------------------------------------


def _bessel(z, m_max):
    """J_0 .. J_m_max by the trapezoid rule of Bessel's integral (exact to rounding)."""
    t = np.arange(256) * (2 * np.pi / 256)
    return np.array([np.mean(np.cos(m * t - z * np.sin(t))) for m in range(m_max + 1)])


class _Ell:
    """H / s as padded rows (column -1: none) with x -> H x / s on [n, S] complex128."""

    def __init__(self, x, s, dr=None):
        n, i, j = x["n"], x["i"], x["j"]
        self.n, self.s, dev = n, s, i.device
        row, col = torch.cat([i, j]), torch.cat([j, i])
        bond = torch.arange(i.shape[0], device=dev).repeat(2)
        order = torch.sort(row * n + col).indices
        row, col, self.bond = row[order], col[order], bond[order]
        deg = torch.bincount(row, minlength=n)
        at = torch.arange(row.shape[0], device=dev) - (torch.cumsum(deg, 0) - deg)[row]
        self.w = int(deg.max())
        self.col = torch.zeros((self.w, n), dtype=torch.int64, device=dev)
        self.col[at, row] = col
        self.ent = torch.full((self.w, n), row.shape[0], dtype=torch.int64, device=dev)
        self.ent[at, row] = torch.arange(row.shape[0], device=dev)
        self.up = order < i.shape[0]
        self.set(x["v"], x["onsite"])
        if dr is not None:
            d = torch.cat([dr, -dr])[order]
            d = torch.cat([d, torch.zeros_like(d[:1])])
            self.dr = [d[self.ent, a] for a in (0, 1)]

    def set(self, v, onsite):
        val = torch.where(self.up, v[self.bond], v[self.bond].conj()) if v.is_complex() else v[self.bond]
        val = torch.cat([val / self.s, torch.zeros_like(val[:1])])
        self.val = val[self.ent][:, :, None]
        self.diag = None if onsite is None else (onsite / self.s)[:, None]

    def __call__(self, x):
        y = torch.zeros_like(x) if self.diag is None else self.diag * x
        for k in range(self.w):
            y = y + self.val[k] * torch.index_select(x, 0, self.col[k])
        return y

    def current(self, x, a):
        y = torch.zeros_like(x)
        for k in range(self.w):
            y = y + self.val[k] * self.dr[a][k][:, None] * torch.index_select(x, 0, self.col[k])
        return -1j * self.s * y


def _step(H, psi, J, sign=1.0):
    """exp(-i sign H tau) psi by the Chebyshev sum."""
    t0, t1 = psi, -1j * sign * H(psi)
    out = J[0] * t0 + 2 * J[1] * t1
    for m in range(2, len(J)):
        t0, t1 = t1, -2j * sign * H(t1) + t0
        out = out + 2 * J[m] * t1
    return out


def _fermi(H, v, s):
    K = 1
    while True:                     # double the sampling until the tail is rounding
        K *= 2
        n = 4 * K
        t = np.arange(n) * (2 * np.pi / n)
        f = 0.5 * (1 - np.tanh(0.5 * BETA * s * np.cos(t)))
        ck = np.fft.rfft(f).real[:K + 1] * 2 / n
        if K >= 16 and np.abs(ck[-8:]).max() < 2e-15:
            break
    t0, t1 = v, H(v)
    out = 0.5 * ck[0] * t0 + ck[1] * t1
    for k in range(2, K + 1):
        t0, t1 = t1, 2 * H(t1) - t0
        if abs(ck[k]) > 1e-17:
            out = out + ck[k] * t1
    return out


def _dos(C, tau, s, n_e):
    """Windowed transform of averaged correlations [..., steps + 1]."""
    nt = C.shape[-1] - 1
    n = torch.arange(1, nt + 1, dtype=torch.float64, device=C.device)
    w = 0.5 * (1 + torch.cos(math.pi * n / nt))
    E = -s + (torch.arange(n_e, dtype=torch.float64, device=C.device) + 0.5) * (2 * s / n_e)
    ph = torch.exp(1j * tau * E[:, None] * n[None, :]) * w
    return tau / math.pi * (0.5 * C[..., :1].real + (ph * C[..., None, 1:]).real.sum(-1))


def exact(case, seed):
    c = case
    if c["kind"] == "bilayer" and 1300 * c["L1"] ** 2 * c["steps"] * c["states"] > 3e9:
        return None
    x = _inputs(c, seed)
    s, steps, tau, S = c["s"], c["steps"], Z / c["s"], c["states"]
    J = _bessel(Z, 20)
    H = _Ell(x, s, x.get("dr") if c["kind"] == "optical" else None)
    off = [0, x["n"]] if x["offsets"] is None else [int(o) for o in x["offsets"]]
    if c["kind"] == "packet":
        psi0 = x["psi0"].T.contiguous()
    else:
        size = torch.cat([torch.full((b - a,), float(b - a), dtype=torch.float64, device="cuda")
                          for a, b in zip(off, off[1:])])
        psi0 = (torch.exp(1j * x["theta"]) / torch.sqrt(size)).T.contiguous()

    def dots(a, b):                 # [samples, states]
        p = a.conj() * b
        return torch.stack([p[lo:hi].sum(0) for lo, hi in zip(off, off[1:])])

    if c["kind"] == "optical":
        if S > 1:
            return None
        p2 = _fermi(H, psi0, s)
        p1 = [H.current(psi0, b) for b in (0, 1)]
        p1 = [p - _fermi(H, p, s) for p in p1]
        C = torch.empty((1, S, 4, steps + 1), dtype=torch.complex128, device="cuda")
        for n in range(steps + 1):
            for a in (0, 1):
                j2 = H.current(p2, a)
                for b in (0, 1):
                    C[0, :, 2 * a + b, n] = (j2.conj() * p1[b]).sum(0)
            if n < steps:
                p2, p1 = _step(H, p2, J), [_step(H, p, J) for p in p1]
        return dict(C=C.cpu().numpy())
    if c["kind"] == "quasi":
        acc = torch.zeros((len(x["energies"]),) + psi0.shape, dtype=torch.complex128, device="cuda")
        for sign in (1, -1):
            psi = psi0
            for n in range(steps + 1):
                w = tau / (2 * math.pi) * 0.5 * (1 + math.cos(math.pi * n / steps))
                if n or sign > 0:
                    for k, E in enumerate(x["energies"]):
                        ph = E * sign * n * tau
                        acc[k] += w * complex(math.cos(ph), math.sin(ph)) * psi
                if n < steps:
                    psi = _step(H, psi, J, sign)
        nn = (acc.abs() ** 2).sum(1)
        psi = (acc / torch.sqrt(nn)[:, None, :]).permute(0, 2, 1).contiguous()
        return dict(psi=psi, norms=nn[:, :, None].cpu().numpy())
    if c["kind"] == "gradient":
        v = x["v"].clone().requires_grad_(True)
        onsite = x["onsite"].clone().requires_grad_(True)

        def one(psi, v_, on_):
            H.set(v_, on_)
            return _step(H, psi, J)

        psi, C = psi0, [dots(psi0, psi0).mean(1)]
        for n in range(steps):
            psi = torch.utils.checkpoint.checkpoint(one, psi, v, onsite, use_reentrant=False)
            C.append(dots(psi0, psi).mean(1))
        D = _dos(torch.stack(C, 1)[0], tau, s, _n_e(c))
        (D * x["weight"]).sum().backward()
        return dict(D=D.detach(), grad_hop=v.grad, grad_onsite=onsite.grad)
    psi, C, norms = psi0, [dots(psi0, psi0)], [dots(psi0, psi0).real]
    for n in range(steps):
        psi = _step(H, psi, J)
        C.append(dots(psi0, psi))
        norms.append(dots(psi, psi).real)
    C, norms = torch.stack(C, 2), torch.stack(norms, 2)
    if c["kind"] == "packet":
        return dict(C=C.cpu().numpy(), psi=psi.T.contiguous())
    D = torch.stack([_dos(a, tau, s, _n_e(c)) for a in C.mean(1)])
    out = dict(C=C.cpu().numpy(), norms=norms.cpu().numpy(), D=D.cpu().numpy())
    if c["kind"] != "whole":
        out["psi"] = psi.T.contiguous()
    return out
