"""What a user of this framework has it do, as cases that can be timed and checked.

A Spectral Quadrature calculation (arXiv:1708.07913) runs the four steps of
``SQSolver`` -- spectral bounds, Chebyshev moments, Fermi level, density and
energies -- once per SCF iteration, alone or for several systems as a batch;
the SCF around it solves a Poisson problem and mixes potentials; a molecular
dynamics step adds the nonlocal forces; and the learned warm start predicts
densities and is trained on the SQ path's own.  The systems are the seeded
FCC-Al-like crystals of ``synth`` (a = 7.65 bohr, four atoms per cell).

Sizes: the grid spacing of the workloads is 0.45 to 0.51 bohr, the region of
influence reaches from 13^3 points (R_cut 3) to 31^3 (R_cut 7, the largest
the library takes), the degree from 24 to 64.  A node's cost does not depend
on how many nodes there are, so one or two cells per axis stand for the
larger grids wherever the region is what matters.

What a context of SQ_FP32 computes has FP32 accuracy and is handed out in the
FP64 arrays of the C interface; such results are returned here in the type
that they were computed in, and so are the network's.
"""
import math
import random

import numpy as np
import torch

import synth
from paper_1708_07913_gb300 import SQ_FP32, SQ_FP64, SQBatch, SQCNN, SQSolver, sq

A_LAT = synth.LATTICE_A
DEVICE = "cuda:0"
NO = 6                       # half order of the finite differences
MIX_HISTORY, MIX_BETA, KERKER = 16, 0.3, (0.5, 0.1)


def _region(kind, name, n, cells, r_cut, npl, kT, fp32, nonlocal_, n_lanczos=40, margin=0.02):
    return dict(name=name, kind=kind, n=n, cells=cells, r_cut=r_cut, npl=npl, kT=kT, fp32=fp32, nonlocal_=nonlocal_,
                n_lanczos=n_lanczos, margin=margin)


def listed():
    return [
        # the smallest calculation: one cell, 13^3 regions, local potential only; launches and waits count here
        _region("step", "step_local_13", 16, 1, 3.0, 24, 0.1, True, False),
        # one SCF iteration's SQ step at the scale workload's region, degree and temperature (29^3, n_pl 64)
        _region("step", "step_29", 32, 2, 7.0, 64, 0.1, True, True),
        # the two region steps by themselves: fresh bounds at the region of the 3- and 4-cell workloads,
        _region("bounds", "bounds_25", 16, 1, 6.0, 48, 0.05, True, True),
        # moments with bounds in hand (an SCF iteration that reuses them) at the scale workload's region,
        _region("moments", "moments_29", 16, 1, 7.0, 64, 0.1, True, True),
        # and at the largest region there is, on a grid of odd size
        _region("moments", "moments_31", 17, 1, 7.0, 32, 0.1, True, True),
        # the FP64 finish of an SCF: a whole step in FP64 at its largest region
        _region("step", "step_fp64_25", 16, 1, 6.0, 48, 0.05, False, True),
        # forces after the last SCF iteration
        _region("forces", "forces_25", 16, 1, 6.0, 48, 0.05, True, True),
        # Fermi level, density and energies from the moments of the 4-cell SCF system
        dict(name="fermi_64", kind="fermi", n1=64, n2=64, n3=64, npl=48, kT=0.05),
        # the SCF update of that system: electrostatics, effective potential, preconditioner, mixing
        dict(name="scf_update_64", kind="scf", n1=64, n2=64, n3=64, mix_steps=8),
        # the warm start's network on that grid, and its loss gradient over a training minibatch
        dict(name="cnn_predict_64", kind="predict", n1=64, n2=64, n3=64, bf16=True),
        dict(name="cnn_grad_8x16", kind="grad", n1=16, n2=16, n3=16, batch=8, bf16=True),
        # uneven systems as one launch: one to two cells, 15^3 to 25^3 regions, with unlike degrees and temperatures
        dict(name="batch_uneven", kind="batch", n="15,16,17,31", cells="1,1,1,2", r_cut="6.0,6.0,5.0,4.0",
             npl="48,24,64,32", kT="0.05,0.1,0.15,0.08", fp32=True),
    ]


def draw(rng: random.Random):
    kind = rng.choice(["step", "step", "bounds", "moments", "moments", "forces", "fermi", "scf", "predict", "grad", "batch"])

    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    if kind in ("step", "bounds", "moments", "forces"):
        fp32 = rng.random() < 0.75
        while True:
            n = rng.randint(11, 33)
            cells = 1 if n < 23 else 2
            h = A_LAT * cells / n
            r_cut = round(min(rng.uniform(2.5, 7.0), h * (15.4 if fp32 else 12.4)), 3)
            npl = rng.choice([24, 32, 48, 64])
            m = int(r_cut / h)
            cost = n ** 3 * (2 * m + 1) ** 3 * (40 + npl) * (1 if fp32 else 12)
            if cost < 2.5e10:
                break
        return dict(kind=kind, n=n, cells=cells, r_cut=r_cut, npl=npl, kT=round(rng.uniform(0.03, 0.2), 4), fp32=fp32,
                    nonlocal_=kind == "forces" or rng.random() < 0.8, n_lanczos=40, margin=0.02)
    if kind == "batch":
        k = rng.randint(2, 5)
        ns = [rng.randint(12, 18) for _ in range(k)]
        return dict(kind="batch", n=",".join(map(str, ns)), cells=",".join("1" for _ in ns),
                    r_cut=",".join(str(round(rng.uniform(3.0, 6.0), 2)) for _ in ns),
                    npl=",".join(str(rng.choice([24, 32, 48, 64])) for _ in ns),
                    kT=",".join(str(round(rng.uniform(0.03, 0.2), 3)) for _ in ns), fp32=rng.random() < 0.8)
    if kind == "fermi":
        return dict(kind=kind, n1=log_int(12, 72), n2=log_int(12, 72), n3=log_int(12, 72), npl=rng.choice([24, 32, 48, 64]),
                    kT=round(rng.uniform(0.03, 0.2), 4))
    if kind == "scf":
        return dict(kind=kind, n1=log_int(14, 72), n2=log_int(14, 72), n3=log_int(14, 72), mix_steps=rng.randint(1, 12))
    if kind == "predict":
        return dict(kind=kind, n1=log_int(14, 80), n2=log_int(14, 80), n3=log_int(14, 80), bf16=rng.random() < 0.7)
    return dict(kind="grad", n1=rng.randint(11, 24), n2=rng.randint(11, 24), n3=rng.randint(11, 24), batch=rng.randint(1, 8),
                bf16=rng.random() < 0.7)


# ---------------------------------------------------------------- inputs

def _crystal(n, cells, nonlocal_, seed):
    """(positions, V on the device, projector types) of a seeded crystal."""
    pos = synth.fcc_positions(cells, 0.15, seed)
    V = synth.local_potential(n, A_LAT * cells, pos)
    return pos, torch.from_numpy(np.ascontiguousarray(V).ravel()).to(DEVICE), synth.projector_types(nonlocal_)


def _fd(h):
    """Weights of the 12th-order Laplacian and gradient, d = 0 .. 6."""
    f = math.factorial
    w = [-sum(1.0 / q ** 2 for q in range(1, NO + 1)) / h ** 2]
    g = [0.0]
    for d in range(1, NO + 1):
        c = (-1) ** (d + 1) * f(NO) ** 2 / (f(NO - d) * f(NO + d))
        w.append(2.0 * c / (h * h * d * d))
        g.append(c / (h * d))
    return w, g


def _enclosure(h, V, n_nodes, seed):
    """Per-node bounds (chi, zeta) around the spectrum of every nodal Hamiltonian, a little uneven as Lanczos bounds are."""
    w, _ = _fd(h)
    kin = -3.0 * (w[0] + sum(w[d] * (-1) ** d for d in range(1, NO + 1)))
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    u = torch.rand(2, n_nodes, dtype=torch.float64, device=DEVICE, generator=g)
    lo = V.min() + 0.8 - 0.3 * u[0]
    hi = kin + V.max() + 0.5 + 0.5 * u[1]
    return 0.5 * (hi + lo), 0.5 * (hi - lo)


def _smooth(shape, seed, modes=6):
    """A smooth periodic field (a few plane waves), x fastest, flat."""
    n1, n2, n3 = shape
    g = np.random.default_rng(seed)
    z, y, x = torch.meshgrid(*(torch.arange(n, dtype=torch.float64, device=DEVICE) * (2 * math.pi / n) for n in (n3, n2, n1)),
                             indexing="ij")
    out = torch.zeros_like(x)
    for _ in range(modes):
        k = g.integers(-2, 3, 3)
        out += float(g.normal()) * torch.cos(k[0] * x + k[1] * y + k[2] * z + float(g.uniform(0, 6.28)))
    return out.reshape(-1) / math.sqrt(modes)


def _noise(n, seed):
    return torch.randn(n, dtype=torch.float64, device=DEVICE, generator=torch.Generator(device=DEVICE).manual_seed(seed))


def _fermi_inputs(c, seed):
    """Moments of a positive local density of states at every node, as the recurrence gives them."""
    N = c["n1"] * c["n2"] * c["n3"]
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    P = 8
    wt = torch.rand(N, P, dtype=torch.float64, device=DEVICE, generator=g)
    wt /= wt.sum(1, keepdim=True)
    x = -0.97 + 1.93 * torch.rand(N, P, dtype=torch.float64, device=DEVICE, generator=g) ** (2.0 / 3.0)   # free-electron-like
    mom = torch.empty(N, c["npl"] + 1, dtype=torch.float64, device=DEVICE)
    tm, t = torch.ones_like(x), x.clone()
    mom[:, 0], mom[:, 1] = 1.0, (wt * x).sum(1)
    for j in range(2, c["npl"] + 1):
        tm, t = t, 2 * x * t - tm
        mom[:, j] = (wt * t).sum(1)
    u = torch.rand(2, N, dtype=torch.float64, device=DEVICE, generator=g)
    return mom, 21.0 + 0.3 * u[0], 23.5 + 0.3 * u[1]


FERMI_FILL = 6.0 / 4096       # occupied states per node of the Al-like crystals (12 electrons on a 16^3 cell)


def _scf_inputs(c, seed):
    """A positive density, the potentials of an iteration and the (V_in, V_out) pairs of the mixing steps."""
    shape = (c["n1"], c["n2"], c["n3"])
    N = shape[0] * shape[1] * shape[2]
    rho = 0.03 * torch.exp(0.4 * _smooth(shape, seed)) + 1e-4 * _noise(N, seed).abs()
    pairs = [(-1.0 + _smooth(shape, seed + 17 * i + 1) + 1e-2 * _noise(N, seed + 17 * i + 1),
              -1.0 + _smooth(shape, seed + 17 * i + 2) + 1e-2 * _noise(N, seed + 17 * i + 2)) for i in range(c["mix_steps"])]
    return dict(rho=rho, V_loc=-1.0 + _smooth(shape, seed + 5), V_in=-1.0 + _smooth(shape, seed + 6), pairs=pairs)


def _cnn_inputs(c, seed):
    shape = (c["n1"], c["n2"], c["n3"])
    out = []
    for i in range(c.get("batch", 1)):
        V = -1.0 + 0.9 * _smooth(shape, 7919 * seed + i) + 0.02 * _noise(shape[0] * shape[1] * shape[2], 31 * seed + i)
        ref = 0.03 * torch.exp(0.5 * _smooth(shape, 104729 * seed + i))
        out.append((shape, V, ref))
    return out


def _cnn_params(seed):
    """Weights of variance 1/fan-in and small biases, flat, in the network's natural order."""
    r, C = np.random.default_rng(seed), 32
    p = [r.standard_normal(C * 125) / math.sqrt(125), 0.1 * r.standard_normal(C), r.standard_normal(C * C * 27) / math.sqrt(C * 27),
         0.1 * r.standard_normal(C), r.standard_normal(C * 27) / math.sqrt(C * 27), 0.1 * r.standard_normal(1)]
    return np.concatenate(p)


def _split(text, to):
    return [to(v) for v in text.split(",")]


def _solver(c, pos, proj):
    return SQSolver((c["n"],) * 3, A_LAT * c["cells"] / c["n"], c["r_cut"], c["npl"], SQ_FP32 if c["fp32"] else SQ_FP64, pos, proj,
                    device=DEVICE)


def _batch_members(c):
    return [dict(n=n, cells=k, r_cut=r, npl=p, kT=t, fp32=c["fp32"]) for n, k, r, p, t in zip(
        _split(c["n"], int), _split(c["cells"], int), _split(c["r_cut"], float), _split(c["npl"], int), _split(c["kT"], float))]


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("step", "bounds", "moments", "forces"):
        pos, V, proj = _crystal(c["n"], c["cells"], c["nonlocal_"], seed)
        s = dict(case=c, solver=_solver(c, pos, proj), V=V, electrons=synth.ELECTRONS_PER_ATOM * len(pos))
        if kind in ("moments", "forces"):
            s["bounds"] = _enclosure(A_LAT * c["cells"] / c["n"], V, c["n"] ** 3, seed)
            s["mu"] = -0.3
        return s
    if kind == "batch":
        members, solvers, Vs, ne, kts = _batch_members(c), [], [], [], []
        for i, m in enumerate(members):
            pos, V, proj = _crystal(m["n"], m["cells"], True, 101 * seed + i)
            solvers.append(_solver(m, pos, proj))
            Vs.append(V)
            ne.append(synth.ELECTRONS_PER_ATOM * len(pos))
            kts.append(m["kT"])
        b = SQBatch(solvers)
        b.set_plan(sq.SQ_BATCH_STREAMS)
        return dict(case=c, batch=b, solvers=solvers, V=Vs, electrons=ne, kT=kts)
    if kind == "fermi":
        shape = (c["n1"], c["n2"], c["n3"])
        mom, chi, zeta = _fermi_inputs(c, seed)
        solver = SQSolver(shape, 0.478125, 0.5, c["npl"], SQ_FP32, device=DEVICE)
        solver.moments.copy_(mom)
        return dict(case=c, solver=solver, chi=chi, zeta=zeta, electrons=2 * FERMI_FILL * chi.numel())
    if kind == "scf":
        shape = (c["n1"], c["n2"], c["n3"])
        N = shape[0] * shape[1] * shape[2]
        solver = SQSolver(shape, 0.478125, 0.5, 8, SQ_FP64, device=DEVICE)
        new = lambda: torch.empty(N, dtype=torch.float64, device=DEVICE)  # noqa: E731
        return dict(_scf_inputs(c, seed), case=c, solver=solver, phi=new(), V_out=new(), V_pre=new(), V_next=new(),
                    mixer=_Mixer(N))
    net = SQCNN(bf16=c["bf16"], seed=0, device=DEVICE)
    net.set_params(_cnn_params(seed), -1.0, 0.8, 0.03)
    return dict(case=c, net=net, items=_cnn_inputs(c, seed))


class _Mixer:
    """A mixer handle, given back with the state."""

    def __init__(self, n):
        self.h = sq.sq_mixer_create(n, MIX_HISTORY, MIX_BETA)

    def __del__(self):
        try:
            sq.sq_mixer_destroy(self.h)
        except Exception:
            pass


# ---------------------------------------------------------------- one pass

def _as_computed(c, outs):
    """The results of an FP32 context in FP32 (see the head of this file)."""
    if not c["fp32"]:
        return outs
    return {k: v.float() if isinstance(v, torch.Tensor) else np.float32(v) for k, v in outs.items()}


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "step":
        o = state["solver"].solve(state["V"], state["electrons"], c["kT"], c["n_lanczos"], c["margin"])
        return _as_computed(c, o)
    if kind == "bounds":
        chi, zeta = state["solver"].bounds(state["V"], c["n_lanczos"], c["margin"])
        return _as_computed(c, dict(chi=chi, zeta=zeta))
    if kind == "moments":
        return _as_computed(c, dict(moments=state["solver"].compute_moments(state["V"], *state["bounds"])))
    if kind == "forces":
        return _as_computed(c, dict(forces=state["solver"].nl_forces(state["V"], state["mu"], c["kT"], *state["bounds"])))
    if kind == "batch":
        state["batch"].run(state["V"], state["electrons"], state["kT"], 40, 0.02)
        res = state["batch"].results()
        return [_as_computed(c, dict(r, rho=s.rho, moments=s.moments, chi=s.chi, zeta=s.zeta))
                for r, s in zip(res, state["solvers"])]
    if kind == "fermi":
        s = state["solver"]
        mu = s.fermi_level(state["electrons"], c["kT"], state["chi"], state["zeta"])
        eb, es, ne = s.density_energy(mu, c["kT"], state["chi"], state["zeta"])
        return dict(mu=mu, e_band=eb, e_ent=es, n_elec=ne, rho=s.rho)
    if kind == "scf":
        s = state["solver"]
        sq.sq_set_stream(s.ctx)
        sq.sq_poisson(s.ctx, state["rho"], state["phi"], 1e-12)
        sq.sq_effective_potential(s.ctx, state["V_loc"], state["phi"], state["rho"], 2.0 / 3.0, state["V_out"])
        r, _ = sq.sq_kerker(s.ctx, state["V_in"], state["V_out"], KERKER[0], KERKER[1], state["V_pre"])
        m = state["mixer"].h
        sq.sq_mixer_reset(m)
        for v_in, v_out in state["pairs"]:
            sq.sq_mixer_step(m, v_in, v_out, state["V_next"])
        return dict(phi=state["phi"], V_out=state["V_out"], resid=r, V_pre=state["V_pre"], V_next=state["V_next"])
    net = state["net"]
    if kind == "predict":
        shape, V, _ = state["items"][0]
        return net.predict(shape, V).float()
    total, rhos = 0.0, []
    for i, (shape, V, ref) in enumerate(state["items"]):
        rho = torch.empty(V.numel(), dtype=torch.float64, device=V.device)
        total += sq.sq_cnn_backward(net.net, shape, V, ref, rho, accumulate=i > 0)
        rhos.append(rho)
    return dict(loss=np.float32(total), grads=sq.sq_cnn_get_grads(net.net).astype(np.float32), rho=torch.stack(rhos).float())


# ---------------------------------------------------------------- the work there is

def _pairs_per_point(c):
    """Projector supports over a region point: atom density times the support sphere."""
    h3 = (A_LAT * c["cells"] / c["n"]) ** 3
    return 4 * c["cells"] ** 3 * (4.0 / 3.0) * math.pi * synth.PROJ_RNL ** 3 / (c["n"] ** 3 * h3)


def _region_flops(c, lanczos, cheb, nonlocal_=True):
    S = 2 * int(math.floor(c["r_cut"] * c["n"] / (A_LAT * c["cells"]) + 1e-12)) + 1
    nl = 16.0 * _pairs_per_point(c) if nonlocal_ else 0.0
    return c["n"] ** 3 * float(S) ** 3 * (lanczos * (56 + nl) + cheb * (52 + nl))


def work(case):
    c, kind = case, case["kind"]
    if kind in ("step", "bounds", "moments", "forces"):
        N, nl = c["n"] ** 3, c["nonlocal_"]
        if kind == "bounds":
            return dict(bytes=24.0 * N, flops=_region_flops(c, c["n_lanczos"], 0, nl))
        if kind == "moments":
            return dict(bytes=8.0 * N * (c["npl"] + 4), flops=_region_flops(c, 0, c["npl"] // 2, nl))
        if kind == "forces":
            return dict(bytes=24.0 * N + 96 * c["cells"] ** 3, flops=_region_flops(c, 0, c["npl"], nl))
        return dict(bytes=8.0 * N * (c["npl"] + 5), flops=_region_flops(c, c["n_lanczos"], c["npl"] // 2, nl))
    if kind == "batch":
        ms = _batch_members(c)
        return dict(bytes=sum(8.0 * m["n"] ** 3 * (m["npl"] + 5) for m in ms),
                    flops=sum(_region_flops(m, 40, m["npl"] // 2) for m in ms))
    N = c["n1"] * c["n2"] * c["n3"]
    if kind == "fermi":
        K = c["npl"] + 1
        return dict(bytes=8.0 * N * (K + 3), flops=2.0 * N * K * K)
    if kind == "scf":
        return dict(bytes=8.0 * N * (6 + 2 * c["mix_steps"]), flops=2.0 * N * (2 * 43 + 12 * c["mix_steps"]))
    if kind == "predict":
        return dict(bytes=16.0 * N, flops=2.0 * N * (32 * 125 + 32 * 32 * 27 + 32 * 27))
    return dict(bytes=24.0 * N * c["batch"], flops=6.0 * N * c["batch"] * (32 * 125 + 32 * 32 * 27 + 32 * 27))


# ---------------------------------------------------------------- the same in 64 bits, in plain torch

class _Plain:
    """The nodal Hamiltonians of a chunk of nodes as dense arrays (region vectors [B, S, S, S], z slowest)."""

    def __init__(self, c, pos, V, proj, nodes):
        n, self.h = c["n"], A_LAT * c["cells"] / c["n"]
        m = int(math.floor(c["r_cut"] / self.h + 1e-12))
        S, B, dev = 2 * m + 1, nodes.numel(), V.device
        self.m, self.S, self.B = m, S, B
        self.w, self.g = _fd(self.h)
        i, j, k = nodes % n, (nodes // n) % n, nodes // (n * n)
        r = torch.arange(-m, m + 1, device=dev)
        self.ax = [q[:, None] + r for q in (i, j, k)]                     # unwrapped grid indices
        x, y, z = (a % n for a in self.ax)
        self.V = V.view(n, n, n)[z[:, :, None, None], y[:, None, :, None], x[:, None, None, :]]
        self.P, self.atom = None, None
        if not proj:
            return
        L, rc, rnl = n * self.h, proj[0][2], proj[0][3]
        E = int(math.ceil((m * self.h + rnl + L) / L)) + 1
        e = torch.arange(-E, E + 1, device=dev, dtype=torch.float64) * L
        R = torch.from_numpy(pos).to(dev)
        img = (R[:, None, None, None, :] + torch.stack(torch.meshgrid(e, e, e, indexing="ij"), -1)[None]).reshape(-1, 3)
        who = torch.arange(len(pos), device=dev).repeat_interleave(e.numel() ** 3)
        q = torch.stack([i, j, k], 1).double() * self.h
        near = ((img[None] - q[:, None]).abs() <= m * self.h + rnl).all(-1)
        C = int(near.sum(1).max())
        order = torch.argsort(near.to(torch.int8), dim=1, descending=True, stable=True)[:, :C]
        ok = torch.gather(near, 1, order)
        pick = img[order]                                                  # [B, C, 3]
        self.atom = torch.where(ok, who[order], torch.full_like(order, len(pos)))
        d = [a[:, None, :].double() * self.h - pick[:, :, s, None] for s, a in enumerate(self.ax)]   # [B, C, S]
        r2 = (d[0] ** 2)[:, :, None, None, :] + (d[1] ** 2)[:, :, None, :, None] + (d[2] ** 2)[:, :, :, None, None]
        chi = torch.exp(-r2 / (2 * rc * rc)) * ((r2 < rnl * rnl) & ok[:, :, None, None, None])
        del r2
        self.P = torch.stack([chi, chi * d[0][:, :, None, None, :], chi * d[1][:, :, None, :, None], chi * d[2][:, :, :, None, None]],
                             2).reshape(B, C * 4, S ** 3)
        As2 = (math.pi * rc * rc) ** -1.5
        gam = {l: gm for l, gm, _, _ in proj}
        h3 = self.h ** 3
        cs, cp = h3 * gam.get(0, 0.0) * As2, h3 * gam.get(1, 0.0) * 2.0 / (rc * rc) * As2
        self.coef = torch.tensor([cs, cp, cp, cp], dtype=torch.float64, device=dev).repeat(C)

    def H(self, t):
        out = (self.V - 3.0 * self.w[0]) * t
        for axis in (1, 2, 3):
            for d in range(1, NO + 1):
                if d < self.S:
                    lo, hi = t.narrow(axis, 0, self.S - d), t.narrow(axis, d, self.S - d)
                    out.narrow(axis, 0, self.S - d).add_(hi, alpha=-0.5 * self.w[d])
                    out.narrow(axis, d, self.S - d).add_(lo, alpha=-0.5 * self.w[d])
        if self.P is not None:
            p = torch.bmm(self.P, t.reshape(self.B, -1, 1))[:, :, 0] * self.coef
            out += torch.bmm(p[:, None, :], self.P).view_as(t)
        return out

    def dot(self, a, b):
        return (a * b).flatten(1).sum(1)

    def bounds(self, n_lanczos, margin):
        v = torch.full((self.B,) + (self.S,) * 3, self.S ** -1.5, dtype=torch.float64, device=self.V.device)
        old, b, al, be = torch.zeros_like(v), torch.zeros(self.B, dtype=torch.float64, device=v.device), [], []
        s = lambda a: a[:, None, None, None]  # noqa: E731
        for _ in range(n_lanczos):
            w = self.H(v) - s(b) * old
            a = self.dot(v, w)
            w -= s(a) * v
            b = self.dot(w, w).sqrt()
            al.append(a)
            be.append(b)
            old, v = v, w / s(b)
        T = torch.diag_embed(torch.stack(al, 1)) + torch.diag_embed(torch.stack(be[:-1], 1), 1) + torch.diag_embed(torch.stack(be[:-1], 1), -1)
        ev = torch.linalg.eigvalsh(T)
        wd = margin * (ev[:, -1] - ev[:, 0]).clamp(min=1.0)
        return 0.5 * (ev[:, -1] + ev[:, 0]), 0.5 * (ev[:, -1] - ev[:, 0]) + wd

    def recur(self, chi, zeta, steps):
        t0 = torch.zeros((self.B,) + (self.S,) * 3, dtype=torch.float64, device=self.V.device)
        t0[:, self.m, self.m, self.m] = 1.0
        s = lambda a: a[:, None, None, None]  # noqa: E731
        yield t0
        t1 = (self.H(t0) - s(chi) * t0) / s(zeta)
        yield t1
        for _ in range(steps - 1):
            t0, t1 = t1, 2.0 * (self.H(t1) - s(chi) * t1) / s(zeta) - t0
            yield t1

    def moments(self, chi, zeta, npl):
        m, half = self.m, npl // 2
        out = torch.empty(self.B, npl + 1, dtype=torch.float64, device=self.V.device)
        prev = None
        for i, t in enumerate(self.recur(chi, zeta, half)):
            out[:, i] = t[:, m, m, m]
            if i and 2 * i > half:
                out[:, 2 * i] = 2.0 * self.dot(t, t) - 1.0
            if i and 2 * i - 1 > half:
                out[:, 2 * i - 1] = 2.0 * self.dot(t, prev) - out[:, 1]
            prev = t
        return out

    def forces(self, chi, zeta, npl, mu, kT, n_atoms):
        K, dev = npl + 1, self.V.device
        k = torch.arange(K, dtype=torch.float64, device=dev)
        th = math.pi * (k + 0.5) / K
        f = 1.0 / (1.0 + torch.exp((chi[:, None] + zeta[:, None] * torch.cos(th) - mu) / kT))
        cj = 2.0 / K * f @ torch.cos(th[:, None] * k[None, :])
        cj[:, 0] *= 0.5
        D = torch.zeros((self.B,) + (self.S,) * 3, dtype=torch.float64, device=dev)
        for j, t in enumerate(self.recur(chi, zeta, npl)):
            D += cj[:, j, None, None, None] * t
        at_q = self.P.view(self.B, -1, self.S, self.S, self.S)[:, :, self.m, self.m, self.m] * self.coef
        F = torch.zeros(n_atoms + 1, 3, dtype=torch.float64, device=dev)
        for ax in range(3):
            g = torch.zeros_like(D)
            for d in range(1, NO + 1):
                lo, hi = D.narrow(3 - ax, 0, self.S - d), D.narrow(3 - ax, d, self.S - d)
                g.narrow(3 - ax, 0, self.S - d).add_(hi, alpha=self.g[d])
                g.narrow(3 - ax, d, self.S - d).sub_(lo, alpha=self.g[d])
            c = -4.0 * at_q * torch.bmm(self.P, g.reshape(self.B, -1, 1))[:, :, 0]
            F[:, ax].index_add_(0, self.atom.reshape(-1), c.view(self.B, -1, 4).sum(2).reshape(-1))
        return F[:n_atoms]


def _weights(mom):
    K = mom.shape[1]
    k = torch.arange(K, dtype=torch.float64, device=mom.device)
    th = math.pi * (k + 0.5) / K
    T = torch.cos(k[:, None] * th[None, :])
    T[0] *= 0.5
    return 2.0 / K * mom @ T, torch.cos(th)


def _fermi(mom, chi, zeta, electrons, kT, h):
    """(mu, E_band, E_ent, N, rho) from moments."""
    W, x = _weights(mom)
    E = chi[:, None] + zeta[:, None] * x
    lo, hi = float((chi - zeta).min()) - 10 * kT, float((chi + zeta).max()) + 10 * kT
    while True:
        mu = 0.5 * (lo + hi)
        if mu in (lo, hi):
            break
        if float(2.0 * (W * torch.special.expit((mu - E) / kT)).sum()) < electrons:
            lo = mu
        else:
            hi = mu
    t = (E - mu) / kT
    g = torch.special.expit(-t)
    ent = torch.special.entr(g) + torch.special.entr(torch.special.expit(t))
    rho = 2.0 / h ** 3 * (W * g).sum(1)
    return dict(mu=mu, e_band=float(2.0 * (W * E * g).sum()), e_ent=float(-2.0 * kT * (W * ent).sum()), n_elec=float(rho.sum() * h ** 3), rho=rho)


def _exact_scf(c, s):
    n1, n2, n3 = c["n1"], c["n2"], c["n3"]
    h, dev = 0.478125, s["rho"].device
    w, _ = _fd(h)
    ax = []
    for n in (n1, n2, n3):
        th = 2 * math.pi * torch.arange(n, dtype=torch.float64, device=dev) / n
        ax.append(-2.0 * (w[0] + sum(w[d] * torch.cos(d * th) for d in range(1, NO + 1))))
    sym = ax[2][:, None, None] + ax[1][None, :, None] + ax[0][None, None, :]
    grid = lambda v: torch.fft.fftn(v.view(n3, n2, n1))  # noqa: E731
    b = grid(4 * math.pi * (s["rho"] - s["rho"].mean()))
    safe = sym.clone()
    safe[0, 0, 0] = 1.0
    ph = b / safe
    ph[0, 0, 0] = 0.0
    phi = torch.fft.ifftn(ph).real.reshape(-1)
    phi -= phi.mean()
    rho = s["rho"]
    v_out = s["V_loc"] + phi + torch.where(rho > 0, -(3.0 * rho.clamp(min=0) / math.pi) ** (1.0 / 3.0), torch.zeros_like(rho))
    f = v_out - s["V_in"]
    k2, amin = KERKER[0] ** 2, KERKER[1]
    v_pre = s["V_in"] + torch.fft.ifftn(grid(f) * (sym + amin * k2) / (sym + k2)).real.reshape(-1)
    X = [p[0] for p in s["pairs"]][-(MIX_HISTORY + 1):]
    F = [p[1] - p[0] for p in s["pairs"]][-(MIX_HISTORY + 1):]
    nxt = X[-1] + MIX_BETA * F[-1]
    if len(F) > 1:
        dF = torch.stack([b - a for a, b in zip(F, F[1:])], 1)
        dX = torch.stack([b - a for a, b in zip(X, X[1:])], 1)
        Q, Rm = torch.linalg.qr(dF)
        g = torch.linalg.solve_triangular(Rm, (Q.T @ F[-1])[:, None], upper=True)
        nxt = nxt - ((dX + MIX_BETA * dF) @ g)[:, 0]
    return dict(phi=phi, V_out=v_out, resid=float(f.norm() / v_out.norm()), V_pre=v_pre, V_next=nxt)


def _bf(x):
    return x.to(torch.bfloat16).double()


def _cnn_weights(seed, bf16, dev):
    p, C = torch.from_numpy(_cnn_params(seed)).float().double().to(dev), 32
    cut = np.cumsum([0, C * 125, C, C * C * 27, C, C * 27, 1])
    W1, b1, W2, b2, W3, b3 = (p[a:b].clone() for a, b in zip(cut, cut[1:]))
    if bf16:
        W1, W2, W3 = _bf(W1), _bf(W2), _bf(W3)
    return W1.view(C, 1, 5, 5, 5), b1, W2.view(C, C, 3, 3, 3), b2, W3.view(1, C, 3, 3, 3), b3


class _Round(torch.autograd.Function):
    """Rounding to bfloat16 with the identity as its derivative."""

    @staticmethod
    def forward(ctx, x):
        return _bf(x)

    @staticmethod
    def backward(ctx, g):
        return g


def _cnn(c, params, shape, V):
    """rho of the network, activations stored in bfloat16 where the network stores them so."""
    W1, b1, W2, b2, W3, b3 = params
    keep = _Round.apply if c["bf16"] else (lambda x: x)

    def conv(x, W, b):
        k = W.shape[-1]
        x = torch.nn.functional.pad(x, (k // 2,) * 6, mode="circular")
        cols = x.unfold(2, k, 1).unfold(3, k, 1).unfold(4, k, 1)            # [1, I, z, y, x, k, k, k]
        return torch.einsum("nizyxabc,oiabc->nozyx", cols, W) + b.view(1, -1, 1, 1, 1)

    n1, n2, n3 = shape
    x0 = keep(((V + 1.0) / 0.8).float().double().view(1, 1, n3, n2, n1))
    a1 = keep(torch.nn.functional.silu(conv(x0, W1, b1)))
    a2 = keep(torch.nn.functional.silu(conv(a1, W2, b2)))
    return 0.03 * torch.nn.functional.softplus(conv(a2, W3, b3)).reshape(-1)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("step", "bounds", "moments", "forces"):
        h = A_LAT * c["cells"] / c["n"]
        S = 2 * int(math.floor(c["r_cut"] / h + 1e-12)) + 1
        steps = dict(step=c["n_lanczos"] + c["npl"] // 2, bounds=c["n_lanczos"], moments=c["npl"] // 2, forces=c["npl"])[kind]
        if c["n"] ** 3 * float(S) ** 3 * steps * (5.0 if c["nonlocal_"] else 1.0) > 2.2e10:
            return None
        pos, V, proj = _crystal(c["n"], c["cells"], c["nonlocal_"], seed)
        N = c["n"] ** 3
        chi, zeta = _enclosure(h, V, N, seed)
        chi, zeta = chi.clone(), zeta.clone()
        mom = torch.empty(N, c["npl"] + 1, dtype=torch.float64, device=V.device)
        F = torch.zeros(len(pos), 3, dtype=torch.float64, device=V.device)
        B = max(1, min(N, int(1e9 / ((S * h + 9.0) ** 3 * 0.036 * S ** 3)) if proj else int(2e8 / S ** 3)))
        for nodes in torch.arange(N, device=V.device).split(B):
            p = _Plain(c, pos, V, proj, nodes)
            if kind in ("step", "bounds"):
                chi[nodes], zeta[nodes] = p.bounds(c["n_lanczos"], c["margin"])
            if kind in ("step", "moments"):
                mom[nodes] = p.moments(chi[nodes], zeta[nodes], c["npl"])
            if kind == "forces":
                F += p.forces(chi[nodes], zeta[nodes], c["npl"], -0.3, c["kT"], len(pos))
            del p
        if kind == "bounds":
            return dict(chi=chi, zeta=zeta)
        if kind == "moments":
            return dict(moments=mom)
        if kind == "forces":
            return dict(forces=F)
        return dict(_fermi(mom, chi, zeta, synth.ELECTRONS_PER_ATOM * len(pos), c["kT"], h), moments=mom, chi=chi, zeta=zeta)
    if kind == "batch":
        return None
    if kind == "fermi":
        mom, chi, zeta = _fermi_inputs(c, seed)
        return _fermi(mom, chi, zeta, 2 * FERMI_FILL * chi.numel(), c["kT"], 0.478125)
    if kind == "scf":
        return _exact_scf(c, _scf_inputs(c, seed))
    items = _cnn_inputs(c, seed)
    params = _cnn_weights(seed, c["bf16"], items[0][1].device)
    if kind == "predict":
        if c["n1"] * c["n2"] * c["n3"] > 300000:
            return None
        with torch.no_grad():
            return _cnn(c, params, items[0][0], items[0][1])
    params = [p.requires_grad_() for p in params]
    total, rhos = 0.0, []
    for shape, V, ref in items:
        rho = _cnn(c, params, shape, V)
        loss = ((rho - ref) ** 2).mean() / 0.03 ** 2
        loss.backward()
        total += float(loss.detach())
        rhos.append(rho.detach())
    return dict(loss=total, grads=torch.cat([p.grad.reshape(-1) for p in params]).cpu().numpy(), rho=torch.stack(rhos))
