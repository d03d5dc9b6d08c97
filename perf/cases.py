"""The work that users of this library have it do, as timed cases.

A case is one call sequence through the public binding
(paper_2105_00448_gb300.hca) on device tensors:

* ``step``: one coupled step of a 3-D lattice and the read-back of its states
  and fields (what a simulation does hour after hour);
* ``batch``: the same for uneven replicates (virtual patients) that advance
  together in one handle;
* ``biopsy``: one coupled step of a flat lattice with piecewise-constant
  voxel maps (the digital biopsy);
* ``o2``: one quasi-steady oxygen solve on given states and a given previous
  field (hca_write_fields, hca_stage, hca_read_fields);
* ``drug``: one drug over one hour in sub-steps (Crank-Nicolson or implicit
  Euler) on a given field: the paper's own time stepping;
* ``cells``: the cell ODEs and the cellular-automaton update on a given
  lattice;
* ``residual``: the allocation-free oxygen residual of caller-owned arrays (a
  monitor called between other work: the smallest call there is);
* ``net_forward`` / ``net_train``: the warm-start network's guess for one
  lattice, and one training step (gradients and Adam) on one solve.

Inputs are seeded Gaussian random fields with the densities of the
repository's map recipe, made on the GPU.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2105_00448_gb300 import hca

DEV = "cuda"
EMPTY, PROLIF, QUIESC, DEAD, VESSEL, STROMA = range(6)

# physical parameters, spelled out (the library's defaults, Table 1)
DX, DT = 10.0, 60.0
D_K, PHI_K, K1, K0, R_K = 1.05e5, 900.0, 2.5, 20.0, 1.88e4
D_G, PSI_G, KAPPA_G = 9.6e3, 1e-2, 2.0
DECAY = (3.93e3 / 2430e3, 0.983e3 / 18e3, 1.75 / 27.0)
DOSE_INTERVAL = 21
NET_SCALE = 64.0
TRAIN_W_RES = 0.03
# the network's convolutions in parameter order: (name, C_in, C_out)
CONVS = (("enc0", 16, 16), ("enc1", 16, 32), ("enc2", 32, 64), ("enc3", 64, 64), ("dec2", 64, 64), ("dec1", 64, 32),
         ("dec0", 32, 16))


def listed():
    return [
        # the plain FP64 method on the smallest lattice of the configurations:
        # 48^3, one drug, hourly steps, Jacobi-preconditioned CG (the library's
        # default preconditioner)
        dict(name="step-f64-48", kind="step", nx=48, ny=48, nz=48, precision="f64", mg=False, n_drugs=1, corr=4.0),
        # a small FP32 lattice, multigrid-preconditioned: parameter studies on
        # 64^3 boxes, where launches and latency count
        dict(name="step-f32-64", kind="step", nx=64, ny=64, nz=64, precision="f32", mg=True, n_drugs=2, corr=4.0),
        # the headline workload: 256^3, oxygen and two drugs
        dict(name="step-f32-256", kind="step", nx=256, ny=256, nz=256, precision="f32", mg=True, n_drugs=2, corr=8.0),
        # the large single tumour portion
        dict(name="step-f32-512", kind="step", nx=512, ny=512, nz=512, precision="f32", mg=True, n_drugs=2, corr=16.0),
        # virtual patients of uneven size in one handle
        dict(name="batch-f32-16", kind="batch", count=16, sizes=7, precision="f32", mg=True, n_drugs=2, corr=8.0),
        # the paper's 2 x 10 voxel biopsy of 200 x 1000 sites
        dict(name="biopsy-f32", kind="biopsy", vox_y=2, vox_x=10, vox_edge=100, precision="f32", mg=True, n_drugs=2,
             ca_mode=0),
        # one oxygen solve on a patient-shaped lattice whose extents fit nothing
        dict(name="o2-f32-ragged", kind="o2", nx=131, ny=90, nz=77, precision="f32", mg=True),
        # the paper's time stepping of one drug: Crank-Nicolson at one minute
        dict(name="drug-cn-96", kind="drug", nx=96, ny=96, nz=96, precision="f32", mg=True, scheme=1, substeps=60),
        # the cell side of a step alone: ODEs and the stochastic automaton
        dict(name="cells-192", kind="cells", nx=192, ny=192, nz=192, precision="f32", ca_mode=0),
        # the allocation-free residual check
        dict(name="residual-48", kind="residual", nx=48, ny=48, nz=48),
        # the warm-start network: its guess, and one training step
        dict(name="net-forward-128", kind="net_forward", nx=128, ny=128, nz=128),
        dict(name="net-train-64", kind="net_train", nx=64, ny=64, nz=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "batch", "biopsy", "o2", "o2", "drug", "cells", "residual",
                       "net_forward", "net_train"))
    if kind == "step":
        if rng.random() < 0.25:
            e = [_log(rng, 16, 64) for _ in range(3)]
            return dict(kind=kind, nx=e[0], ny=e[1], nz=e[2], precision="f64", mg=rng.random() < 0.5,
                        n_drugs=rng.choice((1, 2)), corr=rng.choice((3.0, 4.0)))
        e = [_log(rng, 40, 320) for _ in range(3)]
        if rng.random() < 0.5:   # half of them with rows of whole 16-byte groups
            e[0] = 4 * max(10, round(e[0] / 4))
        return dict(kind=kind, nx=e[0], ny=e[1], nz=e[2], precision="f32", mg=rng.random() < 0.85,
                    n_drugs=rng.choice((1, 2, 2)), corr=rng.choice((4.0, 8.0)))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 16), sizes=rng.randrange(1000), precision="f32", mg=True,
                    n_drugs=rng.choice((1, 2)), corr=rng.choice((4.0, 8.0)))
    if kind == "biopsy":
        return dict(kind=kind, vox_y=rng.randint(1, 4), vox_x=rng.randint(2, 10), vox_edge=rng.randint(50, 100),
                    precision="f32", mg=True, n_drugs=rng.choice((1, 2)), ca_mode=rng.choice((0, 1)))
    if kind == "o2":
        return dict(kind=kind, nx=_log(rng, 24, 200), ny=_log(rng, 24, 200), nz=_log(rng, 24, 160),
                    precision=rng.choice(("f32", "f32", "f64")), mg=True)
    if kind == "drug":
        return dict(kind=kind, nx=_log(rng, 32, 112), ny=_log(rng, 32, 112), nz=_log(rng, 32, 112), precision="f32",
                    mg=True, scheme=rng.choice((0, 1)), substeps=rng.choice((10, 20, 30, 60)))
    if kind == "cells":
        return dict(kind=kind, nx=_log(rng, 64, 256), ny=_log(rng, 64, 256), nz=_log(rng, 64, 256),
                    precision=rng.choice(("f32", "f32", "f64")), ca_mode=rng.choice((0, 1)))
    if kind == "residual":
        return dict(kind=kind, nx=_log(rng, 24, 200), ny=_log(rng, 24, 160), nz=_log(rng, 24, 160))
    hi = 16 if kind == "net_forward" else 10
    e = [8 * rng.randint(3, hi) for _ in range(3)]
    return dict(kind=kind, nx=e[0], ny=e[1], nz=e[2])


# -------------------------------------------------------------- inputs ---
def _grf(shape, corr, g):
    """Zero-mean unit-variance periodic Gaussian random field (float32)."""
    f = torch.fft.rfftn(torch.randn(shape, generator=g, device=DEV))
    for axis, n in enumerate(shape):
        last = axis == len(shape) - 1
        k = torch.fft.rfftfreq(n, device=DEV) if last else torch.fft.fftfreq(n, device=DEV)
        view = [1, 1, 1]
        view[axis] = k.numel()
        f *= torch.exp(-2.0 * math.pi ** 2 * corr ** 2 * k ** 2).view(view)
    z = torch.fft.irfftn(f, s=shape)
    z -= z.mean()
    return z / z.std()


def _maps(shape, corr, g):
    """(p_cell, perf, p_vessel) of the repository's recipe: cell density 0.4
    +- 0.2, lognormal perfusion of mean 1, vessel fraction 0.12."""
    z1, z2 = _grf(shape, corr, g), _grf(shape, corr, g)
    p_cell = (0.4 + 0.2 * z1).clamp_(0.0, 1.0)
    perf = torch.exp(0.5 * z2 - 0.125)
    p_vessel = -torch.expm1(math.log(1.0 - 0.12) * perf)
    return p_cell.contiguous(), perf.contiguous(), p_vessel.contiguous()


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _lattice(shape, maps, g):
    """uint8 states as seeding leaves them, a tenth of the cells quiescent."""
    p_cell, _, p_vessel = maps
    st = torch.zeros(shape, dtype=torch.uint8, device=DEV)
    st[torch.rand(shape, generator=g, device=DEV) < p_cell] = PROLIF
    st[(st == PROLIF) & (torch.rand(shape, generator=g, device=DEV) < 0.1)] = QUIESC
    st[torch.rand(shape, generator=g, device=DEV) < p_vessel] = VESSEL
    return st


def _ca_like_change(st, g):
    """The lattice one automaton update later: about one cell in a hundred
    divided into a free site, a few died."""
    u = torch.rand(st.shape, generator=g, device=DEV)
    new = st.clone()
    new[(st == EMPTY) & (u < 0.008)] = PROLIF
    new[((st == PROLIF) | (st == QUIESC)) & (u < 0.002)] = DEAD
    return new


def _nb_sum(u):
    s = torch.zeros_like(u)
    for ax in range(3):
        n = u.shape[ax]
        if n > 1:
            s.narrow(ax, 0, n - 1).add_(u.narrow(ax, 1, n - 1))
            s.narrow(ax, 1, n - 1).add_(u.narrow(ax, 0, n - 1))
    return s


def _operator(a, c):
    """u -> A u = (c n + a) u - c sum of neighbours, and its diagonal."""
    d = a + c * _nb_sum(torch.ones_like(a))
    return (lambda u: d * u - c * _nb_sum(u)), d


def _cg(A, d, b, x, rtol, maxit):
    """Jacobi-preconditioned CG in the tensors' precision."""
    r = b - A(x)
    z = r / d
    p, rho, stop = z.clone(), (r * z).sum(), rtol ** 2 * (b * b).sum()
    for k in range(maxit):
        q = A(p)
        alpha = rho / (p * q).sum()
        x = x + alpha * p
        r = r - alpha * q
        if k % 8 == 7 and float((r * r).sum()) <= float(stop):
            break
        z = r / d
        rho, old = (r * z).sum(), rho
        p = z + (rho / old) * p
    return x


def _o2_system(st, K_prev):
    """Reaction and right-hand side of the oxygen equation linearised about K_prev (FP64)."""
    cons = (st == PROLIF) | (st == QUIESC) | (st == STROMA)
    a = torch.where(cons, PHI_K / (K1 + K_prev.double()), 0.0) + torch.where(st == VESSEL, R_K, 0.0).double()
    return a, torch.where(st == VESSEL, R_K * K0, 0.0).double()


def _previous_oxygen(st, fixed_points=2, its=48):
    """The field of the steps before: oxygen roughly in equilibrium with st."""
    K = torch.full(st.shape, 12.0, dtype=torch.float64, device=DEV)
    for _ in range(fixed_points):
        a, b = _o2_system(st, K)
        A, d = _operator(a, D_K / DX ** 2)
        K = _cg(A, d, b, K, 0.0, its)
    return K


def _o2_inputs(case, seed):
    """States and the previous oxygen field of one solve."""
    g = _gen(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    maps = _maps(shape, case.get("corr", 6.0), g)
    before = _lattice(shape, maps, g)
    K_prev = _previous_oxygen(before)
    if case.get("precision") != "f64":
        K_prev = K_prev.float()
    return maps, _ca_like_change(before, g), K_prev


def _residual_inputs(case, seed):
    """States, the field before and a half-converged field of one solve (FP64)."""
    _, st, K_prev = _o2_inputs(dict(case, precision="f64"), seed)
    a, b = _o2_system(st, K_prev)
    A, d = _operator(a, D_K / DX ** 2)
    return st, K_prev.contiguous(), _cg(A, d, b, K_prev, 0.0, 6).contiguous()


def _drug_inputs(case, seed):
    """Perfusion, states and a drug field of the hour before."""
    g = _gen(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    maps = _maps(shape, 6.0, g)
    st = _lattice(shape, maps, g)
    G = 0.4 * torch.exp(0.3 * _grf(shape, 6.0, g))
    return maps, st, G.contiguous()


def _net_inputs(case, seed):
    """One oxygen solve as the training data record it: lattice, perfusion, K before and after."""
    maps, st, K_prev = _o2_inputs(dict(case, precision="f32", corr=8.0), seed)
    K_new = None
    if case["kind"] == "net_train":
        a, b = _o2_system(st, K_prev)
        A, d = _operator(a, D_K / DX ** 2)
        K_new = _cg(A, d, b, K_prev.double(), 0.0, 40).float()
    return maps[1], st, K_prev, K_new


def _net_params(seed):
    """Weights of a network in use: He-normal convolutions (taps, C_out, C_in),
    small biases, 16 head weights and the head's bias."""
    rng = np.random.default_rng(int(seed))
    parts = []
    for _, ci, co in CONVS:
        parts += [rng.standard_normal(27 * co * ci) * math.sqrt(2.0 / (27 * ci)), 0.05 * rng.standard_normal(co)]
    return np.concatenate(parts + [0.05 * rng.standard_normal(17)]).astype(np.float32)


# ------------------------------------------------------------- prepare ---
def _config(case, nx, ny, nz, seed, **more):
    common = dict(precision=case.get("precision", "f32"), seed=int(seed) & 0x7FFFFFFF, rtol_o2=1e-8, rtol_drug=1e-8,
                  picard_tol=1e-6, dose_interval=DOSE_INTERVAL,
                  preconditioner=hca.HCA_PC_MG if case.get("mg") else hca.HCA_PC_JACOBI)
    return hca.make_config(nx, ny, nz, **{**common, **more})


class _Run:
    """One handle with the device buffers its user reads into."""

    def __init__(self, sim, mask, n_fields, shapes):
        self.sim, self.mask = sim, mask
        dt = torch.float64 if sim.fp64 else torch.float32
        self.states = [torch.empty(s, dtype=torch.uint8, device=DEV) for s in shapes]
        self.fields = [torch.empty((n_fields, *s), dtype=dt, device=DEV) for s in shapes]

    def read(self):
        out = []
        for r, (s, f) in enumerate(zip(self.states, self.fields)):
            hca.hca_read_states(self.sim.handle, r, s)
            hca.hca_read_fields(self.sim.handle, r, self.mask, f)
            out.append({"states": s, "fields": f})
        return out


def _all_fields(n_drugs):
    mask = hca.FIELD_O2 | hca.FIELD_PHI | hca.FIELD_P53 | hca.FIELD_VEGFC
    for d in range(n_drugs):
        mask |= hca.FIELD_DRUG[d]
    return mask, 4 + n_drugs


def _voxel_maps(case, g):
    """Piecewise-constant maps: the poorly perfused core in the first half of
    each voxel row, the better perfused edge in the second."""
    vy, vx, e = case["vox_y"], case["vox_x"], case["vox_edge"]
    edge = (torch.arange(vx, device=DEV) >= vx // 2).expand(vy, vx)

    def voxels(core, rim):
        u = torch.rand((vy, vx), generator=g, device=DEV)
        lo = torch.where(edge, rim[0], core[0])
        hi = torch.where(edge, rim[1], core[1])
        v = lo + (hi - lo) * u
        return v.repeat_interleave(e, 0).repeat_interleave(e, 1).float()[None].contiguous()

    perf = voxels((0.1, 0.5), (1.0, 2.0))
    p_vessel = voxels((0.005, 0.02), (0.03, 0.08))
    return voxels((0.5, 0.8), (0.3, 0.6)), perf, p_vessel


def _batch_edges(case):
    rng = np.random.default_rng(case["sizes"])
    return [int((64, 96, 128, 192)[i]) for i in rng.integers(0, 4, size=case["count"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        shape = (case["nz"], case["ny"], case["nx"])
        maps = _maps(shape, case["corr"], _gen(seed))
        cfg = _config(case, shape[2], shape[1], shape[0], seed, n_drugs=case["n_drugs"])
        return kind, _Run(hca.Sim(cfg, maps), *_all_fields(case["n_drugs"]), [shape])
    if kind == "batch":
        g, cfgs, maps, shapes = _gen(seed), [], [], []
        for r, n in enumerate(_batch_edges(case)):
            shapes.append((n, n, n))
            maps.append(_maps(shapes[-1], case["corr"], g))
            cfgs.append(_config(case, n, n, n, seed + 1000 * r, n_drugs=case["n_drugs"]))
        return kind, _Run(hca.Sim(cfgs, maps, batch=True), *_all_fields(case["n_drugs"]), shapes)
    if kind == "biopsy":
        maps = _voxel_maps(case, _gen(seed))
        shape = tuple(maps[0].shape)
        cfg = _config(case, shape[2], shape[1], 1, seed, n_drugs=case["n_drugs"], ca_mode=case["ca_mode"])
        return kind, _Run(hca.Sim(cfg, maps), *_all_fields(case["n_drugs"]), [shape])
    if kind == "o2":
        maps, st, K_prev = _o2_inputs(case, seed)
        cfg = _config(case, case["nx"], case["ny"], case["nz"], seed, n_drugs=0)
        sim = hca.Sim(cfg, maps)
        hca.hca_write_states(sim.handle, 0, st)
        return kind, (sim, K_prev, torch.empty_like(K_prev))
    if kind == "drug":
        maps, st, G = _drug_inputs(case, seed)
        cfg = _config(case, case["nx"], case["ny"], case["nz"], seed, n_drugs=1, drug_scheme=case["scheme"],
                      drug_substeps=case["substeps"])
        sim = hca.Sim(cfg, maps)
        hca.hca_write_states(sim.handle, 0, st)
        hca.hca_set_step(sim.handle, 3)
        return kind, (sim, G, torch.empty_like(G))
    if kind == "cells":
        g = _gen(seed)
        shape = (case["nz"], case["ny"], case["nx"])
        maps = _maps(shape, 8.0, g)
        cfg = _config(dict(case, mg=True), shape[2], shape[1], shape[0], seed, n_drugs=1, ca_mode=case["ca_mode"])
        sim = hca.Sim(cfg, maps)
        dt = torch.float64 if sim.fp64 else torch.float32
        st = _lattice(shape, maps, g)
        cell = ((st == PROLIF) | (st == QUIESC)).to(dt)
        # phi uniform over the cycle (about one cell in a hundred commits this
        # hour), p53 and VEGF at the levels of cells a few hours old
        inner = torch.rand((3, *shape), generator=g, device=DEV, dtype=dt) * cell
        inner[1] *= 0.5
        inner[2] *= 0.1
        hca.hca_write_fields(sim.handle, 0, hca.FIELD_DRUG0, (0.2 * torch.exp(0.3 * _grf(shape, 8.0, g))).to(dt))
        return kind, (sim, st, inner, torch.empty_like(st), torch.empty_like(inner))
    if kind == "residual":
        cfg = _config(dict(precision="f64"), case["nx"], case["ny"], case["nz"], seed)
        return kind, (cfg, *_residual_inputs(case, seed))
    # the network
    perf, st, K_prev, K_new = _net_inputs(case, seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    cfg = _config(dict(precision="f32", mg=True), nx, ny, nz, seed)
    net = hca.Net(nz, ny, nx, trainable=kind == "net_train")
    net.set_params(_net_params(seed))
    if kind == "net_forward":
        return kind, (net, cfg, st, perf, K_prev, torch.empty((nz, ny, nx), device=DEV))
    grads = torch.empty(hca.hca_net_param_count(), device=DEV)
    return kind, (net, cfg, st, perf, K_prev, K_new, grads, torch.empty(1, device=DEV))


# ----------------------------------------------------------------- run ---
def run(state):
    kind, s = state
    if kind in ("step", "batch", "biopsy"):
        s.sim.step(1)
        return s.read()
    if kind == "o2":
        sim, K_prev, out = s
        hca.hca_write_fields(sim.handle, 0, hca.FIELD_O2, K_prev)
        sim.stage(hca.STAGE_O2)
        hca.hca_read_fields(sim.handle, 0, hca.FIELD_O2, out)
        return out
    if kind == "drug":
        sim, G, out = s
        hca.hca_write_fields(sim.handle, 0, hca.FIELD_DRUG0, G)
        sim.stage(hca.STAGE_DRUGS)
        hca.hca_read_fields(sim.handle, 0, hca.FIELD_DRUG0, out)
        return out
    if kind == "cells":
        sim, st, inner, st_out, inner_out = s
        mask = hca.FIELD_PHI | hca.FIELD_P53 | hca.FIELD_VEGFC
        hca.hca_write_states(sim.handle, 0, st)
        hca.hca_write_fields(sim.handle, 0, mask, inner)
        sim.stage(hca.STAGE_ODE | hca.STAGE_CA)
        hca.hca_read_states(sim.handle, 0, st_out)
        hca.hca_read_fields(sim.handle, 0, mask, inner_out)
        return {"states": st_out, "inner": inner_out}
    if kind == "residual":
        return hca.hca_o2_residual_noalloc(*s)
    if kind == "net_forward":
        net, cfg, st, perf, K_prev, out = s
        hca.hca_net_forward(net.handle, cfg, st, perf, K_prev, out)
        return out
    net, cfg, st, perf, K_prev, K_new, grads, loss = s
    hca.hca_net_gradients(net.handle, cfg, st, perf, K_prev, K_new, w_mse=1.0, w_res=TRAIN_W_RES, grads=grads,
                          loss=loss)
    hca.hca_net_adam(net.handle, 1e-3)
    return {"grads": grads, "loss": loss}


# ---------------------------------------------------------------- work ---
def work(case):
    """Each input read once, each output written once; the arithmetic of the
    parts that no better algorithm saves (the cells' RK4, the convolutions)."""
    kind = case["kind"]
    w = 8 if case.get("precision") == "f64" else 4
    cells = 0.35            # consuming sites per site
    rk4 = 60 * 45           # flops per cell and hour
    if kind in ("step", "batch", "biopsy"):
        if kind == "batch":
            n = sum(e ** 3 for e in _batch_edges(case))
        elif kind == "biopsy":
            n = case["vox_y"] * case["vox_x"] * case["vox_edge"] ** 2
        else:
            n = case["nx"] * case["ny"] * case["nz"]
        # states, oxygen, drugs, phi, P, Vc in and out, perfusion in
        return {"bytes": n * (2 + w * (2 * (4 + case["n_drugs"]) + 1)), "flops": n * cells * rk4}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "o2":
        return {"bytes": n * (1 + 2 * w), "flops": 0}
    if kind == "drug":      # every sub-step's field depends on the one before
        return {"bytes": n * (1 + w + 2 * w * case["substeps"]), "flops": 0}
    if kind == "cells":     # states, phi, P, Vc in and out, oxygen and one drug in
        return {"bytes": n * (2 + 8 * w), "flops": n * cells * rk4}
    if kind == "residual":
        return {"bytes": n * 17, "flops": n * 14}
    per_site = 2 * 27 * (16 * 16 + 32 * 16 + (16 * 32 + 64 * 32) / 8 + (32 * 64 + 64 * 64) / 64 + 64 * 64 / 512) + 32
    params = hca.hca_net_param_count()
    if kind == "net_forward":
        return {"bytes": n * 13 + 2 * params, "flops": n * per_site}
    return {"bytes": n * 13 + 24 * params, "flops": 3 * n * per_site}


# --------------------------------------------------------------- exact ---
def _exact_o2(case, seed):
    _, st, K_prev = _o2_inputs(case, seed)
    a, b = _o2_system(st, K_prev)
    A, d = _operator(a, D_K / DX ** 2)
    return _cg(A, d, b, K_prev.double(), 1e-13, 2000)


def _plasma(t):
    interval = DOSE_INTERVAL * DT
    return sum(math.exp(-DECAY[0] * (t - n * interval)) for n in range(int(t // interval) + 1)) if t >= 0 else 0.0


def _exact_drug(case, seed):
    maps, st, G = _drug_inputs(case, seed)
    m = case["substeps"]
    h, c = DT / m, D_G / DX ** 2
    vessel = torch.where(st == VESSEL, KAPPA_G * maps[1].double(), 0.0)
    cn = case["scheme"] == 1
    A0, d0 = _operator(PSI_G + vessel, c)
    mass = (2.0 if cn else 1.0) / h
    u = G.double()
    for k in range(m):
        t0 = 3 * DT + k * h
        b = mass * u + vessel * _plasma(t0 + h)
        if cn:
            b = b - A0(u) + vessel * _plasma(t0)
        u = _cg(lambda v: A0(v) + mass * v, d0 + mass, b, u, 1e-12, 2000)
    return u


def _exact_residual(case, seed):
    st, K_prev, K = _residual_inputs(case, seed)
    a, b = _o2_system(st, K_prev)
    A, _ = _operator(a, D_K / DX ** 2)
    return float((b - A(K)).norm() / b.norm())


def _net_f(p, x):
    """The network on (C, D, H, W) features, in the tensors' precision."""
    F = torch.nn.functional
    layer, o = {}, 0
    for name, ci, co in CONVS:
        w = p[o:o + 27 * co * ci].view(27, co, ci).permute(1, 2, 0).reshape(co, ci, 3, 3, 3)
        o += 27 * co * ci
        layer[name] = (w, p[o:o + co])
        o += co
    conv = lambda name, v: F.conv3d(v, *layer[name], padding=1)

    up = lambda v: F.interpolate(v, scale_factor=2, mode="nearest")
    e0 = torch.relu(conv("enc0", x))
    e1 = torch.relu(conv("enc1", F.avg_pool3d(e0, 2)))
    e2 = torch.relu(conv("enc2", F.avg_pool3d(e1, 2)))
    e3 = torch.relu(conv("enc3", F.avg_pool3d(e2, 2)))
    d2 = torch.relu(conv("dec2", up(e3)) + e2)
    d1 = torch.relu(conv("dec1", up(d2)) + e1)
    d0 = torch.relu(conv("dec0", up(d1)) + e0)
    return (d0 * p[o:o + 16].view(1, 16, 1, 1, 1)).sum(1)[0] + p[o + 16]


def _exact_net(case, seed):
    perf, st, K_prev, K_new = _net_inputs(case, seed)
    Kp = K_prev.double()
    a, b = _o2_system(st, Kp)
    A, d = _operator(a, D_K / DX ** 2)
    x = torch.zeros((1, 16, *st.shape), dtype=torch.float64, device=DEV)
    for s in range(6):
        x[0, s] = st == s
    x[0, 6], x[0, 7], x[0, 8] = perf, Kp / K0, NET_SCALE * (b - A(Kp)) / (d * K0)
    p = torch.from_numpy(_net_params(seed)).to(DEV).double()
    if case["kind"] == "net_forward":
        with torch.no_grad():
            return _net_f(p, x)
    p.requires_grad_(True)
    e = _net_f(p, x) - NET_SCALE * (K_new.double() - Kp) / K0
    loss = (e * e).mean() + TRAIN_W_RES * (A(e) ** 2).mean() / (D_K / DX ** 2) ** 2
    loss.backward()
    return {"grads": p.grad, "loss": loss.detach().view(1)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "o2":
        return _exact_o2(case, seed)
    if kind == "drug":
        return _exact_drug(case, seed)
    if kind == "residual":
        return _exact_residual(case, seed)
    if kind in ("net_forward", "net_train"):
        return _exact_net(case, seed)
    return None   # whole steps and the automaton: states depend on every draw before them
