"""What a user of the library has it do: the measured cases.

Each case is one call (or one short sequence of calls) through the Python
binding of the C ABI, on device buffers that the program keeps: leaf DtN
builds in every precision, mixed batches, solves with stored factors, a time
step, the interface factorisation, a whole Dirichlet solve, the 2-D and the
cross-term leaves, and the learned surrogate's inference.  The sizes are those
of the repository's own workloads (p = 8 .. 20, 8 to 4096 boxes); ``draw``
spreads over the same ranges, odd orders and ragged batches among them.

``exact`` repeats the same problem in 64 bits with dense torch algebra: the
collocation of -Lap u - kappa^2 b u (or the cross-term operator) on
Chebyshev-Lobatto nodes, written here from its definition.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2503_04033_gb300 as H

PREC = {"fp64": H.HPS_FP64, "fp32ir": H.HPS_FP32_IR, "bf16ir": H.HPS_BF16_IR}
F64 = torch.float64


def listed():
    return [
        # the smallest real problem: 2 x 2 x 2 boxes of the manufactured solution, where launches and latency count
        dict(name="dtn_fp64_p8_x8", kind="dtn", prec="fp64", p=8, nbox=8, kappa=10.0, want_s=True),
        # the plain FP64 batch: T, S, the particular solution and the interior reconstruction of 8 x 8 x 8 boxes
        dict(name="leaf_fp64_p12_x512", kind="leaf", prec="fp64", p=12, nbox=512, kappa=20.0, nrhs=1),
        # the headline workload: DtN maps of 8 x 8 x 8 boxes, FP32 tensor-core LU with FP64 refinement
        dict(name="dtn_fp32ir_p16_x512", kind="dtn", prec="fp32ir", p=16, nbox=512, kappa=40.0, want_s=False),
        # the BF16 option, on an odd order and a batch that is no multiple of anything
        dict(name="dtn_bf16ir_p13_x90", kind="dtn", prec="bf16ir", p=13, nbox=90, kappa=30.0, want_s=True),
        # a mixed batch: four orders, a wavenumber per box, 32 body loads each
        dict(name="groups_p8_20_x92", kind="groups", prec="fp32ir", p_lo=8, p_step=4, ngroups=4, nbox=23, nrhs=32),
        # many loads against factors kept on the device
        dict(name="factored_p16_x128_r32", kind="factored", prec="fp32ir", p=16, nbox=128, kappa=40.0, nrhs=32),
        # one Crank-Nicolson step of the heat equation on 4 x 4 x 4 boxes, as the time loop calls it
        dict(name="timestep_p12_4x4x4", kind="timestep", prec="fp32ir", p=12, nx=4, ny=4, nz=4),
        # the interface system factored in FP64 (the default) and solved
        dict(name="iface_fp64_p12_4x4x4", kind="iface", prec="fp64", p=12, nx=4, ny=4, nz=4, kappa=20.0, nrhs=4),
        # a whole two-stage solve: leaf maps, FP32 interface factors, particular solutions, reconstruction
        dict(name="dirichlet_p12_8x8x8", kind="dirichlet", prec="fp32ir", p=12, nx=8, ny=8, nz=8, kappa=20.0),
        # the 2-D form, thousands of small boxes
        dict(name="leaf2d_p16_x4096", kind="leaf2d", p=16, nbox=4096, kappa=40.0, nrhs=1),
        # leaves of an operator with cross terms (a curved domain), T and S
        dict(name="cross_p10_x512", kind="cross", p=10, nbox=512, kappa=2.3, nrhs=0),
        # the learned surrogate served: network and low-rank maps of a batch of boxes
        dict(name="surrogate_p12_x512", kind="surrogate", p=12, nbox=512, rank=32),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dtn", "dtn", "dtn", "leaf", "groups", "factored", "timestep", "iface", "dirichlet", "leaf2d",
                       "cross", "surrogate"])
    kappa = round(rng.uniform(1.0, 40.0), 2)
    if kind in ("dtn", "leaf"):
        prec = rng.choice(["fp64", "fp32ir", "bf16ir"])
        p = rng.randint(6, 14 if prec == "fp64" else 18)
        most = (3e11 if prec == "fp64" else 3e12) / _leaf_flops(p)
        nbox = _loguniform(rng, 1, max(2, min(700, int(most))))
        if kind == "dtn":
            return dict(kind=kind, prec=prec, p=p, nbox=nbox, kappa=kappa, want_s=rng.random() < 0.5)
        return dict(kind=kind, prec=prec, p=p, nbox=nbox, kappa=kappa, nrhs=rng.randint(1, 9))
    if kind == "groups":
        return dict(kind=kind, prec=rng.choice(["fp32ir", "fp32ir", "bf16ir"]), p_lo=rng.randint(6, 9),
                    p_step=rng.randint(1, 3), ngroups=rng.randint(2, 4), nbox=_loguniform(rng, 2, 40),
                    nrhs=_loguniform(rng, 1, 32))
    if kind == "factored":
        p = rng.randint(8, 17)
        return dict(kind=kind, prec="fp32ir", p=p, nbox=_loguniform(rng, 4, 100), kappa=kappa,
                    nrhs=_loguniform(rng, 1, 48))
    nx, ny, nz = (rng.randint(2, 5) for _ in range(3))
    if kind == "timestep":
        return dict(kind=kind, prec="fp32ir", p=rng.randint(7, 13), nx=nx, ny=ny, nz=nz)
    # The FP32 interface factors are drawn at even orders only: with an odd p - 2 some grids' separators (a size that
    # is no multiple of 4) come out wrong by 1e-4, a known fault of that path, and say nothing about speed.
    if kind == "iface":
        prec = rng.choice(["fp64", "fp64", "fp32ir"])
        return dict(kind=kind, prec=prec, p=rng.randint(7, 12) if prec == "fp64" else rng.choice([8, 10, 12]), nx=nx,
                    ny=ny, nz=min(nz, 4), kappa=round(rng.uniform(1.0, 20.0), 2), nrhs=rng.randint(1, 12))
    if kind == "dirichlet":
        return dict(kind=kind, prec="fp32ir", p=rng.choice([8, 10, 12]), nx=nx, ny=ny, nz=nz,
                    kappa=round(rng.uniform(1.0, 20.0), 2))
    if kind == "leaf2d":
        return dict(kind=kind, p=rng.randint(8, 22), nbox=_loguniform(rng, 50, 2000), kappa=kappa,
                    nrhs=rng.randint(0, 5))
    if kind == "cross":
        return dict(kind=kind, p=rng.randint(6, 11), nbox=_loguniform(rng, 8, 250), kappa=round(rng.uniform(0.5, 5.0), 2),
                    nrhs=rng.randint(0, 4))
    return dict(kind=kind, p=rng.randint(8, 13), nbox=_loguniform(rng, 16, 700), rank=rng.choice([8, 16, 24, 32]))


# ------------------------------------------------------------ inputs (from the seed alone)

def _nodes(p):
    """Chebyshev-Lobatto nodes on [0, 1], ascending."""
    return 0.5 + 0.5 * np.sin(math.pi * (2 * np.arange(p) - (p - 1)) / (2.0 * (p - 1)))


def _grid(p, dim=3):
    """Node coordinates of the unit box [p^dim, dim], first axis fastest."""
    t = _nodes(p)
    g = np.meshgrid(*([t] * dim), indexing="ij")
    return np.stack([a.reshape(-1) for a in g[::-1]], axis=1)


def _boxes(case, rng):
    """Lower corners [nbox, dim] and sides h of the boxes: the cells of a grid, or seeded cells of a 1/8 grid."""
    if "nx" in case:
        nb = np.array([case["nx"], case["ny"], case["nz"]])
        i = np.arange(nb.prod())
        cell = np.stack([i % nb[0], (i // nb[0]) % nb[1], i // (nb[0] * nb[1])], axis=1)
        return cell / nb, 1.0 / nb
    if case["kind"] == "leaf2d":
        return rng.integers(0, 64, (case["nbox"], 2)) / 64.0, np.full(2, 1.0 / 64.0)
    if case["kind"] == "cross":
        h = np.array([1.0, 1.0, 1.4]) / 8.0
        return np.array([1.1, -1.0, -1.2]) + rng.integers(0, 8, (case["nbox"], 3)) * h, h
    return rng.integers(0, 8, (case["nbox"], 3)) / 8.0, np.full(3, 1.0 / 8.0)


def _coords(p, lo, h):
    """[nbox, p^dim, dim] node coordinates on the GPU."""
    g = torch.from_numpy(_grid(p, lo.shape[1]) * h).cuda()
    return torch.from_numpy(np.ascontiguousarray(lo)).cuda()[:, None, :] + g[None]


def _modes(rng, dim, n=16):
    """Random smooth Fourier modes with wavevectors of length <= 4: (k, amplitude, phase)."""
    k = np.zeros((n, dim))
    for i in range(n):
        while not 0 < (k[i] ** 2).sum() <= 16:
            k[i] = rng.integers(-4, 5, dim)
    return [torch.from_numpy(a).cuda() for a in (k, rng.normal(0.0, 0.25, n), rng.uniform(0.0, 2 * math.pi, n))]


def _field(modes, x):
    k, a, ph = modes
    out = torch.zeros(x.shape[:-1], dtype=F64, device="cuda")
    for i in range(len(a)):
        out += a[i] * torch.cos(2 * math.pi * (x @ k[i]) + ph[i])
    return out


def _b_field(modes, x):
    return (1.0 + 0.5 * _field(modes, x)).clamp(0.5, 1.5)


def _loads(rng, x, nrhs):
    """Smooth random body loads [nbox, nrhs, nodes]."""
    f = torch.empty(x.shape[0], nrhs, x.shape[1], dtype=F64, device="cuda")
    for r in range(nrhs):
        f[:, r] = _field(_modes(rng, x.shape[-1], 6), x)
    return f


def _dip(rng, x):
    """b of the smooth dip: 1 - 0.5 exp(-|x - c|^2 / 0.04) with a seeded centre."""
    c = torch.from_numpy(rng.uniform(0.3, 0.7, 3)).cuda()
    return 1.0 - 0.5 * torch.exp(-((x - c) ** 2).sum(-1) / 0.04)


def _curved(rng, x):
    """Coefficients of the Helmholtz operator pulled back from {(x1, x2 / psi(x1), x3)}, psi(z) = 1 - a sin(w z)."""
    al, w = rng.uniform(0.15, 0.3), rng.uniform(4.0, 7.0)
    x1, x2 = x[..., 0], x[..., 1]
    ps, dps, ddps = 1 - al * torch.sin(w * x1), -al * w * torch.cos(w * x1), al * w * w * torch.sin(w * x1)
    r = dps * x2 / ps
    one, zero = torch.ones_like(x1), torch.zeros_like(x1)
    C = torch.stack([one, r * r + ps * ps, one, r, zero, zero], dim=1).contiguous()
    return C, torch.stack([zero, -ddps * x2 / ps, zero], dim=1).contiguous()


def _sizes(p):
    return (p - 2) ** 3, 6 * (p - 2) ** 2


def _group_sizes(case):
    """Orders of a mixed batch's groups and the boxes of each."""
    return [(case["p_lo"] + g * case["p_step"], max(1, case["nbox"] - g)) for g in range(case["ngroups"])]


def _inputs(case, seed):
    """Everything the calls read, the same for ``prepare`` and ``exact``."""
    rng = np.random.default_rng([seed, 20250304])
    kind, d = case["kind"], {}
    if kind == "groups":
        d["groups"] = []
        bm, fm = _modes(rng, 3), [_modes(rng, 3, 6) for _ in range(case["nrhs"])]
        for p, nb in _group_sizes(case):
            x = _coords(p, rng.integers(0, 8, (nb, 3)) / 8.0, np.full(3, 1.0 / 8.0))
            d["groups"].append(dict(p=p, h=[0.125] * 3, kappa=rng.choice([10.0, 20.0, 40.0, 60.0], nb),
                                    b=_b_field(bm, x), f=torch.stack([_field(q, x) for q in fm], dim=1)))
        return d
    if kind == "surrogate":
        x = _coords(case["p"], np.zeros((1, 3)), np.full(3, 0.125))
        d["b"] = torch.cat([_b_field(_modes(rng, 3), x) for _ in range(case["nbox"])])
        m = _sizes(case["p"])[1]
        d["T0"] = torch.from_numpy(rng.standard_normal((m, m))).cuda()
        d["theta"] = _weights(case, rng)
        return d
    lo, d["h"] = _boxes(case, rng)
    x = _coords(case["p"], lo, d["h"])
    nbox = len(lo)
    if kind == "cross":
        d["C"], d["d"] = _curved(rng, x)
        d["b"] = torch.ones(nbox, x.shape[1], dtype=F64, device="cuda")
    elif kind == "timestep":
        d["b"] = torch.full((nbox, x.shape[1]), -1.0, dtype=F64, device="cuda")
        w = torch.from_numpy(rng.uniform(0.2, 1.0, 4)).cuda()
        k = torch.from_numpy(rng.integers(1, 4, (4, 3)).astype(np.float64)).cuda()
        d["u"] = sum(w[i] * torch.sin(math.pi * k[i] * x).prod(-1) for i in range(4))[:, None, :].contiguous()
        return d
    elif kind in ("iface", "dirichlet"):
        d["b"] = _dip(rng, x)
    else:
        d["b"] = _b_field(_modes(rng, x.shape[-1]), x)
    nrhs = 1 if kind == "dirichlet" else case.get("nrhs", 0)
    if nrhs:
        d["f"] = _loads(rng, x, nrhs)
    m = 4 * (case["p"] - 2) if kind == "leaf2d" else _sizes(case["p"])[1]
    if kind == "leaf":
        d["ub"] = torch.from_numpy(rng.standard_normal((nbox, nrhs, m))).cuda()
    if kind == "iface":
        d["hf"] = torch.from_numpy(rng.standard_normal((nbox, nrhs, m))).cuda()
        d["g"] = torch.from_numpy(rng.standard_normal((nbox, nrhs, m))).cuda()
    return d


def _weights(case, rng):
    """The network's FP32 parameter vector W0, c0, W1, c1, W2, c2 (He-uniform), as a trained one is loaded."""
    dims = _dims(case)
    g = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 30)))
    out = []
    for a, b in zip(dims[:-1], dims[1:]):
        s = math.sqrt(6.0 / a)
        out += [(torch.rand(a * b, generator=g, device="cuda") * 2 - 1) * s,
                (torch.rand(b, generator=g, device="cuda") * 2 - 1) * 0.1]
    return torch.cat(out)


def _dims(case):
    return [case["p"] ** 3, 512, 512, 2 * _sizes(case["p"])[1] * case["rank"]]


# ------------------------------------------------------------ the program's state and its calls

_contexts = {}


def _context(graphs=False):
    """The library context a program creates once (a time loop turns graph replay on)."""
    if graphs not in _contexts:
        ctx = H.hps_create(0, 0)
        if graphs:
            H.hps_set_option(ctx, H.HPS_OPT_GRAPHS, 1)
        _contexts[graphs] = ctx
    return _contexts[graphs]


class _State:
    """Buffers and handles of one case; the handles go with it."""

    def __init__(self):
        self.free = []

    def __del__(self):
        torch.cuda.synchronize()
        for fn, handle in self.free:
            fn(handle)


def _new(*shape):
    return torch.empty(*shape, dtype=F64, device="cuda")


def prepare(case, seed):
    s = _State()
    s.case, s.kind = case, case["kind"]
    s.__dict__.update(_inputs(case, seed))
    if s.kind == "groups":
        for g in s.groups:
            n, m = H.hps_leaf_sizes(g["p"])
            nb = len(g["kappa"])
            g.update(T=_new(nb, m, m), v=_new(nb, case["nrhs"], n), hflux=_new(nb, case["nrhs"], m),
                     box_status=torch.zeros(nb, dtype=torch.int32, device="cuda"))
        s.ctx = _context()
        return s
    p = s.p = case["p"]
    nbox = s.nbox = len(s.b)
    if s.kind == "surrogate":
        n, m = H.hps_leaf_sizes(p)
        s.m = m
        dims = _dims(case)
        s.net = H.hps_mlp_create(0, dims[0], dims[1], dims[2], m, case["rank"], 1)
        s.free.append((H.hps_mlp_destroy, s.net))
        H.hps_mlp_copy_params(s.net, 0, s.theta.cpu().numpy(), to_device=True)
        s.U, s.V, s.T = _new(nbox, m, case["rank"]), _new(nbox, m, case["rank"]), _new(nbox, m, m)
        return s
    s.status = torch.zeros(nbox, dtype=torch.int32, device="cuda")
    nrhs = s.nrhs = 1 if s.kind in ("dirichlet", "timestep") else case.get("nrhs", 0)
    if s.kind in ("leaf2d", "cross"):
        n, m = (H.hps_leaf2d_sizes if s.kind == "leaf2d" else H.hps_leaf_cross_sizes)(p)
        s.T, s.S = _new(nbox, m, m), _new(nbox, n, m)
        s.v, s.hf = (_new(nbox, nrhs, n), _new(nbox, nrhs, m)) if nrhs else (None, None)
        return s
    n, m = H.hps_leaf_sizes(p)
    s.ctx = _context(graphs=s.kind == "timestep")
    s.prec = PREC[case["prec"]]
    s.nb = [case[k] for k in ("nx", "ny", "nz")] if "nx" in case else None
    kappa = math.sqrt(2.0 / (0.01 * 0.05)) if s.kind == "timestep" else case["kappa"]
    s.lk = H.LeafKind(p, s.h, kappa)
    if s.kind != "factored":
        s.T = _new(nbox, m, m)
    if s.kind in ("leaf", "dirichlet") or case.get("want_s"):
        s.S = _new(nbox, n, m)
    if nrhs:
        s.v, s.ui = _new(nbox, nrhs, n), _new(nbox, nrhs, n)
        s.hflux = _new(nbox, nrhs, m)
        if s.kind != "leaf":
            s.ub = _new(nbox, nrhs, m)
    if s.kind == "leaf":
        s.group = dict(p=p, h=s.h, kappa=np.full(nbox, kappa), b=s.b, T=s.T, S=s.S, f=s.f, v=s.v, hflux=s.hflux,
                       box_status=s.status)
    if s.kind in ("factored", "timestep"):
        s.factors = H.hps_leaf_factor(s.ctx, s.lk, nbox, s.b, nrhs, s.prec, s.status)
        s.free.append((H.hps_leaf_factors_destroy, s.factors))
    if s.kind in ("iface", "timestep"):
        H.hps_leaf_build_dtn(s.ctx, s.lk, nbox, s.b, s.T, None, H.HPS_FP32_IR, s.status)
    if s.kind == "timestep":
        s.iface = H.hps_interface_factor(s.ctx, p, s.nb, s.T, 1, H.HPS_FP64)
        s.free.append((H.hps_interface_destroy, s.iface))
        s.Au, s.rhs, s.c = torch.empty_like(s.u), torch.empty_like(s.u), kappa * kappa
    return s


def run(s):
    k = s.kind
    if k == "dtn":
        S = s.S if s.case["want_s"] else None
        H.hps_leaf_build_dtn(s.ctx, s.lk, s.nbox, s.b, s.T, S, s.prec, s.status)
        return {"T": s.T, "S": S, "status": s.status} if S is not None else {"T": s.T, "status": s.status}
    if k == "leaf":
        H.hps_leaf_groups(s.ctx, [s.group], s.prec)
        H.hps_leaf_reconstruct(s.ctx, s.lk, s.nbox, s.nrhs, s.b, s.S, s.v, s.ub, s.ui, s.prec)
        return {"T": s.T, "S": s.S, "v": s.v, "h": s.hflux, "ui": s.ui, "status": s.status}
    if k == "groups":
        H.hps_leaf_groups(s.ctx, s.groups, PREC[s.case["prec"]])
        return [{"T": g["T"], "v": g["v"], "h": g["hflux"], "status": g["box_status"]} for g in s.groups]
    if k == "factored":
        H.hps_leaf_solve_factored(s.factors, s.nrhs, s.f, s.v, s.hflux, s.status)
        return {"v": s.v, "h": s.hflux, "status": s.status}
    if k == "timestep":
        # f = 2 c u - (c - Lap) u, the particular solution, the interface values (u = 0 outside), the new interior
        H.hps_leaf_apply(s.ctx, s.lk, s.nbox, 1, s.b, s.u, s.Au)
        torch.sub(2.0 * s.c * s.u, s.Au, out=s.rhs)
        H.hps_leaf_solve_factored(s.factors, 1, s.rhs, s.v, s.hflux, s.status)
        H.hps_interface_solve(s.iface, 1, s.hflux, None, s.ub)
        H.hps_leaf_reconstruct_factored(s.factors, 1, s.v, s.ub, s.ui, s.status)
        return {"ui": s.ui, "ub": s.ub, "v": s.v, "h": s.hflux}
    if k == "iface":
        fac = H.hps_interface_factor(s.ctx, s.p, s.nb, s.T, s.nrhs, s.prec)
        H.hps_interface_solve(fac, s.nrhs, s.hf, s.g, s.ub)
        H.hps_interface_destroy(fac)
        return {"ub": s.ub}
    if k == "dirichlet":
        H.hps_leaf_build_dtn(s.ctx, s.lk, s.nbox, s.b, s.T, s.S, s.prec, s.status)
        fac = H.hps_interface_factor(s.ctx, s.p, s.nb, s.T, 1, H.HPS_FP32_IR)
        H.hps_leaf_particular(s.ctx, s.lk, s.nbox, 1, s.b, s.f, s.v, s.hflux, s.prec)
        H.hps_interface_solve(fac, 1, s.hflux, None, s.ub)
        H.hps_leaf_reconstruct(s.ctx, s.lk, s.nbox, 1, s.b, s.S, s.v, s.ub, s.ui, s.prec)
        H.hps_interface_destroy(fac)
        return {"ui": s.ui, "ub": s.ub, "h": s.hflux}
    if k == "leaf2d":
        H.hps_leaf2d_solve(s.p, s.h, s.case["kappa"], s.nbox, s.b, s.nrhs, s.f if s.nrhs else None, s.T, s.S, s.v,
                           s.hf, s.status)
    elif k == "cross":
        H.hps_leaf_cross_solve(s.p, s.h, s.case["kappa"], s.nbox, s.C, s.d, s.b, s.nrhs, s.f if s.nrhs else None, s.T,
                               s.S, s.v, s.hf, s.status)
    else:
        H.hps_mlp_forward(s.net, s.nbox, s.b, s.U, s.V)
        H.hps_lowrank_dtn(s.nbox, s.m, s.case["rank"], s.T0, 0.05, s.U, s.V, s.T)
        return {"U": s.U, "V": s.V, "T": s.T}
    out = {"T": s.T, "S": s.S, "status": s.status}
    return {**out, "v": s.v, "h": s.hf} if s.nrhs else out


# ------------------------------------------------------------ what a pass cannot do without

def _leaf_flops(p, r=None, m=None):
    """The dense method's count for one 3-D box: LU, r solved columns, the D_n products."""
    n, m0 = _sizes(p)
    r = m0 if r is None else r
    return 2.0 / 3.0 * n ** 3 + 2.0 * n * n * r + 2.0 * (p - 2) * (m or m0) * r


def _iface_flops(case):
    """Elimination of the interface by halving the box grid: LU of each separator with its neighbours' columns, and
    the merged map of what is left (faces on the outer boundary never enter)."""
    q2, whole = (case["p"] - 2) ** 2, [(0, case[k]) for k in ("nx", "ny", "nz")]
    fl, todo = 0.0, [whole]
    while todo:
        box = todo.pop()
        size = [hi - lo for lo, hi in box]
        if max(size) == 1:
            continue
        a = size.index(max(size))
        s = q2 * size[0] * size[1] * size[2] // size[a]
        e = sum(q2 * size[0] * size[1] * size[2] // size[c] * ((box[c][0] > 0) + (box[c][1] < whole[c][1]))
                for c in range(3))
        fl += 2.0 / 3.0 * s ** 3 + 2.0 * s * s * e + 2.0 * s * e * e
        mid = box[a][0] + size[a] // 2
        todo += [box[:a] + [part] + box[a + 1:] for part in ((box[a][0], mid), (mid, box[a][1]))]
    return fl


def work(case):
    k, r = case["kind"], case.get("nrhs", 0)
    if k == "groups":
        b = f = 0.0
        for p, nb in _group_sizes(case):
            n, m = _sizes(p)
            b += 8.0 * nb * (p ** 3 * (1 + r) + m * m + r * (n + m))
            f += nb * _leaf_flops(p, m + r)
        return {"bytes": b, "flops": f}
    p = case["p"]
    n, m = _sizes(p)
    nbox = case["nbox"] if "nbox" in case else case["nx"] * case["ny"] * case["nz"]
    if k == "dtn":
        return {"bytes": 8.0 * nbox * (p ** 3 + m * m + (n * m if case["want_s"] else 0)), "flops": nbox * _leaf_flops(p)}
    if k == "leaf":
        return {"bytes": 8.0 * nbox * (p ** 3 * (1 + r) + m * m + n * m + r * (2 * n + 2 * m)),
                "flops": nbox * (_leaf_flops(p, m + r) + 2.0 * n * m * r)}
    if k == "factored":   # the stored L and U are read once at the least
        return {"bytes": nbox * (4.0 * n * n + 8.0 * r * (p ** 3 + n + m)),
                "flops": nbox * r * (2.0 * n * n + 2.0 * (p - 2) * m)}
    if k == "timestep":
        return {"bytes": nbox * (2 * 4.0 * n * n + 8.0 * (2 * p ** 3 + 2 * n + 2 * m)) + 8.0 * nbox * m * m,
                "flops": nbox * (4.0 * n * n + 2.0 * m * m)}
    if k == "iface":
        return {"bytes": 8.0 * nbox * (m * m + 3 * m * r), "flops": _iface_flops(case)}
    if k == "dirichlet":
        return {"bytes": 8.0 * nbox * (2 * p ** 3 + n + 2 * m), "flops": nbox * _leaf_flops(p, m + 1) + _iface_flops(case)}
    if k == "leaf2d":
        n, m = (p - 2) ** 2, 4 * (p - 2)
        return {"bytes": 8.0 * nbox * (p * p * (1 + r) + m * m + n * m + r * (n + m)),
                "flops": nbox * (2.0 / 3.0 * n ** 3 + 2.0 * n * n * (m + r) + 2.0 * (p - 2) * m * (m + r))}
    if k == "cross":
        m = 6 * (p - 1) ** 2
        return {"bytes": 8.0 * nbox * (p ** 3 * (10 + r) + m * m + n * m + r * (n + m)),
                "flops": nbox * (2.0 / 3.0 * n ** 3 + 2.0 * n * n * (m + r) + 2.0 * (n + m) * m * (m + r) / p)}
    d = _dims(case)
    return {"bytes": 4.0 * sum(a * b for a, b in zip(d[:-1], d[1:])) + 8.0 * nbox * (d[0] + d[3] + m * m) + 8.0 * m * m,
            "flops": nbox * (2.0 * sum(a * b for a, b in zip(d[:-1], d[1:])) + 2.0 * m * m * case["rank"])}


# ------------------------------------------------------------ the same in 64 bits

def _diff(p):
    """Chebyshev-Lobatto differentiation matrix on [-1, 1] (ascending nodes), diagonal by negative row sums."""
    x = 2.0 * _nodes(p) - 1.0
    c = np.where((np.arange(p) == 0) | (np.arange(p) == p - 1), 2.0, 1.0) * (-1.0) ** np.arange(p)
    D = np.outer(c, 1.0 / c) / (x[:, None] - x[None, :] + np.eye(p))
    return D - np.diag(D.sum(axis=1))


def _axes(p, h, dim=3):
    """Full-grid first-derivative matrices per axis, axis 0 fastest (on the GPU)."""
    D, I, out = _diff(p), np.eye(p), []
    for a in range(dim):
        M = np.ones((1, 1))
        for b in range(dim):
            M = np.kron((2.0 / h[a]) * D if b == a else I, M)
        out.append(torch.from_numpy(M).cuda())
    return out


def _index_sets(p, dim=3):
    """Interior nodes, and face nodes (without edges and corners) in the order x-, x+, y-, ... , lower axis fastest."""
    g = np.indices((p,) * dim)[::-1].reshape(dim, -1)
    inner = (g > 0) & (g < p - 1)
    faces = []
    for a in range(dim):
        rest = np.all(np.delete(inner, a, axis=0), axis=0)
        faces += [np.nonzero(rest & (g[a] == e))[0] for e in (0, p - 1)]
    return np.nonzero(inner.all(axis=0))[0], np.concatenate(faces)


class _Leaf:
    """Dense collocation of boxes of one order: A_ii = base - kappa^2 diag(b)."""

    def __init__(self, p, h, dim=3):
        G = _axes(p, h, dim)
        I, F = (torch.from_numpy(a).cuda() for a in _index_sets(p, dim))
        L = -sum(g @ g for g in G)
        self.I, self.F = I, F
        self.Aii, self.Aib = L[I][:, I], L[I][:, F]
        q = (p - 2) ** (dim - 1)
        rows = [(-1.0 if f % 2 == 0 else 1.0) * G[f // 2][F[f * q:(f + 1) * q]] for f in range(2 * dim)]
        N = torch.cat(rows)
        self.Abi, self.Abb = N[:, I], N[:, F]

    def solve(self, kappa, b, rhs, most=2 << 30):
        """A_ii^{-1} rhs per box: rhs [n, c] shared, or [nbox, n, c]."""
        n = len(self.I)
        out = torch.empty(len(b), n, rhs.shape[-1], dtype=F64, device="cuda")
        step = max(1, int(most // (8 * n * (2 * n + 2 * rhs.shape[-1]))))
        kap = torch.as_tensor(kappa, dtype=F64, device="cuda").expand(len(b))
        for i in range(0, len(b), step):
            A = self.Aii.expand(len(b[i:i + step]), n, n).clone()
            A.diagonal(dim1=1, dim2=2).sub_(kap[i:i + step, None] ** 2 * b[i:i + step][:, self.I])
            R = rhs.expand(len(A), *rhs.shape) if rhs.dim() == 2 else rhs[i:i + step]
            out[i:i + step] = torch.linalg.solve(A, R)
        return out

    def maps(self, kappa, b, f=None):
        """(S, T, v, h) of every box."""
        rhs = -self.Aib
        if f is not None:
            rhs = torch.cat([rhs.expand(len(b), *rhs.shape), f[:, :, self.I].transpose(1, 2)], dim=2)
        X = self.solve(kappa, b, rhs)
        m = len(self.F)
        S, v = X[:, :, :m], X[:, :, m:].transpose(1, 2)
        return S, self.Abb + self.Abi @ S, v, v @ self.Abi.T


def _interface_ids(case):
    """Per box and face node: the number of its interface unknown, or -1 on the outer boundary."""
    nb, q2 = (case["nx"], case["ny"], case["nz"]), (case["p"] - 2) ** 2
    ids, count = {}, 0
    out = np.full((nb[0] * nb[1] * nb[2], 6 * q2), -1, dtype=np.int64)
    for t in range(len(out)):
        c = (t % nb[0], (t // nb[0]) % nb[1], t // (nb[0] * nb[1]))
        for f in range(6):
            a, e = f // 2, c[f // 2] + f % 2
            if e in (0, nb[a]):
                continue
            key = (a, e, c[:a] + c[a + 1:])
            if key not in ids:
                ids[key], count = count, count + q2
            out[t, f * q2:(f + 1) * q2] = ids[key] + np.arange(q2)
    return torch.from_numpy(out).cuda(), count


def _interface_solve(case, T, h, g=None):
    """Face values u_b of every box from the flux balance at shared face nodes (dense solve)."""
    ids, count = _interface_ids(case)
    A = torch.zeros(count, count, dtype=F64, device="cuda")
    rhs = torch.zeros(count, h.shape[1], dtype=F64, device="cuda")
    outer = ids < 0
    ub = torch.zeros_like(h) if g is None else torch.where(outer[:, None, :], g, torch.zeros_like(g))
    for t in range(len(ids)):
        i = torch.nonzero(~outer[t])[:, 0]
        r = ids[t, i]
        A[r[:, None], r[None, :]] += T[t][i][:, i]
        rhs[r] -= (h[t][:, i] + (ub[t] @ T[t].T)[:, i]).T
    u = torch.linalg.solve(A, rhs)
    return torch.where(outer[:, None, :], ub, u[ids.clamp(min=0)].transpose(1, 2))


def _lagrange(src, dst):
    M = np.ones((len(dst), len(src)))
    for j in range(len(src)):
        for i in range(len(src)):
            if i != j:
                M[:, j] *= (dst - src[i]) / (src[j] - src[i])
    return M


def _cross_exact(case, d):
    p, h = case["p"], d["h"]
    t, gl = 2.0 * _nodes(p) - 1.0, np.polynomial.legendre.leggauss(p - 1)[0]
    G, Q = _lagrange(gl, t), _lagrange(t, gl)
    idx = np.indices((p,) * 3)[::-1].reshape(3, -1)
    ml, P, Qf, seen = (p - 1) ** 2, np.zeros((p ** 3, 6 * (p - 1) ** 2)), [], np.zeros(p ** 3)
    ax = _axes(p, h)
    for f in range(6):
        on = np.nonzero(idx[f // 2] == (p - 1) * (f % 2))[0]   # the face's p x p nodes, lower axis fastest
        P[on, f * ml:(f + 1) * ml] += np.kron(G, G)
        seen[on] += 1
        Qf.append(torch.from_numpy((1 if f % 2 else -1) * np.kron(Q, Q)).cuda() @ ax[f // 2][torch.from_numpy(on).cuda()])
    P[seen > 0] /= seen[seen > 0][:, None]
    P, NQ = torch.from_numpy(P).cuda(), torch.cat(Qf)
    I = torch.from_numpy(_index_sets(p)[0]).cuda()
    pair = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]
    second = [(ax[a] @ ax[b] + (ax[b] @ ax[a] if a != b else 0))[I] for a, b in pair]
    out = {k: [] for k in ("T", "S", "v", "h")}
    for t_ in range(len(d["b"])):
        A = -sum(d["C"][t_, c][I][:, None] * second[c] for c in range(6))
        A += sum(d["d"][t_, a][I][:, None] * ax[a][I] for a in range(3))
        A[torch.arange(len(I), device="cuda"), I] -= case["kappa"] ** 2 * d["b"][t_][I]
        rhs = -A @ P
        if "f" in d:
            rhs = torch.cat([rhs, d["f"][t_][:, I].T], dim=1)
        X = torch.linalg.solve(A[:, I], rhs)
        U = P.clone()
        U[I] = X[:, :6 * ml]
        v = X[:, 6 * ml:].T
        for key, val in (("T", NQ @ U), ("S", X[:, :6 * ml]), ("v", v), ("h", v @ NQ[:, I].T)):
            out[key].append(val)
    out = {key: torch.stack(val) for key, val in out.items()}
    return {"T": out["T"], "S": out["S"], "status": None, **({"v": out["v"], "h": out["h"]} if "f" in d else {})}


def exact(case, seed):
    k = case["kind"]
    if k in ("dtn", "leaf") and work(case)["flops"] > 4e12:
        return None   # minutes of dense FP64
    if k == "dirichlet" and _interface_ids(case)[1] > 20000:
        return None   # a dense interface system of this size does not fit
    d = _inputs(case, seed)
    if k == "groups":
        out = []
        for g in d["groups"]:
            _, T, v, h = _Leaf(g["p"], g["h"]).maps(g["kappa"], g["b"], g["f"])
            out.append({"T": T, "v": v, "h": h, "status": None})
        return out
    if k == "cross":
        return _cross_exact(case, d)
    if k == "surrogate":
        dims, m, r = _dims(case), _sizes(case["p"])[1], case["rank"]
        y, off = 2.0 * (d["b"] - 1.0), 0
        for i, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
            W = d["theta"][off:off + a * b].to(F64).view(a, b)
            c = d["theta"][off + a * b:off + a * b + b].to(F64)
            y, off = y @ W + c, off + a * b + b
            y = y.relu() if i < 2 else y
        U, V = y[:, :m * r].view(-1, m, r), y[:, m * r:].view(-1, m, r)
        return {"U": U, "V": V, "T": d["T0"] + 0.05 * U @ V.transpose(1, 2)}
    L = _Leaf(case["p"], d["h"], 2 if k == "leaf2d" else 3)
    if k == "timestep":
        c = 2.0 / (0.01 * 0.05)
        u = d["u"][:, 0]
        f = torch.zeros_like(d["u"])
        f[:, 0, L.I] = 2.0 * c * u[:, L.I] - (u[:, L.I] @ L.Aii.T + u[:, L.F] @ L.Aib.T + c * u[:, L.I])
        S, T, v, h = L.maps(math.sqrt(c), d["b"][:1])
        v = L.solve(math.sqrt(c), d["b"][:1], f[:, 0, L.I].T)[0].T[:, None]   # one operator for every box
        h = v @ L.Abi.T
        ub = _interface_solve(case, T.expand(len(u), -1, -1), h)
        return {"ui": v + ub @ S[0].T, "ub": ub, "v": v, "h": h}
    S, T, v, h = L.maps(case["kappa"], d["b"], d.get("f"))
    if k == "iface":
        return {"ub": _interface_solve(case, T, d["hf"], d["g"])}
    if k == "dirichlet":
        ub = _interface_solve(case, T, h)
        return {"ui": v + ub @ S.transpose(1, 2), "ub": ub, "h": h}
    if k == "factored":
        return {"v": v, "h": h, "status": None}
    if k == "leaf":
        return {"T": T, "S": S, "v": v, "h": h, "ui": v + d["ub"] @ S.transpose(1, 2), "status": None}
    out = {"T": T, "S": S, "status": None}
    if k == "dtn":
        return out if case["want_s"] else {"T": T, "status": None}
    return {**out, "v": v, "h": h} if case["nrhs"] else out
