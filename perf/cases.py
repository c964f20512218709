"""The calls this library is used for, as measurable cases.

A user of the library solves the interstitial Poisson step of an SCF loop for free-standing Pd
clusters (whole solves, alone and in batches, from the density model or from a density on the
grid), runs parts of the step on its own buffers (deposit, two-grid operators, projection),
solves inside the spheres, forms the interstitial H and S, and trains the guess network's
layers.  Each case is one such call with the sizes of this repository's workloads: magic-number
fcc clusters of 13 to 561 atoms (NN 5.20 bohr, sphere radius 2.4), graded meshes of 65 to 385
nodes per axis (0.12 to 0.6 bohr, 10 bohr vacuum), the three-exponent Slater density model, and
the Pd basis of 25 functions per atom.  Atoms are displaced by up to 0.03 bohr and the weights
and nonspherical coefficients are drawn, all from the seed.
"""
from __future__ import annotations

import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_0806_1723_gb300 import binding as B

PI = math.pi
NN, RADIUS, VACUUM, Z_PD = 5.20, 2.4, 10.0, 46.0
ZETA = (1.5, 3.0, 8.0)
N_RAD, R_MIN = 429, 1e-5
SHELL_ATOMS = {1: 13, 2: 55, 3: 147, 4: 309, 5: 561}
# nodes per axis that coarsen to at most 9
NODES = (65, 81, 97, 113, 129, 161, 193, 225, 257, 321, 385)


def listed():
    return [
        # one step of a large cluster's SCF loop: the next density, started from the previous
        # potential (the repository's largest workload)
        {"name": "scf_pd561_385", "kind": "solve", "shells": 5, "n": 385, "graded": True, "mixed": True, "start": "warm"},
        # a fresh mid-size cluster: learned first iterate, mixed precision
        {"name": "solve_pd55_129", "kind": "solve", "shells": 2, "n": 129, "graded": True, "mixed": True,
         "start": "learned"},
        # the same cluster with everything in FP64, for users who want no FP32 anywhere
        {"name": "plain_pd55_129", "kind": "solve", "shells": 2, "n": 129, "graded": True, "mixed": False, "start": "zero"},
        # the smallest whole solve: launch latency and short kernels
        {"name": "plain_pd13_65", "kind": "solve", "shells": 1, "n": 65, "graded": False, "mixed": False, "start": "zero"},
        # many clusters of uneven sizes in one call (screening runs)
        {"name": "batch_uneven_8", "kind": "batch", "members": "1@65 2@129 3@129 1@97 2@97 3@161 2@161 1@129"},
        # a density that comes from an SCF code: values on the grid and tables inside the spheres
        {"name": "raw_pd55_129", "kind": "raw", "shells": 2, "n": 129},
        # the right-hand side alone, for callers with their own solver
        {"name": "deposit_pd147_161", "kind": "deposit", "shells": 3, "n": 161},
        # inside the spheres: the density's harmonics on the radial mesh and the radial solves
        {"name": "spheres_pd55", "kind": "spheres", "shells": 2, "n": 97, "n_rad": 429},
        # interstitial overlap and Hamiltonian of the Slater basis
        {"name": "hs_pd55_97", "kind": "hs", "shells": 2, "n": 97},
        # one layer of the guess network's training (the widest grid, decoder input)
        {"name": "layer_33_48_16", "kind": "layer", "n": 33, "nb": 8, "cin": 48, "cout": 16},
        # callers composing their own multigrid: smoothing, residual, transfers on a ragged grid
        {"name": "twogrid_129x97x113", "kind": "twogrid", "nx": 129, "ny": 97, "nz": 113, "sweeps": 2},
        # the smallest call: potentials back onto the sphere surfaces
        {"name": "project_pd13_65", "kind": "project", "shells": 1, "n": 65},
    ]


def _feasible(shells, most):
    """Mesh sizes whose 0.6 bohr edge spacing covers the box of a cluster."""
    half = shells * NN + RADIUS + VACUUM
    return [n for n in NODES if n <= most and 0.6 * (n - 1) / 2 > 1.05 * half]


def draw(rng):
    kind = rng.choice(["solve", "solve", "scf", "plain", "batch", "raw", "deposit", "spheres", "hs", "layer", "twogrid",
                       "project"])
    if kind in ("solve", "scf"):
        shells = rng.randint(1, 4 if kind == "solve" else 5)
        start = "warm" if kind == "scf" else rng.choice(["zero", "learned"])
        return {"kind": "solve", "shells": shells, "n": rng.choice(_feasible(shells, 225 if kind == "solve" else 321)),
                "graded": True, "mixed": True, "start": start}
    if kind == "plain":
        shells = rng.randint(1, 3)
        return {"kind": "solve", "shells": shells, "n": rng.choice(_feasible(shells, 161)), "graded": rng.random() < 0.7,
                "mixed": False, "start": rng.choice(["zero", "warm"])}
    if kind == "batch":
        members = []
        for _ in range(rng.randint(2, 10)):
            shells = rng.randint(1, 3)
            members.append("%d@%d" % (shells, rng.choice(_feasible(shells, 193))))
        return {"kind": "batch", "members": " ".join(members)}
    if kind in ("raw", "deposit", "project"):
        shells = rng.randint(1, 3 if kind == "raw" else 4)
        return {"kind": kind, "shells": shells, "n": rng.choice(_feasible(shells, 161 if kind == "raw" else 257))}
    if kind == "spheres":
        shells = rng.randint(1, 3)
        return {"kind": "spheres", "shells": shells, "n": 129, "n_rad": rng.randint(150, 500)}
    if kind == "hs":
        shells = rng.randint(1, 2)
        return {"kind": "hs", "shells": shells, "n": rng.choice([n for n in (81, 89, 97, 103, 113) if shells == 1 or n >= 89])}
    if kind == "layer":
        cin, cout = rng.choice([(16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (128, 64), (96, 32), (48, 16)])
        return {"kind": "layer", "n": rng.choice([9, 17, 33]), "nb": rng.randint(1, 12), "cin": cin, "cout": cout}
    nx, ny, nz = (rng.choice([65, 81, 97, 113, 129]) for _ in range(3))
    return {"kind": "twogrid", "nx": nx, "ny": ny, "nz": nz, "sweeps": rng.randint(1, 4)}


# ------------------------------------------------------------------ inputs
def _axis(n, half, h_min, h_max):
    """The graded axis: slope h_min m at the centre and h_max m at the ends (exponent at most 6)."""
    m = (n - 1) / 2
    a, b, p = half, 0.0, 1.0
    if h_max > h_min:
        a = h_min * m
        b = half - a
        p = (h_max * m - a) / b
        if p > 6.0:
            p, b = 6.0, (h_max * m - half) / 5.0
            a = half - b
    xi = (np.arange(n) - m) / m
    x = a * xi + b * np.sign(xi) * np.abs(xi) ** p
    x[0], x[-1] = -half, half
    return x


def _positions(shells, rng):
    """The fcc cuboctahedron with `shells` shells around a centre atom, slightly displaced."""
    r = range(-2 * shells, 2 * shells + 1)
    pts = [(i, j, k) for i in r for j in r for k in r
           if (i + j + k) % 2 == 0 and max(abs(i), abs(j), abs(k)) <= shells and abs(i) + abs(j) + abs(k) <= 2 * shells]
    pos = np.array(pts, dtype=float) * (NN / math.sqrt(2.0))
    return pos + rng.uniform(-0.03, 0.03, pos.shape)


def _densities(na, rng):
    """Slater weights and nonspherical coefficients of one density and of the next one of the loop."""
    u = rng.uniform(0.5, 1.5, (na, 3))
    w = Z_PD * u / u.sum(1, keepdims=True)
    c = rng.normal(0.0, 1e-3, (na, 24))
    w2 = w * (1.0 + 0.01 * rng.normal(size=w.shape))
    w2 = Z_PD * w2 / w2.sum(1, keepdims=True)
    return w, c, w2, c * (1.0 + 0.01 * rng.normal(size=c.shape))


def _cluster(shells, n, graded, seed):
    """One cluster's numbers on the host; its slater_w and c_lm are the density to be solved."""
    rng = np.random.default_rng([seed, shells, n])
    pos = _positions(shells, rng)
    na = len(pos)
    if graded:
        axis = _axis(n, shells * NN + RADIUS + VACUUM, 0.12, 0.6)
    else:
        half = max(12.0, shells * NN + RADIUS + 4.0)
        axis = _axis(n, half, 2 * half / (n - 1), 2 * half / (n - 1))
    w0, c0, w, c = _densities(na, rng)
    return SimpleNamespace(pos=pos, Z=np.full(na, Z_PD), R=np.full(na, RADIUS), slater_w=w, c_lm=c, prev_w=w0, prev_c=c0,
                           slater_zeta=np.tile(np.array(ZETA), (na, 1)), n=n, centre=(0.0, 0.0, 0.0), axis=axis, na=na)


def _device_cluster(c):
    return B.DeviceCluster(c, axes=(c.axis, c.axis, c.axis))


def _set_density(dc, w, clm):
    dc.w.copy_(torch.as_tensor(w))
    dc.clm.copy_(torch.as_tensor(clm))


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _raw_density(c):
    """A density on the nodes and each sphere's spherical component on the radial mesh, as an SCF
    code holds them (here from the density model, in torch)."""
    ax = _cuda(c.axis)
    ne = _slater_sum(c, ax, ax, ax)
    own, d = _owner(c, ax, ax, ax)
    flat = own.reshape(-1)
    inside = torch.nonzero(flat >= 0).reshape(-1)
    _add_nonspherical(c, ne.view(-1), inside, flat[inside], d)
    dx = math.log(RADIUS / R_MIN) / (N_RAD - 1)
    r = RADIUS * torch.exp((torch.arange(N_RAD, dtype=torch.float64, device="cuda") - (N_RAD - 1)) * dx)
    A, Bc, W, z = _neighbour_sums(c)
    rho = (W[:, :, None] * torch.exp(-z[:, None] * r)).sum(1) + _neighbour_average(A, Bc, z, r)
    return ne, rho * math.sqrt(4 * PI)


def _bf16(t):
    return t.to(torch.bfloat16)


def _layer_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    nodes = case["nb"] * case["n"] ** 3
    x = _bf16(torch.relu(torch.randn(nodes, case["cin"], generator=g, device="cuda")))
    w = _bf16(torch.randn(27, case["cin"], case["cout"], generator=g, device="cuda") * math.sqrt(2.0 / (27 * case["cin"])))
    bias = 0.1 * torch.randn(case["cout"], generator=g, device="cuda")
    dy = _bf16(1e-3 * torch.randn(nodes, case["cout"], generator=g, device="cuda")).float()
    saved = torch.relu(torch.randn(nodes, case["cout"], generator=g, device="cuda"))
    return x, w, bias, dy, saved


def _grid_inputs(case, seed):
    """Two-grid inputs: graded ragged axes, a rough field, a right-hand side, a coarse correction."""
    rng = np.random.default_rng(seed)
    n = (case["nx"], case["ny"], case["nz"])
    ax = [_cuda(_axis(m, 20.0, 0.6 * 40.0 / (m - 1), 1.5 * 40.0 / (m - 1)) + rng.uniform(-0.01, 0.01, m)) for m in n]
    g = torch.Generator(device="cuda").manual_seed(seed)
    rand = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    return ax, rand(*n[::-1]), rand(*n[::-1]), rand(*[(m + 1) // 2 for m in n[::-1]])


def _hs_inputs(case, seed):
    c = _cluster(case["shells"], case["n"], True, seed)
    ax = _cuda(c.axis)
    rng = np.random.default_rng([seed, 7])
    V = torch.zeros((c.n,) * 3, dtype=torch.float64, device="cuda")
    for p in c.pos:
        r = _distance(p, ax, ax, ax)
        V -= rng.uniform(8.0, 12.0) * torch.exp(-rng.uniform(0.5, 0.8) * r) / r.clamp_min(0.5)
    return c, ax, V


def _potential_field(c, seed):
    """A smooth potential on the nodes: screened charges at the atoms."""
    ax = _cuda(c.axis)
    rng = np.random.default_rng([seed, 5])
    u = torch.zeros((c.n,) * 3, dtype=torch.float64, device="cuda")
    for p in c.pos:
        u += rng.uniform(1.0, 4.0) * torch.exp(-0.7 * _distance(p, ax, ax, ax))
    return ax, u


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case, kind=kind)
    if kind == "solve":
        c = _cluster(case["shells"], case["n"], case["graded"], seed)
        s.dc = _device_cluster(c)
        s.solver = B.Poisson(n_max=c.n, max_atoms=c.na,
                             precision=B.LASTO_PREC_MIXED if case["mixed"] else B.LASTO_PREC_FP64)
        if case["start"] == "learned":
            s.solver.set_guess()
        s.v = torch.empty((c.na, 25), dtype=torch.float64, device="cuda")
        s.pot = torch.empty(s.dc.N, dtype=torch.float64, device="cuda")
        s.guess = torch.zeros_like(s.pot) if case["start"] == "warm" else None
        # the loop's previous density has been solved in the same buffers
        _set_density(s.dc, c.prev_w, c.prev_c)
        s.solver.solve(s.dc, s.v, potential=s.pot, guess=s.guess)
        if s.guess is not None:
            s.guess.copy_(s.pot)
        _set_density(s.dc, c.slater_w, c.c_lm)
    elif kind == "batch":
        cls = _members(case, seed)
        s.dc = [_device_cluster(c) for c in cls]
        s.solver = B.Poisson(n_max=max(c.n for c in cls), max_atoms=max(c.na for c in cls), max_batch=len(cls),
                             precision=B.LASTO_PREC_MIXED)
        s.solver.set_guess()
        s.v = torch.empty((sum(c.na for c in cls), 25), dtype=torch.float64, device="cuda")
        s.pot = torch.empty(sum(d.N for d in s.dc), dtype=torch.float64, device="cuda")
        for d, c in zip(s.dc, cls):
            _set_density(d, c.prev_w, c.prev_c)
        s.solver.solve(s.dc, s.v, potential=s.pot)
        for d, c in zip(s.dc, cls):
            _set_density(d, c.slater_w, c.c_lm)
    elif kind == "raw":
        c = _cluster(case["shells"], case["n"], True, seed)
        ne, rho00 = _raw_density(c)
        s.rc = B.RawCluster(c.pos, c.Z, c.R, c.axis, c.axis, c.axis, c.centre, 0.99 * ne, 0.99 * rho00, r_min=R_MIN)
        s.solver = B.Poisson(n_max=c.n, max_atoms=c.na, precision=B.LASTO_PREC_MIXED)
        s.v = torch.empty((c.na, 25), dtype=torch.float64, device="cuda")
        s.pot = torch.empty(c.n ** 3, dtype=torch.float64, device="cuda")
        s.solver.solve_raw(s.rc, s.v, potential=s.pot)
        s.rc.density.copy_(ne)
        s.rc.rho00.copy_(rho00)
    elif kind == "deposit":
        s.dc = _device_cluster(_cluster(case["shells"], case["n"], True, seed))
    elif kind == "spheres":
        c = _cluster(case["shells"], case["n"], True, seed)
        s.dc = _device_cluster(c)
        s.v_R = _cuda(np.random.default_rng([seed, 3]).normal(size=(c.na, 25)))
    elif kind == "hs":
        c, s.ax, s.V = _hs_inputs(case, seed)
        s.pos, s.R = _cuda(c.pos), _cuda(c.R)
    elif kind == "layer":
        s.x, s.w, s.bias, s.dy, s.saved = _layer_inputs(case, seed)
        s.wpk, s.wflip, s.wpk_flip = (torch.empty_like(s.w) for _ in range(3))
        s.err = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind == "twogrid":
        s.ax, s.u, s.b, s.ec = _grid_inputs(case, seed)
        s.u32, s.b32 = s.u.float(), s.b.float()
    elif kind == "project":
        c = _cluster(case["shells"], case["n"], True, seed)
        s.ax, s.u = _potential_field(c, seed)
        s.pos, s.R = _cuda(c.pos), _cuda(c.R)
    else:
        raise ValueError(kind)
    return s


def _members(case, seed):
    return [_cluster(int(m.split("@")[0]), int(m.split("@")[1]), True, seed + 1000 * q)
            for q, m in enumerate(case["members"].split())]


def run(s):
    kind = s.kind
    if kind == "solve":
        s.solver.solve(s.dc, s.v, potential=s.pot, guess=s.guess)
        return {"v_lm": s.v, "potential": s.pot}
    if kind == "batch":
        s.solver.solve(s.dc, s.v, potential=s.pot)
        return {"v_lm": s.v, "potential": s.pot}
    if kind == "raw":
        s.solver.solve_raw(s.rc, s.v, potential=s.pot)
        return {"v_lm": s.v, "potential": s.pot}
    if kind == "deposit":
        b, owner, _ = B.lasto_op_deposit(s.dc, precision=B.LASTO_PREC_MIXED)
        return {"b": b, "owner": owner}
    if kind == "spheres":
        rho, _ = B.lasto_op_sphere_density(s.dc, n_rad=s.case["n_rad"], r_min=R_MIN)
        return {"rho": rho, "v": B.lasto_op_inner_solve(s.dc.R, s.dc.Z, rho, s.v_R, r_min=R_MIN)}
    if kind == "hs":
        S, H = B.lasto_op_interstitial_hs(s.ax, s.ax, s.ax, s.pos, s.R, s.V)
        return {"S": S, "H": H}
    if kind == "layer":
        return _run_layer(s)
    if kind == "twogrid":
        u = B.lasto_op_smooth(*s.ax, s.u.clone(), s.b, sweeps=s.case["sweeps"])
        r = B.lasto_op_residual(*s.ax, u, s.b)
        rc = B.lasto_op_restrict(*s.ax, r)
        v = B.lasto_op_prolong_add(*s.ax, s.ec, u.clone())
        return {"u": u, "r": r, "rc": rc, "v": v,
                "u32": B.lasto_op_smooth(*s.ax, s.u32.clone(), s.b32, sweeps=s.case["sweeps"])}
    return {"v_lm": B.lasto_op_project(s.ax, s.ax, s.ax, s.u, s.pos, s.R)[0]}


def _run_layer(s):
    """Forward pass (weights packed after the last update); from the activation that the step's
    forward pass saved: ReLU gradient, data and weight gradients."""
    L, c = B.load(), s.case
    n, nb, cin, cout = c["n"], c["nb"], c["cin"], c["cout"]
    dims = (ctypes.c_int * 3)(n, n, n)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    y = torch.empty(nb * n ** 3, cout, device="cuda")
    dpre, dpre16 = torch.empty_like(y), torch.empty(y.shape, dtype=torch.bfloat16, device="cuda")
    dx = torch.empty(nb * n ** 3, cin, device="cuda")
    dw, db = torch.zeros(27, cin, cout, device="cuda"), torch.zeros(cout, device="cuda")
    rc = L.lasto_nn_pack_weights(cin, cout, p(s.w), p(s.wpk), st)
    rc |= L.lasto_nn_conv3d_fwd_tc(nb, dims, cin, cout, p(s.x), p(s.wpk), p(s.bias), 1, p(y), cout, 0, None, 0, 0,
                                   p(s.err), st)
    rc |= L.lasto_nn_relu_grad(y.numel(), p(s.saved), p(s.dy), p(dpre), p(dpre16), st)
    rc |= L.lasto_nn_conv3d_dgrad_tc(nb, dims, cin, cout, p(dpre16), p(s.w), p(s.wflip), p(s.wpk_flip), p(dx), p(s.err), st)
    rc |= L.lasto_nn_conv3d_wgrad_tc(nb, dims, cin, cout, p(s.x), p(dpre16), p(dpre), p(dw), p(db), p(s.err), st)
    if rc:
        raise RuntimeError("a layer call failed")
    return {"y": y, "dx": dx, "dw": dw, "db": db}


# ------------------------------------------------------------------ work
def work(case):
    kind = case["kind"]
    if kind in ("solve", "batch", "raw"):
        sizes = ([tuple(int(v) for v in m.split("@")) for m in case["members"].split()] if kind == "batch"
                 else [(case["shells"], case["n"])])
        nodes = sum(n ** 3 for _, n in sizes)
        atoms = sum(SHELL_ATOMS[k] for k, _ in sizes)
        reads = (8 if kind == "raw" or case.get("start") == "warm" else 0) * nodes + 300 * atoms
        # the potential is written; the density needs its nearest atoms' three terms (a distance
        # and an exponential each, about 30 operations) and the iteration at least one application
        # of the 7-point operator
        return {"bytes": reads + 8 * nodes + 200 * atoms, "flops": (14 + (0 if kind == "raw" else 90 * 13)) * nodes}
    if kind == "deposit":
        nodes = case["n"] ** 3
        return {"bytes": 12 * nodes, "flops": 90 * 13 * nodes}
    if kind == "spheres":
        na = SHELL_ATOMS[case["shells"]]
        pts = na * case["n_rad"] * 512
        return {"bytes": 2 * 8 * na * 25 * case["n_rad"], "flops": pts * (90 * 13 + 2 * 25)}
    if kind == "hs":
        m = 25 * SHELL_ATOMS[case["shells"]]
        return {"bytes": 8 * case["n"] ** 3 + 16 * m * m, "flops": 2 * case["n"] ** 3 * m * m}   # S and H, half of each
    if kind == "layer":
        nodes = case["nb"] * case["n"] ** 3
        w = 27 * case["cin"] * case["cout"]
        return {"bytes": nodes * (6 * case["cin"] + 8 * case["cout"]) + 8 * w, "flops": 3 * 2 * nodes * w}
    if kind == "twogrid":
        nodes = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": nodes * (16 + 16 + 12 + 2), "flops": nodes * (28 * case["sweeps"] + 14 + 8 + 8)}
    na = SHELL_ATOMS[case["shells"]]
    return {"bytes": na * 512 * 64 + 200 * na, "flops": na * 512 * (14 + 50)}


# ------------------------------------------------------------------ the same in 64 bits, plain torch
def _distance(p, x, y, z):
    return torch.sqrt((x - p[0])[None, None, :] ** 2 + (y - p[1])[None, :, None] ** 2 + (z - p[2])[:, None, None] ** 2)


def _weights(c):
    z = _cuda(np.array(ZETA))
    return _cuda(c.slater_w) * z ** 3 / (8 * PI), z


def _slater_sum(c, x, y, z):
    W, zt = _weights(c)
    W = W.cpu().numpy()
    out = torch.zeros((len(z), len(y), len(x)), dtype=torch.float64, device="cuda")
    for a in range(c.na):
        r = _distance(c.pos[a], x, y, z)
        for k in range(3):
            out += W[a, k] * torch.exp(-ZETA[k] * r)
    return out


def _owner(c, x, y, z):
    """The sphere that holds each node (or -1) and the nodes' distance from its centre."""
    own = torch.full((len(z), len(y), len(x)), -1, dtype=torch.int32, device="cuda")
    d = torch.zeros(own.shape, dtype=torch.float64, device="cuda")
    for a in range(c.na):
        r = _distance(c.pos[a], x, y, z)
        m = r < c.R[a]
        own[m] = a
        d = torch.where(m, r, d)
    return own, d


def _harmonics(u, lmax=4):
    """Real orthonormal y_lm of unit vectors u [..., 3], lm = l*l + l + m, no Condon-Shortley phase."""
    ux, uy, uz = u[..., 0], u[..., 1], u[..., 2]
    cs, sn = [torch.ones_like(ux)], [torch.zeros_like(ux)]
    for m in range(lmax):
        cs, sn = cs + [cs[m] * ux - sn[m] * uy], sn + [cs[m] * uy + sn[m] * ux]
    out = [None] * (lmax + 1) ** 2
    for l in range(lmax + 1):
        for m in range(l + 1):
            poly = np.polynomial.legendre.Legendre.basis(l).convert(kind=np.polynomial.Polynomial)
            coef = (poly.deriv(m) if m else poly).coef
            f = torch.zeros_like(uz)
            for q in coef[::-1]:
                f = f * uz + float(q)
            norm = math.sqrt((2 * l + 1) / (4 * PI) * math.factorial(l - m) / math.factorial(l + m) * (2 if m else 1))
            out[l * l + l + m] = norm * f * cs[m]
            if m:
                out[l * l + l - m] = norm * f * sn[m]
    return torch.stack(out, -1)


def _points(ax, flat):
    """Coordinates [., 3] of nodes given by flat index (three equal axes)."""
    n = len(ax)
    return torch.stack([ax[flat % n], ax[(flat // n) % n], ax[flat // (n * n)]], -1)


def _own_nonspherical(c, a, vec):
    """zeta^3/(8 pi) e^{-zeta r} (1 - r^2/R^2)^2 sum c_lm (r/R)^l y_lm of atoms a at offsets vec."""
    r = torch.sqrt((vec ** 2).sum(-1))
    unit = torch.where(r[..., None] > 0, vec / r.clamp_min(1e-300)[..., None], torch.zeros_like(vec))
    s = r / RADIUS
    l = torch.tensor([int(math.isqrt(lm)) for lm in range(1, 25)], device="cuda")
    ang = (_cuda(c.c_lm)[a] * _harmonics(unit)[..., 1:] * s[..., None] ** l).sum(-1)
    return ZETA[0] ** 3 / (8 * PI) * torch.exp(-ZETA[0] * r) * (1 - s * s) ** 2 * ang


def _add_nonspherical(c, out, inside, own, d):
    ax = _cuda(c.axis)
    for q in range(0, len(inside), 1 << 18):
        f, a = inside[q:q + (1 << 18)], own[q:q + (1 << 18)].long()
        out[f] += _own_nonspherical(c, a, _points(ax, f) - _cuda(c.pos)[a])


def _neighbour_sums(c):
    """A, B of N_i(r) = sum_k 2 A sinh(zeta r)/r - 2 B cosh(zeta r), the neighbours' spherical average."""
    W, z = _weights(c)
    p = _cuda(c.pos)
    D = torch.sqrt(((p[:, None] - p[None]) ** 2).sum(-1))
    off = ~torch.eye(c.na, dtype=torch.bool, device="cuda")
    D = torch.where(off, D, torch.ones_like(D))[:, :, None]
    e = torch.where(off[:, :, None], W[None] * torch.exp(-z * D), torch.zeros_like(D))
    return (e * (1 + z * D) / (2 * D * z * z)).sum(1), (e / (2 * D * z)).sum(1), W, z


def _neighbour_average(A, Bc, z, r):
    """N_i(r) for A, B [., 3] and radii r [.] or per row."""
    zr = z[:, None] * r if r.dim() == 1 and A.dim() == 2 and A.shape[0] != r.shape[0] else None
    if zr is not None:
        return (2 * A[:, :, None] * torch.sinh(zr) / r - 2 * Bc[:, :, None] * torch.cosh(zr)).sum(1)
    zr = r[:, None] * z
    shr = torch.where(zr > 1e-6, torch.sinh(zr) / r.clamp_min(1e-300)[:, None], z * (1 + zr * zr / 6))
    return (2 * A * shr - 2 * Bc * torch.cosh(zr)).sum(-1)


def _quartic(q, rho, drho):
    """a + b r^2 + c r^4 with charge q inside the sphere, value rho and slope drho at its radius."""
    R = RADIUS
    c = (q / (4 * PI) - rho * R ** 3 / 3 + drho * R ** 4 / 15) * 105 / (8 * R ** 7)
    b = drho / (2 * R) - 2 * c * R * R
    return rho - drho * R / 2 + c * R ** 4, b, c


def _pseudo(c):
    A, Bc, W, z = _neighbour_sums(c)
    R = RADIUS
    t, wt = np.polynomial.legendre.leggauss(64)
    r, wr = _cuda(0.5 * R * (t + 1)), _cuda(0.5 * R * wt)
    own = (_cuda(c.slater_w) * (1 - torch.exp(-z * R) * (1 + z * R + 0.5 * (z * R) ** 2))).sum(1)
    zr = z[:, None] * r
    N = (2 * A[:, :, None] * torch.sinh(zr) / r - 2 * Bc[:, :, None] * torch.cosh(zr)).sum(1)
    q = own + 4 * PI * (N * r * r * wr).sum(1) - _cuda(c.Z)
    sh, ch, e = torch.sinh(z * R), torch.cosh(z * R), torch.exp(-z * R)
    rho = (W * e + 2 * A * sh / R - 2 * Bc * ch).sum(1)
    drho = (-z * W * e + 2 * A * (z * ch / R - sh / R ** 2) - 2 * Bc * z * sh).sum(1)
    return _quartic(q, rho, drho), A, Bc, z


def _rhs(c):
    """b = 4 pi rho~ on the nodes and the owners."""
    ax = _cuda(c.axis)
    own, d = _owner(c, ax, ax, ax)
    out = _slater_sum(c, ax, ax, ax)
    flat = own.reshape(-1)
    inside = torch.nonzero(flat >= 0).reshape(-1)
    a = flat[inside].long()
    r = d.reshape(-1)[inside]
    (qa, qb, qc), A, Bc, z = _pseudo(c)
    W = _weights(c)[0]
    rho0 = (W[a] * torch.exp(-r[:, None] * z)).sum(-1) + _neighbour_average(A[a], Bc[a], z, r)
    v = out.view(-1)
    v[inside] += qa[a] + qb[a] * r ** 2 + qc[a] * r ** 4 - rho0
    _add_nonspherical(c, v, inside, flat[inside], d)
    return 4 * PI * out, own


def _raw_rhs(c):
    """The same from the density on the nodes and the tables inside the spheres."""
    ne, rho00 = _raw_density(c)
    n, R = N_RAD, RADIUS
    h = math.log(R / R_MIN) / (n - 1)
    r = R * torch.exp((torch.arange(n, dtype=torch.float64, device="cuda") - (n - 1)) * h)
    s4 = math.sqrt(4 * PI)
    q = s4 * (rho00[:, 0] * R_MIN ** 3 / 3 + _segments(rho00 * r ** 3, h).sum(-1)) - Z_PD
    f = rho00
    drho = (25 * f[:, -1] - 48 * f[:, -2] + 36 * f[:, -3] - 16 * f[:, -4] + 3 * f[:, -5]) / (12 * h) / (R * s4)
    qa, qb, qc = _quartic(q, f[:, -1] / s4, drho)
    ax = _cuda(c.axis)
    own, d = _owner(c, ax, ax, ax)
    flat = own.reshape(-1)
    inside = torch.nonzero(flat >= 0).reshape(-1)
    a, rr = flat[inside].long(), d.reshape(-1)[inside]
    t = torch.log(rr.clamp_min(R_MIN) / R_MIN) / h
    j = t.floor().long().clamp(1, n - 3)
    s = t - j
    l = (-s * (s - 1) * (s - 2) / 6, (s + 1) * (s - 1) * (s - 2) / 2, -(s + 1) * s * (s - 2) / 2, (s + 1) * s * (s - 1) / 6)
    rho = sum(l[m] * f[a, j - 1 + m] for m in range(4))
    line = f[a, 0] + (f[a, 1] - f[a, 0]) * (rr - R_MIN) / (r[1] - r[0])
    rho = torch.where(rr <= R_MIN, line, rho)
    ne.view(-1)[inside] += qa[a] + qb[a] * rr ** 2 + qc[a] * rr ** 4 - rho / s4
    return 4 * PI * ne


def _segments(g, h):
    """Integral over each interval of the cubic through its four nearest samples (last axis)."""
    mid = h / 24 * (-g[..., :-3] + 13 * g[..., 1:-2] + 13 * g[..., 2:-1] - g[..., 3:])
    first = h / 24 * (9 * g[..., :1] + 19 * g[..., 1:2] - 5 * g[..., 2:3] + g[..., 3:4])
    last = h / 24 * (g[..., -4:-3] - 5 * g[..., -3:-2] + 19 * g[..., -2:-1] + 9 * g[..., -1:])
    return torch.cat([first, mid, last], -1)


def _dual(x):
    d = torch.zeros_like(x)
    d[1:-1] = 0.5 * (x[2:] - x[:-2])
    d[0], d[-1] = 0.5 * (x[1] - x[0]), 0.5 * (x[-1] - x[-2])
    return d


def _stencil(x):
    hm, hp = x[1:-1] - x[:-2], x[2:] - x[1:-1]
    return 2 / ((hm + hp) * hm), 2 / ((hm + hp) * hp)


def _poisson(ax, b):
    """The 7-point equation with the l <= 4 multipole faces, solved directly in the 1-D operators'
    eigenvectors (three equal axes)."""
    n = len(ax)
    vol = _dual(ax)
    l = torch.tensor([int(math.isqrt(lm)) for lm in range(25)], device="cuda", dtype=torch.float64)
    Q = torch.zeros(25, dtype=torch.float64, device="cuda")
    u = torch.zeros_like(b)
    for k in range(n):
        p = torch.stack([ax[None, :].expand(n, n), ax[:, None].expand(n, n), ax[k].expand(n, n)], -1)
        r = torch.sqrt((p ** 2).sum(-1))
        y = _harmonics(torch.where(r[..., None] > 0, p / r.clamp_min(1e-300)[..., None], torch.zeros_like(p)))
        wgt = b[k] / (4 * PI) * vol[k] * vol[:, None] * vol[None, :]
        rl = torch.where(l > 0, r[..., None] ** l, torch.ones_like(y))
        Q += (wgt[..., None] * rl * y).sum((0, 1))
    coef = -4 * PI / (2 * l + 1) * Q
    for k in range(n):
        p = torch.stack([ax[None, :].expand(n, n), ax[:, None].expand(n, n), ax[k].expand(n, n)], -1)
        face = torch.ones(n, n, dtype=torch.bool, device="cuda")
        if 0 < k < n - 1:
            face[1:-1, 1:-1] = False
        pf = p[face]
        r = torch.sqrt((pf ** 2).sum(-1))
        u[k][face] = (coef * _harmonics(pf / r[:, None]) / r[:, None] ** (l + 1)).sum(-1)
    cm, cp = _stencil(ax)
    f = b[1:-1, 1:-1, 1:-1].clone()
    f[:, :, 0] -= cm[0] * u[1:-1, 1:-1, 0]
    f[:, :, -1] -= cp[-1] * u[1:-1, 1:-1, -1]
    f[:, 0, :] -= cm[0] * u[1:-1, 0, 1:-1]
    f[:, -1, :] -= cp[-1] * u[1:-1, -1, 1:-1]
    f[0] -= cm[0] * u[0, 1:-1, 1:-1]
    f[-1] -= cp[-1] * u[-1, 1:-1, 1:-1]
    s = torch.sqrt(vol[1:-1])
    T = torch.diag(-(cm + cp)) + torch.diag(cp[:-1], 1) + torch.diag(cm[1:], -1)
    T = s[:, None] * T / s[None, :]
    lam, V = torch.linalg.eigh(0.5 * (T + T.T))
    to = (V * s[:, None]).T.contiguous()          # eigenvector components of f sqrt(vol)
    back = V / s[:, None]
    g = torch.einsum("ai,kji->kja", to, f)
    g = torch.einsum("bj,kja->kba", to, g)
    g = torch.einsum("ck,kba->cba", to, g)
    g = g / (lam[:, None, None] + lam[None, :, None] + lam[None, None, :])
    g = torch.einsum("kc,cba->kba", back, g)
    g = torch.einsum("jb,kba->kja", back, g)
    u[1:-1, 1:-1, 1:-1] = torch.einsum("ia,kja->kji", back, g)
    return u


def _quadrature(n_theta=16, n_phi=32):
    t, w = np.polynomial.legendre.leggauss(n_theta)
    ph = 2 * PI * np.arange(n_phi) / n_phi
    st = np.sqrt(1 - t * t)
    u = np.stack([st[:, None] * np.cos(ph), st[:, None] * np.sin(ph), np.broadcast_to(t[:, None], (n_theta, n_phi))], -1)
    return _cuda(u.reshape(-1, 3)), _cuda(np.repeat(w * 2 * PI / n_phi, n_phi))


def _project(ax, u, pos):
    pts, w = _quadrature()
    P = _cuda(pos)[:, None, :] + RADIUS * pts[None]
    n = len(ax)
    cell, t = [], []
    for d in range(3):
        c = (torch.searchsorted(ax, P[..., d].contiguous(), right=True) - 1).clamp(0, n - 2)
        cell.append(c)
        t.append((P[..., d] - ax[c]) / (ax[c + 1] - ax[c]))
    V = 0.0
    for k in range(2):
        for j in range(2):
            for i in range(2):
                wt = (t[0] if i else 1 - t[0]) * (t[1] if j else 1 - t[1]) * (t[2] if k else 1 - t[2])
                V = V + wt * u[cell[2] + k, cell[1] + j, cell[0] + i]
    return torch.einsum("aq,q,ql->al", V, w, _harmonics(pts))


def _exact_solve(c, raw=False):
    ax = _cuda(c.axis)
    u = _poisson(ax, _raw_rhs(c) if raw else _rhs(c)[0])
    return _project(ax, u, c.pos), u.reshape(-1)


def _exact_spheres(case, seed):
    c = _cluster(case["shells"], case["n"], True, seed)
    n, R = case["n_rad"], RADIUS
    h = math.log(R / R_MIN) / (n - 1)
    r = R * torch.exp((torch.arange(n, dtype=torch.float64, device="cuda") - (n - 1)) * h)
    pts, w = _quadrature()
    yw = _harmonics(pts) * w[:, None]
    W = _weights(c)[0].cpu().numpy()
    pos = _cuda(c.pos)
    rho = torch.empty(c.na, 25, n, dtype=torch.float64, device="cuda")
    off = r[:, None, None] * pts[None]
    for a in range(c.na):
        f = torch.zeros(n, len(pts), dtype=torch.float64, device="cuda")
        for t in range(c.na):
            d = torch.sqrt(((off + (pos[a] - pos[t])) ** 2).sum(-1))
            for k in range(3):
                f += W[t, k] * torch.exp(-ZETA[k] * d)
        f[:-1] += _own_nonspherical(c, torch.full((n - 1, len(pts)), a, device="cuda"), off[:-1])
        rho[a] = torch.einsum("jq,ql->lj", f, yw)
    vR = _cuda(np.random.default_rng([seed, 3]).normal(size=(c.na, 25)))
    v = torch.empty_like(rho)
    for lm in range(25):
        L = math.isqrt(lm)
        g1, g2 = rho[:, lm] * r ** (L + 3), rho[:, lm] * r ** (2 - L)
        zero = torch.zeros(c.na, 1, dtype=torch.float64, device="cuda")
        I1 = g1[:, :1] / (L + 3) + torch.cat([zero, _segments(g1, h).cumsum(-1)], -1)
        s2 = _segments(g2, h)
        I2 = torch.cat([s2.flip(-1).cumsum(-1).flip(-1), zero], -1)
        v[:, lm] = vR[:, lm:lm + 1] * (r / R) ** L - 4 * PI / (2 * L + 1) * (
            I1 / r ** (L + 1) + r ** L * I2 - r ** L * I1[:, -1:] / R ** (2 * L + 1))
        if L == 0:
            v[:, lm] += math.sqrt(4 * PI) * Z_PD * (1 / r - 1 / R)
    return {"rho": rho, "v": v}


def _exact_hs(case, seed):
    c, ax, V = _hs_inputs(case, seed)
    own, _ = _owner(c, ax, ax, ax)
    nodes = torch.nonzero(own.reshape(-1) < 0).reshape(-1)
    n, M = len(ax), 25 * c.na
    dual = _dual(ax)
    S, H = (torch.zeros(M, M, dtype=torch.float64, device="cuda") for _ in range(2))
    pos = _cuda(c.pos)
    for q in range(0, len(nodes), 1 << 16):
        f = nodes[q:q + (1 << 16)]
        sv = torch.sqrt(dual[f % n] * dual[(f // n) % n] * dual[f // (n * n)])
        d = _points(ax, f)[:, None, :] - pos[None]
        r = torch.sqrt((d ** 2).sum(-1))
        Y = _harmonics(d / r[..., None], 3)
        phi, til = [], []
        for bn, bl, bz in B.PD_BASIS:
            e = torch.exp(-bz * r)
            rad = r ** (bn - 1) * e
            kin = 0.5 * ((bl * (bl + 1) - bn * (bn - 1)) * r ** (bn - 3) + 2 * bz * bn * r ** (bn - 2)
                         - bz * bz * r ** (bn - 1)) * e
            y = Y[..., bl * bl:(bl + 1) ** 2]
            phi.append(rad[..., None] * y)
            til.append((kin + V.reshape(-1)[f][:, None] * rad)[..., None] * y)
        phi = (torch.cat(phi, -1) * sv[:, None, None]).reshape(len(f), M)
        til = (torch.cat(til, -1) * sv[:, None, None]).reshape(len(f), M)
        S += phi.T @ phi
        H += phi.T @ til
    return {"S": S, "H": 0.5 * (H + H.T)}


def _exact_layer(case, seed):
    x, w, bias, dy, saved = _layer_inputs(case, seed)
    n, nb, cin, cout = case["n"], case["nb"], case["cin"], case["cout"]
    xg = torch.zeros(nb, n + 2, n + 2, n + 2, cin, dtype=torch.float64, device="cuda")
    xg[:, 1:-1, 1:-1, 1:-1] = x.double().view(nb, n, n, n, cin)
    taps = [(a, b, d) for a in range(3) for b in range(3) for d in range(3)]
    cut = lambda g, t: g[:, t[0]:t[0] + n, t[1]:t[1] + n, t[2]:t[2] + n].reshape(nb * n ** 3, -1)
    w64 = w.double()
    y = sum(cut(xg, t) @ w64[q] for q, t in enumerate(taps)) + bias.double()
    g = torch.where(saved > 0, dy.double(), torch.zeros_like(y))
    gg = torch.zeros(nb, n + 2, n + 2, n + 2, cout, dtype=torch.float64, device="cuda")
    gg[:, 1:-1, 1:-1, 1:-1] = g.view(nb, n, n, n, cout)
    dx = sum(cut(gg, (2 - t[0], 2 - t[1], 2 - t[2])) @ w64[q].T for q, t in enumerate(taps))
    dw = torch.stack([cut(xg, t).T @ g for t in taps])
    return {"y": torch.relu(y), "dx": dx, "dw": dw, "db": g.sum(0)}


def _operator(ax, u):
    (xm, xp), (ym, yp), (zm, zp) = (_stencil(a) for a in ax)
    c = u[1:-1, 1:-1, 1:-1]
    off = (xm * u[1:-1, 1:-1, :-2] + xp * u[1:-1, 1:-1, 2:] + ym[:, None] * u[1:-1, :-2, 1:-1] + yp[:, None] * u[1:-1, 2:, 1:-1]
           + zm[:, None, None] * u[:-2, 1:-1, 1:-1] + zp[:, None, None] * u[2:, 1:-1, 1:-1])
    diag = (xm + xp) + (ym + yp)[:, None] + (zm + zp)[:, None, None]
    return off, diag, c


def _sweeps(ax, u, b, count):
    n = u.shape
    idx = sum(torch.meshgrid(*[torch.arange(1, m - 1, device="cuda") for m in n], indexing="ij"))
    for _ in range(count):
        for colour in (1, 0):     # interior (1, 1, 1) has odd index sum; even sums are red, first
            off, diag, c = _operator(ax, u)
            new = (off - b[1:-1, 1:-1, 1:-1]) / diag
            u[1:-1, 1:-1, 1:-1] = torch.where(idx % 2 == (1 - colour), new, c)
    return u


def _exact_twogrid(case, seed):
    ax, u0, b, ec = _grid_inputs(case, seed)
    u = _sweeps(ax, u0.clone(), b, case["sweeps"])
    r = torch.zeros_like(u)
    off, diag, c = _operator(ax, u)
    r[1:-1, 1:-1, 1:-1] = b[1:-1, 1:-1, 1:-1] - (off - diag * c)
    P = []
    for x in ax:                       # linear interpolation from every other node
        n = len(x)
        p = torch.zeros(n, (n + 1) // 2, dtype=torch.float64, device="cuda")
        p[torch.arange(0, n, 2), torch.arange((n + 1) // 2)] = 1.0
        i = torch.arange(1, n, 2, device="cuda")
        p[i, (i - 1) // 2] = (x[i + 1] - x[i]) / (x[i + 1] - x[i - 1])
        p[i, (i + 1) // 2] = (x[i] - x[i - 1]) / (x[i + 1] - x[i - 1])
        P.append(p)
    rc = r * _dual(ax[0]) * _dual(ax[1])[:, None] * _dual(ax[2])[:, None, None]
    rc = torch.einsum("kc,jb,ia,kji->cba", P[2], P[1], P[0], rc)
    rc = rc / (_dual(ax[0][::2]) * _dual(ax[1][::2])[:, None] * _dual(ax[2][::2])[:, None, None])
    inner = torch.zeros_like(rc)
    inner[1:-1, 1:-1, 1:-1] = rc[1:-1, 1:-1, 1:-1]
    v = u.clone()
    v[1:-1, 1:-1, 1:-1] += torch.einsum("kc,jb,ia,cba->kji", P[2], P[1], P[0], ec)[1:-1, 1:-1, 1:-1]
    u32 = _sweeps(ax, u0.float().double(), b.float().double(), case["sweeps"])
    return {"u": u, "r": r, "rc": inner, "v": v, "u32": u32}


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        if SHELL_ATOMS[case["shells"]] * case["n"] ** 3 > 3e9:
            return None
        v, u = _exact_solve(_cluster(case["shells"], case["n"], case["graded"], seed))
        return {"v_lm": v, "potential": u}
    if kind == "batch":
        got = [_exact_solve(c) for c in _members(case, seed)]
        return {"v_lm": torch.cat([g[0] for g in got]), "potential": torch.cat([g[1] for g in got])}
    if kind == "raw":
        v, u = _exact_solve(_cluster(case["shells"], case["n"], True, seed), raw=True)
        return {"v_lm": v, "potential": u}
    if kind == "deposit":
        if SHELL_ATOMS[case["shells"]] * case["n"] ** 3 > 3e9:
            return None
        b, own = _rhs(_cluster(case["shells"], case["n"], True, seed))
        return {"b": b, "owner": own}
    if kind == "spheres":
        return _exact_spheres(case, seed)
    if kind == "hs":
        return _exact_hs(case, seed)
    if kind == "layer":
        return _exact_layer(case, seed)
    if kind == "twogrid":
        return _exact_twogrid(case, seed)
    c = _cluster(case["shells"], case["n"], True, seed)
    ax, u = _potential_field(c, seed)
    return {"v_lm": _project(ax, u, c.pos)}
