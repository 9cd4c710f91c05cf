"""What a user of this framework has it do, as measurable cases.

Every case is one pass through the public Python entry points of `paper_2309_06225_gb300` on data
that the path meets in earnest: puncture metrics with a scalar field, the couplings, boundaries and
schemes of the evolution, its diagnostics and its differentiation. `listed()` gives the cases,
`draw` more of the same ranges, `prepare` the inputs and buffers a program holds before the call,
`run` one pass, `work` the bytes and operations a pass cannot do without, and `exact` the outputs
from a plain torch evaluation of the same equations in 64 bits.

A pass that advances a state starts from the given initial data each time (a copy of the initial
state into the working buffer, as a program does that starts another run).
"""
import math

import numpy as np
import torch

import paper_2309_06225_gb300 as grf
from paper_2309_06225_gb300.diff import sphere as _sphere

NF = 27
DEV = "cuda"
PERIODIC, FROZEN, SOMMERFELD = grf.GRF_BC_PERIODIC, grf.GRF_BC_FROZEN, grf.GRF_BC_SOMMERFELD

# Operations of one right-hand side with dissipation and stage update at one point (adds and products
# one each, a fused multiply-add two): the pointwise equations and the 4th-order stencils.
POINT_FLOPS = 6615
R3 = range(3)


# ------------------------------------------------------------------------------------ the cases
def listed():
    """The work by use: single steps and runs of one box from the smallest to the production size,
    the schemes and boundaries, box sets, host-resident states, diagnostics, and derivatives."""
    return [
        # A tiny box advanced alone: what a user's first experiments and unit checks do; latency.
        _case("step_16", "rk4", n=(16, 16, 16), dx=0.5, steps=1),
        # The single-puncture run of the README: 32^3 on [-4, 4]^3, ten steps in one call.
        _case("puncture_32", "rk4", n=(32, 32, 32), dx=0.25, steps=10, lam=0.01, g2=0.01),
        # One refinement box of an AMR hierarchy: uneven extents, ghosts given by the parent level.
        _case("refined_box", "rk4", n=(75, 50, 61), dx=0.125, steps=2, bc=FROZEN, beta=1),
        # The throughput workload: two punctures and scalar bumps in 256^3 points.
        _case("pair_256", "rk4", n=(256, 256, 256), dx=0.125, steps=1, data="pair", beta=1, lam=0.05, g2=0.01),
        # A production setup: 6th-order stencils, lopsided advection, radiative outer boundary.
        _case("order6_outer", "rk4", n=(96, 96, 96), dx=0.25, steps=1, bc=SOMMERFELD, ng=4, adv=1, data="pair",
              beta=1, lam=0.05),
        # A set of uneven AMR-like boxes with their own couplings, advanced by one batched call.
        _case("box_set", "batch", n=(48, 64, 24), dx=0.25, steps=1, boxes=16, bc=FROZEN),
        # One box held as 2 x 2 x 2 patches with a halo exchange after every stage.
        _case("patches_8", "patches", n=(96, 80, 96), dx=0.25, steps=1, data="pair", beta=1, lam=0.05),
        # A state that lives in page-locked host memory, stepped from host to host.
        _case("host_step", "host", n=(96, 96, 96), dx=0.25, steps=1, data="pair", beta=1, lam=0.05),
        # One right-hand side for a user's own integrator, then dissipation of its strength on top.
        _case("rhs_call", "rhs", n=(80, 64, 72), dx=0.25, data="pair", beta=1, lam=0.05),
        # Monitoring of an output step: constraints with norms, Psi_4, and its modes on a sphere.
        _case("diagnostics", "diag", n=(72, 72, 60), dx=0.25, data="pair", beta=1, lam=0.05),
        # Gradient of the sphere signal: checkpointed evolution, then the reverse sweep.
        _case("adjoint", "adjoint", n=(36, 32, 30), dx=0.5, steps=2, lam=0.2, g2=0.1),
        # Forward-mode derivatives of the same signal, three directions at once.
        _case("tangents", "tangent", n=(40, 32, 36), dx=0.5, steps=1, lam=0.2, g2=0.1),
    ]


def _case(name, kind, n, dx, steps=1, bc=PERIODIC, ng=3, adv=0, beta=0, lam=0.01, g2=0.01, g3=0.0, dec=0,
          data="single", boxes=1):
    return {"name": name, "kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "dx": dx, "steps": steps, "bc": bc,
            "ng": ng, "adv": adv, "beta": beta, "lam": lam, "g2": g2, "g3": g3, "dec": dec, "data": data,
            "boxes": boxes}


def draw(rng):
    """One more case of the ranges above: kinds by how often they are used, sizes over the logarithm
    of the range with odd ones among them, any coupling, scheme and boundary a kind accepts."""
    kind = rng.choice(["rk4"] * 5 + ["batch", "batch", "patches", "host", "rhs", "diag", "adjoint", "tangent"])
    hi = {"rk4": 160, "batch": 64, "patches": 112, "host": 112, "rhs": 112, "diag": 96, "adjoint": 40,
          "tangent": 48}[kind]
    lo = {"rk4": 12, "batch": 16, "patches": 24, "host": 16, "rhs": 12, "diag": 32, "adjoint": 24, "tangent": 24}[kind]
    edge = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    n = tuple(max(lo, min(hi, int(round(edge * rng.uniform(0.75, 1.25))))) for _ in range(3))
    if rng.random() < 0.4:  # a round size: a multiple of 8
        n = tuple(max(16, 8 * (m // 8)) for m in n)
    c = _case("", kind, n, dx=rng.choice([0.125, 0.2, 0.25, 0.5]))
    c["beta"] = rng.choice([0, 1, 1, 2])
    c["lam"] = round(rng.uniform(0.0, 0.1), 4)
    c["g2"] = round(rng.uniform(0.0, 0.05), 4)
    c["data"] = rng.choice(["single", "pair"])
    if kind in ("adjoint", "tangent", "diag"):
        c["dx"] = 0.5 if kind != "diag" else 0.25
    if kind in ("rk4", "patches", "host", "batch", "rhs"):
        c["adv"] = rng.choice([0, 0, 1])
        c["dec"] = rng.choice([0, 0, 0, 1])
        c["g3"] = rng.choice([0.0, 0.0, 0.02])
    if kind in ("rk4", "rhs"):
        c["bc"] = rng.choice([PERIODIC, PERIODIC, FROZEN, SOMMERFELD])
        c["ng"] = rng.choice([3, 3, 4])
    elif kind in ("patches", "host"):
        c["bc"] = rng.choice([PERIODIC, FROZEN])
    elif kind == "batch":
        c["bc"] = rng.choice([PERIODIC, FROZEN])
        c["boxes"] = rng.randint(4, 16)
    if kind == "rk4":
        c["steps"] = 10 if max(n) <= 40 else rng.choice([1, 2])
    elif kind == "adjoint":
        c["steps"] = 2
    del c["name"]
    return c


# ------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _boxes(case):
    """The case's boxes: one, or a set of extents and spacings around the case's own."""
    n = (case["nx"], case["ny"], case["nz"])
    out = []
    for b in range(case["boxes"]):
        m, dx = n, case["dx"]
        if case["boxes"] > 1:
            scale = (1.0, 0.75, 0.5, 1.25)[b % 4]
            m = tuple(max(16, min(64, int(round(n[(b + d) % 3] * scale)) + (b % 2) * d)) for d in R3)
            dx = dx * (1.0, 0.5, 0.25)[b % 3]
        out.append(grf.make_box(*m, dx, *(-0.5 * (x - 1) * dx for x in m), bc=case["bc"], ng=case["ng"]))
    return out


def _params(case, b=0):
    lam, g2 = case["lam"], case["g2"]
    if case["boxes"] > 1:  # a coupling sweep over the set
        lam, g2 = 0.1 * (b + 1) / case["boxes"], 0.05 * (case["boxes"] - b) / case["boxes"]
    return grf.grf_params(0.1, 0.0, 1.0, 0.75, 1.0, 0.2, 0.4, lam, g2, 0.3, 1e-4, 1e-4, case["beta"], 1, case["dec"],
                          case["adv"], 1.0, case["g3"])


def _initial(case, box, seed, b=0):
    """Puncture data in the ghosted layout: a conformally flat metric with one or two punctures, a
    scalar field, and small smooth perturbations of every field (an evolved state has no exact
    zeros), all from the seed."""
    g = _gen(1000003 * seed + 7919 * b + 17)
    ng = box.ng
    ax = [torch.arange(m + 2 * ng, dtype=torch.float64, device=DEV) - ng for m in (box.nx, box.ny, box.nz)]
    X = (box.x0 + ax[0] * box.dx)[None, None, :]
    Y = (box.y0 + ax[1] * box.dx)[None, :, None]
    Z = (box.z0 + ax[2] * box.dx)[:, None, None]

    def u(a, c, *shape):
        return a + (c - a) * torch.rand(shape, generator=g, dtype=torch.float64, device=DEV)

    s = _fields(box)
    v = s[..., :box.nx + 2 * ng]
    half = 0.5 * box.dx * min(box.nx, box.ny, box.nz)
    if case["data"] == "pair":
        sep = min(3.0, 0.4 * half)
        m = u(0.4, 0.6, 2).tolist()
        cz = [sep + 0.31 * box.dx, -sep + 0.31 * box.dx]
    else:
        m, cz = u(0.9, 1.1, 1).tolist(), [0.31 * box.dx]
    o = 0.27 * box.dx
    psi = 1.0
    for mm, c in zip(m, cz):
        psi = psi + mm / (2.0 * torch.sqrt((X - o) ** 2 + (Y + o) ** 2 + (Z - c) ** 2))
    v[0] = psi ** -4
    v[18] = psi ** -2
    for f in (1, 4, 6):
        v[f] = 1.0
    nb = 4
    cen = u(-half, half, nb, 3).tolist()
    wid = u(1.0, 3.0, nb).tolist()
    amp = u(-1e-2, 1e-2, nb).tolist()
    for c, w, a in zip(cen, wid, amp):
        v[25] += a * torch.exp(-((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2) / w ** 2)
    # perturbations that decay from the centre and repeat with the box's period
    ph = u(0.0, 2 * math.pi, NF, 3).tolist()
    am = u(-1.0, 1.0, NF).tolist()
    k = [2 * math.pi / (q * box.dx) for q in (box.nx, box.ny, box.nz)]
    for f in range(NF):
        v[f] += (2e-3 if f not in (0, 18) else 1e-4) * am[f] * (
            torch.sin(k[0] * X + ph[f][0]) * torch.cos(k[1] * Y + ph[f][1]) * torch.sin(k[2] * Z + ph[f][2]))
    return s


def _signal_sphere(box):
    """A sphere well inside the box, about its centre."""
    r = 0.3 * box.dx * (min(box.nx, box.ny, box.nz) - 1)
    return _sphere(r, (0.02, -0.03, 0.01))


def _fields(box, n=NF):
    """Zeroed fields in the padded, ghosted layout."""
    return torch.zeros((n, box.nz + 2 * box.ng, box.ny + 2 * box.ng, box.pitch), dtype=torch.float64, device=DEV)


def _dt(box):
    return 0.25 * box.dx


def prepare(case, seed):
    boxes = _boxes(case)
    st = {"case": case, "boxes": boxes, "params": [_params(case, b) for b in range(len(boxes))],
          "u0": [_initial(case, bx, seed, b) for b, bx in enumerate(boxes)]}
    box, kind = boxes[0], case["kind"]
    if kind in ("rk4", "batch"):
        st["u"] = [torch.empty_like(x) for x in st["u0"]]
    if kind == "rk4":
        st["ws"] = grf.alloc_workspace(grf.grf_workspace_bytes(box, grf.GRF_OP_RK4))
    elif kind == "batch":
        st["cfg"] = grf.batch_config(grf.GRF_BATCH_GRAPH)
        st["items"] = grf.batch_items(boxes, st["u"], list(range(len(boxes))), [_dt(b) for b in boxes])
        st["parr"] = grf.params_array(st["params"])
        st["ws"] = grf.alloc_workspace(grf.grf_batched_workspace_bytes(st["items"], st["cfg"]))
    elif kind == "patches":
        st["level"] = grf.patch_level(box, 2, 2, 2)
        st["patches"] = grf.patch_states(st["level"])
        st["ws"] = grf.alloc_workspace(grf.grf_patches_workspace_bytes(st["level"]))
    elif kind == "host":
        st["hin"] = st["u0"][0].cpu().pin_memory()
        st["hout"] = torch.empty_like(st["hin"]).pin_memory()
        st["u"] = [torch.empty_like(st["u0"][0])]
        st["ws"] = grf.alloc_workspace(grf.grf_workspace_bytes(box, grf.GRF_OP_RK4))
    elif kind == "rhs":
        st["out"] = _fields(box)
    elif kind == "diag":
        st["out4"], st["psi"] = _fields(box, 4), _fields(box, 2)
        st["ws"] = grf.alloc_workspace(grf.grf_workspace_bytes(box, grf.GRF_OP_CONSTRAINTS))
        st["wse"] = grf.alloc_workspace(grf.grf_extract_workspace_bytes(24, 4))
    elif kind == "adjoint":
        st["u"] = [torch.empty_like(st["u0"][0])]
        n, every = case["steps"], 2
        st["ck"] = torch.zeros((grf.checkpoint_count(n, every),) + tuple(st["u0"][0].shape), dtype=torch.float64,
                               device=DEV)
        nb = grf.grf_adjoint_workspace_bytes(box, every)
        st["ws"] = grf.alloc_workspace(nb)
    elif kind == "tangent":
        st["u"] = [torch.empty_like(st["u0"][0])]
        # direction 2: the amplitude of the scalar (the state's own phi); 0, 1: lambda and g2
        st["t0"] = _fields(box, 3 * NF).view(3, NF, *st["u0"][0].shape[1:])
        st["t0"][2, 25].copy_(st["u0"][0][25])
        st["t"] = torch.empty_like(st["t0"])
        st["ws"] = grf.alloc_workspace(grf.grf_tlm_workspace_bytes(box))
    return st


# ------------------------------------------------------------------------------------ one pass
_DPARAMS = [1.0, 0.0, 0.0, 1.0, 0.0, 0.0]  # d(lambda, g2) along the three tangent directions


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    box, params, steps = st["boxes"][0], st["params"][0], case["steps"]
    if kind == "rk4":
        st["u"][0].copy_(st["u0"][0])
        grf.grf_rk4_step(box, params, st["u"][0], _dt(box), steps, ws=st["ws"])
        return st["u"][0]
    if kind == "batch":
        for a, b in zip(st["u"], st["u0"]):
            a.copy_(b)
        grf.grf_batched_rk4(st["items"], st["parr"], steps, st["cfg"], ws=st["ws"], sync_status=False)
        return st["u"]
    if kind == "patches":
        grf.grf_patch_copy(st["level"], st["u0"][0], st["patches"], 0)
        grf.grf_patches_rk4(st["level"], params, st["patches"], _dt(box), steps, ws=st["ws"], sync_status=False)
        return st["patches"]
    if kind == "host":
        grf.grf_rk4_step_host(box, params, st["hin"], st["hout"], st["u"][0], _dt(box), steps, ws=st["ws"])
        return st["hout"]
    if kind == "rhs":
        grf.grf_rhs(box, params, st["u0"][0], st["out"])
        grf.grf_ko_dissipation(box, 0.1, st["u0"][0], st["out"])
        return st["out"]
    if kind == "diag":
        norms = grf.grf_constraints(box, params, st["u0"][0], st["out4"], ws=st["ws"])
        grf.grf_weyl_psi4(box, params, st["u0"][0], st["psi"])
        sp = _signal_sphere(box)
        modes = grf.grf_extract_modes(box, st["psi"][0], st["psi"][1], -2, sp.radius, (sp.cx, sp.cy, sp.cz), 24, 48, 4,
                                      ws=st["wse"])
        return {"constraints": st["out4"], "norms": norms, "psi4": st["psi"], "modes": modes}
    if kind == "adjoint":
        st["u"][0].copy_(st["u0"][0])
        sp = _signal_sphere(box)
        loss = torch.zeros(1, dtype=torch.float64, device=DEV)
        grf.grf_signal_forward(box, params, st["u"][0], _dt(box), steps, sp, 2, st["ck"], loss, ws=st["ws"])
        sbar = torch.zeros_like(st["u"][0])
        pbar = torch.zeros(2, dtype=torch.float64, device=DEV)
        grf.grf_adjoint_rk4(box, params, st["ck"], _dt(box), steps, sp, 2, 1.0, sbar, pbar, ws=st["ws"])
        return {"state": st["u"][0], "signal": loss, "d_state": sbar, "d_couplings": pbar}
    if kind == "tangent":
        st["u"][0].copy_(st["u0"][0])
        st["t"].copy_(st["t0"])
        loss = torch.zeros(4, dtype=torch.float64, device=DEV)
        grf.grf_tlm_rk4(box, params, _DPARAMS, st["u"][0], st["t"], _dt(box), steps, _signal_sphere(box), loss,
                        ws=st["ws"])
        return {"state": st["u"][0], "tangents": st["t"], "signal": loss}
    raise ValueError(kind)


def work(case):
    """Bytes: the state read once and written once (the outputs, for calls that do not advance it).
    Operations: one pointwise right-hand side per point and stage; a reverse sweep needs about
    three, three tangents about four times a stage's, besides the evolution itself."""
    pts = sum(b.nx * b.ny * b.nz for b in _boxes(case))
    kind, steps = case["kind"], case["steps"]
    fields = {"rhs": 54, "diag": 27 + 6, "adjoint": 108, "tangent": 216}.get(kind, 54)
    evals = {"rhs": 1, "diag": 2, "adjoint": 4 * 5 * steps, "tangent": 16 * steps}.get(kind, 4 * steps)
    return {"bytes": 8 * fields * pts, "flops": POINT_FLOPS * evals * pts}


# ------------------------------------------------------------------------------------ plain 64-bit evaluation
# The equations with tensors of grid values as scalars: v[f], d1[f][k], d2[f][i][j] are 1D tensors over
# the points. Fields: 0 chi, 1-6 h, 7 K, 8-13 A, 14 Theta, 15-17 Gamma, 18 lapse, 19-21 shift, 22-24 B,
# 25 phi, 26 Pi.
SYM = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))
POS = [[0, 1, 2], [1, 3, 4], [2, 4, 5]]


def _sym(x):
    return [[x[POS[i][j]] for j in R3] for i in R3]


def _symf(f):
    x = [f(i, j) for i, j in SYM]
    return _sym(x)


def _mat(f):
    return [[f(i, j) for j in R3] for i in R3]


def _sum(it):
    it = iter(it)
    s = next(it)
    for x in it:
        s = s + x
    return s


def _dot(a, b):
    return _sum(a[i][j] * b[i][j] for i in R3 for j in R3)


def _inv3(h):
    c = _symf(lambda i, j: h[(i + 1) % 3][(j + 1) % 3] * h[(i + 2) % 3][(j + 2) % 3]
              - h[(i + 1) % 3][(j + 2) % 3] * h[(i + 2) % 3][(j + 1) % 3])
    det = _sum(h[0][j] * c[0][j] for j in R3)
    return _mat(lambda i, j: c[i][j] / det), det


def _point(P, v, d1, d2, adv, xyz=None):
    """Right-hand side of the 27 fields, constraints and (with xyz, the coordinates) Psi_4."""
    chi, K, Th, al, phi, Pi = v[0], v[7], v[14], v[18], v[25], v[26]
    h, A = _sym(v[1:7]), _sym(v[8:14])
    hi, _ = _inv3(h)
    gd, gu = _mat(lambda i, j: h[i][j] / chi), _mat(lambda i, j: chi * hi[i][j])
    dh = [_sym([d1[1 + m][k] for m in range(6)]) for k in R3]
    dA = [_sym([d1[8 + m][k] for m in range(6)]) for k in R3]
    ddh = _mat(lambda i, j: _sym([d2[1 + m][i][j] for m in range(6)]))  # ddh[i][j][a][b]
    dchi, dK, dTh, dal, dphi, dPi = d1[0], d1[7], d1[14], d1[18], d1[25], d1[26]
    Gh, be, Bf = v[15:18], v[19:22], v[22:25]
    db = _mat(lambda j, i: d1[19 + i][j])  # d_j beta^i
    divb = _sum(db[i][i] for i in R3)
    # conformal connection
    G1 = [_symf(lambda i, j: 0.5 * (dh[i][l][j] + dh[j][l][i] - dh[l][i][j])) for l in R3]
    G2 = [_symf(lambda i, j: _sum(hi[k][l] * G1[l][i][j] for l in R3)) for k in R3]
    Gl = [_dot(hi, G1[l]) for l in R3]
    Gt = [_sum(hi[k][l] * Gl[l] for l in R3) for k in R3]
    dhi = []
    for m in R3:
        t = _mat(lambda a, c: _sum(hi[a][b] * dh[m][b][c] for b in R3))
        dhi.append(_symf(lambda a, c: -_sum(t[a][b] * hi[b][c] for b in R3)))
    dGl = _mat(lambda m, l: _dot(dhi[m], G1[l]) + _sum(hi[i][j] * (ddh[m][i][l][j] - 0.5 * ddh[m][l][i][j])
                                                       for i in R3 for j in R3))
    hdchi = [_sum(hi[k][l] * dchi[l] for l in R3) for k in R3]

    def gp(k, i, j):
        t = G2[k][i][j] + h[i][j] * hdchi[k] / (2 * chi)
        if k == i:
            t = t - dchi[j] / (2 * chi)
        if k == j:
            t = t - dchi[i] / (2 * chi)
        return t

    Gp = [_symf(lambda i, j: gp(k, i, j)) for k in R3]
    # Ricci tensor of gamma = h / chi
    U = [[[_sum(hi[l][m] * G2[k][l][i] for l in R3) for i in R3] for m in R3] for k in R3]
    Q = _mat(lambda i, j: _sum(U[k][m][i] * G1[j][k][m] for k in R3 for m in R3))
    DDc = _symf(lambda i, j: d2[0][i][j] - _sum(G2[k][i][j] * dchi[k] for k in R3))
    lapc, dc2 = _dot(hi, DDc), _sum(dchi[k] * hdchi[k] for k in R3)
    Ric = _symf(lambda i, j: -0.5 * _sum(hi[l][m] * ddh[l][m][i][j] for l in R3 for m in R3)
                + 0.5 * (dGl[i][j] + dGl[j][i]) - _sum(Gt[k] * G1[k][i][j] for k in R3) + Q[i][j] + Q[j][i]
                + _sum(U[k][l][i] * G1[k][l][j] for k in R3 for l in R3)
                + (DDc[i][j] + h[i][j] * lapc) / (2 * chi)
                - (dchi[i] * dchi[j] + 3 * h[i][j] * dc2) / (4 * chi * chi))
    Rs = _dot(Ric, gu)
    # Z_i and R_ij + 2 D_(i Z_j)
    hG = [_sum(h[i][k] * Gh[k] for k in R3) for i in R3]
    Zl = [0.5 * (hG[i] - Gl[i]) for i in R3]
    Zu = [0.5 * chi * (Gh[k] - Gt[k]) for k in R3]
    dZ = _mat(lambda j, i: 0.5 * (_sum(dh[j][i][k] * Gh[k] + h[i][k] * d1[15 + k][j] for k in R3) - dGl[j][i]))
    RZ = _symf(lambda i, j: Ric[i][j] + dZ[i][j] + dZ[j][i] - 2 * _sum(Gp[k][i][j] * Zl[k] for k in R3))
    RZs = _dot(RZ, gu)
    DDa = _symf(lambda i, j: d2[18][i][j] - _sum(Gp[k][i][j] * dal[k] for k in R3))
    DDp = _symf(lambda i, j: d2[25][i][j] - _sum(Gp[k][i][j] * dphi[k] for k in R3))
    lapa = _dot(DDa, gu)
    # extrinsic curvature
    Kp = _mat(lambda i, j: (A[i][j] + h[i][j] * K / 3) / chi)
    Aud = _mat(lambda i, j: _sum(hi[i][k] * A[k][j] for k in R3))
    Kud = _mat(lambda i, j: Aud[i][j] + K / 3 if i == j else Aud[i][j])
    Au = _mat(lambda i, j: _sum(Aud[i][k] * hi[k][j] for k in R3))
    AA, trK = _dot(A, Au), K + _sum(Aud[i][i] for i in R3)
    KK = _symf(lambda i, j: _sum(Kp[i][k] * Kud[k][j] for k in R3))
    dKp = [_symf(lambda i, j: (dA[k][i][j] + h[i][j] * dK[k] / 3 + dh[k][i][j] * K / 3 - Kp[i][j] * dchi[k]) / chi)
           for k in R3]
    aA, ah = _sym(adv[8:14]), _sym(adv[1:7])
    LbK = _symf(lambda i, j: (aA[i][j] + h[i][j] * adv[7] / 3 + ah[i][j] * K / 3 - Kp[i][j] * adv[0]) / chi
                + _sum(Kp[i][k] * db[j][k] + Kp[k][j] * db[i][k] for k in R3))

    def bk(k, i, j):  # B_kij = D_i K_kj - D_j K_ki
        return (dKp[i][k][j] - dKp[j][k][i]
                - _sum(Gp[l][i][k] * Kp[l][j] - Gp[l][j][k] * Kp[l][i] for l in R3))

    Bk = [[[None] * 3 for _ in R3] for _ in R3]
    for k in R3:
        for i, j in ((0, 1), (0, 2), (1, 2)):
            Bk[k][i][j] = bk(k, i, j)
            Bk[k][j][i] = -Bk[k][i][j]
    Bv = [_sum(gu[a][b] * Bk[a][b][j] for a in R3 for b in R3 if b != j) for j in R3]
    # Gauss block
    S = _symf(lambda i, j: Ric[i][j] + trK * Kp[i][j] - KK[i][j])
    Ss = _dot(S, gu)
    GS = _symf(lambda i, j: S[i][j] - 0.5 * gd[i][j] * Ss)
    t = _mat(lambda i, j: _sum(gu[i][a] * GS[a][j] for a in R3))
    GSu = _symf(lambda i, j: _sum(t[i][a] * gu[a][j] for a in R3))
    # scalar
    lam, g2, g3 = P["lam"], P["g2"], P["g3"]
    if P["beta"] == 0:
        b1, b2 = lam + 0.0 * phi, 0.0 * phi
    elif P["beta"] == 1:
        b1, b2 = lam * phi, lam + 0.0 * phi
    else:
        e = torch.exp(-phi * phi)
        b1, b2 = lam * phi * e, lam * e * (1 - 2 * phi * phi)
    pu = [_sum(gu[i][j] * dphi[j] for j in R3) for i in R3]
    dp2 = _sum(dphi[i] * pu[i] for i in R3)
    X = 0.5 * (Pi * Pi - dp2)
    fX, XX = 1 + 2 * g2 * X, X + g2 * X * X
    H = _symf(lambda i, j: DDp[i][j] + Kp[i][j] * Pi)
    Hn = [dPi[i] + _sum(Kud[k][i] * dphi[k] for k in R3) for i in R3]
    F = _symf(lambda i, j: b1 * H[i][j] + b2 * dphi[i] * dphi[j])
    Fn = [b1 * Hn[i] + b2 * Pi * dphi[i] for i in R3]
    Fm = _mat(lambda i, k: _sum(F[i][j] * gu[j][k] for j in R3))
    Fu = _symf(lambda i, j: _sum(gu[i][k] * Fm[k][j] for k in R3))
    Fnu = [_sum(gu[i][j] * Fn[j] for j in R3) for i in R3]
    trF = _sum(Fm[i][i] for i in R3)
    trH = _dot(H, gu)
    Hd = [_sum(H[i][k] * pu[k] for k in R3) for i in R3]
    Hdd, Hnd = _sum(pu[i] * Hd[i] for i in R3), _sum(pu[i] * Hn[i] for i in R3)
    dec = P["dec"]
    zero = 0.0 * phi
    rho, S8 = zero, [zero] * 3
    S1 = _sym([zero] * 6)
    Y = _sym([zero] * 6)
    if not dec:
        rho = 0.5 * fX * Pi * Pi - 0.5 * XX - 4 * _dot(GS, Fu) + 0.5 * g3 * (Pi * Pi * trH - Hdd)
        S8 = [4 * (_sum(GS[i][k] * Fnu[k] for k in R3) + trF * Bv[i] - _sum(Fm[i][l] * Bv[l] for l in R3)
                   + _sum(Bk[k][i][l] * Fu[k][l] for k in R3 for l in R3 if l != i))
              - 0.5 * fX * Pi * dphi[i]
              - 0.5 * g3 * ((Pi * trH - Hnd) * dphi[i] + Pi * Pi * Hn[i] - Pi * Hd[i]) for i in R3]
        S1 = _symf(lambda i, j: 0.5 * fX * dphi[i] * dphi[j] + 0.5 * XX * gd[i][j])
        BF = _sum(Bv[i] * Fnu[i] for i in R3)
        Y = _symf(lambda i, j: Bv[j] * Fn[i] + Bv[i] * Fn[j] - 2 * BF * gd[i][j]
                  + _sum(Bk[i][j][l] * Fnu[l] for l in R3 if l != j) + _sum(Bk[j][i][l] * Fnu[l] for l in R3 if l != i))

    def qof(Xm):
        xf, tx = _dot(Xm, Fu), _dot(Xm, gu)
        return _symf(lambda i, j: gd[i][j] * (xf - tx * trF) + trF * Xm[i][j] + tx * F[i][j]
                     - _sum(Fm[i][k] * Xm[k][j] + Fm[j][k] * Xm[i][k] for k in R3))

    C0 = _symf(lambda i, j: (DDa[i][j] - LbK[i][j]) / al + KK[i][j])
    bdPi = adv[26]
    dadp = _sum(dal[i] * pu[i] for i in R3)
    Hnn0 = -(bdPi + dadp) / al
    Fnn0 = b1 * Hnn0 + b2 * Pi * Pi
    # L_GB at d_t K_ij = 0
    Buu = _sum(Bk[k][i][j] * _sum(gu[k][a] * gu[i][b] * gu[j][c] * Bk[a][b][c] for a in R3 for b in R3 for c in R3
                                  if b != c) for k in R3 for i in R3 for j in R3 if i != j)
    BvBv = _sum(Bv[i] * gu[i][j] * Bv[j] for i in R3 for j in R3)
    L0 = 8 * _dot(C0, GSu) - 4 * Buu + 8 * BvBv
    # CCZ4 without S_ij
    k1, k2, k3, shF, eta, a0, b0 = 0.1, 0.0, 1.0, 0.75, 1.0, 0.2, 0.4
    bK, bTh = 3 * b0 / (4 * (1 + b0)), 1 / (2 * (1 + b0))
    r = [None] * NF
    r[0] = adv[0] + 2.0 / 3.0 * chi * (al * K - divb)
    hd = _symf(lambda i, j: ah[i][j] - 2 * al * A[i][j] - 2.0 / 3.0 * divb * h[i][j]
               + _sum(h[i][k] * db[j][k] + h[j][k] * db[i][k] for k in R3))
    K2 = K - 2 * Th
    Hb = Rs - AA + 2.0 / 3.0 * K * K - 2 * rho - 2 * k1 * (2 + k2) * Th
    Kd = adv[7] + al * (K * K2 + RZs) - 3 * k1 * (1 + k2) * al * Th - lapa - 1.5 * al * rho - bK * al * Hb
    Xa = _symf(lambda i, j: al * RZ[i][j] - DDa[i][j])
    trX = _dot(Xa, hi)
    Ad = _symf(lambda i, j: aA[i][j] + chi * (Xa[i][j] - h[i][j] * trX / 3) + (al * K2 - 2.0 / 3.0 * divb) * A[i][j]
               + _sum(A[i][k] * (db[j][k] - 2 * al * Aud[k][j]) + A[j][k] * db[i][k] for k in R3))
    r[14] = adv[14] + al * (0.5 * (RZs - Rs) - Th * K) - _sum(Zu[i] * dal[i] for i in R3) + bTh * al * Hb
    hZ = [_sum(hi[i][j] * Zl[j] for j in R3) for i in R3]
    for i in R3:
        wb = [Bv[j] - S8[j] + dTh[j] - k1 * Zl[j] - _sum(Kud[k][j] * Zl[k] for k in R3) for j in R3]
        x = adv[15 + i] + 2 * al * (_dot(G2[i], Au) - 1.5 / chi * _sum(Au[i][j] * dchi[j] for j in R3)
                                    - 2.0 / 3.0 * _sum(hi[i][j] * dK[j] for j in R3))
        x = x - 2 * _sum(Au[i][j] * dal[j] for j in R3) + _sum(hi[a][b] * d2[19 + i][a][b] for a in R3 for b in R3)
        x = x + _sum(hi[k][i] * (_sum(d2[19 + l][k][l] for l in R3) / 3
                                 + 2 * (al * dTh[k] - Th * dal[k] - 2.0 / 3.0 * al * K * Zl[k]))
                     - Gt[k] * db[k][i] for k in R3)
        x = x + 2.0 / 3.0 * divb * Gt[i] + (4.0 / 3.0 * k3 * divb - 2 * al * k1) * hZ[i]
        x = x - 2 * k3 * _sum(hZ[j] * db[j][i] for j in R3) - 2 * al * _sum(hi[i][j] * S8[j] for j in R3)
        x = x - 2 * b0 / (1 + b0) * al * _sum(hi[i][j] * wb[j] for j in R3)
        r[15 + i] = x
        r[22 + i] = x - eta * Bf[i]
        r[19 + i] = shF / (1 + a0) * Bf[i] - a0 / (1 + a0) * al * chi * _sum(hi[i][j] * dal[j] for j in R3)
    r[18] = adv[18] - 2 / (1 + a0) * al * K2
    r[25] = adv[25] + al * Pi
    # the system for (d_t K_ij, d_t Pi)
    D = fX + 2 * g2 * Pi * Pi + 2 * g3 * trH
    PP = _symf(lambda i, j: Pi * Pi * gu[i][j] - pu[i] * pu[j])
    S3, S3w, E3 = _sym([zero] * 6), _sym([zero] * 6), zero
    if g3 != 0.0:
        Hm = _mat(lambda i, k: _sum(H[i][j] * gu[j][k] for j in R3))
        HH = _sum(Hm[i][k] * Hm[k][i] for i in R3 for k in R3)
        HnHn = _sum(Hn[i] * gu[i][j] * Hn[j] for i in R3 for j in R3)
        E3 = g3 * (trH * trH + 2 * HnHn - HH - 2 * Pi * _sum(Bv[i] * pu[i] for i in R3)
                   - _sum(S[i][j] * pu[i] * pu[j] for i in R3 for j in R3) - _dot(C0, PP))
        if not dec:
            S3 = _symf(lambda i, j: g3 * (0.5 * Hnn0 * (Pi * Pi * gd[i][j] - dphi[i] * dphi[j])
                                          + 0.5 * trH * dphi[i] * dphi[j]
                                          + 0.5 * Pi * (Hn[i] * dphi[j] + Hn[j] * dphi[i])
                                          - 0.5 * (Hd[i] * dphi[j] + Hd[j] * dphi[i])
                                          + gd[i][j] * (0.5 * Hdd - Pi * Hnd)))
            S3w = _symf(lambda i, j: 0.5 * g3 * (Pi * Pi * gd[i][j] - dphi[i] * dphi[j]))  # times w / alpha
    src = fX * trH + 4 * g2 * Pi * Hnd - 2 * g2 * Hdd + b1 * L0 + E3

    def lop(x):  # x - gamma tr(x) / 2
        tr = _dot(x, gu)
        return _symf(lambda i, j: x[i][j] - 0.5 * gd[i][j] * tr)

    U0 = _symf(lambda i, j: (Ad[i][j] + h[i][j] * Kd / 3 + hd[i][j] * K / 3 - Kp[i][j] * r[0]) / chi)
    M = [[zero] * 7 for _ in range(7)]
    b = [None] * 7
    for m, (i, j) in enumerate(SYM):
        M[m][m] = zero + 1.0
        b[m] = U0[i][j]
    if not dec:
        LGS, QC = lop(GS), qof(C0)
        LS = lop(_symf(lambda i, j: S1[i][j] + S3[i][j] - 4 * (GS[i][j] * Fnn0 + Y[i][j] + QC[i][j])))
        LW = lop(S3w)
        for m, (i, j) in enumerate(SYM):
            b[m] = b[m] - al * LS[i][j]
            M[m][6] = LW[i][j] - 4 * b1 * LGS[i][j]
        for c, (a, bb) in enumerate(SYM):
            E = _symf(lambda i, j: zero + (1.0 if (i, j) in ((a, bb), (bb, a)) else 0.0))
            LQ = lop(qof(E))
            for m, (i, j) in enumerate(SYM):
                M[m][c] = M[m][c] - 4 * LQ[i][j]
    for c, (a, bb) in enumerate(SYM):
        w2 = 1.0 if a == bb else 2.0
        M[6][c] = w2 * (g3 * PP[a][bb] - 8 * b1 * GSu[a][bb]) / D
    M[6][6] = zero + 1.0
    b[6] = bdPi + dadp + al / D * src
    sol = torch.linalg.solve(torch.stack([torch.stack(row, -1) for row in M], -2), torch.stack(b, -1).unsqueeze(-1))
    u, w = _sym([sol[..., m, 0] for m in range(6)]), sol[..., 6, 0]
    S8f = _sym([zero] * 6)
    if not dec:
        Qu, Fnn = qof(u), Fnn0 + b1 * w / al
        S8f = _symf(lambda i, j: S1[i][j] + S3[i][j] + S3w[i][j] * w / al
                    - 4 * (GS[i][j] * Fnn + Y[i][j] + Qu[i][j] / al + QC[i][j]))
    r[7] = Kd + 0.5 * al * _dot(S8f, gu)
    trS = _dot(S8f, hi)
    for m, (i, j) in enumerate(SYM):
        r[1 + m] = hd[i][j]
        r[8 + m] = Ad[i][j] - al * chi * (S8f[i][j] - h[i][j] * trS / 3)
    r[26] = w
    con = [Ss - 2 * rho] + [Bv[i] - S8[i] for i in R3]
    psi = None
    if xyz is not None:
        x, y, z = xyz
        e = [[x, y, z], [x * z, y * z, -(x * x + y * y)], [-y, x, 0.0 * z]]
        for a in R3:
            for q in range(a):
                d = _sum(gd[i][j] * e[a][i] * e[q][j] for i in R3 for j in R3)
                e[a] = [e[a][i] - d * e[q][i] for i in R3]
            nrm = torch.sqrt(_sum(gd[i][j] * e[a][i] * e[a][j] for i in R3 for j in R3))
            e[a] = [c / nrm for c in e[a]]

        def form(s, p, q):
            return _sum(s[i][j] * p[i] * q[j] for i in R3 for j in R3)

        er, et, ep = e
        Rn = _symf(lambda i, j: (u[i][j] - LbK[i][j] + DDa[i][j]) / al + KK[i][j])
        Krr, Krt, Krp = form(Kp, er, er), form(Kp, er, et), form(Kp, er, ep)
        E1 = (0.5 * (form(Rn, et, et) - form(Rn, ep, ep)), -form(Rn, et, ep))
        E3p = (0.5 * (form(Ric, et, et) - form(Ric, ep, ep)) + 0.5 * Krr * (form(Kp, et, et) - form(Kp, ep, ep))
               - 0.5 * (Krt * Krt - Krp * Krp), -form(Ric, et, ep) - Krr * form(Kp, et, ep) + Krt * Krp)

        def tri(p, q):
            return _sum(Bk[i][k][j] * p[i] * er[k] * q[j] for i in R3 for k in R3 for j in R3 if k != j)

        E2 = (0.5 * (tri(et, et) - tri(ep, ep)), -0.5 * (tri(et, ep) + tri(ep, et)))
        psi = [0.5 * E1[q] - E2[q] + 0.5 * E3p[q] for q in (0, 1)]
    return r, con, psi


# first and second differences, dissipation, advection biased towards the shift, by ghost width
_W1 = {3: (12.0, {1: 8.0, 2: -1.0}), 4: (60.0, {1: 45.0, 2: -9.0, 3: 1.0})}
_W2 = {3: (12.0, -30.0, {1: 16.0, 2: -1.0}), 4: (180.0, -490.0, {1: 270.0, 2: -27.0, 3: 2.0})}
_WL = {3: {-1: -3.0, 0: -10.0, 1: 18.0, 2: -6.0, 3: 1.0},
       4: {-2: 2.0, -1: -24.0, 0: -35.0, 1: 80.0, 2: -30.0, 3: 8.0, 4: -1.0}}
_WK = {3: (64.0, -20.0, {1: 15.0, 2: -6.0, 3: 1.0}), 4: (-256.0, 70.0, {1: -56.0, 2: 28.0, 3: -8.0, 4: 1.0})}


def _shift(a, off, ng, n):
    """a[..., z, y, x] of the ghosted box at offset (x, y, z) from the interior points."""
    return a[..., ng + off[2]:ng + off[2] + n[2], ng + off[1]:ng + off[1] + n[1], ng + off[0]:ng + off[0] + n[0]]


def _derivs(P, s):
    """v, d1, d2, adv, ko of the ghosted fields s (27, nz + 2 ng, ny + 2 ng, nx + 2 ng)."""
    ng, dx, adv_on = P["ng"], P["dx"], P["adv"]
    n = (s.shape[3] - 2 * ng, s.shape[2] - 2 * ng, s.shape[1] - 2 * ng)
    den, w1 = _W1[ng]
    den2, w20, w2 = _W2[ng]
    denk, wk0, wk = _WK[ng]

    def at(f, *offs):
        o = [0, 0, 0]
        for d, r in offs:
            o[d] += r
        return _shift(s[f], o, ng, n).reshape(-1)

    def D(f, d, *more):
        return _sum(w * (at(f, (d, r), *more) - at(f, (d, -r), *more)) for r, w in w1.items()) / (den * dx)

    v = [at(f) for f in range(NF)]
    d1 = [[D(f, d) for d in R3] for f in range(NF)]
    d2 = [None] * NF
    for f in [0, 1, 2, 3, 4, 5, 6, 18, 19, 20, 21, 25]:
        diag = [(_sum(w * (at(f, (d, r)) + at(f, (d, -r))) for r, w in w2.items()) + w20 * v[f]) / (den2 * dx * dx)
                for d in R3]
        mixed = {(a, b): _sum(w * (D(f, b, (a, r)) - D(f, b, (a, -r))) for r, w in w1.items()) / (den * dx)
                 for a, b in ((0, 1), (0, 2), (1, 2))}
        d2[f] = _mat(lambda i, j: diag[i] if i == j else mixed[(min(i, j), max(i, j))])
    if adv_on:
        def up(f, d):
            b = v[19 + d]
            fw = _sum(w * at(f, (d, r)) for r, w in _WL[ng].items())
            bw = _sum(w * at(f, (d, -r)) for r, w in _WL[ng].items())
            return b.abs() * torch.where(b >= 0, fw, bw) / (den * dx)

        adv = [_sum(up(f, d) for d in R3) for f in range(NF)]
    else:
        adv = [_sum(v[19 + d] * d1[f][d] for d in R3) for f in range(NF)]
    ko = [_sum(w * (at(f, (d, r)) + at(f, (d, -r))) for d in R3 for r, w in wk.items()) + 3 * wk0 * v[f]
          for f in range(NF)]
    return v, d1, d2, adv, [k / (denk * dx) for k in ko]


def _xrhs(P, s, sigma=0.3):
    """The dissipated right-hand side at the interior points, (27, nz, ny, nx), by slabs of planes."""
    ng = P["ng"]
    nz, ny, nx = (m - 2 * ng for m in s.shape[1:])
    planes = max(1, (1 << 21) // (ny * nx))
    out = []
    for k in range(0, nz, planes):
        m = min(planes, nz - k)
        v, d1, d2, adv, ko = _derivs(P, s[:, k:k + m + 2 * ng])
        r, _, _ = _point(P, v, d1, d2, adv)
        out.append(torch.stack([r[f] + sigma * ko[f] for f in range(NF)]).view(NF, m, ny, nx))
    return out[0] if len(out) == 1 else torch.cat(out, 1)


def _wrap(P, s):
    """The ghosts of the interior's periodic images."""
    ng = P["ng"]
    for d in (1, 2, 3):
        m = s.shape[d] - 2 * ng
        idx = torch.arange(-ng, m + ng, device=s.device) % m + ng
        s = s.index_select(d, idx)
    return s


def _enforce(x):
    hi, _ = _inv3(_sym([x[1 + m] for m in range(6)]))
    tr = _dot(hi, _sym([x[8 + m] for m in range(6)]))
    rows = list(x.unbind(0))
    for m in range(6):
        rows[8 + m] = rows[8 + m] - rows[1 + m] * tr / 3
    rows[0], rows[18] = rows[0].clamp(min=1e-4), rows[18].clamp(min=1e-4)
    return torch.stack(rows)


def _radiative(P, s):
    """d_t u = -(u - u_inf) / r - x^i d_i u / r everywhere, one-sided differences beyond the interior."""
    ng, dx = P["ng"], P["dx"]
    tot, xs = 0.0, []
    for d, ax in enumerate((3, 2, 1)):
        N = s.shape[ax]
        x = P["origin"][d] + (torch.arange(N, dtype=torch.float64, device=s.device) - ng) * dx
        xs.append(x.view([-1 if q == ax else 1 for q in (1, 2, 3)]))

        def at(i, ax=ax):
            return s.index_select(ax, i)

        i = torch.arange(N, device=s.device)
        c = (at((i + 1).clamp(max=N - 1)) - at((i - 1).clamp(min=0))) / (2 * dx)
        f = (-3 * s + 4 * at((i + 1).clamp(max=N - 1)) - at((i + 2).clamp(max=N - 1))) / (2 * dx)
        b = (3 * s - 4 * at((i - 1).clamp(min=0)) + at((i - 2).clamp(min=0))) / (2 * dx)
        lo, hi = (i < ng).view_as(xs[-1]), (i >= N - ng).view_as(xs[-1])
        tot = tot + xs[-1] * torch.where(lo, f, torch.where(hi, b, c))
    r = torch.sqrt(xs[0] ** 2 + xs[1] ** 2 + xs[2] ** 2)
    flat = torch.zeros(NF, 1, 1, 1, dtype=torch.float64, device=s.device)
    for f in (0, 1, 4, 6, 18):
        flat[f] = 1.0
    return -((s - flat) + tot) / r


def _xstep(P, s, dt, rhs):
    """One RK4 step of the ghosted fields."""
    ng, bc = P["ng"], P["bc"]
    inner = (slice(None),) + (slice(ng, -ng),) * 3

    def embed(new, ghosts):
        if bc == PERIODIC:
            pad = torch.nn.functional.pad(new, (ng,) * 6)
            return _wrap(P, pad)
        out = ghosts.clone()
        out[inner] = new
        return out

    un, cur, acc, gacc = s[inner], s, None, None
    for w, c in ((1.0, 0.5), (2.0, 0.5), (2.0, 1.0), (1.0, 1.0 / 6.0)):
        k = rhs(cur)
        acc = k if acc is None else acc + w * k
        ghosts = s
        if bc == SOMMERFELD:
            gk = _radiative(P, cur)
            gacc = gk if gacc is None else gacc + w * gk
            ghosts = s + dt * c * (gacc if c < 0.2 else gk)
        cur = embed(_enforce(un + dt * c * (acc if c < 0.2 else k)), ghosts)
    return cur


def _pars(case, box, params):
    return {"ng": box.ng, "dx": box.dx, "bc": box.bc, "adv": params.advection, "beta": params.beta_kind,
            "lam": params.lambda_, "g2": params.g2, "g3": params.g3, "dec": params.decoupled,
            "origin": (box.x0, box.y0, box.z0)}


def _ghosted(box, s):
    return s[..., :box.nx + 2 * box.ng]


def _advance(case, box, params, s0, steps):
    P = _pars(case, box, params)
    s = _ghosted(box, s0)
    if box.bc == PERIODIC:
        s = _wrap(P, s)
    for _ in range(steps):
        s = _xstep(P, s, _dt(box), lambda x: _xrhs(P, x))
    out = s0.clone()
    _ghosted(box, out).copy_(s)
    return out


_S2, _S3 = 0.5 ** 0.5, 3.0 ** -0.5


def _rule():
    """The 26-point rule of degree 7 on the unit sphere."""
    pts = [(s * (d == 0), s * (d == 1), s * (d == 2), 1.0 / 21.0) for d in R3 for s in (1.0, -1.0)]
    for a in (_S2, -_S2):
        for b in (_S2, -_S2):
            pts += [(a, b, 0.0, 4.0 / 105.0), (a, 0.0, b, 4.0 / 105.0), (0.0, a, b, 4.0 / 105.0)]
    pts += [(a * _S3, b * _S3, c * _S3, 9.0 / 280.0) for a in (1, -1) for b in (1, -1) for c in (1, -1)]
    return pts


def _signal(box, sp, s):
    """sum_q w_q phi(c + R x_q) with trilinear interpolation."""
    tot = 0.0
    for x, y, z, w in _rule():
        p = [(c + sp.radius * q - o) / box.dx for c, q, o in zip((sp.cx, sp.cy, sp.cz), (x, y, z), (box.x0, box.y0, box.z0))]
        i = [math.floor(q) for q in p]
        t = [q - m for q, m in zip(p, i)]
        for c in range(8):
            b = [c & 1, (c >> 1) & 1, (c >> 2) & 1]
            wt = math.prod(t[d] if b[d] else 1.0 - t[d] for d in R3)
            tot = tot + w * wt * s[25, i[2] + b[2] + box.ng, i[1] + b[1] + box.ng, i[0] + b[0] + box.ng]
    return tot


def _modes(box, fre, fim, sp, nth, nph, lmax):
    """Spin -2 modes of the field on the sphere: Gauss-Legendre in cos(theta), equal phi, cubic Lagrange."""
    mu, w = np.polynomial.legendre.leggauss(nth)
    th, ph = np.arccos(mu)[:, None], 2 * np.pi * np.arange(nph)[None, :] / nph
    n = (np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th) + 0 * ph)
    f = (_ghosted(box, fre) + 1j * _ghosted(box, fim)).cpu().numpy()
    p = [(c + sp.radius * q - o) / box.dx + box.ng for c, q, o in zip((sp.cx, sp.cy, sp.cz), n, (box.x0, box.y0, box.z0))]
    i0 = [np.floor(q).astype(int) for q in p]
    L = []
    for q, i in zip(p, i0):
        t = q - i
        L.append([-t * (t - 1) * (t - 2) / 6, (t + 1) * (t - 1) * (t - 2) / 2, -(t + 1) * t * (t - 2) / 2,
                  (t + 1) * t * (t - 1) / 6])
    v = sum(L[2][c] * L[1][b] * L[0][a] * f[i0[2] - 1 + c, i0[1] - 1 + b, i0[0] - 1 + a]
            for c in range(4) for b in range(4) for a in range(4))
    out = np.zeros((lmax + 1) ** 2, dtype=complex)
    fa, s = math.factorial, -2
    for l in range(2, lmax + 1):
        for m in range(-l, l + 1):
            pre = (-1.0) ** m * math.sqrt(fa(l + m) * fa(l - m) * (2 * l + 1) / (4 * math.pi * fa(l + s) * fa(l - s)))
            tot = sum(math.comb(l - s, r) * math.comb(l + s, r + s - m) * (-1.0) ** (l - r - s)
                      * np.sqrt((1 + mu) / (1 - mu)) ** (2 * r + s - m)
                      for r in range(l - s + 1) if 0 <= r + s - m <= l + s)
            y = pre * ((1 - mu) / 2) ** l * tot
            ring = (v * np.exp(-1j * m * ph)).sum(1) * 2 * np.pi / nph
            out[l * l + l + m] = (w * y * ring).sum()
    return out


def _diag(case, box, params, s0):
    P = _pars(case, box, params)
    s = _wrap(P, _ghosted(box, s0)) if box.bc == PERIODIC else _ghosted(box, s0)
    ng = box.ng
    v, d1, d2, adv, _ = _derivs(P, s)
    shape = (box.nz, box.ny, box.nx)
    ax = [torch.arange(m, dtype=torch.float64, device=DEV) * box.dx + o
          for m, o in ((box.nx, box.x0), (box.ny, box.y0), (box.nz, box.z0))]
    xyz = [ax[0][None, None, :].expand(shape).reshape(-1), ax[1][None, :, None].expand(shape).reshape(-1),
           ax[2][:, None, None].expand(shape).reshape(-1)]
    _, con, psi = _point(P, v, d1, d2, adv, xyz)
    out4, out2 = _fields(box, 4), _fields(box, 2)
    for o, x in ((out4, con), (out2, psi)):
        _ghosted(box, o)[:, ng:-ng, ng:-ng, ng:-ng] = torch.stack(x).view(-1, *shape)
    norms = np.array([q for x in con for q in (float(x.square().mean().sqrt()), float(x.abs().max()))])
    return {"constraints": out4, "norms": norms, "psi4": out2,
            "modes": _modes(box, out2[0], out2[1], _signal_sphere(box), 24, 48, 4)}


def _evolve_signal(case, box, params, s, lam, g2, steps, rhs_wrap):
    P = dict(_pars(case, box, params), lam=lam, g2=g2)
    sp, tot = _signal_sphere(box), 0.0
    s = _wrap(P, s)
    for _ in range(steps):
        s = _xstep(P, s, _dt(box), lambda x: rhs_wrap(lambda y, a, c: _xrhs(dict(P, lam=a, g2=c), y), x, lam, g2))
        tot = tot + _dt(box) * _signal(box, sp, s)
    return s, tot


def exact(case, seed):
    kind, boxes = case["kind"], _boxes(case)
    box, params = boxes[0], _params(case)
    u0 = [_initial(case, bx, seed, b) for b, bx in enumerate(boxes)]
    if kind in ("rk4", "host"):
        return _advance(case, box, params, u0[0], case["steps"])
    if kind == "batch":
        return [_advance(case, bx, _params(case, b), u0[b], case["steps"]) for b, bx in enumerate(boxes)]
    if kind == "patches":
        whole = _ghosted(box, _advance(case, box, params, u0[0], case["steps"]))
        out = []
        for q in range(8):
            cut = [[(a * m) // 2, ((a + 1) * m) // 2] for a, m in zip((q & 1, (q >> 1) & 1, q >> 2),
                                                                      (box.nx, box.ny, box.nz))]
            (x, x1), (y, y1), (z, z1) = cut
            w = x1 - x + 6
            t = torch.zeros((NF, z1 - z + 6, y1 - y + 6, (w + 3) // 4 * 4), dtype=torch.float64, device=DEV)
            t[..., :w] = whole[:, z:z1 + 6, y:y1 + 6, x:x1 + 6]
            out.append(t)
        return out
    if kind == "rhs":
        P = _pars(case, box, params)
        s = _ghosted(box, u0[0])
        if box.bc == PERIODIC:
            s = _wrap(P, s)
        out, ng = _fields(box), box.ng
        if box.bc == SOMMERFELD:
            _ghosted(box, out).copy_(_radiative(P, s))
        _ghosted(box, out)[:, ng:-ng, ng:-ng, ng:-ng] = _xrhs(P, s, 0.3 + 0.1)
        return out
    if kind == "diag":
        return _diag(case, box, params, u0[0])
    if box.nx * box.ny * box.nz > 50000:  # the derivatives' records would not fit beside the rest
        return None
    s0, dev = _ghosted(box, u0[0]), DEV
    if kind == "adjoint":
        from torch.utils.checkpoint import checkpoint
        lam = torch.tensor(params.lambda_, dtype=torch.float64, device=dev, requires_grad=True)
        g2 = torch.tensor(params.g2, dtype=torch.float64, device=dev, requires_grad=True)
        x = s0.clone().requires_grad_(True)
        s, L = _evolve_signal(case, box, params, x, lam, g2, case["steps"],
                              lambda f, *a: checkpoint(f, *a, use_reentrant=False))
        gx, gl, gg = torch.autograd.grad(L, (x, lam, g2))
        state, sbar = u0[0].clone(), torch.zeros_like(u0[0])
        _ghosted(box, state).copy_(s.detach())
        _ghosted(box, sbar).copy_(gx)
        return {"state": state, "signal": L.detach().reshape(1), "d_state": sbar, "d_couplings": torch.stack([gl, gg])}
    if kind == "tangent":
        import torch.autograd.forward_ad as fwd
        tang, sig, state = torch.zeros((3,) + tuple(u0[0].shape), dtype=torch.float64, device=dev), [], u0[0].clone()
        base = [torch.tensor(q, dtype=torch.float64, device=dev) for q in (params.lambda_, params.g2)]
        for k in R3:
            with fwd.dual_level(), torch.no_grad():
                dirs = [torch.tensor(_DPARAMS[2 * k + q], dtype=torch.float64, device=dev) for q in (0, 1)]
                dx = torch.zeros_like(s0)
                if k == 2:
                    dx[25] = s0[25]
                s, L = _evolve_signal(case, box, params, fwd.make_dual(s0.clone(), dx), fwd.make_dual(base[0], dirs[0]),
                                      fwd.make_dual(base[1], dirs[1]), case["steps"], lambda f, *a: f(*a))
                sv, st = fwd.unpack_dual(s)
                Lv, Lt = fwd.unpack_dual(L)
                _ghosted(box, state).copy_(sv)
                tang[k][..., :box.nx + 6].copy_(st)
                sig = sig or [Lv.clone()]
                sig.append(Lt.clone())
        return {"state": state, "tangents": tang, "signal": torch.stack(sig)}
    return None
